// Fused D3Q15 adjoint step for the FP32 path on non-periodic grids (exact discrete adjoint of the
// fused forward step; structure of Alg. 2, Eqs. arho, au, as and the adjoint equilibrium), as a
// z-march of warps that hold several rows of a tile in registers.
//
// A block of NW warps covers 32 columns x (R NW) rows of lambda and marches along z over a chunk of
// planes; lane = column, each warp owns R consecutive rows.  The gather of F~_i(y) = mu_rho(y + c_i) +
// c_i . mu_u(y + c_i) into the moments runs one axis at a time:
//   z  in registers: a thread keeps its nodes' mu in planes p - 1 and p and meets plane p + 1;
//   y  in registers between a warp's rows, through shared memory at the R-row seams (five values a
//      column and seam, one block barrier a plane);
//   x  by warp shuffles (ten values a node).
// Each axis turns the two sources of a direction pair into their sum and difference, so the eight
// corner directions cost 36 additions a node and no node is read by more than one thread.  The
// transposed gradient takes 9 S~ from the columns beside by shuffles, from the rows beside in
// registers or through the same seams one plane later, and from the planes beside in registers.
//
// Per plane: lambda^n (float4, by TMA into a ring) has received the boundary copies' transpose, the
// objective source and the Brinkman transpose in k_adj_prep, so mu is lambda on interior nodes and 0
// on boundary nodes and outside the grid; moments of F~; lambda^{n-1} = (R~, 3 U~ + 9 S~ u -
// 3 R~ u + D^T(2 A S~)), the transposed gradient in its central form; k_adj_bcorr adds the
// one-sided parts of boundary rows from the 2 A S~ values stored here for face nodes.
//
// Bound by instruction issue (FP32 adds and shuffles, 55 % active) and the waits for its rings: 260
// instructions a node, where a kernel of one node a thread that passed twelve values a node through
// shared memory took 502.  256^3: 213 us, k_adj_prep 26 (41 where the body's swing makes the footprint
// box large) and k_adj_bcorr 16, before 317 with 13 + 17 around it; a step by events 244 us against
// 314, at 128^3 58 against 63.  Two blocks of up to seven warps an SM rather than one of
// fourteen: one block's barrier leaves the other running.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "lks_device.cuh"
#include "lks_march3d.h"
#include "lks_tma.cuh"

namespace lks {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int R = 4;              // rows per warp
constexpr int NSLOT = 3;          // lambda planes in the ring
constexpr int NUSLOT = 2;         // planes of u^{n-1}
constexpr int kSeam = 8;          // values a column publishes at a seam: 5 of F~, 3 of S~
constexpr int kMaxWarps = 7;      // two such blocks per SM at 128 registers

struct Args {
    int n[3];
    float4* lam_out;
    float* face;           // 2 A S~_{.beta} on the six faces
    long long face_off[6];
    int* err;
    int zchunk;
    float A9;              // A / 9
};

__device__ __forceinline__ float left(float v) { return __shfl_up_sync(FULL, v, 1); }
__device__ __forceinline__ float right(float v) { return __shfl_down_sync(FULL, v, 1); }

// Store of a record under a predicate, without a branch.
__device__ __forceinline__ void st_if(float4* p, const float4& v, bool go) {
    asm volatile(
        "{ .reg .pred p; setp.ne.s32 p, %5, 0;"
        " @p st.global.v4.f32 [%4], {%0, %1, %2, %3}; }" ::"f"(v.x),
        "f"(v.y), "f"(v.z), "f"(v.w), "l"(p), "r"((int)go)
        : "memory");
}

// What a row of planes p - 1, p + 1 sends to the rows beside it: to the row below (its source above)
// P, P1, X0, X1 and mu_rho + mu_y, to the row above M, M1, X0, X1 and mu_rho - mu_y.
struct RowZ {
    float P, M, P1, M1, X0, X1, yp, ym;
};

__device__ __forceinline__ RowZ row_z(const float4& n, const float3& m1, const float4& c) {
    // n: mu of plane p + 1; m1: (mu_rho - mu_z, mu_x, mu_y) of plane p - 1; c: mu of plane p
    const float ep = n.x + n.w;
    const float E0 = ep + m1.x, E1 = ep - m1.x;
    const float Y0 = n.z + m1.z, Y1 = n.z - m1.z;
    RowZ z;
    z.P = E0 + Y0;
    z.M = E0 - Y0;
    z.P1 = E1 + Y1;
    z.M1 = E1 - Y1;
    z.X0 = n.y + m1.y;
    z.X1 = n.y - m1.y;
    z.yp = c.x + c.z;
    z.ym = c.x - c.z;
    return z;
}

// FACE: the tiles start at the low x face (org 0 in adj_march_tiles), else two columns before it.  Two
// instances: with the choice at run time the other grids' march took 4 % longer (64^3 33.7 us a step
// against 32.2).
template <bool FACE>
__global__ void __launch_bounds__(32 * kMaxWarps, 2)
    k_adj_march(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap umap,
                const __grid_constant__ Args a) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
    const int lane = threadIdx.x, wid = threadIdx.y, nw = blockDim.y;
    const int rows = R * nw;
    const unsigned plane_bytes = 512u * rows;
    float4* ring = reinterpret_cast<float4*>(smem);
    // seams[parity][warp][up: to the warp above / down][value][lane]
    float* seams = reinterpret_cast<float*>(smem + (size_t)(NSLOT + NUSLOT) * plane_bytes);
    const int seam_warp = 2 * kSeam * 32, seam_buf = nw * seam_warp;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)(NSLOT + NUSLOT) * plane_bytes +
                                                 (size_t)2 * seam_buf * 4);
    uint64_t* ubars = bars + NSLOT;
    const int x0 = blockIdx.x * kAdjTileX + (FACE ? 2 : 0), y0 = blockIdx.y * (rows - 4);
    const int q0 = blockIdx.z * a.zchunk, q1 = min(nz, q0 + a.zchunk);
    const int nplanes = q1 - q0 + 4;   // lambda planes q0 - 2 .. q1 + 1
    const bool leader = lane == 0 && wid == 0;
    if ((smem_addr(smem) & 127u) != 0u) {
        if (leader) atomicOr(a.err, 16);
        return;
    }
    if (leader) {
        for (int s = 0; s < NSLOT + NUSLOT; ++s) mbar_init(smem_addr(&bars[s]));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int k = 0; k < NSLOT && k < nplanes; ++k)
            tma_load_box(smem_addr(ring + (size_t)k * (plane_bytes / 16)), &tmap, x0 - 2, y0 - 2,
                         q0 - 2 + k, smem_addr(&bars[k]), plane_bytes);
        // u^{n-1} of plane q0 (the first whose output is kept)
        tma_load_box(smem_addr(ring + (size_t)(NSLOT + (q0 & 1)) * (plane_bytes / 16)), &umap, x0 - 2,
                     y0 - 2, q0, smem_addr(&ubars[q0 & 1]), plane_bytes);
    }
    __syncthreads();

    const int x = x0 - 2 + lane, yr = y0 - 2 + R * wid;   // column, first row
    // With FACE the first and the last tile also own the halo columns on their face's side: nothing comes
    // in from beyond a face, where a shuffle returns the lane's own value, which is zero for mu on a face.
    // (A face column in lane 0 or 31 also takes its own 9 S~ for its neighbour's; k_adj_bcorr's one-sided
    // part takes it out.)
    bool xown = lane >= 2 && lane < 2 + kAdjTileX && x < nx;
    if (FACE)
        xown = x < nx && (lane >= 2 || blockIdx.x == 0) &&
               (lane < 30 || blockIdx.x == gridDim.x - 1);
    int fl = 0;   // bits r: interior in x and y, OWN + r: an output row
    constexpr int OWN = 4;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int y = yr + r, row = R * wid + r;
        if (x >= 1 && y >= 1 && x <= nx - 2 && y <= ny - 2) fl |= 1 << r;
        if (xown && row >= 2 && row < rows - 2 && y < ny) fl |= 1 << (OWN + r);
    }
    const bool edge = __any_sync(FULL, (fl & ((1 << R) - 1)) != (1 << R) - 1);
    // does the warp store values of face nodes?
    const bool any_face = __any_sync(FULL, xown && (x == 0 || x == nx - 1)) || yr <= 0 ||
                          yr + R - 1 >= ny - 1;
    const float A9 = a.A9;
    // node offset of row 0 in the next plane of the ring (node counts are below 2^31)
    const int zst = nx * ny;
    int at = (q0 - 2) * zst + yr * nx + x;


    int kc = 0, slot = 0;   // next plane of the ring, its slot and parity
    int par = 0;
    bool ok = true, late = false;   // late: a wait for u^{n-1} ran out
    const unsigned ring0 = smem_addr(ring) + (unsigned)(R * wid * 32 + lane) * 16u;
    // mu of the lane's own rows in the next plane of the ring
    auto take = [&](float4 (&v)[R]) -> bool {
        const bool good = mbar_wait_once(smem_addr(&bars[slot]), par);
        const int gz = q0 - 2 + kc;
        const bool zin = gz >= 1 && gz <= nz - 2;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(v[r].x), "=f"(v[r].y), "=f"(v[r].z), "=f"(v[r].w)
                         : "r"(ring0 + slot * plane_bytes + r * 512));
        }
        if (edge || !zin) {   // uniform
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (!zin || !(fl >> r & 1)) v[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        ++kc;
        at += zst;
        if (++slot == NSLOT) {
            slot = 0;
            par ^= 1;
        }
        return good;
    };
    // every thread has read plane k: its slot takes plane k + NSLOT
    auto refill = [&](int k) {
        if (leader && k + NSLOT < nplanes) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            const int s = k % NSLOT;
            tma_load_box(smem_addr(ring + (size_t)s * (plane_bytes / 16)), &tmap, x0 - 2, y0 - 2,
                         q0 - 2 + k + NSLOT, smem_addr(&bars[s]), plane_bytes);
        }
    };

    float3 m1[R];      // (mu_rho - mu_z, mu_x, mu_y) of plane p - 1
    float4 c[R];       // mu of plane p
    float4 o[R];       // lambda^{n-1} of plane p - 1 but for the seams' and plane p's 9 S~
    float sxz[R], syz[R], szz[R];   // 9 S~_{.z} of plane p - 1
    float sxy0 = 0.f, syy0 = 0.f, sxy3 = 0.f, syy3 = 0.f;   // of the seam rows 0 and R - 1
    {
        float4 v[R];
        bool good = take(v);
#pragma unroll
        for (int r = 0; r < R; ++r) m1[r] = make_float3(v[r].x - v[r].w, v[r].y, v[r].z);
        good = take(c) && good;
        ok = !__syncthreads_or(!good);
        refill(0);
        refill(1);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        o[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        sxz[r] = syz[r] = szz[r] = 0.f;
    }
    const int wlo = max(wid - 1, 0), whi = min(wid + 1, nw - 1);
#pragma unroll 1
    for (int p = q0 - 1; ok && p <= q1; ++p) {
        float4 n[R];
        const int kn = kc;
        const int pofs = at - zst;   // row 0 of plane p
        const bool good = take(n);   // mu of plane p + 1
        const bool pout = p >= q0 && p < q1;
        float* sb = seams + (p & 1) * seam_buf;
        {
            float* s = sb + wid * seam_warp + lane;   // to the warp below, then to the warp above
            const RowZ z0 = row_z(n[0], m1[0], c[0]), z3 = row_z(n[R - 1], m1[R - 1], c[R - 1]);
            s[0 * 32] = z0.P;
            s[1 * 32] = z0.P1;
            s[2 * 32] = z0.X0;
            s[3 * 32] = z0.X1;
            s[4 * 32] = z0.yp;
            s[5 * 32] = sxy0;
            s[6 * 32] = syy0;
            s[7 * 32] = syz[0];
            s += kSeam * 32;
            s[0 * 32] = z3.M;
            s[1 * 32] = z3.M1;
            s[2 * 32] = z3.X0;
            s[3 * 32] = z3.X1;
            s[4 * 32] = z3.ym;
            s[5 * 32] = sxy3;
            s[6 * 32] = syy3;
            s[7 * 32] = syz[R - 1];
        }
        if (__syncthreads_or(!good || late)) {
            ok = false;
            break;
        }
        refill(kn);
        // u^{n-1} of plane p + 1, into the slot plane p - 1 was read from before the barrier
        if (leader && p >= q0 && p + 1 < q1) {
            const int us = (p + 1) & 1;
            tma_load_box(smem_addr(ring + (size_t)(NSLOT + us) * (plane_bytes / 16)), &umap, x0 - 2,
                         y0 - 2, p + 1, smem_addr(&ubars[us]), plane_bytes);
        }
        bool ugood = true;
        if (pout) ugood = mbar_wait_once(smem_addr(&ubars[p & 1]), (p - q0) >> 1 & 1);
        const unsigned uaddr = ring0 + (unsigned)(NSLOT + (p & 1)) * plane_bytes;
        const float* sa = sb + whi * seam_warp + lane;                 // row R - 1's row above
        const float* sl = sb + wlo * seam_warp + kSeam * 32 + lane;    // row 0's row below
        // the seams' part of the transposed gradient of plane p - 1 (its y neighbours)
        {
            const float bxy = sl[5 * 32], byy = sl[6 * 32], byz = sl[7 * 32];
            o[0].y = fmaf(A9, bxy, o[0].y);
            o[0].z = fmaf(A9, byy, o[0].z);
            o[0].w = fmaf(A9, byz, o[0].w);
            const float txy = sa[5 * 32], tyy = sa[6 * 32], tyz = sa[7 * 32];
            o[R - 1].y = fmaf(-A9, txy, o[R - 1].y);
            o[R - 1].z = fmaf(-A9, tyy, o[R - 1].z);
            o[R - 1].w = fmaf(-A9, tyz, o[R - 1].w);
        }
        // moments of plane p row by row; prev: the row below's values
        float bM, bM1, bX0, bX1, bym;   // from the row below
        bM = sl[0 * 32];
        bM1 = sl[1 * 32];
        bX0 = sl[2 * 32];
        bX1 = sl[3 * 32];
        bym = sl[4 * 32];
        RowZ zc = row_z(n[0], m1[0], c[0]);
        float pxy = 0.f, pyy = 0.f, pyz = 0.f;      // 9 S~_{.y} of the row below, same plane
        const bool write = p > q0;
        float nsxy0 = 0.f, nsyy0 = 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            RowZ zn;   // the row above
            if (r < R - 1) {
                zn = row_z(n[r + 1], m1[r + 1], c[r + 1]);
            } else {
                zn.P = sa[0 * 32];
                zn.P1 = sa[1 * 32];
                zn.X0 = sa[2 * 32];
                zn.X1 = sa[3 * 32];
                zn.yp = sa[4 * 32];
                zn.M = zn.M1 = zn.ym = 0.f;
            }
            const float sa_ = zn.P + bM, sb_ = zn.P - bM, sa1 = zn.P1 + bM1, sb1 = zn.P1 - bM1;
            const float sc_ = zn.X0 + bX0, sd_ = zn.X0 - bX0, sc1 = zn.X1 + bX1, sd1 = zn.X1 - bX1;
            const float ay = zn.yp + bym, dy = zn.yp - bym;
            const float4 cc = c[r];
            const float g0 = right(sa_ + sc_), h0 = left(sa_ - sc_);
            const float g1 = right(sb_ + sd_), h1 = left(sb_ - sd_);
            const float g2 = right(sa1 + sc1), h2 = left(sa1 - sc1);
            const float g3 = right(sb1 + sd1), h3 = left(sb1 - sd1);
            const float xr = right(cc.x + cc.y), xl = left(cc.x - cc.y);
            const float ep = n[r].x + n[r].w, em = m1[r].x;
            const float G = g0 + h0, ax = xr + xl, az = ep + em;
            using Wf = Wts<float, 3>;
            const float s2G = Wf::s_2 * G;
            const float Rm = Wf::w0 * cc.x + Wf::w1 * (ax + ay + az) + Wf::w2 * G;
            const float Ux = Wf::w3_1 * (xr - xl) + Wf::w3_2 * (g0 - h0);
            const float Uy = Wf::w3_1 * dy + Wf::w3_2 * (g1 + h1);
            const float Uz = Wf::w3_1 * (ep - em) + Wf::w3_2 * (g2 + h2);
            const float Sxx = ax + s2G, Syy = ay + s2G, Szz = az + s2G;   // s_1 = 1
            const float Sxy = Wf::s_2 * (g1 - h1), Sxz = Wf::s_2 * (g2 - h2);
            const float Syz = Wf::s_2 * (g3 + h3);
            // plane p - 1 is complete with this plane's 9 S~_{.z}
            {
                float4 w = o[r];
                w.y = fmaf(-A9, Sxz, w.y);
                w.z = fmaf(-A9, Syz, w.z);
                w.w = fmaf(-A9, Szz, w.w);
                st_if(a.lam_out + (pofs - zst + r * nx), w, write && (fl >> (OWN + r) & 1));
            }
            // lambda^{n-1} of plane p: the adjoint equilibrium, the gradient along x, along z from
            // plane p - 1, along y between the warp's own rows
            float4 v;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                         : "r"(uaddr + r * 512));
            const float R3 = 3.f * Rm;
            const float tx = (left(Sxx) - right(Sxx)) + sxz[r];
            const float ty = (left(Sxy) - right(Sxy)) + syz[r];
            const float tz = (left(Sxz) - right(Sxz)) + szz[r];
            o[r].x = Rm;
            o[r].y = (Ux - R3 * v.y) + (Sxx * v.y + Sxy * v.z + Sxz * v.w);
            o[r].z = (Uy - R3 * v.z) + (Sxy * v.y + Syy * v.z + Syz * v.w);
            o[r].w = (Uz - R3 * v.w) + (Sxz * v.y + Syz * v.z + Szz * v.w);
            if (r > 0) {
                o[r].y = fmaf(A9, tx + pxy, o[r].y);
                o[r].z = fmaf(A9, ty + pyy, o[r].z);
                o[r].w = fmaf(A9, tz + pyz, o[r].w);
                o[r - 1].y = fmaf(-A9, Sxy, o[r - 1].y);
                o[r - 1].z = fmaf(-A9, Syy, o[r - 1].z);
                o[r - 1].w = fmaf(-A9, Syz, o[r - 1].w);
            } else {
                o[r].y = fmaf(A9, tx, o[r].y);
                o[r].z = fmaf(A9, ty, o[r].z);
                o[r].w = fmaf(A9, tz, o[r].w);
                nsxy0 = Sxy;
                nsyy0 = Syy;
            }
            pxy = Sxy;
            pyy = Syy;
            pyz = Syz;
            sxz[r] = Sxz;
            syz[r] = Syz;
            szz[r] = Szz;
            // boundary nodes keep 2 A S~_{.beta} for the one-sided parts of D^T
            if (pout && (any_face || p == 0 || p == nz - 1) && (fl >> (OWN + r) & 1)) {
                const float A2 = 2.f * A9;
                const int y = yr + r;
                if (x == 0 || x == nx - 1) {
                    float* f = a.face + a.face_off[x == 0 ? 0 : 1] + 3 * ((long long)p * ny + y);
                    f[0] = A2 * Sxx;
                    f[1] = A2 * Sxy;
                    f[2] = A2 * Sxz;
                }
                if (y == 0 || y == ny - 1) {
                    float* f = a.face + a.face_off[y == 0 ? 2 : 3] + 3 * ((long long)p * nx + x);
                    f[0] = A2 * Sxy;
                    f[1] = A2 * Syy;
                    f[2] = A2 * Syz;
                }
                if (p == 0 || p == nz - 1) {
                    float* f = a.face + a.face_off[p == 0 ? 4 : 5] + 3 * ((long long)y * nx + x);
                    f[0] = A2 * Sxz;
                    f[1] = A2 * Syz;
                    f[2] = A2 * Szz;
                }
            }
            bM = zc.M;
            bM1 = zc.M1;
            bX0 = zc.X0;
            bX1 = zc.X1;
            bym = zc.ym;
            zc = zn;
            m1[r] = make_float3(cc.x - cc.w, cc.y, cc.z);
            c[r] = n[r];
        }
        sxy0 = nsxy0;
        syy0 = nsyy0;
        sxy3 = pxy;
        syy3 = pyy;
        late = late || !ugood;
    }
    if (!ok) {
        // a copy did not land in time: record it, then give the copies still in flight a bounded
        // chance to finish before the block's shared memory goes away
        if (leader) {
            atomicOr(a.err, 8);
            const long long t0 = clock64();
            while (clock64() - t0 < (1LL << 28)) {
            }
        }
        __syncthreads();
    }
}

}  // namespace

March3d adj_march_tiles(const Geom& g, int org, int warps) {
    return march_tiles(MarchCost{kAdjTileX, R, 4, kMaxWarps, 2 * kMaxWarps, 11.0, 50.0, 13.0},
                       std::max(org == 0 ? g.n[0] - 4 : g.n[0], 1), g.n[1], g.n[2], warps);
}

cudaError_t launch_adj_march(const Geom& g, const V4<float>* lam_in, V4<float>* lam_out,
                             const V4<float>* sp, float* face, int* err, cudaStream_t st,
                             const March3d& t, int org) {
    Args a;
    for (int k = 0; k < 3; ++k) a.n[k] = g.n[k];
    a.lam_out = reinterpret_cast<float4*>(lam_out);
    a.face = face;
    FaceOffsets fo;
    long long tot;
    face_offsets(g, fo, tot);
    for (int f = 0; f < 6; ++f) a.face_off[f] = fo.off[f];
    a.err = err;
    a.A9 = (float)(g.A / 9.0);
    a.zchunk = t.zchunk;
    const size_t per_warp = (NSLOT + NUSLOT) * 512 * R + 2 * 2 * kSeam * 32 * 4;
    const size_t bars = (NSLOT + NUSLOT) * 8, smem = per_warp * t.warps + bars;
    static std::atomic<unsigned> attr{0};   // devices whose shared-memory limit is raised
    if (!device_done(attr)) {
        for (const void* k : {(const void*)k_adj_march<false>, (const void*)k_adj_march<true>}) {
            const cudaError_t r =
                cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(per_warp * kMaxWarps + bars));
            if (r != cudaSuccess) return r;
        }
        device_mark(attr);
    }
    CUtensorMap map, umap;
    if (!encode_state_map(&map, lam_in, g, 32, R * t.warps) ||
        !encode_state_map(&umap, sp, g, 32, R * t.warps))
        return cudaErrorInvalidValue;
    const dim3 grid(t.tiles_x, t.tiles_y, t.chunks), block(32, t.warps);
    if (org == 0) k_adj_march<true><<<grid, block, smem, st>>>(map, umap, a);
    else k_adj_march<false><<<grid, block, smem, st>>>(map, umap, a);
    return cudaGetLastError();
}

}  // namespace lks
