// Fused D3Q15 LKS step for the FP32 path on non-periodic grids, as a z-march of warps that hold
// several rows of a tile in registers (Algorithm 1's stencil part: Eqs. rho, u with the viscosity term
// of f^eq, the Brinkman update of Eq. u_ex_2), and the tiling of the 3D z-march kernels.
//
// A block of NW warps evaluates f^eq on 32 columns x (R NW) rows of one plane after another over a
// chunk of planes; lane = column, each warp owns R consecutive rows.  The node state comes by TMA into
// a ring of planes one node wider on every side.  The sums over c_i f_i^eq(x - c_i) run one axis at a
// time:
//   y  in registers between a warp's rows; at the R-row seams through shared memory, after the x part
//      (five values a column and seam, one block barrier a plane);
//   x  by warp shuffles, per c_z group the sums and the differences of the two rows' values (ten a
//      node);
//   z  in registers: the groups c_z = -1, 0, +1 of plane p complete plane p - 1, add to plane p and
//      start plane p + 1.
// Every f^eq is evaluated once per block; with the halo columns, rows and planes and the parts of the
// last tiles outside the grid that makes 1.38 of them an output node at 256^3 and 1.75 at 128^3.  The 12
// values a node sends out no longer pass through shared memory.  kappa and u_S of the footprint box come by TMA too: outside
// the box the copy fills zeros, so the update needs no test.  The boundary copies (Eqs. bc_rho, bc_u)
// follow in k_bc_shell3d: written here by the threads that hold their sources they made the blocks at
// the faces, and so the launch, longer by more than that kernel (256^3: 239 us a step against 198).
//
// Bound by instruction issue (67 % active): 250 instructions a node, 299 with one node a thread and
// twelve values a node through shared memory.  256^3: 168 us and k_bc_shell3d 10; 178 us a step by
// events against 202 of that z-march.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "lks_march3d.h"
#include "lks_tma.cuh"
#include "lks_units.cuh"

namespace lks {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int R = 4;              // rows per warp
constexpr int NSLOT = 3;          // state planes in the ring
constexpr int NKSLOT = 3;         // planes of kappa, u_S
constexpr int RX = 34;            // columns of a ring row
constexpr int kOutX = 30;         // output columns of a tile
constexpr int kSeam = 5;          // values a column publishes at a seam
constexpr int kMaxWarps = 7;      // two such blocks per SM at 128 registers

struct Args {
    int n[3];
    int blo[3], bn[3], box;       // footprint box (box = 0: none)
    const float4* src;            // the state the tensor map describes (planes two off a z face)
    float4* out;
    int* err;
    int zchunk;
    float A, bf[3];
};

__device__ __forceinline__ float left(float v) { return __shfl_up_sync(FULL, v, 1); }
__device__ __forceinline__ float right(float v) { return __shfl_down_sync(FULL, v, 1); }

__device__ __forceinline__ float4 lds(unsigned a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a));
    return v;
}
__device__ __forceinline__ void st_if(float4* p, const float4& v, bool go) {
    asm volatile(
        "{ .reg .pred p; setp.ne.s32 p, %5, 0;"
        " @p st.global.v4.f32 [%4], {%0, %1, %2, %3}; }" ::"f"(v.x),
        "f"(v.y), "f"(v.z), "f"(v.w), "l"(p), "r"((int)go)
        : "memory");
}

__global__ void __launch_bounds__(32 * kMaxWarps, 2)
    k_step_march(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap kmap,
                 const __grid_constant__ Args a) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
    const int lane = threadIdx.x, wid = threadIdx.y, nw = blockDim.y, rows = R * nw;
    // ring planes of (rows + 2) x RX records and kappa planes of rows x 32, each a multiple of 128
    // bytes
    const unsigned pbytes = (unsigned)(rows + 2) * RX * 16u, pslot = (pbytes + 127u) & ~127u;
    const unsigned kbytes = (unsigned)rows * 512u;
    const unsigned kbase = smem_addr(smem) + NSLOT * pslot;
    const int seam_warp = 2 * kSeam * 32;
    float* seams = reinterpret_cast<float*>(smem + NSLOT * pslot + NKSLOT * kbytes);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + NSLOT * pslot + NKSLOT * kbytes +
                                                 (size_t)2 * nw * seam_warp * 4);
    uint64_t* kbars = bars + NSLOT;
    // first output column, row and plane of the block; f^eq from one less
    const int x0 = 1 + blockIdx.x * kOutX, y0 = 1 + blockIdx.y * (rows - 2);
    const int q0 = 1 + blockIdx.z * a.zchunk, q1 = min(nz - 1, q0 + a.zchunk);
    const int nplanes = q1 - q0 + 4;   // state planes q0 - 2 .. q1 + 1
    const bool leader = lane == 0 && wid == 0;
    if ((smem_addr(smem) & 127u) != 0u) {
        if (leader) atomicOr(a.err, 16);
        return;
    }
    // planes whose outputs meet the footprint box (the same for all threads of the block)
    const bool bxy = a.box && x0 + kOutX > a.blo[0] && x0 < a.blo[0] + a.bn[0] &&
                     y0 + rows - 2 > a.blo[1] && y0 < a.blo[1] + a.bn[1];
    const int kq0 = bxy ? max(q0, a.blo[2]) : 1, kq1 = bxy ? min(q1, a.blo[2] + a.bn[2]) : 0;
    auto load_k = [&](int q, int s) {   // kappa, u_S of plane q into slot s
        tma_load_box(kbase + s * kbytes, &kmap, x0 - 1 - a.blo[0], y0 - 1 - a.blo[1], q - a.blo[2],
                     smem_addr(&kbars[s]), kbytes);
    };
    if (leader) {
        for (int s = 0; s < NSLOT + NKSLOT; ++s) mbar_init(smem_addr(&bars[s]));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int k = 0; k < NSLOT && k < nplanes; ++k)
            tma_load_box(smem_addr(smem) + k * pslot, &tmap, x0 - 2, y0 - 2, q0 - 2 + k,
                         smem_addr(&bars[k]), pbytes);
        for (int q = kq0; q < kq1 && q < kq0 + 2; ++q) load_k(q, q - kq0);
    }
    __syncthreads();

    const int x = x0 - 1 + lane, yr = y0 - 1 + R * wid;   // column, first row
    const bool xout = lane >= 1 && lane <= kOutX && x <= nx - 2;
    const bool xlo = x == 0, xhi = x == nx - 1;
    const bool xface = __any_sync(FULL, xlo || xhi);
    const bool yface = yr == 0 || (yr <= ny - 1 && yr + R - 1 >= ny - 1);
    // own node of row 0 in a ring plane; the node offset of row 0 in plane p - 1
    const unsigned own = smem_addr(smem) + (unsigned)(((R * wid + 1) * RX) + lane + 1) * 16u;
    constexpr unsigned ROW = RX * 16u;
    const unsigned kown = kbase + (unsigned)(R * wid * 32 + lane) * 16u;
    const int zst = nx * ny;   // node counts are below 2^31
    int at = (q0 - 2) * zst + yr * nx + x;
    int fout = 0;   // bit r: row r is an output row
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int j = R * wid + r;
        if (xout && j >= 1 && j <= rows - 2 && yr + r <= ny - 2) fout |= 1 << r;
    }
    const float A = a.A;
    float3 um[R];      // u of plane p - 1
    float4 c[R];       // node of plane p
    float4 acc[R];     // rho, u of plane p - 1 but for the c_z = -1 group of plane p
    float3 nxt[R];     // c_z = +1 group of plane p - 1: its sum (rho and u_z), u_x, u_y
    bool ok;
    {
        bool good = mbar_wait(smem_addr(&bars[0]), 0);
        good = mbar_wait(smem_addr(&bars[1]), 0) && good;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 v = lds(own + r * ROW);
            um[r] = make_float3(v.y, v.z, v.w);
            c[r] = lds(own + pslot + r * ROW);
            acc[r] = make_float4(0.f, 0.f, 0.f, 0.f);
            nxt[r] = make_float3(0.f, 0.f, 0.f);
        }
        ok = !__syncthreads_or(!good);
        if (leader && NSLOT < nplanes) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tma_load_box(smem_addr(smem), &tmap, x0 - 2, y0 - 2, q0 - 2 + NSLOT,
                         smem_addr(&bars[0]), pbytes);
        }
    }
    const int wlo = max(wid - 1, 0), whi = min(wid + 1, nw - 1);
    int k = 1;   // ring index of plane p (p = q0 - 2 + k)
    int s0 = 1, s1 = 2, par = 0;   // slots of planes p and p + 1, parity of the latter
    int ks = 0, kpar = 0;          // the same for the next plane of kappa
    // rho, u of plane q = p - 1 in row r to global memory (Eq. u_ex_2), kappa and u_S from the ring
    auto emit = [&](int r, float4 o, bool box, unsigned kaddr, bool go) {
        o.y += a.bf[0];
        o.z += a.bf[1];
        o.w += a.bf[2];
        if (box) {
            const float4 ks = lds(kaddr + r * 512u);
            const float inv = __frcp_rn(1.f + ks.x);
            o.y = fmaf(ks.x, ks.y, o.y) * inv;
            o.z = fmaf(ks.x, ks.z, o.z) * inv;
            o.w = fmaf(ks.x, ks.w, o.w) * inv;
        }
        st_if(a.out + (at + r * nx), o, go && (fout >> r & 1));
    };
#pragma unroll 1
    for (int p = q0 - 1; ok && p <= q1; ++p, ++k, at += zst) {
        bool good = mbar_wait_once(smem_addr(&bars[s1]), par);
        const unsigned o0 = own + s0 * pslot, o1 = own + s1 * pslot;
        const int q = p - 1;
        const bool box = q >= kq0 && q < kq1, go = q >= q0;
        if (box) good = mbar_wait_once(smem_addr(&kbars[ks]), kpar) && good;
        const unsigned kaddr = kown + ks * kbytes;
        float* sb = seams + ((p & 1) * nw + wid) * seam_warp + lane;
        Feq<float> f;
        float upP[2], upM[2], upY;   // what row r - 1 sends up, to row r
        float md[5];                 // row r - 1: f0, xp, xm, zp, zm
        float lowP[2], lowM[2], lowY;   // what row r - 2 sent up, to row r - 1
        lowP[0] = lowP[1] = lowM[0] = lowM[1] = lowY = 0.f;
        float4 fin0 = make_float4(0.f, 0.f, 0.f, 0.f), fin3 = fin0;
#pragma unroll
        for (int r = 0; r <= R; ++r) {
            if (r < R) {
                const float4 n = lds(o1 + r * ROW);
                const float4 e = lds(o0 + r * ROW + 16u), w = lds(o0 + r * ROW - 16u);
                const float4 cc = c[r];
                const float4 hi = r < R - 1 ? c[r + 1] : lds(o0 + R * ROW);
                // the row below: its node of plane p is in um / c by now (see the end of the loop)
                const float4 lo = r > 0 ? make_float4(0.f, um[r - 1].x, um[r - 1].y, um[r - 1].z)
                                        : lds(o0 - ROW);
                float Dxx = e.y - w.y, Dyx = e.z - w.z, Dzx = e.w - w.w;
                float Dxy = hi.y - lo.y, Dyy = hi.z - lo.z, Dzy = hi.w - lo.w;
                float Dxz = n.y - um[r].x, Dyz = n.z - um[r].y, Dzz = n.w - um[r].z;
                if (xface) {   // one-sided along x on a face column
                    const float4 t = lds(o0 + r * ROW + (xhi ? -32 : (xlo ? 32 : 0)));
                    if (xlo || xhi) {
                        const float4 i1 = xhi ? w : e;
                        Dxx = onesided(xhi, cc.y, i1.y, t.y);
                        Dyx = onesided(xhi, cc.z, i1.z, t.z);
                        Dzx = onesided(xhi, cc.w, i1.w, t.w);
                    }
                }
                if (yface && (yr + r == 0 || yr + r == ny - 1)) {   // along y on a face row
                    const bool h = yr + r != 0;
                    const float4 t = lds(o0 + r * ROW + (h ? -2 * (int)ROW : 2 * (int)ROW));
                    const float4 i1 = h ? lo : hi;
                    Dxy = onesided(h, cc.y, i1.y, t.y);
                    Dyy = onesided(h, cc.z, i1.z, t.z);
                    Dzy = onesided(h, cc.w, i1.w, t.w);
                }
                if (p == 0 || p == nz - 1) {   // along z on a face plane: the second plane inward
                    const bool h = p != 0;     // is not in the ring
                    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (x < nx && yr + r < ny)
                        t = __ldg(a.src + ((h ? nz - 3 : 2) * zst + (yr + r) * nx + x));
                    Dxz = onesided(h, cc.y, h ? um[r].x : n.y, t.y);
                    Dyz = onesided(h, cc.z, h ? um[r].y : n.z, t.z);
                    Dzz = onesided(h, cc.w, h ? um[r].z : n.w, t.w);
                }
                feq<float>(cc.x, cc.y, cc.z, cc.w, A, Dxx, Dyx, Dzx, Dxy, Dyy, Dzy, Dxz, Dyz, Dzz, f);
                um[r] = make_float3(cc.y, cc.z, cc.w);
                c[r] = n;
                if (r == 0) {   // what row 0 sends down, x-combined, to the warp below
                    const float lp = left(f.dp[0]), rp = right(f.dp[1]);
                    const float lm = left(f.dm[0]), rm = right(f.dm[1]);
                    sb[0 * 32] = lp + rp;
                    sb[1 * 32] = lp - rp;
                    sb[2 * 32] = lm + rm;
                    sb[3 * 32] = lm - rm;
                    sb[4 * 32] = f.ym;
                }
                if (r == R - 1) {   // what row R - 1 sends up, to the warp above
                    const float lp = left(f.up[0]), rp = right(f.up[1]);
                    const float lm = left(f.um[0]), rm = right(f.um[1]);
                    float* s = sb + kSeam * 32;
                    s[0 * 32] = lp + rp;
                    s[1 * 32] = lp - rp;
                    s[2 * 32] = lm + rm;
                    s[3 * 32] = lm - rm;
                    s[4 * 32] = f.yp;
                }
            } else {   // nothing comes down from inside the warp to row R - 1
                f.dp[0] = f.dp[1] = f.dm[0] = f.dm[1] = f.ym = 0.f;
            }
            if (r > 0) {   // row i = r - 1: the y sums inside the warp, then x, then z
                const int i = r - 1;
                const float lp = left(lowP[0] + f.dp[0]), rp = right(lowP[1] + f.dp[1]);
                const float lpt = left(lowP[0] - f.dp[0]), rpt = right(lowP[1] - f.dp[1]);
                const float lm = left(lowM[0] + f.dm[0]), rm = right(lowM[1] + f.dm[1]);
                const float lmt = left(lowM[0] - f.dm[0]), rmt = right(lowM[1] - f.dm[1]);
                const float lx = left(md[1]), rx = right(md[2]);
                const float all_m = (lm + rm) + md[4], all_p = (lp + rp) + md[3];
                float4 o;
                o.x = acc[i].x + all_m;
                o.y = acc[i].y + (lm - rm);
                o.z = acc[i].z + (lmt + rmt);
                o.w = acc[i].w - all_m;
                acc[i].x = nxt[i].x + ((md[0] + lowY) + ((lx + rx) + f.ym));
                acc[i].y = nxt[i].y + (lx - rx);
                acc[i].z = nxt[i].z + (lowY - f.ym);
                acc[i].w = nxt[i].x;
                nxt[i] = make_float3(all_p, lp - rp, lpt + rpt);
                if (i == 0) fin0 = o;
                else if (i == R - 1) fin3 = o;
                else emit(i, o, box, kaddr, go);
            }
            if (r < R) {
                if (r > 0) {
                    lowP[0] = upP[0];
                    lowP[1] = upP[1];
                    lowM[0] = upM[0];
                    lowM[1] = upM[1];
                    lowY = upY;
                }
                upP[0] = f.up[0];
                upP[1] = f.up[1];
                upM[0] = f.um[0];
                upM[1] = f.um[1];
                upY = f.yp;
                md[0] = f.f0;
                md[1] = f.xp;
                md[2] = f.xm;
                md[3] = f.zp;
                md[4] = f.zm;
            }
        }
        if (__syncthreads_or(!good)) {
            ok = false;
            break;
        }
        if (leader) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            // plane p is read by all: its slot takes plane p + NSLOT; so is plane q - 1 of kappa
            if (k + NSLOT < nplanes)
                tma_load_box(smem_addr(smem) + s0 * pslot, &tmap, x0 - 2, y0 - 2,
                             q0 - 2 + k + NSLOT, smem_addr(&bars[s0]), pbytes);
            if (box && q + 2 < kq1) load_k(q + 2, ks == 0 ? 2 : ks - 1);
        }
        {   // the seams: row 0 from the warp below, row R - 1 from the warp above
            const float* s = seams + ((p & 1) * nw + wlo) * seam_warp + kSeam * 32 + lane;
            const float ap = s[0 * 32], bp = s[1 * 32], am = s[2 * 32], bm = s[3 * 32], fy = s[4 * 32];
            nxt[0].x += ap;
            nxt[0].y += bp;
            nxt[0].z += ap;
            acc[0].x += fy;
            acc[0].z += fy;
            fin0.x += am;
            fin0.y += bm;
            fin0.z += am;
            fin0.w -= am;
            emit(0, fin0, box, kaddr, go);
        }
        {
            const float* s = seams + ((p & 1) * nw + whi) * seam_warp + lane;
            const float ap = s[0 * 32], bp = s[1 * 32], am = s[2 * 32], bm = s[3 * 32], fy = s[4 * 32];
            nxt[R - 1].x += ap;
            nxt[R - 1].y += bp;
            nxt[R - 1].z -= ap;
            acc[R - 1].x += fy;
            acc[R - 1].z -= fy;
            fin3.x += am;
            fin3.y += bm;
            fin3.z -= am;
            fin3.w -= am;
            emit(R - 1, fin3, box, kaddr, go);
        }
        s0 = s1;
        if (++s1 == NSLOT) {
            s1 = 0;
            par ^= 1;
        }
        if (box && ++ks == NKSLOT) {
            ks = 0;
            kpar ^= 1;
        }
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

March3d march_tiles(const MarchCost& m, int out_x, int out_y, int nz, int warps) {
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    March3d best{};
    double best_cost = 1e300;
    for (int w = m.max_warps; w >= 2; --w) {
        if (warps > 0 ? w != warps : w < 4) continue;
        const int out = m.rows * w - m.halo;
        const long long tx = (out_x + m.tile_x - 1) / m.tile_x, ty = (out_y + out - 1) / out;
        const int per_sm = m.room / w;
        for (int c = 1; c <= std::max(1, nz / 8); ++c) {
            const int zc = (nz + c - 1) / c;
            const long long chunks = (nz + zc - 1) / zc, blocks = tx * ty * chunks;
            const long long slots = (long long)nsm * per_sm, full = blocks / slots, rem = blocks % slots;
            const double last = rem ? m.wave + (double)((rem + nsm - 1) / nsm * w) : 0.0;
            const double cost = ((double)full * (m.wave + per_sm * w) + last + m.tail) *
                                (zc + m.start + 8.0 / per_sm);
            if (cost < best_cost * (1.0 - 1e-9)) {
                best_cost = cost;
                best = March3d{w, (int)tx, (int)ty, zc, (int)chunks, cost};
            }
        }
    }
    return best;
}

March3d step_march_tiles(const Geom& g) {
    return march_tiles(MarchCost{kOutX, R, 2, kMaxWarps, 2 * kMaxWarps, 27.0, 33.0, 1.0}, g.n[0] - 2,
                       g.n[1] - 2, g.n[2] - 2, 0);
}

cudaError_t launch_step_march(const Geom& g, const V4<float>* src, const V4<float>* kus,
                              V4<float>* dst, int* err, cudaStream_t st, const March3d& t) {
    Args a;
    for (int k = 0; k < 3; ++k) {
        a.n[k] = g.n[k];
        a.blo[k] = g.blo[k];
        a.bn[k] = g.bn[k];
        a.bf[k] = (float)g.body[k];
    }
    a.box = g.boxN > 0;
    a.src = reinterpret_cast<const float4*>(src);
    a.out = reinterpret_cast<float4*>(dst);
    a.err = err;
    a.A = (float)g.A;
    a.zchunk = t.zchunk;
    auto smem_of = [](int w) {
        const size_t plane = ((size_t)(R * w + 2) * RX * 16 + 127) / 128 * 128;
        return NSLOT * plane + (size_t)NKSLOT * R * w * 512 + (size_t)2 * w * 2 * kSeam * 32 * 4 +
               (NSLOT + NKSLOT) * 8;
    };
    static std::atomic<unsigned> attr{0};   // devices whose shared-memory limit is raised
    if (!device_done(attr)) {
        const cudaError_t r = cudaFuncSetAttribute(
            k_step_march, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(kMaxWarps));
        if (r != cudaSuccess) return r;
        device_mark(attr);
    }
    CUtensorMap map, kmap;
    if (!encode_state_map(&map, src, g, RX, R * t.warps + 2)) return cudaErrorInvalidValue;
    kmap = map;
    if (a.box) {
        Geom b = g;
        for (int k = 0; k < 3; ++k) b.n[k] = g.bn[k];
        if (!encode_state_map(&kmap, kus, b, 32, R * t.warps)) return cudaErrorInvalidValue;
    }
    k_step_march<<<dim3(t.tiles_x, t.tiles_y, t.chunks), dim3(32, t.warps), smem_of(t.warps), st>>>(
        map, kmap, a);
    return cudaGetLastError();
}

}  // namespace lks
