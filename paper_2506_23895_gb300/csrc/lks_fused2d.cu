// D2Q9 kernels over instance tables (lks_table.h): every launch covers all instances of a plan.
//
//   k_t_design_pos  x_ref, y_ref of every design node (Sec. 2.3) for a group of steps;
//   k_t_transfer2d  kappa and u_S on every footprint-box node for a group of steps: the transfer
//                   depends on the motion and the design only, so the transfers of many steps
//                   are one launch with full grids instead of a short launch before each step;
//   k_t_step        the LKS step (Alg. 1; Sec. 2.2 f^eq with the viscosity term, Eqs. rho, u,
//                   u_ex_2, bc_rho, bc_u), any number of steps in one launch;
//   k_t_adj         the exact adjoint step (structure of Alg. 2, Eqs. arho, au, as): lambda plus
//                   the transpose of the boundary copies, to mu (Brinkman transpose and the kappa
//                   sensitivity density e), moments of F~, adjoint equilibrium and the full
//                   transposed velocity gradient including the one-sided boundary rows;
//   k_t_sens        dJ/dgamma gather per design node (Sec. 2.4) for a group of steps;
//   k_t_objective   the objective of one level, in parts (Sec. 2.5);
//   k_t_begin, k_t_end, k_t_result   what a run does once, over all instances.
//
// The two stencils march a warp up a strip of columns, lane = column.  What they need from the
// rows below and above stays in registers, what they need from the columns beside comes by warp
// shuffles, so a strip runs without shared memory, barriers or index arithmetic per node.  A
// warp's 32 columns give 28 outputs (f^eq, or the adjoint's moments, need one column of halo and
// the values they read one more).  The 32 x 8 tile kernels these replace spent 410 (step) and 418
// (adjoint) instructions per node, over half of them on tile index arithmetic and shared-memory
// traffic, and waited at four barriers.
#include <cuda_runtime.h>

#include <algorithm>

#include "lks_table.h"
#include "lks_units.cuh"

namespace lks {

namespace {

constexpr int NT = 256;
constexpr int kSensThreads = 64;     // small blocks: a design has few nodes, each a long loop
constexpr int kStripThreads = 256;   // at most eight strips (warps) per block
constexpr unsigned FULL = 0xffffffffu;

// Resident blocks of eight warps the strip kernels are compiled for.
template <class T>
constexpr int strip_minb() {
    return sizeof(T) == 4 ? 2 : 1;
}

// Loads of a node record through L2 (another SM may have written it earlier in the same launch)
// and through the read-only path.
__device__ __forceinline__ V4<float> ldcg4(const V4<float>* p) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
    return V4<float>{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ V4<double> ldcg4(const V4<double>* p) {
    const double2 a = __ldcg(reinterpret_cast<const double2*>(p));
    const double2 b = __ldcg(reinterpret_cast<const double2*>(p) + 1);
    return V4<double>{a.x, a.y, b.x, b.y};
}
template <class V>
__device__ __forceinline__ V ldcg3(const V4<float>* p) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
    return V{v.x, v.y, v.z};
}
template <class V>
__device__ __forceinline__ V ldcg3(const V4<double>* p) {
    const double2 a = __ldcg(reinterpret_cast<const double2*>(p));
    return V{a.x, a.y, __ldcg(reinterpret_cast<const double*>(p) + 2)};
}
template <class V>
__device__ __forceinline__ V ldg3(const V4<float>* p) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    return V{v.x, v.y, v.z};
}
template <class V>
__device__ __forceinline__ V ldg3(const V4<double>* p) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p));
    return V{a.x, a.y, __ldg(reinterpret_cast<const double*>(p) + 2)};
}

// A record from shared memory and to global memory as whole vectors (the pointers come from memory,
// so the compiler does not know their space, and it would split the struct).
__device__ __forceinline__ V4<float> lds4(const V4<float>* p) {
    V4<float> v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.r), "=f"(v.x), "=f"(v.y), "=f"(v.z)
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
    return v;
}
__device__ __forceinline__ V4<double> lds4(const V4<double>* p) {
    V4<double> v;
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.r), "=d"(v.x) : "r"(a));
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v.y) : "r"(a + 16));
    v.z = 0.0;
    return v;
}
__device__ __forceinline__ void stg4(V4<float>* p, const V4<float>& v) {
    asm volatile("st.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.r), "f"(v.x),
                 "f"(v.y), "f"(v.z)
                 : "memory");
}
__device__ __forceinline__ void stg4(V4<double>* p, const V4<double>& v) {
    asm volatile("st.global.v2.f64 [%0], {%1, %2};" ::"l"(p), "d"(v.r), "d"(v.x) : "memory");
    asm volatile("st.global.v2.f64 [%0], {%1, %2};" ::"l"(reinterpret_cast<char*>(p) + 16),
                 "d"(v.y), "d"(v.z)
                 : "memory");
}
// One record of V4<T> from global to shared memory, asynchronously and through L2: skipped unless
// `go`, zeros instead of the record unless `in`; and the groups such copies are counted in.
template <class T>
__device__ __forceinline__ void cp_record(V4<T>* dst, const V4<T>* src, bool go, bool in) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int bytes = in ? 16 : 0;
#pragma unroll
    for (int o = 0; o < (int)sizeof(V4<T>); o += 16)
        asm volatile(
            "{ .reg .pred p; setp.ne.s32 p, %3, 0;"
            " @p cp.async.cg.shared.global [%0], [%1], 16, %2; }" ::"r"(d + o),
            "l"(reinterpret_cast<const char*>(src) + o), "r"(bytes), "r"((int)go)
            : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Instance of work unit u: the last i with pre[i] <= u (pre has count + 1 entries).
__device__ __forceinline__ int find_inst(const int* __restrict__ pre, int count, int u) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(pre + mid) <= u) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int wrap_any(int i, int n) {
    i %= n;
    return i < 0 ? i + n : i;
}

template <class T>
__device__ __forceinline__ const Inst<T>* table(const Plan& p) {
    return (const Inst<T>*)p.tab;
}

template <class T>
__device__ __forceinline__ V4<T>* buf(const Inst<T>& I, int b) {
    return b < BUF_POOL ? (V4<T>*)I.bufs[b]
                        : (V4<T>*)(I.pool + (long long)(b - BUF_POOL) * I.snap);
}

// ---------------------------------------------------------------- transfer

// Design positions of steps n0 .. n0 + n - 1 into position slots 0 .. n - 1.
template <class T>
__global__ void __launch_bounds__(NT) k_t_design_pos(Plan p, int noff, int n) {
    const int* pre = p.pre + U_DCOL * (p.count + 1);
    const int n0 = __ldg(p.nbase) + noff, total = p.total[U_DCOL];
    for (int w = blockIdx.x; w < total * n; w += gridDim.x) {
        const int s = w / total, u = w - s * total;
        const int i = find_inst(pre, p.count, u);
        const Inst<T>& I = table<T>(p)[i];
        const long long k = (long long)(u - pre[i]) * kUnitThreads + threadIdx.x;
        if (k >= I.d.ncol) continue;
        int2 b;
        V4<T> sc;
        col_pos_sc<T>(I.d, I.motion[n0 + s], k, b, sc);
        I.pos_b[s * I.d.ncol + k] = b;
        I.pos_sc[s * I.d.ncol + k] = sc;
    }
}

// One 32 x 16 tile of the footprint box of one step per work unit.  The design nodes whose taps reach
// the tile (integer base in the 35 x 19 cells from two below it to one above) go to shared memory
// ordered by cell (x fastest) and then by design index.  A thread gathers a run of kTrRun nodes of one
// column: a design node serves up to four of them, and the four cells of a row of its support are one
// range of the list.  A tile with more design nodes than the lists hold scans the candidates of each
// node: the bounds' answer only, since the unit squares of a tile's nodes lie in its 35 x 19 cells widened
// by sqrt(2) / 2, which is room for 743.  Bound by instruction issue; 64 channels of side 128 to 512, per step: 55 us (one thread a
// node, 16 cells each with a list of its own: 98 us).
constexpr int kTrRun = 4;
constexpr int kTrThreads = kBoxTileX * kBoxTileY / kTrRun;
constexpr int kTrCX = kBoxTileX + 3, kTrCY = kBoxTileY + 3, kTrCells = kTrCX * kTrCY;
constexpr int kTrPer = (kTrCells + kTrThreads - 1) / kTrThreads;   // cells a thread lists
// a unit-spaced rotated lattice puts at most two nodes in one cell, and about one
constexpr int kTrCap = 4, kTrList = 768;
constexpr int kTrRow = 64;   // a window row's nodes: at most 34.4 + 2 (4 / sqrt 2) + 1 of them

template <class T>
struct TrSmem {
    union {
        V4<T> sc[kTrList];   // sin, cos of the fractions
        struct {             // before these: the cells' unordered lists
            int cnt[kTrCells];
            unsigned short ent[kTrCells * kTrCap];
        };
    };
    V4<T> kx[kTrList];    // kappa_ref, xi - xi_G, the cell's x
    int warp[kTrThreads / 32];
    int full;
    unsigned short start[kTrCells + 1];
    unsigned short key[kTrList];   // window row and place of a listed node
};

template <class T>
__global__ void __launch_bounds__(kTrThreads, sizeof(T) == 4 ? 8 : 4)
    k_t_transfer2d(Plan p, int noff, int nsteps, int kslot0) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    TrSmem<T>& S = *reinterpret_cast<TrSmem<T>*>(smem_raw);
    const int* pre = p.pre + U_BOX * (p.count + 1);
    const int n0 = __ldg(p.nbase) + noff, nbox = p.total[U_BOX];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int NW = kTrThreads / 32;
    for (int w = blockIdx.x; w < nbox * nsteps; w += gridDim.x) {
        const int step = w / nbox, u = w - step * nbox;
        const int i = find_inst(pre, p.count, u);
        const Inst<T>& I = table<T>(p)[i];
        const Design& d = I.d;
        const Geom& g = I.g;
        const Motion& m = I.motion[n0 + step];
        const int2* __restrict__ pb = I.pos_b + (long long)step * d.ncol;
        const V4<T>* __restrict__ psc = I.pos_sc + (long long)step * d.ncol;
        const T* __restrict__ kref = I.kref;
        V4<T>* kus = kslot0 < 0 ? I.kus : I.kus_tape + (long long)(kslot0 + step) * g.boxN;
        const int ntx = (g.bn[0] + kBoxTileX - 1) / kBoxTileX;
        const int t = u - pre[i];
        const int bx0 = (t % ntx) * kBoxTileX, by0 = (t / ntx) * kBoxTileY;
        const int lx = tid % kBoxTileX, ly = tid / kBoxTileX * kTrRun;
        // the tile's window of candidates through the inverse rigid map, in single precision with a
        // margin far above its rounding (it only has to contain the support)
        const float c = m.cf, s = m.sf, ac = fabsf(c), as = fabsf(s);
        const float hx = 0.5f * (kBoxTileX - 1), hy = 0.5f * (kBoxTileY - 1);
        const float px = (float)(g.blo[0] + bx0) + hx - m.xgf[0];
        const float py = (float)(g.blo[1] + by0) + hy - m.xgf[1];
        const float ic = c * px + s * py + d.xiGf[0], jc = -s * px + c * py + d.xiGf[1];
        const float ri = ac * (hx + 2.f) + as * (hy + 2.f) + 0.05f;
        const float rj = as * (hx + 2.f) + ac * (hy + 2.f) + 0.05f;
        const int wi0 = max(0, (int)ceilf(ic - ri)), wi1 = min(d.L[0] - 1, (int)floorf(ic + ri));
        const int wj0 = max(0, (int)ceilf(jc - rj)), wj1 = min(d.L[1] - 1, (int)floorf(jc + rj));
        T kap[kTrRun], m0[kTrRun], m1x[kTrRun], m1y[kTrRun];
#pragma unroll
        for (int j = 0; j < kTrRun; ++j) kap[j] = m0[j] = m1x[j] = m1y[j] = (T)0;
        if (wi0 <= wi1 && wj0 <= wj1) {   // uniform over the block
            const int cx0 = g.blo[0] + bx0 - 2, cy0 = g.blo[1] + by0 - 2;   // first cell
            __syncthreads();   // the previous unit's lists are no longer read
            if (tid == 0) S.full = 0;
            for (int e = tid; e < kTrCells; e += kTrThreads) S.cnt[e] = 0;
            __syncthreads();
            // count the listed nodes of each cell, a warp per window row, over the part of the row
            // that can lie in the cells
            const float ox = m.xgf[0] - c * d.xiGf[0] - (float)cx0;
            const float oy = m.xgf[1] - s * d.xiGf[0] - (float)cy0;
            const float rc = __fdividef(1.f, c), rs = __fdividef(1.f, s);   // used where not near 0
            auto span = [&](int j, int& i0, int& i1) {
                const float dj = (float)j - d.xiGf[1];
                const float xj = ox - s * dj, yj = oy + c * dj;   // of node i = 0, from the first cell
                float lo = (float)wi0, hi = (float)wi1;
                if (ac > 0.2f) {
                    const float e0 = -xj * rc, e1 = ((float)kTrCX - xj) * rc;
                    lo = fmaxf(lo, fminf(e0, e1) - 0.1f);
                    hi = fminf(hi, fmaxf(e0, e1) + 0.1f);
                }
                if (as > 0.2f) {
                    const float e0 = -yj * rs, e1 = ((float)kTrCY - yj) * rs;
                    lo = fmaxf(lo, fminf(e0, e1) - 0.1f);
                    hi = fminf(hi, fmaxf(e0, e1) + 0.1f);
                }
                i0 = (int)ceilf(lo) + lane;
                i1 = j <= wj1 ? (int)floorf(hi) : -1;
            };
            auto put = [&](int j, int ii, const int2& bk) {
                const int cx = bk.x - cx0, cy = bk.y - cy0;
                if ((unsigned)cx >= (unsigned)kTrCX || (unsigned)cy >= (unsigned)kTrCY) return;
                const int cell = cy * kTrCX + cx;
                const int slot = atomicAdd(&S.cnt[cell], 1);
                if (slot < kTrCap)
                    S.ent[cell * kTrCap + slot] = (unsigned short)((j - wj0) * kTrRow + (ii - wi0));
                else S.full = 1;
            };
            constexpr int RB = 3;   // rows whose loads are in flight together
            for (int j = wj0 + wid; j <= wj1; j += RB * NW) {
                int i0[RB], i1[RB];
                int2 bk[RB];
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    span(j + r * NW, i0[r], i1[r]);
                    if (i0[r] <= i1[r]) bk[r] = __ldg(pb + (j + r * NW) * d.L[0] + i0[r]);
                }
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    if (i0[r] <= i1[r]) put(j + r * NW, i0[r], bk[r]);
                    for (int ii = i0[r] + 32; ii <= i1[r]; ii += 32)
                        put(j + r * NW, ii, __ldg(pb + (j + r * NW) * d.L[0] + ii));
                }
            }
            __syncthreads();
            // list offsets: kTrPer consecutive cells per thread, summed over the block
            int nc[kTrPer], sum = 0;
#pragma unroll
            for (int e = 0; e < kTrPer; ++e) {
                const int cell = tid * kTrPer + e;
                nc[e] = cell < kTrCells ? S.cnt[cell] : 0;
                sum += nc[e];
            }
            int at = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(FULL, at, o);
                if (lane >= o) at += v;
            }
            if (lane == 31) S.warp[wid] = at;
            __syncthreads();
            int total = 0;
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                if (k < wid) at += S.warp[k];
                total += S.warp[k];
            }
            at -= sum;
            if (!S.full && total <= kTrList) {
#pragma unroll
                for (int e = 0; e < kTrPer; ++e) {
                    const int cell = tid * kTrPer + e;
                    if (cell >= kTrCells) break;
                    S.start[cell] = (unsigned short)at;
                    if (nc[e] == 0) continue;
                    // in design index order (the order of the slots is not fixed)
                    unsigned short* ent = S.ent + cell * kTrCap;
                    for (int a1 = 1; a1 < nc[e]; ++a1)
                        for (int a2 = a1; a2 > 0 && ent[a2 - 1] > ent[a2]; --a2) {
                            const unsigned short tmp = ent[a2];
                            ent[a2] = ent[a2 - 1];
                            ent[a2 - 1] = tmp;
                        }
                    for (int a1 = 0; a1 < nc[e]; ++a1) {
                        S.key[at + a1] = ent[a1];
                        S.kx[at + a1].z = (T)(cell % kTrCX);
                    }
                    at += nc[e];
                }
                if (tid == 0) S.start[kTrCells] = (unsigned short)total;
                __syncthreads();
#pragma unroll 3
                for (int e = tid; e < total; e += kTrThreads) {
                    const int key = S.key[e], ii = wi0 + key % kTrRow, j = wj0 + key / kTrRow;
                    const int k = j * d.L[0] + ii;
                    S.sc[e] = psc[k];
                    S.kx[e].r = kref[k];
                    S.kx[e].x = (T)ii - (T)d.xiG[0];
                    S.kx[e].y = (T)j - (T)d.xiG[1];
                }
                __syncthreads();
#pragma unroll
                for (int dy = -2; dy <= kTrRun; ++dy) {   // cell row against the run's first node
                    const int c0 = (ly + dy + 2) * kTrCX + lx;
                    const int e1 = S.start[c0 + 4];
#pragma unroll 1
                    for (int e = S.start[c0]; e < e1; ++e) {
                        const V4<T> A = S.sc[e], B = S.kx[e];
                        const T wx = tap_weight<T>(lx + 3 - (int)B.z, A.r, A.x);
#pragma unroll
                        for (int j = 0; j < kTrRun; ++j) {
                            const int qy = j + 1 - dy;
                            if (qy < 0 || qy > 3) continue;
                            const T W = wx * tap_weight<T>(qy, A.y, A.z);
                            kap[j] += W * B.r;
                            m0[j] += W;
                            m1x[j] += W * B.x;
                            m1y[j] += W * B.y;
                        }
                    }
                }
            } else {
                const int x = g.blo[0] + bx0 + lx, y0 = g.blo[1] + by0 + ly;
                for (int j = wj0; j <= wj1; ++j)
                    for (int ii = wi0; ii <= wi1; ++ii) {
                        const int k = j * d.L[0] + ii;
                        const int2 b = __ldg(pb + k);
                        const int qx = x - b.x + 1, q0 = y0 - b.y + 1;
                        if ((unsigned)qx > 3u || q0 > 3 || q0 + kTrRun - 1 < 0) continue;
                        const V4<T> A = psc[k];
                        const T wx = tap_weight<T>(qx, A.r, A.x);
#pragma unroll
                        for (int r = 0; r < kTrRun; ++r) {
                            if ((unsigned)(q0 + r) > 3u) continue;
                            const T W = wx * tap_weight<T>(q0 + r, A.y, A.z);
                            kap[r] += W * kref[k];
                            m0[r] += W;
                            m1x[r] += W * ((T)ii - (T)d.xiG[0]);
                            m1y[r] += W * ((T)j - (T)d.xiG[1]);
                        }
                    }
            }
        }
        const bool f32 = sizeof(T) == 4;
        const T om = f32 ? (T)m.omf : (T)m.om, cT = f32 ? (T)m.cf : (T)m.c,
                sT = f32 ? (T)m.sf : (T)m.s;
        const T ug0 = f32 ? (T)m.ugf[0] : (T)m.uG[0], ug1 = f32 ? (T)m.ugf[1] : (T)m.uG[1];
        if (bx0 + lx >= g.bn[0]) continue;
#pragma unroll
        for (int j = 0; j < kTrRun; ++j) {
            if (by0 + ly + j >= g.bn[1]) break;
            V4<T> o;
            o.r = kap[j];
            o.x = (-sT * m1x[j] - cT * m1y[j]) * om + ug0 * m0[j];
            o.y = (cT * m1x[j] - sT * m1y[j]) * om + ug1 * m0[j];
            o.z = (T)0;
            kus[(long long)(by0 + ly + j) * g.bn[0] + bx0 + lx] = o;
        }
    }
}

// Sensitivity gather of steps noff + n - 1 down to noff: one thread per design node sums its
// 4 x 4 taps of every step's e, and adds kappa' times each sum to dJ/dgamma in step order (FP64).
template <class T>
__global__ void __launch_bounds__(kSensThreads) k_t_sens(Plan p, int noff, int nsteps, int eslot0) {
    const int* pre = p.pre + U_DCOL * (p.count + 1);
    const int n0 = __ldg(p.nbase) + noff;
    constexpr int SUB = kUnitThreads / kSensThreads;
    for (int w = blockIdx.x; w < p.total[U_DCOL] * SUB; w += gridDim.x) {
        const int u = w / SUB;
        const int i = find_inst(pre, p.count, u);
        const Inst<T>& I = table<T>(p)[i];
        const long long k = (long long)(u - pre[i]) * kUnitThreads + (w % SUB) * kSensThreads +
                            threadIdx.x;
        if (k >= I.d.ncol) continue;
        const double kp = (double)I.kprime[k];
        double acc = I.gacc[k];
#pragma unroll 2
        for (int s = nsteps - 1; s >= 0; --s)
            acc += kp * (double)sens2d_sum<T>(I.d, I.g, I.motion[n0 + s],
                                              I.e + (long long)(eslot0 + s) * I.g.boxN, k);
        I.gacc[k] = acc;
    }
}

// ---------------------------------------------------------------- objective (Sec. 2.5)

// Partial sum `part` of the objective over the target list at one level, by one warp: FP64, fixed
// order.
template <class T>
__device__ __forceinline__ void objective_part(const Inst<T>& I, const V4<T>* s, int n, int part,
                                               int lane) {
    const Geom& g = I.g;
    const int tot = (int)g.ocount, np = I.jparts;
    const int per = (tot + np - 1) / np, k1 = min(tot, (part + 1) * per);
    double acc = 0.0;
#pragma unroll 4
    for (int k = part * per + lane; k < k1; k += 32) {
        const V4<T> v = ldcg4(s + g.otarget[k]);
        acc += g.okind == 0 ? (double)v.r : g.odir[0] * (double)v.x + g.odir[1] * (double)v.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
    if (lane == 0) I.jpart[(long long)n * np + part] = acc;
}

// Unit u of the objective units: instance and part, skipped outside the window.
template <class T>
__device__ __forceinline__ void objective_unit(const Plan& p, int u, int n, int b, int lane) {
    const int* pre = p.pre + U_OBJ * (p.count + 1);
    const int i = find_inst(pre, p.count, u);
    const Inst<T>& I = table<T>(p)[i];
    if (n < I.win_begin || n > I.win_end) return;   // uniform over the warp
    objective_part<T>(I, buf(I, b), n, u - pre[i], lane);
}

template <class T>
__global__ void __launch_bounds__(NT) k_t_objective(Plan p, int noff, int b) {
    const int u = blockIdx.x * (NT / 32) + threadIdx.x / 32;
    if (u < p.total[U_OBJ])
        objective_unit<T>(p, u, __ldg(p.nbase) + noff, b, threadIdx.x & 31);
}

// Start of a run: the error words, and for an adjoint run lambda^N and dJ/dgamma, to zero.
template <class T>
__global__ void __launch_bounds__(NT) k_t_begin(Plan p, int adjoint) {
    const Inst<T>& I = table<T>(p)[blockIdx.y];
    const int t = blockIdx.x * NT + threadIdx.x, nt = gridDim.x * NT;
    if (t < 4) I.flags[t] = 0;
    if (!adjoint) return;
    uint4* l = (uint4*)buf(I, BUF_LAM0);
    const int n = (int)(I.g.nodes * (sizeof(V4<T>) / 16));
    for (int k = t; k < n; k += nt) l[k] = make_uint4(0u, 0u, 0u, 0u);
    for (long long k = t; k < I.d.nd; k += nt) I.gacc[k] = 0.0;
}

// End of a run: buffer src to dst, and on a forward run the divergence check of that state.
template <class T>
__global__ void __launch_bounds__(NT) k_t_end(Plan p, int dst, int src, int check) {
    const Inst<T>& I = table<T>(p)[blockIdx.y];
    const V4<T>* a = buf(I, src);
    V4<T>* b = buf(I, dst);
    const int n = (int)I.g.nodes;
    for (int k = blockIdx.x * NT + threadIdx.x; k < n; k += gridDim.x * NT) {
        const V4<T> v = a[k];
        b[k] = v;
        const T m = fabs(v.x) + fabs(v.y) + fabs(v.z);
        if (check && (!(m < (T)0.5) || !(fabs(v.r) < (T)1e30))) atomicOr(I.flags + 2, 1);
    }
}

// Per instance: j = -(rho0 + mean(rho - rho0))/3 (J1) or -mean(n.u) (J2) of every step of the
// window up to n_last from the parts, J = h sum_n j_n (fixed order), and the error words.
template <class T>
__global__ void __launch_bounds__(NT) k_t_result(Plan p, int n_last, int adjoint, RunResult* out) {
    const Inst<T>& I = table<T>(p)[blockIdx.x];
    __shared__ double red[NT];
    double acc = 0.0;
    if (!adjoint) {
        const int w1 = min(I.win_end, n_last);
        const double h = 1.0 / (double)(I.win_end - I.win_begin + 1);
        for (int n = I.win_begin + threadIdx.x; n <= w1; n += NT) {
            double sum = 0.0;
            for (int q = 0; q < I.jparts; ++q) sum += I.jpart[(long long)n * I.jparts + q];
            acc += h * (I.g.okind == 0 ? -(I.g.rho0 + sum / I.g.ocount) / 3.0 : -sum / I.g.ocount);
        }
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = NT / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x].J = red[0];
    if (threadIdx.x < 4) out[blockIdx.x].flags[threadIdx.x] = I.flags[threadIdx.x];
}

__global__ void k_set_int(int* dst, int v) { *dst = v; }

// Buffer src of every instance to its buffer dst (whole records of 16 bytes).
template <class T>
__global__ void __launch_bounds__(NT) k_t_copy(Plan p, int dst, int src) {
    const Inst<T>& I = table<T>(p)[blockIdx.y];
    const uint4* a = (const uint4*)buf(I, src);
    uint4* b = (uint4*)buf(I, dst);
    const int n = (int)(I.g.nodes * (sizeof(V4<T>) / 16));
    for (int k = blockIdx.x * NT + threadIdx.x; k < n; k += gridDim.x * NT) b[k] = a[k];
}

// ---------------------------------------------------------------- strips

// All blocks of a cooperative launch meet for the `round`-th time (1, 2, ...): *bar counts arrivals
// from zero, so that one release and the polling of one word do (an arrival count that the last
// block turns into a generation costs a second trip to L2: 3.0 us a meeting against 2.0).  The wait
// is bounded (about a second); a block that gives up sets the error word and returns false, and so
// do the others after it.
__device__ __forceinline__ bool grid_meet(const Plan& p, int nblocks, int round) {
    __shared__ int ok;
    __syncthreads();
    if (nblocks == 1) return true;
    if (threadIdx.x == 0) {
        int good = 1;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p.bar) : "memory");
        const int want = nblocks * round;
        const long long t0 = clock64();
        while (ld_acquire(p.bar) < want)
            if (clock64() - t0 > (1LL << 31)) {
                atomicOr(p.err, 8);
                good = 0;
                break;
            }
        ok = good;
    }
    __syncthreads();
    return ok != 0;
}

// The arithmetic below is written with explicitly rounded operations, which the compiler neither
// contracts nor reorders: every strip height then computes bitwise the same state.
template <class T>
__device__ __forceinline__ T fma_(T a, T b, T c);
template <>
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <>
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
template <class T>
__device__ __forceinline__ T mul_(T a, T b);
template <>
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
template <>
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
template <class T>
__device__ __forceinline__ T add_(T a, T b);
template <>
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
template <>
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
template <class T>
__device__ __forceinline__ T sub_(T a, T b);
template <>
__device__ __forceinline__ float sub_(float a, float b) { return __fsub_rn(a, b); }
template <>
__device__ __forceinline__ double sub_(double a, double b) { return __dsub_rn(a, b); }
template <class T>
__device__ __forceinline__ T inv_(T a);
template <>
__device__ __forceinline__ float inv_(float a) { return __frcp_rn(a); }
template <>
__device__ __forceinline__ double inv_(double a) { return __drcp_rn(a); }

template <class T>
__device__ __forceinline__ T from_left(T v) { return __shfl_up_sync(FULL, v, 1); }
template <class T>
__device__ __forceinline__ T from_right(T v) { return __shfl_down_sync(FULL, v, 1); }

template <class T>
struct V3 {
    T r, x, y;
};

// Geometry of a strip as its lane sees it.
struct Strip {
    int x;          // this lane's column, wrapped on a periodic axis
    int xs;         // the strip's first output column
    int ya, yb;     // first and last row of the strip (clipped to the grid)
    bool in;        // column inside the grid
    bool own;       // one of the strip's output columns
    int mode;       // kInner, kSide or kGeneral
};

// What a strip and its halo of two nodes and two more rows touch: no face and no node next to one;
// only x faces of a grid without wraps and static solids, no node next to both; anything else.
enum { kInner = 0, kSide = 1, kGeneral = 2 };

template <class T>
__device__ __forceinline__ Strip strip_of(const Inst<T>& I, int local, int rows, int lane) {
    const Geom& g = I.g;
    const int n0 = g.n[0], n1 = g.n[1];
    const int ns = strip_count(n0, kStripW, g.periodic[0]);
    const int kc = local / ns, kx = local - kc * ns;
    Strip s;
    s.xs = kx * kStripW - strip_origin(n0, kStripW, g.periodic[0]);
    const int xr = s.xs - 2 + lane;
    s.own = lane >= 2 && lane < 2 + kStripW && xr >= 0 && xr < n0;
    s.x = g.periodic[0] ? wrap_any(xr, n0) : xr;
    s.in = s.x >= 0 && s.x < n0;
    s.ya = kc * rows;
    s.yb = min(s.ya + rows, n1) - 1;
    // (along an x axis of three nodes the inner column lies next to both faces, where a kSide lane
    // serves one)
    const bool plain = n0 > 3 && !g.periodic[0] && !g.periodic[1] && !g.ks && s.ya >= 4 &&
                       s.yb <= n1 - 5;
    const bool xmid = s.xs >= 4 && s.xs + kStripW + 1 <= n0 - 3;
    // (the adjoint's kSide path finds the face column in the lane beside a node next to it)
    const bool xcut = s.xs - 2 + 31 == n0 - 2;
    s.mode = !plain || xcut ? kGeneral : (xmid ? kInner : kSide);
    return s;
}

// The value bc_value gives a boundary node of face f from its source's value, with the face's values
// rounded once on the host.
template <class T>
__device__ __forceinline__ V4<T> face_value2(const Inst<T>& I, int f, const V4<T>& o) {
    const V4<T> p = I.bcf[f];
    const bool keep = I.bckeep[f] != 0;
    V4<T> b;
    b.r = keep ? o.r : p.r;
    b.x = keep || f >= 2 ? p.x : o.x;
    b.y = keep || f < 2 ? p.y : o.y;
    b.z = (T)0;
    return b;
}

// Boundary copies sourced by interior node (x, y) of value o (Eqs. bc_rho, bc_u): the node beside
// it on an x face, on a y face, and the corner of the two with the face that wins there.  (Along
// an axis of three nodes one node lies next to both faces: the general rule.)
template <class T>
__device__ __forceinline__ void write_bc2(const Inst<T>& I, int x, int y, const V4<T>& o,
                                          V4<T>* out) {
    const Geom& g = I.g;
    const int n0 = g.n[0], n1 = g.n[1];
    const bool xl = !g.periodic[0] && x == 1, xh = !g.periodic[0] && x == n0 - 2;
    const bool yl = !g.periodic[1] && y == 1, yh = !g.periodic[1] && y == n1 - 2;
    if ((xl && xh) || (yl && yh)) {
        write_bc_from(g, x, y, 0, o, out);
        return;
    }
    const int fx = xh ? 1 : 0, fy = yh ? 3 : 2;
    const int bx = xl ? 0 : n0 - 1, by = yl ? 0 : n1 - 1;
    if (xl || xh) stg4(out + (y * n0 + bx), face_value2<T>(I, fx, o));
    if (yl || yh) stg4(out + (by * n0 + x), face_value2<T>(I, fy, o));
    if ((xl || xh) && (yl || yh))
        stg4(out + (by * n0 + bx), face_value2<T>(I, I.corner[fx + 2 * (fy - 2)], o));
}

// One strip of the forward step.  F-row f evaluates f_i^eq at the lane's node (x, f); each output
// row collects three F-rows.  Per output node the directions are grouped by c_x: the node's own
// column adds f0 + f2 + f4 to rho and f2 - f4 to u_y; the column to the left sends
// P = f1 + f5 + f8 and Tp = f5 - f8, the column to the right M = f3 + f6 + f7 and Tm = f6 - f7
// (rho takes P + M, u_x P - M, u_y Tp + Tm): four values by shuffle instead of six.
// State rows, and kappa and u_S, pass through rings in shared memory (per lane: each lane reads
// only the records it copied), copied kAhead rows before they are read, so that the march holds no
// loads in flight in registers.  The mode changes which nodes are special, not the arithmetic.
constexpr int kAhead = 4, kRing = 8;
static_assert(kAhead + 3 <= kRing && (kRing & (kRing - 1)) == 0, "ring slots by mask");

template <class T, int MODE>
__device__ __forceinline__ void step_strip(const Inst<T>& I, const Strip& s, const V4<T>* src,
                                           V4<T>* out, const V4<T>* kus, V4<T>* ring) {
    using W = Wts<T, 2>;
    constexpr bool GEN = MODE == kGeneral, SIDE = MODE != kInner;
    V4<T>* ringk = ring + kRing * 32;   // kappa, u_S
    const Geom& g = I.g;
    const int n0 = g.n[0], n1 = g.n[1];
    const bool p0 = GEN && g.periodic[0], p1 = GEN && g.periodic[1];
    const int ya = !GEN || p1 ? s.ya : max(s.ya, 1), yb = !GEN || p1 ? s.yb : min(s.yb, n1 - 2);
    if (ya > yb) return;   // uniform
    const int x = s.x;
    const bool xin = !SIDE || s.in;
    const bool ocol = s.own && (!SIDE || p0 || (x >= 1 && x <= n0 - 2));
    const int sx = !SIDE || p0 ? 0 : (x == 0 ? -1 : (x == n0 - 1 ? 1 : 0));
    const bool xface = SIDE && (!GEN || __any_sync(FULL, sx != 0));
    const bool xnear = GEN && __any_sync(FULL, ocol && !p0 && (x == 1 || x == n0 - 2));
    // kSide: the face column a node next to it writes, and its prescribed values
    const int wf = SIDE && !GEN && ocol ? (x == 1 ? 0 : (x == n0 - 2 ? 1 : -1)) : -1;
    const int bx = x - g.blo[0], bn0 = g.bn[0], bn1 = g.bn[1], by0 = g.blo[1];
    const bool bcol = g.boxN > 0 && ocol && bx >= 0 && bx < bn0;
    const bool bany = __any_sync(FULL, bcol) && ya < by0 + bn1 && yb >= by0;
    const T* ks_st = GEN ? (const T*)g.ks : nullptr;
    const T A = I.A, bfx = I.bf[0], bfy = I.bf[1];
    const V4<T>* scol = src + (xin ? x : 0);
    const V4<T>* kcol = kus + (bcol ? bx : 0);
    V4<T>* ocl = out + (ocol ? x : 0);
    // a state row, and kappa, u_S two rows below it (the output row that completes when the state
    // row is first read), as one copy group; node indices fit 32 bits (checked at create)
    auto issue = [&](int row) {
        int r = row;
        bool in = xin;
        if (GEN) {
            if (p1) r += r < 0 ? n1 : (r >= n1 ? -n1 : 0);
            in = xin && r >= 0 && r < n1;
            if (!in) r = 0;
        }
        cp_record<T>(ring + (row & (kRing - 1)) * 32, scol + r * n0, row <= yb + 2, in);
        if (bany) {
            const int kr = row - 2 - by0;
            const bool kin = bcol && (unsigned)kr < (unsigned)bn1;
            cp_record<T>(ringk + ((row - 2) & (kRing - 1)) * 32, kcol + (kin ? kr * bn0 : 0),
                         row - 2 <= yb, kin);
        }
        cp_commit();
    };
    // sums of output row f - 1 (a) and f (b) as F-row f is reached: the directions already met
    T a_r = (T)0, a_y = (T)0, a_P = (T)0, a_Tp = (T)0, a_M = (T)0, a_Tm = (T)0;
    T b_2 = (T)0, b_5 = (T)0, b_6 = (T)0;
    auto march = [&](int f, bool emit) {   // emit: uniform, the row completes an output row
        issue(f + 1 + kAhead);
        cp_wait<kAhead>();   // row f + 1 has landed
        const int y = f - 1;   // output row this F-row completes
        V4<T> v0, vp, vm, kv;
        v0 = lds4(ring + (f & (kRing - 1)) * 32);
        vp = lds4(ring + ((f + 1) & (kRing - 1)) * 32);
        vm = lds4(ring + ((f - 1) & (kRing - 1)) * 32);
        kv.r = kv.x = kv.y = (T)0;
        if (emit && bany) kv = lds4(ringk + (y & (kRing - 1)) * 32);
        T kst = (T)0;
        if (GEN && emit && ks_st && ocol) kst = ks_st[y * n0 + x];
        // twice the velocity gradient, D_ab = 2 d u_a / d x_b
        const T l1x = from_left(v0.x), l1y = from_left(v0.y);
        const T r1x = from_right(v0.x), r1y = from_right(v0.y);
        T Dxx = sub_<T>(r1x, l1x), Dyx = sub_<T>(r1y, l1y);
        T Dxy = sub_<T>(vp.x, vm.x), Dyy = sub_<T>(vp.y, vm.y);
        if (xface) {   // one-sided along x on a boundary column
            const T l2x = __shfl_up_sync(FULL, v0.x, 2), l2y = __shfl_up_sync(FULL, v0.y, 2);
            const T r2x = __shfl_down_sync(FULL, v0.x, 2), r2y = __shfl_down_sync(FULL, v0.y, 2);
            if (sx < 0) {
                Dxx = fma_<T>((T)-3, v0.x, fma_<T>((T)4, r1x, -r2x));
                Dyx = fma_<T>((T)-3, v0.y, fma_<T>((T)4, r1y, -r2y));
            } else if (sx > 0) {
                Dxx = fma_<T>((T)3, v0.x, fma_<T>((T)-4, l1x, l2x));
                Dyx = fma_<T>((T)3, v0.y, fma_<T>((T)-4, l1y, l2y));
            }
        }
        if (GEN && !p1 && (f == 0 || f == n1 - 1)) {   // one-sided along y on a boundary row
            V3<T> far;
            far.r = far.x = far.y = (T)0;
            if (xin) far = ldcg3<V3<T>>(scol + (f == 0 ? 2 : n1 - 3) * n0);
            if (f == 0) {
                Dxy = fma_<T>((T)-3, v0.x, fma_<T>((T)4, vp.x, -far.x));
                Dyy = fma_<T>((T)-3, v0.y, fma_<T>((T)4, vp.y, -far.y));
            } else {
                Dxy = fma_<T>((T)3, v0.x, fma_<T>((T)-4, vm.x, far.x));
                Dyy = fma_<T>((T)3, v0.y, fma_<T>((T)-4, vm.y, far.y));
            }
        }
        // f_i^eq = w_i (rho - rho0 - 1.5 u^2 + 4.5 (c.u)^2 + A c.S.c + 3 c.u), opposite directions
        // sharing their symmetric part; the weight products are those of Wts<T, 2>
        const T ux = v0.x, uy = v0.y;
        const T P = fma_<T>((T)-1.5, fma_<T>(ux, ux, mul_<T>(uy, uy)), v0.r);
        const T sd = add_<T>(Dxx, Dyy), so = add_<T>(Dxy, Dyx);
        const T cp = add_<T>(ux, uy), cm = sub_<T>(uy, ux);
        const T ex = fma_<T>(mul_<T>(W::h_1, ux), ux, mul_<T>(W::w1, fma_<T>(A, Dxx, P)));
        const T ey = fma_<T>(mul_<T>(W::h_1, uy), uy, mul_<T>(W::w1, fma_<T>(A, Dyy, P)));
        const T ep = fma_<T>(mul_<T>(W::h_2, cp), cp,
                             mul_<T>(W::w2, fma_<T>(A, add_<T>(sd, so), P)));
        const T em = fma_<T>(mul_<T>(W::h_2, cm), cm,
                             mul_<T>(W::w2, fma_<T>(A, sub_<T>(sd, so), P)));
        const T f0 = mul_<T>(W::w0, P);
        const T f1 = fma_<T>(W::w3_1, ux, ex), f3 = fma_<T>(-W::w3_1, ux, ex);
        const T f2 = fma_<T>(W::w3_1, uy, ey), f4 = fma_<T>(-W::w3_1, uy, ey);
        const T f5 = fma_<T>(W::w3_2, cp, ep), f7 = fma_<T>(-W::w3_2, cp, ep);
        const T f6 = fma_<T>(W::w3_2, cm, em), f8 = fma_<T>(-W::w3_2, cm, em);
        if (emit) {
            const T Pl = from_left(add_<T>(a_P, f8)), Tl = from_left(sub_<T>(a_Tp, f8));
            const T Mr = from_right(add_<T>(a_M, f7)), Tr = from_right(sub_<T>(a_Tm, f7));
            V4<T> o;
            o.r = add_<T>(add_<T>(a_r, f4), add_<T>(Pl, Mr));
            o.x = add_<T>(sub_<T>(Pl, Mr), bfx);
            o.y = add_<T>(add_<T>(sub_<T>(a_y, f4), add_<T>(Tl, Tr)), bfy);
            o.z = (T)0;
            if (bany || (GEN && ks_st)) {   // off the body kappa = 0: times 1, plus 0
                T den = add_<T>((T)1, kv.r);
                if (GEN) den = add_<T>(den, kst);
                const T inv = inv_<T>(den);
                o.x = mul_<T>(fma_<T>(kv.r, kv.x, o.x), inv);
                o.y = mul_<T>(fma_<T>(kv.r, kv.y, o.y), inv);
            }
            if (ocol) {
                stg4(ocl + y * n0, o);
                if (GEN) {
                    if (xnear || (!p1 && (y == 1 || y == n1 - 2))) write_bc2<T>(I, x, y, o, out);
                } else if (wf >= 0) {
                    stg4(ocl + y * n0 + (wf == 0 ? -1 : 1), face_value2<T>(I, wf, o));
                }
            }
        }
        a_r = add_<T>(b_2, f0);
        a_y = b_2;
        a_P = add_<T>(b_5, f1);
        a_Tp = b_5;
        a_M = add_<T>(b_6, f3);
        a_Tm = b_6;
        b_2 = f2;
        b_5 = f5;
        b_6 = f6;
    };
    for (int r = ya - 2; r < ya + kAhead; ++r) issue(r);
    // one copy of the body: with the two rows before the first output apart and the loop unrolled by
    // two, warps in three modes ran out of the instruction cache (64 channels of side 128 to 512:
    // gradient 59.4 ms so, 51.6 ms with one)
#pragma unroll 1
    for (int f = ya - 1; f <= yb + 1; ++f) march(f, f > ya);
    cp_wait<0>();
}

// The general path out of line, so that its registers do not weigh on the interior strips.
template <class T>
__device__ __noinline__ void step_strip_gen(const Inst<T>& I, const Strip& s, const V4<T>* src,
                                             V4<T>* out, const V4<T>* kus, V4<T>* ring) {
    step_strip<T, kGeneral>(I, s, src, out, kus, ring);
}

// Each warp's copy of the instance record it works on, staged when the warp moves to another
// instance: geometry then comes from shared memory, which the stores to global memory cannot
// alias.
template <class T>
__device__ __forceinline__ void stage_inst(const Plan& p, int i, int& cur, Inst<T>& sI, int lane) {
    if (i != cur) {
        __syncwarp();
        const int* src = reinterpret_cast<const int*>(table<T>(p) + i);
        int* dst = reinterpret_cast<int*>(&sI);
        for (int k = lane; k < (int)(sizeof(Inst<T>) / 4); k += 32) dst[k] = __ldg(src + k);
        __syncwarp();
        cur = i;
    }
}

// A warp's shared memory: its rings of rows (2 x kRing rows forward, 4 x kARing in the adjoint) and
// its instance record.
template <class T>
struct StripWarp {
    V4<T> ring[16 * 32];
    Inst<T> inst;
};

template <class T>
__global__ void __launch_bounds__(kStripThreads, strip_minb<T>())
    k_t_step(Plan p, int unit, int rows, StripRun r) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    StripWarp<T>& sw = reinterpret_cast<StripWarp<T>*>(smem_raw)[wid];
    Inst<T>& sI = sw.inst;
    V4<T>* ring = sw.ring + lane;
    const int* pre = p.pre + unit * (p.count + 1);
    const int total = p.total[unit], warps = gridDim.x * wpb;
    const int nb = __ldg(p.nbase);
    int cur = -1, su = -1;
    Strip s;
    for (int k = r.k0; k < r.k0 + r.n; ++k) {
        const int src = r.taped ? r.buf + k - 1 : BUF_S0 + ((r.buf + k - 1) & 1);
        const int dst = r.taped ? r.buf + k : BUF_S0 + ((r.buf + k) & 1);
        // the objective of the level this step reads; the last level of the launch has its own
        const int nobj = r.obj && k > r.k0 ? p.total[U_OBJ] : 0;
        for (int u = wid * gridDim.x + blockIdx.x; u < total + nobj; u += warps) {
            if (u >= total) {
                objective_unit<T>(p, u - total, nb + k - 1, src, lane);
                continue;
            }
            if (u != su) {   // a warp with one strip finds it once per launch
                const int i = find_inst(pre, p.count, u);
                stage_inst<T>(p, i, cur, sI, lane);
                s = strip_of<T>(sI, u - __ldg(pre + i), rows, lane);
                su = u;
            }
            const Inst<T>& I = sI;
            const V4<T>* kus = r.kslot == kBoxBuffer
                                   ? I.kus : I.kus_tape + (long long)(r.kslot + k) * I.g.boxN;
            if (s.mode == kInner) step_strip<T, kInner>(I, s, buf(I, src), buf(I, dst), kus, ring);
            else if (s.mode == kSide) step_strip<T, kSide>(I, s, buf(I, src), buf(I, dst), kus, ring);
            else step_strip_gen<T>(I, s, buf(I, src), buf(I, dst), kus, ring);
        }
        if (k + 1 < r.k0 + r.n && !grid_meet(p, gridDim.x, k - r.k0 + 1)) return;
    }
}

// ---------------------------------------------------------------- adjoint strips

template <class T>
__device__ __forceinline__ bool in_target2(const Geom& g, int x, int y) {
    if (x < g.obox[0] || x > g.obox[1] || y < g.obox[2] || y > g.obox[3]) return false;
    if (g.ocyl_r > 0.0) {   // the same FP64 test as the host's target list
        const double dx = x - g.ocyl_c[0], dy = y - g.ocyl_c[1];
        if (dx * dx + dy * dy > g.ocyl_r * g.ocyl_r) return false;
    }
    return true;
}

// The transpose of the boundary copies an interior node next to a face sources (Eqs. bc_rho,
// bc_u): the copied components of those boundary nodes, with their objective source.
template <class T>
__device__ __noinline__ V3<T> bcT_general(const Inst<T>& I, const V4<T>* lam, bool on, int x,
                                          int y, V3<T> v) {
    const Geom& g = I.g;
    for_each_sourced_boundary(g, x, y, 0, [&](int bx, int by, int, int f) {
        V4<T> lb = ldcg4(lam + node_index(g, bx, by, 0));
        if (on && in_target2<T>(g, bx, by)) {
            lb.r += I.src_r;
            lb.x += I.src_x;
            lb.y += I.src_y;
        }
        if (I.bckeep[f]) v.r += lb.r;
        else if (f < 2) v.x += lb.x;
        else v.y += lb.y;
    });
    return v;
}

// The same for a node next to at most one face per axis: its node on the x face, on the y face,
// and the corner of the two.
template <class T>
__device__ __forceinline__ V3<T> bcT_fold(const Inst<T>& I, const V4<T>* lam, bool on, int x,
                                          int y, V3<T> v) {
    const Geom& g = I.g;
    const int n0 = g.n[0], n1 = g.n[1];
    const bool xl = !g.periodic[0] && x == 1, xh = !g.periodic[0] && x == n0 - 2;
    const bool yl = !g.periodic[1] && y == 1, yh = !g.periodic[1] && y == n1 - 2;
    if ((xl && xh) || (yl && yh)) return bcT_general<T>(I, lam, on, x, y, v);
    const bool ex = xl || xh, ey = yl || yh;
    const int fx = xh ? 1 : 0, fy = yh ? 3 : 2;
    const int bx = xl ? 0 : n0 - 1, by = yl ? 0 : n1 - 1;
    auto fold = [&](bool go, int cx, int cy, int f) {
        if (!go) return;
        V4<T> lb = ldcg4(lam + (cy * n0 + cx));
        if (on && in_target2<T>(g, cx, cy)) {
            lb.r = add_<T>(lb.r, I.src_r);
            lb.x = add_<T>(lb.x, I.src_x);
            lb.y = add_<T>(lb.y, I.src_y);
        }
        if (I.bckeep[f]) v.r = add_<T>(v.r, lb.r);
        else if (f < 2) v.x = add_<T>(v.x, lb.x);
        else v.y = add_<T>(v.y, lb.y);
    };
    fold(ex, bx, y, fx);
    fold(ey, x, by, fy);
    fold(ex && ey, bx, by, I.corner[fx + 2 * (fy - 2)]);
    return v;
}

// One strip of the adjoint step.  Row m forms mu at the lane's nodes of row m + 1 and the moments
// of F~_i(y) = mu_rho(y + c_i) + c_i . mu_u(y + c_i) at row m, then lambda^{n-1} of row m - 1.
// Per node the directions are grouped by c_x again: the column to the right sends its axis value
// and, over rows m - 1 and m + 1, the sum and the difference of its two diagonal values, the
// column to the left the same.  EDGE as in the forward step.
// lambda, kappa and u_S, u^n (for e) and u^{n-1} pass through rings as in the forward step.
constexpr int kARing = 4, kAAhead = kARing - 1;

template <class T, int MODE>
__device__ __forceinline__ void adj_strip(const Inst<T>& I, const Strip& s, bool on,
                                          const V4<T>* lam, V4<T>* out, const V4<T>* __restrict__ sn,
                                          const V4<T>* __restrict__ sp,
                                          const V4<T>* __restrict__ kus, T* __restrict__ eo,
                                          V4<T>* ring) {
    using W = Wts<T, 2>;
    constexpr bool GEN = MODE == kGeneral, SIDE = MODE != kInner;
    const Geom& g = I.g;
    const int n0 = g.n[0], n1 = g.n[1];
    const bool p0 = GEN && g.periodic[0], p1 = GEN && g.periodic[1];
    const int ya = s.ya, yb = s.yb, x = s.x;
    if (ya > yb) return;   // uniform
    const bool own = s.own, xin = !SIDE || s.in;
    const bool icol = !SIDE || p0 || (x >= 1 && x <= n0 - 2);   // not on an x face, in the grid
    const bool xface = SIDE && !p0 && (!GEN || __any_sync(FULL, x == 0 || x == n0 - 1));
    const bool xnear = GEN && !p0 && __any_sync(FULL, x == 1 || x == n0 - 2);
    // kSide: the face whose column a node next to it collects
    const int wf = SIDE && !GEN ? (x == 1 ? 0 : (x == n0 - 2 ? 1 : -1)) : -1;
    const int bx = x - g.blo[0], bn0 = g.bn[0], bn1 = g.bn[1], by0 = g.blo[1];
    const bool bcol = g.boxN > 0 && xin && bx >= 0 && bx < bn0;
    // (a halo row of a wrapping strip may fall in the box from the other side)
    const bool bany = __any_sync(FULL, bcol) && (p1 || (ya - 2 < by0 + bn1 && yb + 2 >= by0));
    const int ty0 = g.obox[2], ty1 = g.obox[3];
    const bool tany = on && __any_sync(FULL, xin && x >= g.obox[0] && x <= g.obox[1]) &&
                      (p1 || (ya - 2 <= ty1 && yb + 2 >= ty0));
    const T* ks_st = GEN ? (const T*)g.ks : nullptr;
    const T A9 = I.A9;
    // coefficients of the face columns' 9 S~ in the x part of the transposed gradient: the
    // one-sided stencil less the central one, for columns 0, 1, 2 and n-1, n-2, n-3
    T cxl = (T)0, cxh = (T)0;
    int lane_l = 0, lane_h = 0;
    if (xface) {
        const int dl = x, dh = n0 - 1 - x;
        const unsigned ml = __ballot_sync(FULL, dl == 0), mh = __ballot_sync(FULL, dh == 0);
        lane_l = ml ? __ffs(ml) - 1 : 0;
        lane_h = mh ? __ffs(mh) - 1 : 0;
        if (ml) cxl = dl == 0 ? (T)-3 : (dl == 1 ? (T)3 : (dl == 2 ? (T)-1 : (T)0));
        if (mh) cxh = dh == 0 ? (T)3 : (dh == 1 ? (T)-3 : (dh == 2 ? (T)1 : (T)0));
    }
    // first and last moment row: the boundary rows' one-sided parts reach rows 2 and n - 3, also
    // where the strip starts or ends there
    const int ma = GEN && !p1 && ya == 2 ? 0 : ya - 1;
    const int mb = GEN && !p1 && yb == n1 - 3 ? n1 - 1 : yb + 1;
    V4<T>* ringk = ring + kARing * 32;
    V4<T>* ringn = ring + 2 * kARing * 32;
    V4<T>* ringp = ring + 3 * kARing * 32;
    const V4<T>* lcol = lam + (xin ? x : 0);
    const V4<T>* kcol = kus + (bcol ? bx : 0);
    const V4<T>* ncol = sn + (own ? x : 0);
    const V4<T>* pcol = sp + (own ? x : 0);
    V4<T>* ocl = out + (own ? x : 0);
    auto wrap = [&](int row) { return p1 ? row + (row < 0 ? n1 : (row >= n1 ? -n1 : 0)) : row; };
    struct Q {
        V3<T> l, k, u;   // lambda, (kappa, u_S), u^n of one row
    };
    auto direct = [&](int row0) -> Q {   // (u^n is for e on the strip's own rows, from the ring)
        Q q;
        q.l.r = q.l.x = q.l.y = q.k.r = q.k.x = q.k.y = q.u.r = q.u.x = q.u.y = (T)0;
        const int row = wrap(row0), kr = row - by0;
        if (xin && (!GEN || (row >= 0 && row < n1))) q.l = ldcg3<V3<T>>(lcol + row * n0);
        if (bany && bcol && (unsigned)kr < (unsigned)bn1) q.k = ldg3<V3<T>>(kcol + kr * bn0);
        return q;
    };
    // a row of lambda, kappa, u_S and u^n, and u^{n-1} two rows below it, as one copy group
    auto issue = [&](int row0) {
        const int slot = (row0 & (kARing - 1)) * 32;
        const int row = wrap(row0);
        const bool go = row0 <= mb + 1, in = xin && (!GEN || (row >= 0 && row < n1));
        cp_record<T>(ring + slot, lcol + (GEN && !in ? 0 : row * n0), go, in);
        if (bany) {
            const int kr = row - by0;
            const bool kin = bcol && (unsigned)kr < (unsigned)bn1;
            cp_record<T>(ringk + slot, kcol + (kin ? kr * bn0 : 0), go, kin);
            const bool nin = kin && own && row0 >= ya && row0 <= yb;
            cp_record<T>(ringn + slot, ncol + (nin ? row * n0 : 0), go, nin);
        }
        const int pr = row0 - 2;
        cp_record<T>(ringp + (pr & (kARing - 1)) * 32, pcol + (pr >= ya && pr <= yb ? pr * n0 : 0),
                     pr >= ya && pr <= yb, own);
        cp_commit();
    };
    // mu of a row from its loaded values: 0 on boundary nodes and outside the grid; the
    // transposed boundary copies, the objective source, the Brinkman transpose, and e on own nodes
    auto to_mu = [&](int row0, const Q& q) -> V3<T> {
        V3<T> v = q.l;
        const int row = wrap(row0);
        if (SIDE && !GEN) {   // the face column's lambda sits in the lane beside
            V3<T> b;
            const bool hi = wf == 1;
            const T br = from_left(v.r), bxv = from_left(v.x);
            const T cr = from_right(v.r), cx = from_right(v.x);
            b.r = hi ? cr : br;
            b.x = hi ? cx : bxv;
            if (wf >= 0) {
                if (on && in_target2<T>(g, hi ? n0 - 1 : 0, row)) {
                    b.r = add_<T>(b.r, I.src_r);
                    b.x = add_<T>(b.x, I.src_x);
                }
                if (I.bckeep[wf]) v.r = add_<T>(v.r, b.r);
                else v.x = add_<T>(v.x, b.x);
            }
        }
        if (SIDE && !(icol && (!GEN || p1 || (row >= 1 && row <= n1 - 2)))) {
            v.r = v.x = v.y = (T)0;
        } else {
            if (GEN && (xnear || (!p1 && (row == 1 || row == n1 - 2))))
                v = bcT_fold<T>(I, lam, on, x, row, v);
            if (tany && row >= ty0 && row <= ty1 && in_target2<T>(g, x, row)) {
                v.r = add_<T>(v.r, I.src_r);
                v.x = add_<T>(v.x, I.src_x);
                v.y = add_<T>(v.y, I.src_y);
            }
            if (bany || (GEN && ks_st)) {
                const T kst = GEN && ks_st ? ks_st[row * n0 + x] : (T)0;
                const int kr = row - by0;
                const bool box = bany && bcol && (unsigned)kr < (unsigned)bn1;
                if (box || (GEN && kst != (T)0)) {
                    T den = add_<T>((T)1, q.k.r);
                    if (GEN) den = add_<T>(den, kst);
                    const T inv = inv_<T>(den);
                    v.x = mul_<T>(v.x, inv);
                    v.y = mul_<T>(v.y, inv);
                    if (box && own && row0 >= ya && row0 <= yb)
                        eo[kr * bn0 + bx] = fma_<T>(v.x, sub_<T>(q.k.x, q.u.x),
                                                    mul_<T>(v.y, sub_<T>(q.k.y, q.u.y)));
                }
            }
        }
        return v;
    };
    // row m - 1 (its lower diagonal and axis values), row m (its axis values)
    T d_P, d_Q, d_y, c_r, c_a, c_b, c_P, c_Q, c_y;
    {
        const Q qa = direct(ma - 1), qb = direct(ma);
        for (int i = 1; i <= kARing; ++i) issue(ma + i);
        V3<T> a, b = qa.l;
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {   // one copy of to_mu
            a = b;
            b = to_mu(ma - 1 + i, i == 0 ? qa : qb);
        }
        d_P = sub_<T>(add_<T>(a.r, a.x), a.y);
        d_Q = sub_<T>(sub_<T>(a.r, a.x), a.y);
        d_y = sub_<T>(a.r, a.y);
        c_r = b.r;
        c_a = add_<T>(b.r, b.x);
        c_b = sub_<T>(b.r, b.x);
        c_P = sub_<T>(c_a, b.y);
        c_Q = sub_<T>(c_b, b.y);
        c_y = sub_<T>(b.r, b.y);
    }
    // moments of row m - 1, its x differences, 9 S~ of row m - 2 and of boundary row 0
    T R = (T)0, Ux = (T)0, Uy = (T)0, Sxx = (T)0, Sxy = (T)0, Syy = (T)0, gx = (T)0, gy = (T)0;
    T Sxy2 = (T)0, Syy2 = (T)0, S0xy = (T)0, S0yy = (T)0;
    V4<T> o;
    o.r = o.x = o.y = o.z = (T)0;
    auto march = [&](int m, bool emit) {   // emit: uniform, row m - 1 is an output row
        const int y = m - 1;   // output row
        cp_wait<kAAhead>();    // row m + 1 has landed
        Q q;
        {
            const int slot = ((m + 1) & (kARing - 1)) * 32;
            const V4<T> l = lds4(ring + slot);
            q.l = V3<T>{l.r, l.x, l.y};
            q.k.r = q.k.x = q.k.y = q.u.r = q.u.x = q.u.y = (T)0;
            if (bany) {
                const V4<T> k = lds4(ringk + slot), n = lds4(ringn + slot);
                q.k = V3<T>{k.r, k.x, k.y};
                q.u = V3<T>{n.r, n.x, n.y};
            }
        }
        V4<T> u;   // u^{n-1} of the output row
        u.r = u.x = u.y = u.z = (T)0;
        if (emit) u = lds4(ringp + (y & (kARing - 1)) * 32);
        issue(m + 1 + kARing);   // into the slots just read
        const V3<T> v = to_mu(m + 1, q);
        const T va = add_<T>(v.r, v.x), vb = sub_<T>(v.r, v.x);
        const T uP = add_<T>(va, v.y), uQ = add_<T>(vb, v.y), uy = add_<T>(v.r, v.y);
        // from the right (c_x = +1) and left (c_x = -1) columns
        const T Ap = from_right(c_a), Am = from_left(c_b);
        const T Dp = from_right(add_<T>(uP, d_P)), Ep = from_right(sub_<T>(uP, d_P));
        const T Dm = from_left(add_<T>(uQ, d_Q)), Em = from_left(sub_<T>(uQ, d_Q));
        const T ax = add_<T>(Ap, Am), ay = add_<T>(uy, d_y), ds = add_<T>(Dp, Dm);
        const T nR = fma_<T>(W::w2, ds, fma_<T>(W::w1, add_<T>(ax, ay), mul_<T>(W::w0, c_r)));
        const T nUx = fma_<T>(W::w3_1, sub_<T>(Ap, Am), mul_<T>(W::w3_2, sub_<T>(Dp, Dm)));
        const T nUy = fma_<T>(W::w3_1, sub_<T>(uy, d_y), mul_<T>(W::w3_2, add_<T>(Ep, Em)));
        T nSxx = fma_<T>(W::s_2, ds, ax), nSyy = fma_<T>(W::s_2, ds, ay);   // s_1 = 1
        T nSxy = mul_<T>(W::s_2, sub_<T>(Ep, Em));
        if (SIDE && (!xin || (GEN && !p1 && (m < 0 || m >= n1)))) nSxx = nSyy = nSxy = (T)0;
        T ngx = sub_<T>(from_left(nSxx), from_right(nSxx));
        T ngy = sub_<T>(from_left(nSxy), from_right(nSxy));
        if (xface) {
            const T lxx = __shfl_sync(FULL, nSxx, lane_l), lxy = __shfl_sync(FULL, nSxy, lane_l);
            const T hxx = __shfl_sync(FULL, nSxx, lane_h), hxy = __shfl_sync(FULL, nSxy, lane_h);
            ngx = fma_<T>(cxh, hxx, fma_<T>(cxl, lxx, ngx));
            ngy = fma_<T>(cxh, hxy, fma_<T>(cxl, lxy, ngy));
        }
        if (GEN && !p1) {
            if (m == 0) {
                S0xy = nSxy;
                S0yy = nSyy;
            }
            if (m == n1 - 1 && y - 1 >= ya && own) {
                // the high boundary row's one-sided part reaches row n - 3, written by the
                // previous iteration: add it now
                o.x = fma_<T>(A9, nSxy, o.x);
                o.y = fma_<T>(A9, nSyy, o.y);
                stg4(ocl + (y - 1) * n0, o);
            }
        }
        if (emit && (!GEN || y <= yb)) {   // uniform
            T tx = add_<T>(gx, sub_<T>(Sxy2, nSxy)), ty = add_<T>(gy, sub_<T>(Syy2, nSyy));
            if (GEN && !p1) {
                if (y <= 2) {
                    const T cy = y == 0 ? (T)-3 : (y == 1 ? (T)3 : (T)-1);
                    tx = fma_<T>(cy, S0xy, tx);
                    ty = fma_<T>(cy, S0yy, ty);
                }
                if (y == n1 - 1) {
                    tx = fma_<T>((T)3, Sxy, tx);
                    ty = fma_<T>((T)3, Syy, ty);
                } else if (y == n1 - 2) {
                    tx = fma_<T>((T)-3, nSxy, tx);
                    ty = fma_<T>((T)-3, nSyy, ty);
                }
            }
            const T R3 = mul_<T>((T)3, R);
            T lx = fma_<T>(-R3, u.x, Ux), ly = fma_<T>(-R3, u.y, Uy);
            lx = fma_<T>(Sxy, u.y, fma_<T>(Sxx, u.x, lx));
            ly = fma_<T>(Syy, u.y, fma_<T>(Sxy, u.x, ly));
            o.r = R;
            o.x = fma_<T>(A9, tx, lx);
            o.y = fma_<T>(A9, ty, ly);
            if (own) stg4(ocl + y * n0, o);
        }
        Sxy2 = Sxy;
        Syy2 = Syy;
        R = nR;
        Ux = nUx;
        Uy = nUy;
        Sxx = nSxx;
        Sxy = nSxy;
        Syy = nSyy;
        gx = ngx;
        gy = ngy;
        d_P = c_P;
        d_Q = c_Q;
        d_y = c_y;
        c_r = v.r;
        c_a = va;
        c_b = vb;
        c_P = sub_<T>(va, v.y);
        c_Q = sub_<T>(vb, v.y);
        c_y = sub_<T>(v.r, v.y);
    };
    // (two rows before the first output, three from boundary row 0; one copy of the body as above)
#pragma unroll 1
    for (int m = ma; m <= mb; ++m) march(m, m > ya);
    cp_wait<0>();
}

template <class T>
__device__ __noinline__ void adj_strip_gen(const Inst<T>& I, const Strip& s, bool on,
                                            const V4<T>* lam, V4<T>* out, const V4<T>* sn,
                                            const V4<T>* sp, const V4<T>* kus, T* eo,
                                            V4<T>* ring) {
    adj_strip<T, kGeneral>(I, s, on, lam, out, sn, sp, kus, eo, ring);
}

template <class T>
__global__ void __launch_bounds__(kStripThreads, strip_minb<T>())
    k_t_adj(Plan p, int unit, int rows, StripRun r) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    StripWarp<T>& sw = reinterpret_cast<StripWarp<T>*>(smem_raw)[wid];
    Inst<T>& sI = sw.inst;
    V4<T>* ring = sw.ring + lane;
    const int* pre = p.pre + unit * (p.count + 1);
    const int total = p.total[unit], warps = gridDim.x * wpb;
    const int nb = __ldg(p.nbase);
    int cur = -1, su = -1;
    Strip s;
    for (int j = 0; j < r.n; ++j) {
        const int k = r.k0 - j, par = (r.buf + j) & 1;
        for (int u = wid * gridDim.x + blockIdx.x; u < total; u += warps) {
            if (u != su) {   // a warp with one strip finds it once per launch
                const int i = find_inst(pre, p.count, u);
                stage_inst<T>(p, i, cur, sI, lane);
                s = strip_of<T>(sI, u - __ldg(pre + i), rows, lane);
                su = u;
            }
            const Inst<T>& I = sI;
            const long long bn = I.g.boxN;
            const V4<T>* kus =
                r.kslot == kBoxBuffer ? I.kus : I.kus_tape + (long long)(r.kslot + k) * bn;
            const bool on = nb + k >= I.win_begin && nb + k <= I.win_end;
            T* eo = I.e + (long long)(r.eslot + k) * bn;
            const V4<T>* lam = buf(I, BUF_LAM0 + par);
            V4<T>* lo = buf(I, BUF_LAM0 + 1 - par);
            const V4<T>*sn = buf(I, r.tape + k), *sp = buf(I, r.tape + k - 1);
            if (s.mode == kInner) adj_strip<T, kInner>(I, s, on, lam, lo, sn, sp, kus, eo, ring);
            else if (s.mode == kSide) adj_strip<T, kSide>(I, s, on, lam, lo, sn, sp, kus, eo, ring);
            else adj_strip_gen<T>(I, s, on, lam, lo, sn, sp, kus, eo, ring);
        }
        if (j + 1 < r.n && !grid_meet(p, gridDim.x, j + 1)) return;
    }
}

// ---------------------------------------------------------------- host side

int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

int cap_grid(long long units, int per_sm) {
    const long long g = (long long)sm_count() * std::max(per_sm, 1);
    return (int)std::max(1LL, std::min(units, g));
}

// The shared-memory limit of the strip kernels, raised once per device to what eight warps take: the
// limit belongs to the kernel, not to a context, so a launch must not set it to its own size while
// another thread's context is about to launch a larger one.
template <class T>
cudaError_t raise_strip_limits() {
    static std::atomic<unsigned> attr{0};
    if (device_done(attr)) return cudaSuccess;
    constexpr int most = (int)sizeof(StripWarp<T>) * (kStripThreads / 32);
    for (const void* kern : {(const void*)k_t_step<T>, (const void*)k_t_adj<T>}) {
        const cudaError_t e =
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return e;
    }
    device_mark(attr);
    return cudaSuccess;
}

// Blocks and warps per block of a strip kernel over `units` strips: the strips spread over all
// SMs, eight warps to a block at most; a launch of several steps keeps every block resident and
// loops over the rest.
template <class K>
cudaError_t launch_strips(K kern, size_t warp_bytes, long long units, bool meet, const Plan& p,
                          int unit, int rows, const StripRun& r, cudaStream_t st) {
    const int sms = sm_count();
    const int wpb = (int)std::min<long long>(kStripThreads / 32, (units + sms - 1) / sms);
    const int w = units <= kStripThreads / 32 ? (int)units : wpb;   // a few strips: one block
    const size_t smem = warp_bytes * w;
    long long grid = (units + w - 1) / w;
    if (meet && grid > sms) {
        int per = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, 32 * w, smem);
        if (e != cudaSuccess) return e;
        grid = std::min<long long>(grid, (long long)sms * std::max(per, 1));
    }
    if (!meet || grid == 1) {
        kern<<<(unsigned)grid, 32 * w, smem, st>>>(p, unit, rows, r);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(p.bar, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    Plan pp = p;
    int un = unit, ro = rows;
    StripRun rr = r;
    void* args[] = {&pp, &un, &ro, &rr};
    return cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)grid), dim3(32 * w), args,
                                       smem, st);
}

}  // namespace

int default_strips(const Plan& p, int type_size) {
    // the shortest strips that are all resident at once: a small grid's step is one march, whose
    // length is its latency (512^2: 2, 4, 8, 16, 32 rows took 29.6, 25.0, 27.8, 36.4, 54.1 ms over
    // 600 steps and their adjoint); but where taller ones fit one block, whose barrier is its own,
    // those
    const int per = kStripThreads / 32;
    const int room = sm_count() * per * (type_size == 4 ? strip_minb<float>() : strip_minb<double>());
    int k = 0;
    while (k + 1 < kStripCfgs && p.total[U_STRIP0 + k] > room) ++k;
    if (p.total[U_STRIP0 + k] > per && k + 1 < kStripCfgs && p.total[U_STRIP0 + k + 1] <= per) ++k;
    return k;
}

template <class T>
cudaError_t launch_t_transfer(const Plan& p, int noff, int n, int kslot0, cudaStream_t st) {
    if (p.total[U_DCOL] == 0 || p.total[U_BOX] == 0 || n <= 0) return cudaSuccess;
    k_t_design_pos<T><<<cap_grid((long long)p.total[U_DCOL] * n, 8), NT, 0, st>>>(p, noff, n);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    constexpr size_t smem = sizeof(TrSmem<T>);
    static std::atomic<unsigned> attr{0};
    if (!device_done(attr)) {
        e = cudaFuncSetAttribute(k_t_transfer2d<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem);
        if (e != cudaSuccess) return e;
        device_mark(attr);
    }
    const long long units = (long long)p.total[U_BOX] * n;
    k_t_transfer2d<T><<<cap_grid(units, sizeof(T) == 4 ? 8 : 4), kTrThreads, smem, st>>>(p, noff, n, kslot0);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_t_step(const Plan& p, int cfg, const StripRun& r, cudaStream_t st) {
    if (cfg < 0 || cfg >= kStripCfgs) return cudaErrorInvalidValue;
    const cudaError_t e = raise_strip_limits<T>();
    if (e != cudaSuccess) return e;
    const int unit = U_STRIP0 + cfg;
    return launch_strips(k_t_step<T>, sizeof(StripWarp<T>),
                         p.total[unit] + (r.obj && r.n > 1 ? p.total[U_OBJ] : 0), r.n > 1, p, unit,
                         strip_rows(cfg), r, st);
}

template <class T>
cudaError_t launch_t_adj(const Plan& p, int cfg, const StripRun& r, cudaStream_t st) {
    if (cfg < 0 || cfg >= kStripCfgs) return cudaErrorInvalidValue;
    const cudaError_t e = raise_strip_limits<T>();
    if (e != cudaSuccess) return e;
    const int unit = U_STRIP0 + cfg;
    return launch_strips(k_t_adj<T>, sizeof(StripWarp<T>), p.total[unit], r.n > 1, p, unit,
                         strip_rows(cfg), r, st);
}

template <class T>
cudaError_t launch_t_objective(const Plan& p, int noff, int src, cudaStream_t st) {
    const int per = NT / 32;
    k_t_objective<T><<<(p.total[U_OBJ] + per - 1) / per, NT, 0, st>>>(p, noff, src);
    return cudaGetLastError();
}

// Blocks per instance of the element-wise kernels.
inline int per_instance(const Plan& p) { return std::max(1, 8 * sm_count() / p.count); }

template <class T>
cudaError_t launch_t_begin(const Plan& p, bool adjoint, cudaStream_t st) {
    k_t_begin<T><<<dim3(adjoint ? per_instance(p) : 1, p.count), NT, 0, st>>>(p, adjoint);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_t_end(const Plan& p, int dst, int src, int n_last, bool adjoint, RunResult* out,
                         cudaStream_t st) {
    k_t_end<T><<<dim3(per_instance(p), p.count), NT, 0, st>>>(p, dst, src, !adjoint);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_t_result<T><<<p.count, NT, 0, st>>>(p, n_last, adjoint, out);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_t_sens(const Plan& p, int noff, int n, int eslot0, cudaStream_t st) {
    if (p.total[U_DCOL] == 0 || n <= 0) return cudaSuccess;
    const long long units = (long long)p.total[U_DCOL] * (kUnitThreads / kSensThreads);
    k_t_sens<T><<<cap_grid(units, 32), kSensThreads, 0, st>>>(p, noff, n, eslot0);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_t_copy(const Plan& p, int dst, int src, cudaStream_t st) {
    k_t_copy<T><<<dim3(per_instance(p), p.count), NT, 0, st>>>(p, dst, src);
    return cudaGetLastError();
}

cudaError_t launch_set_int(int* dst, int v, cudaStream_t st) {
    k_set_int<<<1, 1, 0, st>>>(dst, v);
    return cudaGetLastError();
}

#define LKS_INST_2D(T)                                                                      \
    template cudaError_t launch_t_transfer<T>(const Plan&, int, int, int, cudaStream_t);    \
    template cudaError_t launch_t_step<T>(const Plan&, int, const StripRun&, cudaStream_t); \
    template cudaError_t launch_t_adj<T>(const Plan&, int, const StripRun&, cudaStream_t);  \
    template cudaError_t launch_t_objective<T>(const Plan&, int, int, cudaStream_t);        \
    template cudaError_t launch_t_begin<T>(const Plan&, bool, cudaStream_t);                \
    template cudaError_t launch_t_end<T>(const Plan&, int, int, int, bool, RunResult*,      \
                                         cudaStream_t);                                     \
    template cudaError_t launch_t_sens<T>(const Plan&, int, int, int, cudaStream_t);        \
    template cudaError_t launch_t_copy<T>(const Plan&, int, int, cudaStream_t);

LKS_INST_2D(float)
LKS_INST_2D(double)

}  // namespace lks
