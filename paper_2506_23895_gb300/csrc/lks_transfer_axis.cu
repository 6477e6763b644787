// Transfer and sensitivity gather for a design grid rotating about a general 3D axis (Sec. 2.3,
// Eqs. brinkman_ref, velocity_ref with R(theta) from Rodrigues' formula).  The kernel weight
// no longer separates into a column part and a z part, so the gather goes through cell lists:
//   k_ga_bin   x_ref of every design node (FP64) as integer base and fraction; the sine and cosine
//              of each fraction, from which all its tap weights follow, and its place in the list
//              of the footprint-box cell that holds it (at most 8: the preimage of a unit cell is a
//              unit cube, which holds at most 8 points at mutual distance >= 1);
//   k_ga_fill  kappa = sum W kappa_ref and u_S = omega a x (R m1) + u_G m0 on every box node,
//              gathered from the cells based in [x - 2, x + 1]^3 whose taps cover it, in design
//              index order within a cell;
//   k_ga_sens  per design node, sum of W e(x) over its 4^3 taps, times kappa' (FP64).
// The list order within a cell is not fixed, the order it is read in is: deterministic results.
#include <algorithm>

#include "lks_units.cuh"

namespace lks {

namespace {

constexpr int kThreads = 256;
inline unsigned grid_for(long long n, int t = kThreads) { return (unsigned)((n + t - 1) / t); }

// Per design node: rec[0] = sin, cos of (pi f / 2) for x and y, rec[1] = those of z and kappa_ref,
// rec[2] = xi - xi_G.  Weights from these take one multiply-add a tap; evaluating the cosine
// kernel at every (box node, design node) pair cost three cosines a pair, 64 pairs a node.
template <class T>
__global__ void __launch_bounds__(kThreads)
    k_ga_bin(Design d, Geom g, Motion m, const T* __restrict__ kref, int4* __restrict__ base,
             V4<T>* __restrict__ rec, int* __restrict__ cnt, int* __restrict__ idx) {
    const unsigned k = blockIdx.x * kThreads + threadIdx.x;   // design nodes fit 32 bits
    if (k >= (unsigned)d.nd) return;
    const unsigned r = k / (unsigned)d.L[0];
    const int i = (int)(k - r * (unsigned)d.L[0]);
    const int l = (int)(r / (unsigned)d.L[1]), j = (int)(r - (unsigned)l * (unsigned)d.L[1]);
    const double dv[3] = {i - d.xiG[0], j - d.xiG[1], l - d.xiG[2]};
    int b[3];
    T S[3], C[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double xr = m.R[3 * a] * dv[0] + m.R[3 * a + 1] * dv[1] + m.R[3 * a + 2] * dv[2] +
                          m.xG[a];   // Eq. rigid_body_position
        const double fl = floor(xr);
        b[a] = (int)fl;
        sincospi_half<T>((T)(xr - fl), S[a], C[a]);
    }
    base[k] = make_int4(b[0], b[1], b[2], 0);
    V4<T>* o = rec + 3 * (size_t)k;
    o[0] = V4<T>{S[0], C[0], S[1], C[1]};
    o[1] = V4<T>{S[2], C[2], kref[k], (T)0};
    o[2] = V4<T>{(T)dv[0], (T)dv[1], (T)dv[2], (T)0};
    long long c;
    if (in_box(g, b[0], b[1], b[2], c)) {
        const int slot = atomicAdd(cnt + c, 1);
        if (slot < kCellMax) idx[c * kCellMax + slot] = (int)k;
    }
}

// One 8 x 8 x 8 tile of the footprint box per block.  The design nodes in the 11^3 cells whose taps
// reach the tile go to shared memory, ordered by cell (x fastest) and then by design index; each
// thread gathers a run of kGaRun nodes of one column, so that a design node serves up to four of
// them, and the four cells of a row of its support are one range of the staged list.  Tiles farther
// from the design box than the kernel reaches (most of a box that holds the turning body at every
// angle) are zero without a look at the cells.  Bound by the latency of the staging and the serial
// sums of the few hundred tiles that hold design nodes.  36^3 design, 62^3 box, FP32: one thread per
// box node reading the lists of 64 cells from global memory, with three cosines a pair, took 340 us;
// a thread per run of four with the trigonometry tabled 100 us; staged 40 us.
constexpr int kGaTile = 8, kGaRun = 4, kGaCells = kGaTile + 3;
constexpr int kGaThreads = kGaTile * kGaTile * kGaTile / kGaRun;
constexpr int kGaCell3 = kGaCells * kGaCells * kGaCells;
constexpr int kGaPer = (kGaCell3 + kGaThreads - 1) / kGaThreads;   // cells a thread lists
// a unit lattice puts about one node in a cell (1331), a few more at the rims of a small design
constexpr int kGaList = 1536;

template <class T>
struct GaSmem {
    V4<T> a[kGaList], b[kGaList], c[kGaList];   // rec, with the cell's x in b.z
    int k[kGaList];
    unsigned short start[kGaCell3 + 1];
    int warp[kGaThreads / 32];
};

// kappa, m0, m1 of a node.
template <class T>
struct GaSum {
    T kap, m0, x, y, z;
};

// Adds design node (A, B, D) to a run whose first node is dz cells above its cell.
template <class T>
__device__ __forceinline__ void ga_add(GaSum<T> (&s)[kGaRun], int dz, int qx, int qy, const V4<T>& A,
                                       const V4<T>& B, const V4<T>& D) {
    const T wxy = tap_weight<T>(qx, A.r, A.x) * tap_weight<T>(qy, A.y, A.z);
#pragma unroll
    for (int j = 0; j < kGaRun; ++j) {
        const int qz = j + 1 - dz;   // static where dz is
        if (qz < 0 || qz > 3) continue;
        const T W = wxy * tap_weight<T>(qz, B.r, B.x);
        s[j].kap += W * B.y;
        s[j].m0 += W;
        s[j].x += W * D.r;
        s[j].y += W * D.x;
        s[j].z += W * D.y;
    }
}

// The next node of a cell's list in design index order, after `last`.
__device__ __forceinline__ int next_in_cell(const int* __restrict__ list, int nc, int last) {
    int k = 0x7fffffff;
    for (int f = 0; f < nc; ++f) {
        const int kf = __ldg(list + f);
        if (kf > last && kf < k) k = kf;
    }
    return k;
}

template <class T>
__global__ void __launch_bounds__(kGaThreads, 2)
    k_ga_fill(Design d, Geom g, Motion m, const int* __restrict__ cnt, const int* __restrict__ idx,
              const V4<T>* __restrict__ rec, V4<T>* __restrict__ kus) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    GaSmem<T>& S = *reinterpret_cast<GaSmem<T>*>(smem_raw);
    const int plane = g.bn[0] * g.bn[1];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int lx = tid % kGaTile, ly = tid / kGaTile % kGaTile, lz = tid / (kGaTile * kGaTile) * kGaRun;
    const int nxt = (g.bn[0] + kGaTile - 1) / kGaTile, nzt = (g.bn[2] + kGaTile - 1) / kGaTile;
    for (int tz = blockIdx.y; tz < nzt; tz += gridDim.y) {
        const int bx0 = (int)blockIdx.x % nxt * kGaTile, by0 = (int)blockIdx.x / nxt * kGaTile;
        const int bz0 = tz * kGaTile;
        // the tile's middle in design coordinates, against the design box widened by the reach of
        // the kernel (2 sqrt 3), half the tile's diagonal and a margin for single precision
        const float half = 0.5f * (kGaTile - 1);
        const float p[3] = {(float)((double)(g.blo[0] + bx0) - m.xG[0]) + half,
                            (float)((double)(g.blo[1] + by0) - m.xG[1]) + half,
                            (float)((double)(g.blo[2] + bz0) - m.xG[2]) + half};
        bool near = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float xi = (float)m.R[a] * p[0] + (float)m.R[3 + a] * p[1] +
                             (float)m.R[6 + a] * p[2] + (float)d.xiG[a];
            const float reach = 1.7321f * (2.f + half) + 0.05f;
            near = near && xi >= -reach && xi <= (float)(d.L[a] - 1) + reach;
        }
        GaSum<T> s[kGaRun];
#pragma unroll
        for (int j = 0; j < kGaRun; ++j) s[j].kap = s[j].m0 = s[j].x = s[j].y = s[j].z = (T)0;
        if (near) {   // uniform over the block
            const int cx0 = bx0 - 2, cy0 = by0 - 2, cz0 = bz0 - 2;   // first cell
            auto cell = [&](int c) -> int {   // box index of tile cell c, -1 outside the box
                const int z = c / (kGaCells * kGaCells), r = c - z * kGaCells * kGaCells;
                const int y = r / kGaCells, x = r - y * kGaCells;
                const int ex = cx0 + x, ey = cy0 + y, ez = cz0 + z;
                return c < kGaCell3 && (unsigned)ex < (unsigned)g.bn[0] &&
                               (unsigned)ey < (unsigned)g.bn[1] && (unsigned)ez < (unsigned)g.bn[2]
                           ? ez * plane + ey * g.bn[0] + ex
                           : -1;
            };
            // list offsets: counts of kGaPer consecutive cells per thread, summed over the block
            // (the first two nodes of every list come along: few cells hold more, and a load
            // that waits for a count would make the staging a chain)
            int nc[kGaPer], sum = 0;
            int2 k01[kGaPer];
#pragma unroll
            for (int i = 0; i < kGaPer; ++i) {
                const int c = cell(tid * kGaPer + i);
                nc[i] = c >= 0 ? __ldg(cnt + c) : 0;
                k01[i] = __ldg(reinterpret_cast<const int2*>(idx + (size_t)max(c, 0) * kCellMax));
            }
#pragma unroll
            for (int i = 0; i < kGaPer; ++i) {
                nc[i] = min(nc[i], kCellMax);
                sum += nc[i];
            }
            int pre = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, pre, o);
                if (lane >= o) pre += v;
            }
            __syncthreads();   // the previous tile's lists are no longer read
            if (lane == 31) S.warp[wid] = pre;
            __syncthreads();
            int total = 0;
#pragma unroll
            for (int w = 0; w < kGaThreads / 32; ++w) {
                if (w < wid) pre += S.warp[w];
                total += S.warp[w];
            }
            pre -= sum;
            const bool fits = total <= kGaList;
            if (fits) {
#pragma unroll
                for (int i = 0; i < kGaPer; ++i) {
                    const int c = tid * kGaPer + i;
                    const T cx = (T)(c % kGaCells);
                    if (c < kGaCell3) S.start[c] = (unsigned short)pre;
                    if (nc[i] > 2) {
                        const int* list = idx + (size_t)cell(c) * kCellMax;
                        int last = -1;
                        for (int e = 0; e < nc[i]; ++e) {
                            last = next_in_cell(list, nc[i], last);
                            S.k[pre + e] = last;
                            S.b[pre + e].z = cx;
                        }
                    } else {
                        const bool two = nc[i] == 2;
                        if (nc[i] > 0) {
                            S.k[pre] = two ? min(k01[i].x, k01[i].y) : k01[i].x;
                            S.b[pre].z = cx;
                        }
                        if (two) {
                            S.k[pre + 1] = max(k01[i].x, k01[i].y);
                            S.b[pre + 1].z = cx;
                        }
                    }
                    pre += nc[i];
                }
                if (tid == 0) S.start[kGaCell3] = (unsigned short)total;
                __syncthreads();
                for (int e = tid; e < total; e += kGaThreads) {
                    const V4<T>* r = rec + 3 * (size_t)S.k[e];
                    const V4<T> A = r[0], B = r[1], D = r[2];
                    S.a[e] = A;
                    S.b[e].r = B.r;
                    S.b[e].x = B.x;
                    S.b[e].y = B.y;
                    S.c[e] = D;
                }
                __syncthreads();
#pragma unroll
                for (int dz = -2; dz <= kGaRun; ++dz)
#pragma unroll 1
                    for (int qy = 3; qy >= 0; --qy) {   // cell rows from y - 2 to y + 1
                        const int c0 = ((lz + dz + 2) * kGaCells + (ly + 3 - qy)) * kGaCells + lx;
                        const int e1 = S.start[c0 + 4];
                        for (int e = S.start[c0]; e < e1; ++e) {
                            const V4<T> A = S.a[e], B = S.b[e], D = S.c[e];
                            ga_add<T>(s, dz, lx + 3 - (int)B.z, qy, A, B, D);
                        }
                    }
            } else {   // more design nodes than the list holds: the lists in global memory
#pragma unroll
                for (int dz = -2; dz <= kGaRun; ++dz)
#pragma unroll 1
                    for (int qy = 3; qy >= 0; --qy)
#pragma unroll 1
                        for (int qx = 3; qx >= 0; --qx) {
                            const int c = cell(((lz + dz + 2) * kGaCells + (ly + 3 - qy)) * kGaCells +
                                               lx + 3 - qx);
                            const int n = c >= 0 ? min(__ldg(cnt + c), kCellMax) : 0;
                            int last = -1;
                            for (int e = 0; e < n; ++e) {
                                last = next_in_cell(idx + (size_t)c * kCellMax, n, last);
                                const V4<T>* r = rec + 3 * (size_t)last;
                                ga_add<T>(s, dz, qx, qy, r[0], r[1], r[2]);
                            }
                        }
            }
        }
        // u_S = omega a x (R m1) + u_G m0 (u_ref is affine in xi, Eq. rigid_body_velocity)
        const int bx = bx0 + lx, by = by0 + ly;
        if (bx >= g.bn[0] || by >= g.bn[1]) continue;
        const T ax = (T)m.ax[0], ay = (T)m.ax[1], az = (T)m.ax[2], om = (T)m.om;
#pragma unroll
        for (int j = 0; j < kGaRun; ++j) {
            const int bz = bz0 + lz + j;
            if (bz >= g.bn[2]) break;
            V4<T> o;
            o.r = s[j].kap;
            o.x = o.y = o.z = (T)0;
            if (near) {
                T rm[3];
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    rm[a] = (T)m.R[3 * a] * s[j].x + (T)m.R[3 * a + 1] * s[j].y +
                            (T)m.R[3 * a + 2] * s[j].z;
                o.x = om * (ay * rm[2] - az * rm[1]) + (T)m.uG[0] * s[j].m0;
                o.y = om * (az * rm[0] - ax * rm[2]) + (T)m.uG[1] * s[j].m0;
                o.z = om * (ax * rm[1] - ay * rm[0]) + (T)m.uG[2] * s[j].m0;
            }
            kus[(long long)bz * plane + (by * g.bn[0] + bx)] = o;
        }
    }
}

// Four threads per design node, one per tap plane: a design has too few nodes to fill the GPU with
// one thread each.
template <class T>
__global__ void __launch_bounds__(kThreads)
    k_ga_sens(Design d, Geom g, const int4* __restrict__ base, const V4<T>* __restrict__ rec,
              const T* __restrict__ e, const T* __restrict__ kprime, double* __restrict__ gacc) {
    const long long t = blockIdx.x * (long long)kThreads + threadIdx.x;
    const long long k = min(t >> 2, d.nd - 1);   // (lanes past the end repeat the last node)
    const int tz = (int)(t & 3);
    const int4 b = base[k];
    const V4<T> A = rec[3 * k], B = rec[3 * k + 1];
    T acc = (T)0;
    const int ez = b.z - 1 + tz - g.blo[2];
    if (ez >= 0 && ez < g.bn[2]) {
        const T* ep = e + (long long)ez * g.bn[1] * g.bn[0];
#pragma unroll
        for (int ty = 0; ty < 4; ++ty) {
            const int ey = b.y - 1 + ty - g.blo[1];
            if (ey < 0 || ey >= g.bn[1]) continue;
            const T wy = tap_weight<T>(ty, A.y, A.z);
#pragma unroll
            for (int tx = 0; tx < 4; ++tx) {
                const int ex = b.x - 1 + tx - g.blo[0];
                if (ex < 0 || ex >= g.bn[0]) continue;
                acc += (tap_weight<T>(tx, A.r, A.x) * wy) * ep[ey * g.bn[0] + ex];
            }
        }
        acc *= tap_weight<T>(tz, B.r, B.x);
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    if (tz == 0 && (t >> 2) < d.nd) gacc[k] += (double)kprime[k] * (double)acc;
}

}  // namespace

template <class T>
void launch_transfer_axis(const Design& d, const Geom& g, const Motion& m, AxisScratch as,
                          const T* kref, V4<T>* kus, cudaStream_t st) {
    if (d.nd == 0 || g.boxN == 0) return;
    cudaMemsetAsync(as.cnt, 0, (size_t)g.boxN * sizeof(int), st);
    k_ga_bin<T><<<grid_for(d.nd), kThreads, 0, st>>>(d, g, m, kref, as.base, (V4<T>*)as.rec,
                                                     as.cnt, as.idx);
    const int nt[3] = {(g.bn[0] + kGaTile - 1) / kGaTile, (g.bn[1] + kGaTile - 1) / kGaTile,
                       (g.bn[2] + kGaTile - 1) / kGaTile};
    static std::atomic<unsigned> attr{0};   // devices whose shared-memory limit is raised
    if (!device_done(attr)) {
        cudaFuncSetAttribute(k_ga_fill<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(GaSmem<T>));
        device_mark(attr);
    }
    k_ga_fill<T><<<dim3(nt[0] * nt[1], std::min(nt[2], 65535)), kGaThreads, sizeof(GaSmem<T>), st>>>(d, g, m, as.cnt, as.idx, (const V4<T>*)as.rec, kus);
}

template <class T>
void launch_sens_axis(const Design& d, const Geom& g, AxisScratch as, const T* e,
                      const T* kprime, double* gacc, cudaStream_t st) {
    if (d.nd == 0 || g.boxN == 0) return;
    k_ga_sens<T><<<grid_for(4 * d.nd), kThreads, 0, st>>>(d, g, as.base, (const V4<T>*)as.rec, e,
                                                          kprime, gacc);
}

template void launch_transfer_axis<float>(const Design&, const Geom&, const Motion&, AxisScratch,
                                          const float*, V4<float>*, cudaStream_t);
template void launch_transfer_axis<double>(const Design&, const Geom&, const Motion&,
                                           AxisScratch, const double*, V4<double>*, cudaStream_t);
template void launch_sens_axis<float>(const Design&, const Geom&, AxisScratch, const float*,
                                      const float*, double*, cudaStream_t);
template void launch_sens_axis<double>(const Design&, const Geom&, AxisScratch, const double*,
                                       const double*, double*, cudaStream_t);

}  // namespace lks
