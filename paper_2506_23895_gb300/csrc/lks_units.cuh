// Per-unit device bodies shared by the single-context kernels and the instance-table kernels
// (one launch over many contexts), so both run exactly the same arithmetic per node, design
// column or boundary node.
#pragma once

#include "lks_device.cuh"

namespace lks {

__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

// ---------------------------------------------------------------- equilibrium (Sec. 2.2)
// The 15 values of f^eq at a node: rest and axes, and the corners [s_x > 0 ? 0 : 1] for s_y = +1 (u)
// and -1 (d), s_z = +1 (p) and -1 (m).
template <class T>
struct Feq {
    T f0, xp, xm, yp, ym, zp, zm;
    T up[2], um[2], dp[2], dm[2];
};

// f^eq (Sec. 2.2) from rho - rho0, u and D_ab = 2 d u_a / d x_b: the symmetric part of each pair of
// opposite directions is formed once, 68 operations in all.
template <class T>
__device__ __forceinline__ void feq(T r, T ux, T uy, T uz, T A, T Dxx, T Dyx, T Dzx, T Dxy, T Dyy,
                                    T Dzy, T Dxz, T Dyz, T Dzz, Feq<T>& f) {
    using W = Wts<T, 3>;
    const T hA = (T)0.5 * A;
    const T ASxx = A * Dxx, ASyy = A * Dyy, ASzz = A * Dzz;
    const T ASxy = hA * (Dxy + Dyx), ASxz = hA * (Dxz + Dzx), ASyz = hA * (Dyz + Dzy);
    const T P = r - (T)1.5 * (ux * ux + uy * uy + uz * uz);
    f.f0 = W::w0 * P;
    const T bx = fma_(W::h_1 * ux, ux, W::w1 * (P + ASxx));
    f.xp = fma_(W::w3_1, ux, bx);
    f.xm = fma_(-W::w3_1, ux, bx);
    const T by = fma_(W::h_1 * uy, uy, W::w1 * (P + ASyy));
    f.yp = fma_(W::w3_1, uy, by);
    f.ym = fma_(-W::w3_1, uy, by);
    const T bz = fma_(W::h_1 * uz, uz, W::w1 * (P + ASzz));
    f.zp = fma_(W::w3_1, uz, bz);
    f.zm = fma_(-W::w3_1, uz, bz);
    const T T0 = W::w2 * (P + ASxx + ASyy + ASzz);
    const T s1 = ux + uy, d1 = ux - uy, w2x2 = (T)2 * W::w2;
    const T q1 = ASxz + ASyz, q2 = ASyz - ASxz;
    {   // (+,+,+) and (-,-,-)
        const T cu = s1 + uz;
        const T s = fma_(W::h_2 * cu, cu, fma_(w2x2, ASxy + q1, T0));
        f.up[0] = fma_(W::w3_2, cu, s);
        f.dm[1] = fma_(-W::w3_2, cu, s);
    }
    {   // (-,+,+) and (+,-,-)
        const T cu = uz - d1;
        const T s = fma_(W::h_2 * cu, cu, fma_(w2x2, q2 - ASxy, T0));
        f.up[1] = fma_(W::w3_2, cu, s);
        f.dm[0] = fma_(-W::w3_2, cu, s);
    }
    {   // (+,-,+) and (-,+,-)
        const T cu = uz + d1;
        const T s = fma_(W::h_2 * cu, cu, fma_(-w2x2, ASxy + q2, T0));
        f.dp[0] = fma_(W::w3_2, cu, s);
        f.um[1] = fma_(-W::w3_2, cu, s);
    }
    {   // (-,-,+) and (+,+,-)
        const T cu = uz - s1;
        const T s = fma_(W::h_2 * cu, cu, fma_(w2x2, ASxy - q1, T0));
        f.dp[1] = fma_(W::w3_2, cu, s);
        f.um[0] = fma_(-W::w3_2, cu, s);
    }
}

// Second-order one-sided 2 d/dx at a low (hi = false) or high boundary node from it and its
// neighbours one and two nodes inward.
template <class T>
__device__ __forceinline__ T onesided(bool hi, T c, T n1, T n2) {
    const T d = fma_((T)-3, c, fma_((T)4, n1, -n2));
    return hi ? -d : d;
}

// ---------------------------------------------------------------- 2D transfer (table path)
// Design column k for the D2Q9 instance-table kernels: integer base of x_ref, y_ref and, per axis,
// S = sin(pi f/2), C = cos(pi f/2) of the fraction f.  The four
// taps of the cosine kernel then follow without further trigonometry: for an analysis node at
// base + q, q = -1, 0, 1, 2, w = (1 - S)/4, (1 + C)/4, (1 + S)/4, (1 - C)/4 (w(r) =
// (1 + cos(pi r/2))/4 at r = q - f).
// x_ref = x_G + a da - b db of one axis in single precision without losing the fraction:
// Dekker's exact product split (with fma) and Knuth's two-sum carry the rounding errors, so
// base + frac equals x_ref to about 1e-12 although every operation is FP32 (GB300's FP64 rate is
// a small fraction of its FP32 rate).  Returns the integer base; frac in [0, 1).
__device__ __forceinline__ int ref_coord(float ah, float al, float da, float bh, float bl,
                                         float db, int gi, float gh, float gl, float& frac) {
    const float p = ah * da, pe = fmaf(ah, da, -p);     // a_hi da = p + pe exactly
    const float q = bh * db, qe = fmaf(bh, db, -q);     // b_hi db = q + qe exactly
    const float r = p - q, rb = r - p;
    const float re = (p - (r - rb)) + (-q - rb);        // p - q = r + re exactly
    const float t = r + gh, tb = t - r;
    const float te = (r - (t - tb)) + (gh - tb);        // r + gh = t + te exactly
    const float lo = ((te + re) + (pe - qe)) + (fmaf(al, da, -bl * db) + gl);
    float fl = floorf(t);
    float f = (t - fl) + lo;                            // t - floor(t) is exact
    if (f < 0.f) {
        f += 1.f;
        fl -= 1.f;
    } else if (f >= 1.f) {
        f -= 1.f;
        fl += 1.f;
    }
    frac = f;
    return gi + (int)fl;
}

// sin and cos of pi f / 2.
template <class T>
__device__ __forceinline__ void sincospi_half(T f, T& s, T& c);
template <>
__device__ __forceinline__ void sincospi_half<float>(float f, float& s, float& c) {
    sincospif(0.5f * f, &s, &c);
}
template <>
__device__ __forceinline__ void sincospi_half<double>(double f, double& s, double& c) {
    sincospi(0.5 * f, &s, &c);
}

template <class T>
__device__ __forceinline__ void col_pos_sc(const Design& d, const Motion& m, long long k, int2& b,
                                           V4<T>& sc);

template <>
__device__ __forceinline__ void col_pos_sc<float>(const Design& d, const Motion& m, long long k,
                                                  int2& b, V4<float>& sc) {
    const int i = (int)((unsigned)k % (unsigned)d.L[0]), j = (int)((unsigned)k / (unsigned)d.L[0]);
    const float dx = (float)i - d.xiGf[0], dy = (float)j - d.xiGf[1];
    float fx, fy;   // Eq. rigid_body_position: x_ref = c dx - s dy + x_G, y_ref = s dx + c dy + y_G
    b.x = ref_coord(m.ch, m.cl, dx, m.sh, m.sl, dy, m.xgi[0], m.xgh[0], m.xgl[0], fx);
    b.y = ref_coord(m.sh, m.sl, dx, -m.ch, -m.cl, dy, m.xgi[1], m.xgh[1], m.xgl[1], fy);
    sincospi_half<float>(fx, sc.r, sc.x);
    sincospi_half<float>(fy, sc.y, sc.z);
}

template <>
__device__ __forceinline__ void col_pos_sc<double>(const Design& d, const Motion& m, long long k,
                                                   int2& b, V4<double>& sc) {
    const int i = (int)((unsigned)k % (unsigned)d.L[0]), j = (int)((unsigned)k / (unsigned)d.L[0]);
    const double dx = i - d.xiG[0], dy = j - d.xiG[1];
    const double xr = m.c * dx - m.s * dy + m.xG[0], yr = m.s * dx + m.c * dy + m.xG[1];
    const double bx = floor(xr), by = floor(yr);
    b = make_int2((int)bx, (int)by);
    sincospi_half<double>(xr - bx, sc.r, sc.x);
    sincospi_half<double>(yr - by, sc.y, sc.z);
}

// Weight of tap q1 - 1 = -1, 0, 1, 2 from S = sin(pi f/2), C = cos(pi f/2) of the fraction f.
template <class T>
__device__ __forceinline__ T tap_weight(int q1, T S, T C) {
    const T t = q1 == 0 ? -S : (q1 == 1 ? C : (q1 == 2 ? S : -C));
    return (T)0.25 * ((T)1 + t);
}

// ---------------------------------------------------------------- design positions (Sec. 2.3)
// x_ref, y_ref of design column k (FP64) as integer base, and sin, cos of (pi f / 2) of the fractions
// f in [0,1): every tap weight then takes one multiply-add, where evaluating the kernel takes a
// cosine at each (analysis column, design column) pair.
template <class T>
__device__ __forceinline__ void design_col_pos(const Design& d, const Motion& m,
                                               const TransferScratch& ts, long long k) {
    const int i = (int)((unsigned)k % (unsigned)d.L[0]), j = (int)((unsigned)k / (unsigned)d.L[0]);
    const double dx = i - d.xiG[0], dy = j - d.xiG[1];
    const double xr = m.c * dx - m.s * dy + m.xG[0];   // Eq. rigid_body_position
    const double yr = m.s * dx + m.c * dy + m.xG[1];
    const double bx = floor(xr), by = floor(yr);
    ts.col_base[2 * k] = (int)bx;
    ts.col_base[2 * k + 1] = (int)by;
    V4<T> sc;
    sincospi_half<T>((T)(xr - bx), sc.r, sc.x);
    sincospi_half<T>((T)(yr - by), sc.y, sc.z);
    ((V4<T>*)ts.col_sc)[k] = sc;
}

// sum of W e(x) over the 4 x 4 taps of design node k (the transpose of the kappa transfer) with
// the tap weights of the transfer, the node's position at the step formed here.
template <class T>
__device__ __forceinline__ T sens2d_sum(const Design& d, const Geom& g, const Motion& m,
                                        const T* __restrict__ e, long long k) {
    int2 b;
    V4<T> sc;
    col_pos_sc<T>(d, m, k, b, sc);
    const int ex0 = b.x - 1 - g.blo[0], ey0 = b.y - 1 - g.blo[1];
    T acc = (T)0;
#pragma unroll
    for (int ty = 0; ty < 4; ++ty) {
        const int ey = ey0 + ty;
        if (ey < 0 || ey >= g.bn[1]) continue;
        const T wy = tap_weight<T>(ty, sc.y, sc.z);
#pragma unroll
        for (int tx = 0; tx < 4; ++tx) {
            const int ex = ex0 + tx;
            if (ex < 0 || ex >= g.bn[0]) continue;
            acc += (tap_weight<T>(tx, sc.r, sc.x) * wy) * e[(long long)ey * g.bn[0] + ex];
        }
    }
    return acc;
}

// ---------------------------------------------------------------- sensitivity gather (Sec. 2.4)
// For design column k and kSensRun planes from z0: sum_x W(x - x_ref) e(x) over the support (the
// transpose of the kappa transfer), times kappa', added to dJ/dgamma in FP64.  The z shift is
// the same for every design plane, so each analysis plane's 4 x 4 x-y tap sum is formed once
// and the four z weights slide over them.
constexpr int kSensRun = 4;

template <class T>
__device__ __forceinline__ void sens_run(const Design& d, const Geom& g, const TransferScratch& ts,
                                         const T* __restrict__ e, const T* __restrict__ kprime,
                                         double* __restrict__ gacc, long long t) {
    const unsigned k = (unsigned)t % (unsigned)d.ncol;   // design column
    const int z0 = (int)((unsigned)t / (unsigned)d.ncol) * kSensRun;
    const int z1 = min(d.L[2], z0 + kSensRun);
    const int bx = ts.col_base[2 * k], by = ts.col_base[2 * k + 1];
    const V4<T> sc = ((const V4<T>*)ts.col_sc)[k];
    const T zs = ((const T*)ts.dz_sc)[0], zc = ((const T*)ts.dz_sc)[1];
    T wx[4], wy[4], wz[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        wx[q] = tap_weight<T>(q, sc.r, sc.x);
        wy[q] = tap_weight<T>(q, sc.y, sc.z);
        wz[q] = (g.dim == 3) ? tap_weight<T>(q, zs, zc) : (q == 1 ? (T)1 : (T)0);
    }
    const int ex0 = bx - 1 - g.blo[0], ey0 = by - 1 - g.blo[1];
    // x-y tap sum of analysis plane z (0 outside the box, where W vanishes)
    auto plane_sum = [&](int z) -> T {
        const int ez = z - g.blo[2];
        if (ez < 0 || ez >= g.bn[2]) return (T)0;
        const T* ep = e + (long long)ez * g.bn[1] * g.bn[0];
        T acc = (T)0;
#pragma unroll
        for (int ty = 0; ty < 4; ++ty) {
            const int ey = ey0 + ty;
            if (ey < 0 || ey >= g.bn[1] || wy[ty] == (T)0) continue;
#pragma unroll
            for (int tx = 0; tx < 4; ++tx) {
                const int ex = ex0 + tx;
                const T W = wx[tx] * wy[ty];
                if (ex < 0 || ex >= g.bn[0] || W == (T)0) continue;
                acc += W * ep[(long long)ey * g.bn[0] + ex];
            }
        }
        return acc;
    };
    const int zb0 = (g.dim == 3) ? ts.dz_base[z0] : 0;   // analysis base plane of design plane z0
    T s0 = plane_sum(zb0 - 1), s1 = plane_sum(zb0), s2 = plane_sum(zb0 + 1);
    for (int zeta = z0; zeta < z1; ++zeta) {
        const int zb = zb0 + (zeta - z0);
        const T s3 = (g.dim == 3) ? plane_sum(zb + 2) : (T)0;
        const T acc = wz[0] * s0 + wz[1] * s1 + wz[2] * s2 + wz[3] * s3;
        const long long dn = (long long)zeta * d.ncol + k;
        gacc[dn] += (double)kprime[dn] * (double)acc;
        s0 = s1;
        s1 = s2;
        s2 = s3;
    }
}

// ---------------------------------------------------------------- objective (Sec. 2.5)
// j = -(rho0 + mean(rho - rho0))/3 (J1) or -mean(n.u) (J2) over the target list, one block of
// kObjThreads threads, fixed-order FP64 reduction.
constexpr int kObjThreads = 256;

template <class T>
__device__ __forceinline__ void objective_block(const Geom& g, const V4<T>* __restrict__ s,
                                                double* jstep) {
    __shared__ double red[kObjThreads];
    const int tot = (int)g.ocount;
    double acc = 0.0;
    for (int k = threadIdx.x; k < tot; k += kObjThreads) {
        const V4<T> v = s[g.otarget[k]];
        if (g.okind == 0)
            acc += (double)v.r;
        else
            acc += g.odir[0] * (double)v.x + g.odir[1] * (double)v.y + g.odir[2] * (double)v.z;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = kObjThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double sum = red[0];
        jstep[0] = (g.okind == 0) ? -(g.rho0 + sum / g.ocount) / 3.0 : -sum / g.ocount;
    }
    __syncthreads();
}

// Objective's direct adjoint source at one node (h = window weight or 0 outside the window).
// Objective source h_n dj/ds at a target node (Sec. 2.5) in the precision T of the state, formed
// on the host in FP64 and rounded once: the device never divides in FP64.
template <class T>
struct ObjAdd {
    T r, x, y, z;
    int on;   // h_n != 0
};
template <class T>
inline ObjAdd<T> obj_add(const Geom& g, double h) {
    ObjAdd<T> o;
    o.on = h != 0.0;
    o.r = o.x = o.y = o.z = (T)0;
    if (h == 0.0) return o;
    if (g.okind == 0) {
        o.r = (T)(-h / (3.0 * g.ocount));
    } else {
        o.x = (T)(-h * g.odir[0] / g.ocount);
        o.y = (T)(-h * g.odir[1] / g.ocount);
        o.z = (T)(-h * g.odir[2] / g.ocount);
    }
    return o;
}

template <class T>
__device__ __forceinline__ void obj_source(const Geom& g, int x, int y, int z, const ObjAdd<T>& o,
                                           V4<T>& l) {
    if (!o.on || !in_target(g, x, y, z)) return;
    if (g.okind == 0) {
        l.r += o.r;
    } else {
        l.x += o.x;
        l.y += o.y;
        l.z += o.z;
    }
}

// ---------------------------------------------------------------- boundary transpose
// Transpose of the boundary copies at interior node (x, y, z): it collects the copied
// components of the boundary nodes it sources (WALL/INLET copy rho, OUTLET copies the normal
// velocity), after their objective source.  Boundary nodes are read only; later kernels treat
// them as zero.
// bcT_gather adds those components to acc (the node's own value); bcT_node stores the sum.
template <class T>
__device__ __forceinline__ void bcT_gather(const Geom& g, const V4<T>* lam, const ObjAdd<T>& h,
                                           int x, int y, int z, V4<T>& acc) {
    for_each_sourced_boundary(g, x, y, z, [&](int bx, int by, int bz, int f) {
        V4<T> lb = lam[node_index(g, bx, by, bz)];
        obj_source(g, bx, by, bz, h, lb);
        const int t = g.bc[f];
        if (t == BC_WALL || t == BC_INLET) {
            acc.r += lb.r;
        } else {
            const int na = f / 2;
            if (na == 0) acc.x += lb.x;
            if (na == 1) acc.y += lb.y;
            if (na == 2) acc.z += lb.z;
        }
    });
}

template <class T>
__device__ __forceinline__ void bcT_node(const Geom& g, V4<T>* lam, const ObjAdd<T>& h, int x,
                                         int y, int z) {
    if (!sources_boundary(g, x, y, z)) return;
    const long long m = node_index(g, x, y, z);
    V4<T> acc = lam[m];
    bcT_gather<T>(g, lam, h, x, y, z, acc);
    lam[m] = acc;
}

// Shell enumeration: slab s (0..5) is the interior layer next to face s (axis s/2, low or
// high side); a node next to several faces is handled by the first slab that contains it.
__device__ __forceinline__ bool shell_node(const Geom& g, long long t, int& x, int& y, int& z) {
    const unsigned per0 = (unsigned)g.n[1] * g.n[2], per1 = (unsigned)g.n[0] * g.n[2],
                   per2 = (unsigned)g.n[0] * g.n[1];
    unsigned r = (unsigned)t;
    int slab = 0;
    while (slab < 6) {
        const unsigned pa = slab < 2 ? per0 : (slab < 4 ? per1 : per2);
        if (r < pa) break;
        r -= pa;
        ++slab;
    }
    t = r;
    if (slab >= 6) return false;
    const int a = slab / 2;
    if (a >= g.dim || g.periodic[a]) return false;
    const int fixed = (slab & 1) ? g.n[a] - 2 : 1;
    int c[3];
    const int b0 = (a == 0) ? 1 : 0, b1 = (a == 2) ? 1 : 2;
    c[a] = fixed;
    c[b0] = (int)((unsigned)t % (unsigned)g.n[b0]);
    c[b1] = (int)((unsigned)t / (unsigned)g.n[b0]);
    // owned by an earlier slab?
    for (int e = 0; e < slab; ++e) {
        const int ae = e / 2;
        if (ae >= g.dim || g.periodic[ae]) continue;
        if (c[ae] == ((e & 1) ? g.n[ae] - 2 : 1)) return false;
    }
    x = c[0];
    y = c[1];
    z = c[2];
    return !is_boundary(g, x, y, z);
}


}  // namespace lks
