// What the fused D3Q15 adjoint step does beside its z-march (lks_march3d_adj.cu) on non-periodic grids:
//   k_adj_prep   (lks_plain.cu) before it, in place on lambda^n: the transpose of the boundary
//                copies, the objective source and, in the footprint box, the Brinkman transpose with e;
//   k_adj_bcorr  after it: the one-sided rows of the transposed velocity gradient.
#include <algorithm>

#include "lks_march3d.h"
#include "lks_units.cuh"

namespace lks {

namespace {

// One-sided parts of the transposed gradient on non-periodic axes: node z within two rows of
// a face gets delta * (2 A S~_{.beta}) of the face node it projects to, with delta = -3/2,
// +3/2, -1/2 at rows 0, 1, 2 (low face) and +3/2, -3/2, +1/2 at rows n-1, n-2, n-3 (high face):
// the exact one-sided stencil minus the central one the fused kernel applied.  Where the march took
// an x face's own value for the one beyond it (its lane 0 or 31), 1/2 of it comes out too: x_lo and x_hi are
// delta at row 0 of those faces.
__global__ void k_adj_bcorr(Geom g, const float* __restrict__ face, FaceOffsets fo, float x_lo,
                            float x_hi, float4* __restrict__ lam) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    // enumerate slabs of thickness 3 next to each face; a node near several faces is owned by
    // the first slab containing it
    const long long per[3] = {3LL * g.n[1] * g.n[2], 3LL * g.n[0] * g.n[2], 3LL * g.n[0] * g.n[1]};
    long long r = t;
    int slab = 0;
    while (slab < 6 && r >= per[slab / 2]) {
        r -= per[slab / 2];
        ++slab;
    }
    if (slab >= 6) return;
    const int ax = slab / 2;
    int c[3];
    const int b0 = (ax == 0) ? 1 : 0, b1 = (ax == 2) ? 1 : 2;
    const int layer = (int)((unsigned)r % 3u);
    const unsigned rr = (unsigned)r / 3u;
    c[ax] = (slab & 1) ? g.n[ax] - 1 - layer : layer;
    c[b0] = (int)(rr % (unsigned)g.n[b0]);
    c[b1] = (int)(rr / (unsigned)g.n[b0]);
    for (int e = 0; e < slab; ++e) {
        const int ae = e / 2;
        const int d = (e & 1) ? g.n[ae] - 1 - c[ae] : c[ae];
        if (d >= 0 && d <= 2) return;
    }
    float sx = 0.f, sy = 0.f, sz = 0.f;
#pragma unroll
    for (int f = 0; f < 6; ++f) {
        const int a = f / 2;
        const int d = (f & 1) ? g.n[a] - 1 - c[a] : c[a];
        if (d > 2) continue;
        const float row0 = f == 0 ? x_lo : (f == 1 ? x_hi : ((f & 1) ? 1.5f : -1.5f));
        const float s = (f & 1) ? -1.f : 1.f;
        const float delta = d == 0 ? row0 : (d == 1 ? 1.5f * s : -0.5f * s);
        const int e0 = (a == 0) ? 1 : 0, e1 = (a == 2) ? 1 : 2;
        const float* fp = face + fo.off[f] + 3 * ((long long)c[e1] * g.n[e0] + c[e0]);
        sx += delta * fp[0];
        sy += delta * fp[1];
        sz += delta * fp[2];
    }
    const long long m = ((long long)c[2] * g.n[1] + c[1]) * g.n[0] + c[0];
    float4 v = lam[m];
    v.y += sx;
    v.z += sy;
    v.w += sz;
    lam[m] = v;
}

}  // namespace

void face_offsets(const Geom& g, FaceOffsets& fo, long long& total) {
    long long off = 0;
    for (int f = 0; f < 6; ++f) {
        const int a = f / 2;
        const int e0 = (a == 0) ? 1 : 0, e1 = (a == 2) ? 1 : 2;
        fo.off[f] = off;
        off += 3LL * g.n[e0] * g.n[e1];
    }
    total = off;
}

cudaError_t launch_fused_adj3d(const Geom& g, const Step3dPlan& plan, V4<float>* lam_in,
                               V4<float>* lam_out,
                               const V4<float>* kus, const V4<float>* sn, const V4<float>* sp,
                               float* e, float* face, double h, int* err, cudaStream_t st,
                               int variant) {
    launch_adj_prep<float>(g, lam_in, kus, sn, e, h, st);
    cudaError_t r = cudaGetLastError();
    if (r != cudaSuccess) return r;
    r = launch_adj_march(g, lam_in, lam_out, sp, face, err, st, plan.adj[variant], plan.adj_org);
    if (r != cudaSuccess) return r;
    FaceOffsets fo;
    long long tot;
    face_offsets(g, fo, tot);
    const long long shell = 6LL * ((long long)g.n[1] * g.n[2] + (long long)g.n[0] * g.n[2] +
                                   (long long)g.n[0] * g.n[1]);
    const bool lo_own = plan.adj_org == 0, hi_own = lo_own && g.n[0] > 4 && (g.n[0] - 4) % kAdjTileX == 0;
    k_adj_bcorr<<<(unsigned)((shell + 255) / 256), 256, 0, st>>>(
        g, face, fo, lo_own ? -2.f : -1.5f, hi_own ? 2.f : 1.5f, reinterpret_cast<float4*>(lam_out));
    return cudaGetLastError();
}

}  // namespace lks
