// Instance tables: the D2Q9 kernels that take a table of contexts of one precision and cover all
// of them in one launch (one context is a table of one).  Each kernel walks a list of work units
// (strips, box tiles, design columns, ...) concatenated over the instances; a prefix array per
// unit kind maps a unit to its instance.
#pragma once

#include <limits.h>

#include "lks_internal.h"

namespace lks {

// Buffers of a context addressed by index, so that a captured launch sequence names buffers
// the same way for every instance: the two working states, the initial state, the two adjoint
// buffers, the end states of the last forward and adjoint runs, then the snapshot/tape pool.
enum { BUF_S0 = 0, BUF_S1 = 1, BUF_INIT = 2, BUF_LAM0 = 3, BUF_LAM1 = 4, BUF_SEND = 5,
       BUF_LEND = 6, BUF_POOL = 7 };

template <class T>
struct Inst {
    Geom g;
    Design d;
    int2* pos_b;              // design positions of several steps: integer base of
    V4<T>* pos_sc;            // x_ref, y_ref and sin, cos of (pi f / 2) of their fractions
    const Motion* motion;     // rows 0..max_steps with cos/sin already evaluated (device)
    void* bufs[BUF_POOL];     // the buffers before the pool
    char* pool;               // and the pool, slots of snap bytes
    long long snap;
    const T* kref;            // kappa_ref per design node
    const T* kprime;          // d kappa_ref / d gamma
    V4<T>* kus;               // kappa, u_S on the footprint box
    V4<T>* kus_tape;          // kappa, u_S of several steps (slots of boxN records) or null
    T* e;                     // dJ/dkappa density of several steps (slots of boxN)
    double* gacc;             // dJ/dgamma accumulator
    int* flags;               // the context's error words
    double* jpart;            // objective partial sums, jparts per step
    int jparts;
    int win_begin, win_end;
    T A, A9, bf[2];           // A, A / 9 and the body force
    T src_r, src_x, src_y;    // h_n d j / d (rho, ux, uy) at a target node, inside the window
    V4<T> bcf[4];             // per face: prescribed rho - rho0 (r) and ux, uy (x, y)
    int bckeep[4];            // per face: 1 keeps the source's rho (wall, inlet), 0 prescribes
                              // it and copies the normal velocity (outlet)
    int corner[4];            // winning face of the corner (x side + 2 y side)
};

// A strip unit of the step and adjoint kernels: kStripW output columns (a warp's 32 columns less
// two of halo on each side) by strip_rows(k) rows, k one of kStripCfgs row counts.
constexpr int kStripW = 28;
constexpr int kStripCfgs = 5;
__host__ __device__ constexpr int strip_rows(int k) { return 2 << k; }   // 2, 4, 8, 16, 32

// Work-unit kinds: design columns in blocks of kUnitThreads, footprint-box tiles, objective parts,
// strips of each row count.
constexpr int kUnitThreads = 256;
constexpr int kBoxTileX = 32, kBoxTileY = 16;   // box tiles of the 2D transfer
enum { U_DCOL = 0, U_BOX, U_OBJ, U_STRIP0, U_COUNT = U_STRIP0 + kStripCfgs };

// Parts the objective's target list is summed in, one warp each: about eight values per lane.
constexpr int kObjMaxParts = 32;
__host__ __device__ inline int obj_parts(double count) {
    const double p = (count + 255.0) / 256.0;
    return p < 1.0 ? 1 : (p > kObjMaxParts ? kObjMaxParts : (int)p);
}

struct Plan {
    const void* tab;          // device, Inst<T> per instance
    const int* pre;           // device, [U_COUNT][count + 1]
    int count;
    int total[U_COUNT];
    const int* nbase;         // device: step index base added to each launch's offset
    int* bar;                 // device: arrival count of the grid barrier
    int* err;                 // device error word (8: a barrier wait ran out)
};

// Origin of the first strip along an axis of n nodes for strips of T: -o with o in {0, 2} chosen
// so that the nodes 0..2 and n-3..n-1 of a non-periodic axis each fall in one strip (the one-sided
// gradient rows of boundary nodes reach two nodes inward, and the adjoint's transposed
// gradient then finds them among its own lanes).
__host__ __device__ inline int strip_origin(int n, int T, int periodic) {
    if (periodic) return 0;
    const int r1 = (n - 1) % T, r2 = (n - 2) % T;
    return (r1 == 0 || r2 == 0) ? 2 : 0;
}
__host__ __device__ inline int strip_count(int n, int T, int periodic) {
    return (n + strip_origin(n, T, periodic) + T - 1) / T;
}

// A run of steps.  Forward: level k - 1 to level k for k = k0 .. k0 + n - 1, the levels in
// consecutive buffers from `buf` (level 0) when `taped`, else in the two working buffers
// starting from working buffer `buf`.  Adjoint: step k down to k - n + 1 for k = k0, lambda
// starting in adjoint buffer `buf`, the levels in consecutive buffers from `tape` (level 0).
// kslot: kappa, u_S of step k are in slot kslot + k (kBoxBuffer: all steps read the box buffer).
// eslot: e of step k goes to slot eslot + k.
struct StripRun {
    int k0, n, taped, buf, tape, kslot, eslot, obj;
};
constexpr int kBoxBuffer = INT_MIN;

// Launchers (stream st; noff = step offset from *nbase; kslot0 < 0: the box buffer).
// Design positions of n steps into position slots 0..n-1, then their transfers into slots
// kslot0 .. kslot0 + n - 1.
template <class T>
cudaError_t launch_t_transfer(const Plan& p, int noff, int n, int kslot0, cudaStream_t st);
// n steps (or adjoint steps) with strips of configuration cfg in one launch; more than one step
// needs a cooperative launch, whose blocks meet at a grid barrier after each step.
template <class T>
cudaError_t launch_t_step(const Plan& p, int cfg, const StripRun& r, cudaStream_t st);
template <class T>
cudaError_t launch_t_adj(const Plan& p, int cfg, const StripRun& r, cudaStream_t st);
// Objective partial sums of the level at offset noff in buffer src.
template <class T>
cudaError_t launch_t_objective(const Plan& p, int noff, int src, cudaStream_t st);
// Start and end of a run over every instance.  begin: error words to zero, and for an adjoint run
// lambda^N and dJ/dgamma too.  end: buffer src copied to dst (and checked as a state, forward); then J up to
// step n_last (forward) and the error words into one RunResult per instance.
struct RunResult {
    double J;
    int flags[4];
};
template <class T>
cudaError_t launch_t_begin(const Plan& p, bool adjoint, cudaStream_t st);
template <class T>
cudaError_t launch_t_end(const Plan& p, int dst, int src, int n_last, bool adjoint, RunResult* out,
                         cudaStream_t st);
// dJ/dgamma gather of the steps noff .. noff + n - 1 (last first), e in slots eslot0 ...
template <class T>
cudaError_t launch_t_sens(const Plan& p, int noff, int n, int eslot0, cudaStream_t st);
// Buffer src of every instance copied to its buffer dst.
template <class T>
cudaError_t launch_t_copy(const Plan& p, int dst, int src, cudaStream_t st);
cudaError_t launch_set_int(int* dst, int v, cudaStream_t st);
// The strip configuration a single context runs with.
int default_strips(const Plan& p, int type_size);

}  // namespace lks
