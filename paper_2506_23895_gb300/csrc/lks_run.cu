// Run machinery of the host engine: the rigid motion of each step, transfers (with the 3D
// side-stream prefetch), the forward and adjoint steps on the per-context and instance-table
// kernels, runs of steps over a group of contexts (captured into CUDA graphs on the table path),
// and the forward and reverse execution of the binomial checkpoint schedule (Algorithm 1 with
// the objective of Sec. 2.5; the exact discrete adjoint in the structure of Algorithm 2).
#include "lks_engine.h"

namespace lks {
namespace eng {

bool timing_begin(lks_ctx* c, int n, int which) {
    if (c->timing_stride <= 0 || (n % c->timing_stride) != 0) return false;
    std::vector<cudaEvent_t>& v = c->tev[which];
    if (c->tused[which] + 2 > v.size()) {
        cudaEvent_t a, b;
        if (cudaEventCreate(&a) != cudaSuccess) return false;
        if (cudaEventCreate(&b) != cudaSuccess) {
            cudaEventDestroy(a);
            return false;
        }
        v.push_back(a);
        v.push_back(b);
    }
    cudaEventRecord(v[c->tused[which]], c->st);
    return true;
}

void timing_end(lks_ctx* c, int which) {
    cudaEventRecord(c->tev[which][c->tused[which] + 1], c->st);
    c->tused[which] += 2;
}

Motion motion_row(const lks_ctx* c, const double* r) {
    Motion m;
    m.c = std::cos(r[0]);
    m.s = std::sin(r[0]);
    m.om = r[1];
    for (int a = 0; a < 3; ++a) {
        m.xG[a] = r[2 + a];
        m.uG[a] = r[5 + a];
        m.ugf[a] = (float)m.uG[a];
    }
    m.ch = (float)m.c;
    m.cl = (float)(m.c - (double)m.ch);
    m.sh = (float)m.s;
    m.sl = (float)(m.s - (double)m.sh);
    for (int a = 0; a < 2; ++a) {
        const double fl = std::floor(m.xG[a]);
        m.xgi[a] = (int)fl;
        m.xgh[a] = (float)(m.xG[a] - fl);
        m.xgl[a] = (float)((m.xG[a] - fl) - (double)m.xgh[a]);
        m.xgf[a] = (float)m.xG[a];
    }
    m.cf = (float)m.c;
    m.sf = (float)m.s;
    m.omf = (float)m.om;
    // R(theta) about the unit axis a by Rodrigues' formula (the z axis gives the plane rotation)
    const double* a = c->axis;
    const double cc = m.c, ss = m.s, oc = 1.0 - cc;
    if (!c->gaxis) {
        const double Rz[9] = {cc, -ss, 0.0, ss, cc, 0.0, 0.0, 0.0, 1.0};
        for (int k = 0; k < 9; ++k) m.R[k] = Rz[k];
        m.ax[0] = 0.0;
        m.ax[1] = 0.0;
        m.ax[2] = 1.0;
    } else {
        m.R[0] = cc + oc * a[0] * a[0];
        m.R[1] = oc * a[0] * a[1] - ss * a[2];
        m.R[2] = oc * a[0] * a[2] + ss * a[1];
        m.R[3] = oc * a[1] * a[0] + ss * a[2];
        m.R[4] = cc + oc * a[1] * a[1];
        m.R[5] = oc * a[1] * a[2] - ss * a[0];
        m.R[6] = oc * a[2] * a[0] - ss * a[1];
        m.R[7] = oc * a[2] * a[1] + ss * a[0];
        m.R[8] = cc + oc * a[2] * a[2];
        for (int k = 0; k < 3; ++k) m.ax[k] = a[k];
    }
    return m;
}

// ---------------------------------------------------------------- single-context steps

// The transfer of step n into buffer set x on stream st (3D and plain 2D paths).
template <class T>
lks_status transfer_into(lks_ctx* c, int n, const lks_ctx::XSlot& x, cudaStream_t st) {
    const Motion m = motion_row(c, &c->motion[8 * (size_t)n]);
    if (c->gaxis) {
        launch_transfer_axis<T>(c->d, c->g, m, x.as, (const T*)c->kref, st4<T>(x.kus), st);
        LAUNCHED();
        c->stats[4] += 2;
        return LKS_OK;
    }
    launch_design_pos<T>(c->d, c->g, m, x.ts, st);
    LAUNCHED();
    launch_transfer<T>(c->d, c->g, m, x.ts, (const T*)c->kref_t, (T*)x.k2, st4<T>(x.kus), st);
    LAUNCHED();
    return LKS_OK;
}

void use_set(lks_ctx* c, int i) {
    c->xcur = i;
    c->kus = c->xs[i].kus;
    c->k2 = c->xs[i].k2;
    c->ts = c->xs[i].ts;
    c->as = c->xs[i].as;
}

// The streams and events of a 3D context's overlapped work, created once: the run stream at
// the highest priority, the side stream at the lowest.
lks_status ensure_streams(lks_ctx* c) {
    if (c->run_st) return LKS_OK;
    int least = 0, greatest = 0;
    CU(cudaDeviceGetStreamPriorityRange(&least, &greatest));
    CU(cudaStreamCreateWithPriority(&c->side, cudaStreamNonBlocking, least));
    for (cudaEvent_t* e : {&c->ev_main, &c->ev_pf, &c->ev_join, &c->ev_adj, &c->ev_sens[0],
                           &c->ev_sens[1], &c->ev_fork, &c->ev_back})
        CU(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
    CU(cudaStreamCreateWithPriority(&c->run_st, cudaStreamNonBlocking, greatest));
    return LKS_OK;
}

// Fork a 3D context's run onto its high-priority stream (after the work on the caller's
// stream) and join it back afterwards.
lks_status run_fork(lks_ctx* c) {
    c->user_st = c->st;
    if (!c->pf_on) return LKS_OK;
    lks_status s = ensure_streams(c);
    if (s != LKS_OK) return s;
    CU(cudaEventRecord(c->ev_fork, c->user_st));
    CU(cudaStreamWaitEvent(c->run_st, c->ev_fork, 0));
    c->st = c->run_st;
    return LKS_OK;
}

lks_status run_join(lks_ctx* c, lks_status s) {
    if (c->pf_on && c->st == c->run_st && c->run_st) {
        cudaError_t e1 = cudaEventRecord(c->ev_back, c->run_st);
        cudaError_t e2 = cudaStreamWaitEvent(c->user_st, c->ev_back, 0);
        c->st = c->user_st;
        if (s == LKS_OK && (e1 != cudaSuccess || e2 != cudaSuccess))
            return fail(c, LKS_ERR_CUDA, "join of the run's stream failed");
    }
    c->st = c->user_st;
    return s;
}

// The context's stream waits for all side-stream work (prefetches, sensitivity gathers); a
// prefetch in flight is dropped, the current set keeps its step.
lks_status transfer_settle(lks_ctx* c) {
    if (c->side) {
        CU(cudaEventRecord(c->ev_join, c->side));
        CU(cudaStreamWaitEvent(c->st, c->ev_join, 0));
    }
    c->pf_step = -1;
    return LKS_OK;
}

// Settle and forget the current set too: no side work outlives a run, and the next run
// (after a possible change of design or motion) starts from fresh transfers.
lks_status transfer_join(lks_ctx* c) {
    lks_status s = transfer_settle(c);
    c->cur_step = -1;
    c->pf_last = -1;
    c->pf_dir = 0;
    return s;
}

// kappa and u_S of step n in the current buffer set.  3D: the transfer depends on the motion
// and the design only, so while the step n kernels run, the transfer of the step the run is
// heading to (n + 1 going forward, n - 1 going backward) is computed into the other set on a
// side stream, ordered by events; a later request for that step swaps the sets.  A request for
// the step the current set already holds (the adjoint's first step after a tape segment)
// launches nothing.
template <class T>
lks_status transfer_at(lks_ctx* c, int n) {
    if (c->d.nd == 0 || c->g.boxN == 0) return LKS_OK;
    if (c->fused2d) {
        CU(launch_set_int(c->nbase, n, c->st));
        CU(launch_t_transfer<T>(c->plan, 0, 1, -1, c->st));
        c->stats[4] += 3;
        return LKS_OK;
    }
    if (!c->pf_on) return transfer_into<T>(c, n, c->xs[c->xcur], c->st);
    {
        lks_status s = ensure_streams(c);
        if (s != LKS_OK) return s;
    }
    if (c->pf_step == n) {
        CU(cudaStreamWaitEvent(c->st, c->ev_pf, 0));
        use_set(c, 1 - c->xcur);
        c->pf_step = -1;
    } else if (c->cur_step != n) {
        // the current set may still be read by a sensitivity gather on the side stream (a run
        // that changed direction or jumped): wait for the side stream before overwriting it
        CU(cudaEventRecord(c->ev_join, c->side));
        CU(cudaStreamWaitEvent(c->st, c->ev_join, 0));
        lks_status s = transfer_into<T>(c, n, c->xs[c->xcur], c->st);
        if (s != LKS_OK) return s;
    }
    c->cur_step = n;
    // direction of the run: one step on from the previous request, or the same step again (a
    // tape segment's last step, then the adjoint of that segment: the run turns around)
    int dir = 0;
    if (c->pf_last >= 0 && std::abs(n - c->pf_last) == 1) dir = n - c->pf_last;
    else if (c->pf_last == n) dir = -c->pf_dir;
    c->pf_dir = dir;
    c->pf_last = n;
    const int next = n + dir;
    if (dir != 0 && next >= 1 && next <= c->cfg.max_steps && c->pf_step != next) {
        // a stale prefetch still in flight is overwritten after it, in side-stream order
        // the other set was last read by work already on the context's stream
        CU(cudaEventRecord(c->ev_main, c->st));
        CU(cudaStreamWaitEvent(c->side, c->ev_main, 0));
        lks_status s = transfer_into<T>(c, next, c->xs[1 - c->xcur], c->side);
        if (s != LKS_OK) return s;
        CU(cudaEventRecord(c->ev_pf, c->side));
        c->pf_step = next;
    }
    return LKS_OK;
}

// Variant of the fused 3D step for this context: the requested one, else each variant timed on
// the step src -> dst (three launches after one warm-up, CUDA events) and the fastest kept.
// Every variant writes the same dst, so the timing launches leave the step done.
lks_status choose_step3d(lks_ctx* c, const void* src, void* dst) {
    if (c->step3d_req >= 0) {
        c->step3d_var = c->step3d_req;
        return LKS_OK;
    }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CU(cudaStreamIsCapturing(c->st, &cap));
    if (cap != cudaStreamCaptureStatusNone) {
        c->step3d_var = 1;
        return LKS_OK;
    }
    cudaEvent_t e0, e1;
    CU(cudaEventCreate(&e0));
    CU(cudaEventCreate(&e1));
    float best = 1e30f;
    int bv = 1;
    cudaError_t err = cudaSuccess;
    for (int v = 0; v < kStep3dVariants && err == cudaSuccess; ++v) {
        for (int r = 0; r < 4 && err == cudaSuccess; ++r) {
            if (r == 1) err = cudaEventRecord(e0, c->st);
            if (err == cudaSuccess)
                err = launch_fused_step3d(c->g, c->plan3d, (const V4<float>*)src,
                                          (const V4<float>*)c->kus, (V4<float>*)dst, c->flags + 3,
                                          c->st, v);
        }
        if (err == cudaSuccess) err = cudaEventRecord(e1, c->st);
        if (err == cudaSuccess) err = cudaEventSynchronize(e1);
        float ms = 0.f;
        if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e0, e1);
        if (err == cudaSuccess && ms < best) {
            best = ms;
            bv = v;
        }
        c->stats[4] += 4;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (err != cudaSuccess) return fail(c, LKS_ERR_CUDA, "step variant timing: %s", cudaGetErrorString(err));
    c->step3d_var = bv;
    return LKS_OK;
}

// One forward step n: src -> dst (3D / FP64 / plain paths).
template <class T>
lks_status forward_step(lks_ctx* c, int n, const void* src, void* dst) {
    lks_status s = transfer_at<T>(c, n);
    if (s != LKS_OK) return s;
    const bool tm = timing_begin(c, n, 0);
    if (sizeof(T) == 4 && c->fused3d && !c->g.ks) {
        if (c->step3d_var < 0) {
            s = choose_step3d(c, src, dst);
            if (s != LKS_OK) return s;
        }
        cudaError_t e = launch_fused_step3d(c->g, c->plan3d, (const V4<float>*)src,
                                            (const V4<float>*)c->kus, (V4<float>*)dst,
                                            c->flags + 3, c->st, c->step3d_var);
        if (e != cudaSuccess) return fail(c, LKS_ERR_CUDA, "fused step: %s", cudaGetErrorString(e));
        ++c->stats[4];
    } else {
        launch_feq<T>(c->g, (const V4<T>*)src, (T*)c->F, c->st);
        LAUNCHED();
        launch_gather<T>(c->g, (const T*)c->F, (const V4<T>*)c->kus, (V4<T>*)dst, c->st);
        LAUNCHED();
    }
    if (tm) timing_end(c, 0);
    return LKS_OK;
}

char* slot_ptr(lks_ctx* c, int slot) { return c->pool + (size_t)slot * c->snap_bytes; }

lks_status copy_state(lks_ctx* c, void* dst, const void* src, cudaStream_t st) {
    CU(cudaMemcpyAsync(dst, src, (size_t)c->g.nodes * 4 * c->tsz, cudaMemcpyDeviceToDevice, st));
    return LKS_OK;
}

// One adjoint step n on the per-context kernels: lambda^n (lam[lam_par]) -> lambda^{n-1}.
template <class T>
lks_status adjoint_step(lks_ctx* c, int n, const void* sn, const void* sp) {
    const double h = 1.0 / (double)(c->cfg.win_end - c->cfg.win_begin + 1);
    const double hn = (n >= c->cfg.win_begin && n <= c->cfg.win_end) ? h : 0.0;
    lks_status s = transfer_at<T>(c, n);
    if (s != LKS_OK) return s;
    V4<T>* lc = st4<T>(c->lam[c->lam_par]);
    V4<T>* ln = st4<T>(c->lam[1 - c->lam_par]);
    const bool side_sens = c->pf_on && c->side && c->d.nd > 0 && c->g.boxN > 0;
    if (side_sens) {   // e alternates between two buffers; wait for the gather that read this one
        c->e = c->ebuf[c->epar];
        CU(cudaStreamWaitEvent(c->st, c->ev_sens[c->epar], 0));
    }
    const bool tm = timing_begin(c, n, 1);
    if (sizeof(T) == 4 && c->fused3d && !c->g.ks) {
        cudaError_t e = launch_fused_adj3d(c->g, c->plan3d, (V4<float>*)lc, (V4<float>*)ln,
                                           (const V4<float>*)c->kus, (const V4<float>*)sn,
                                           (const V4<float>*)sp, (float*)c->e, c->face, hn,
                                           c->flags + 3, c->st, c->adj3d_var);
        if (e != cudaSuccess) return fail(c, LKS_ERR_CUDA, "fused adjoint: %s", cudaGetErrorString(e));
        c->stats[4] += 3;
    } else {
        const V4<T>* mu = lc;
        if (c->g.ks || c->u3) {
            launch_adj_bcT<T>(c->g, lc, hn, c->st);
            LAUNCHED();
            launch_adj_mu<T>(c->g, lc, (const V4<T>*)c->kus, (const V4<T>*)sn, st4<T>(c->mu),
                             (T*)c->e, hn, c->st, (const V4<T>*)c->u3);
            mu = st4<T>(c->mu);
        } else {
            launch_adj_prep<T>(c->g, lc, (const V4<T>*)c->kus, (const V4<T>*)sn, (T*)c->e, hn, c->st);
        }
        LAUNCHED();
        launch_adj_moments<T>(c->g, mu, (const V4<T>*)sp, ln, (T*)c->phi, c->st,
                              (V4<T>*)c->u3);
        LAUNCHED();
        launch_adj_divT<T>(c->g, (const T*)c->phi, ln, c->st);
        LAUNCHED();
    }
    if (tm) timing_end(c, 1);
    if (c->d.nd > 0 && c->g.boxN > 0) {
        // on the side stream (3D): after this step's adjoint kernels, before the prefetch that
        // will next overwrite this step's transfer set; dJ/dgamma sums stay in step order
        cudaStream_t ss = c->st;
        if (side_sens) {
            CU(cudaEventRecord(c->ev_adj, c->st));
            CU(cudaStreamWaitEvent(c->side, c->ev_adj, 0));
            ss = c->side;
        }
        if (c->gaxis)
            launch_sens_axis<T>(c->d, c->g, c->as, (const T*)c->e, (const T*)c->kprime, c->gacc,
                                ss);
        else
            launch_sens<T>(c->d, c->g, c->ts, (const T*)c->e, (const T*)c->kprime, c->gacc, ss);
        LAUNCHED();
        if (side_sens) {
            CU(cudaEventRecord(c->ev_sens[c->epar], c->side));
            c->epar ^= 1;
        }
    }
    c->lam_par ^= 1;
    return LKS_OK;
}

int seg_start(const lks_ctx* c, int a) { return a * c->K; }
int seg_end(const lks_ctx* c, int a) { return std::min((a + 1) * c->K, c->n_fwd); }
// ---------------------------------------------------------------- groups of contexts
// A group runs one checkpoint schedule for contexts of identical step count and snapshot pool:
// the single-context calls use a group of one, lks_batch_* a group over all its contexts.  On
// the instance-table path (D2Q9) every phase of a step is one launch over the whole group,
// and a run of steps can be captured once into a CUDA graph and replayed.


lks_status gfail(Group& G, lks_status s, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    for (int i = 0; i < G.count; ++i) G.cs[i]->err = buf;
    return s;
}

#define GCU(call)                                                                         \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess)                                                            \
            return gfail(G, LKS_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_));       \
    } while (0)

Group self_group(lks_ctx*& c) {
    Group G;
    G.cs = &c;
    G.count = 1;
    G.table = c->fused2d;
    G.plan = &c->plan;
    G.nbase = c->nbase;
    G.result = (RunResult*)c->scal;
    G.tile_fwd = c->tile_fwd;
    G.tile_adj = c->tile_adj;
    G.st = c->st;
    return G;
}

// Every context of the group keeps the transfers of a whole tape segment (2D table path).
bool tape_transfers(const Group& G) {
    if (!G.table) return false;
    for (int i = 0; i < G.count; ++i)
        if (G.cs[i]->d.nd > 0 && G.cs[i]->K + 1 > G.cs[i]->slots.k) return false;
    return true;
}

// Steps of a run handled by one launch: at most kRunSteps (which bounds a launch to some
// milliseconds) and as many as there are slots for their transfers (unless those are kept: kt) and, in
// the adjoint, for their e.
constexpr int kRunSteps = 512;
int group_chunk(const Group& G, bool kt, bool adjoint) {
    int n = kRunSteps;
    for (int i = 0; i < G.count; ++i) {
        if (G.cs[i]->d.nd == 0) continue;
        if (!kt) n = std::min(n, G.cs[i]->slots.k);
        if (adjoint) n = std::min(n, G.cs[i]->slots.e);
    }
    return std::max(n, 1);
}

// Transfers of steps k .. k + n - 1 (offsets from *nbase) into slots slot .. slot + n - 1.
template <class T>
cudaError_t table_transfers(const Group& G, int k, int n, int slot, int& nl) {
    int pos = n;
    for (int i = 0; i < G.count; ++i)
        if (G.cs[i]->d.nd > 0) pos = std::min(pos, G.cs[i]->slots.pos);
    for (int j = 0; j < n; j += pos) {
        const cudaError_t e =
            launch_t_transfer<T>(*G.plan, k + j, std::min(pos, n - j), slot + j, G.st);
        if (e != cudaSuccess) return e;
        nl += 2;
    }
    return cudaSuccess;
}

// Run table-path steps from base: fn(nl, direct) issues them and counts launches.  With a graph
// cache the sequence is captured once per key and replayed.
template <class Fn>
lks_status table_run(Group& G, std::tuple<int, int, int, int, int, int> key, int base, Fn fn) {
    GCU(launch_set_int(G.nbase, base, G.st));
    ++G.launches;
    if (!G.graphs) {
        int nl = 0;
        const cudaError_t e = fn(nl, true);
        if (e != cudaSuccess)
            return gfail(G, LKS_ERR_CUDA, "table kernel launch: %s", cudaGetErrorString(e));
        G.launches += nl;
        return LKS_OK;
    }
    auto it = G.graphs->execs.find(key);
    if (it == G.graphs->execs.end()) {
        GCU(cudaStreamBeginCapture(G.st, cudaStreamCaptureModeThreadLocal));
        int nl = 0;
        cudaError_t e = fn(nl, false);
        cudaGraph_t graph = nullptr;
        cudaError_t e2 = cudaStreamEndCapture(G.st, &graph);
        if (e != cudaSuccess || e2 != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            return gfail(G, LKS_ERR_CUDA, "graph capture: %s",
                         cudaGetErrorString(e != cudaSuccess ? e : e2));
        }
        cudaGraphExec_t exec = nullptr;
        e = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return gfail(G, LKS_ERR_CUDA, "graph instantiate: %s",
                                           cudaGetErrorString(e));
        it = G.graphs->execs.emplace(key, exec).first;
        G.graphs->nodes[key] = nl;
    }
    GCU(cudaGraphLaunch(it->second, G.st));
    G.launches += G.graphs->nodes[key];
    return LKS_OK;
}

// ---------------------------------------------------------------- schedule over a group

// Advance every context of the group from from_level to to_level.  Without a tape the two
// working buffers alternate; with a tape (segment tape_seg, whose start level sits in tape slot
// 0) every level is written straight into its own tape slot and the working buffer keeps
// from_level.
template <class T>
lks_status run_steps(Group& G, int from_level, int to_level, bool with_obj, int tape_seg) {
    lks_ctx* c0 = G.cs[0];
    const int len = to_level - from_level;
    if (len > 0 && G.table) {
        const int w0 = c0->work;
        const int toff = tape_seg >= 0 ? from_level - tape_seg * c0->K : 0;
        // the objective kernel only where some instance's window meets these steps
        bool obj = false;
        for (int i = 0; i < G.count && with_obj; ++i)
            obj = obj || (G.cs[i]->cfg.win_begin <= to_level &&
                          G.cs[i]->cfg.win_end > from_level);
        // a taped step leaves its transfer in the slot of its level, for the adjoint
        const bool kt = tape_seg >= 0 && tape_transfers(G);
        auto fn = [&](int& nl, bool direct) -> cudaError_t {
            lks_ctx* timed = direct && G.count == 1 && c0->timing_stride > 0 ? c0 : nullptr;
            const int chunk = group_chunk(G, kt, false);
            for (int k0 = 1; k0 <= len; k0 += chunk) {
                const int n = std::min(chunk, len - k0 + 1);
                const int slot = kt ? toff + k0 : 0;
                cudaError_t e = table_transfers<T>(G, k0, n, slot, nl);
                if (e != cudaSuccess) return e;
                StripRun r;
                r.taped = tape_seg >= 0;
                r.buf = tape_seg >= 0 ? BUF_POOL + toff : w0;
                r.tape = 0;
                r.kslot = slot - k0;
                r.eslot = 0;
                r.obj = obj;
                // one launch for the chunk; with timing on, one per step with events around it
                for (int k = k0; k < k0 + n; k += r.n) {
                    r.k0 = k;
                    r.n = timed ? 1 : n;
                    const bool tm = timed && timing_begin(timed, from_level + k, 0);
                    if ((e = launch_t_step<T>(*G.plan, G.tile_fwd, r, G.st)) != cudaSuccess)
                        return e;
                    if (tm) timing_end(timed, 0);
                    ++nl;
                    if (!obj) continue;
                    const int kl = k + r.n - 1;
                    const int last = tape_seg >= 0 ? BUF_POOL + toff + kl : BUF_S0 + ((w0 + kl) & 1);
                    if ((e = launch_t_objective<T>(*G.plan, kl, last, G.st)) != cudaSuccess)
                        return e;
                    ++nl;
                }
            }
            return cudaSuccess;
        };
        const auto key = std::make_tuple(tape_seg >= 0 ? 1 : 0, obj ? 1 : 0, len,
                                         tape_seg >= 0 ? toff : w0, G.tile_fwd, kt ? 1 : 0);
        lks_status s = table_run(G, key, from_level, fn);
        if (s != LKS_OK) return s;
        for (int i = 0; i < G.count; ++i) {
            lks_ctx* c = G.cs[i];
            if (tape_seg >= 0) {
                c->last = slot_ptr(c, toff + len);
            } else {
                c->work = (w0 + len) & 1;
                c->last = c->s[c->work];
            }
            c->stats[with_obj ? 0 : 1] += len;
        }
    } else if (len > 0) {
        lks_ctx* c = c0;
        for (int n = from_level + 1; n <= to_level; ++n) {
            const void* src;
            void* dst;
            if (tape_seg >= 0) {
                src = slot_ptr(c, n - 1 - tape_seg * c->K);
                dst = slot_ptr(c, n - tape_seg * c->K);
            } else {
                src = c->s[c->work];
                dst = c->s[1 - c->work];
            }
            lks_status s = forward_step<T>(c, n, src, dst);
            if (s != LKS_OK) return s;
            if (tape_seg < 0) c->work = 1 - c->work;
            c->last = dst;
            if (with_obj && n >= c->cfg.win_begin && n <= c->cfg.win_end) {
                launch_objective<T>(c->g, (const V4<T>*)dst, c->jstep + n, c->st);
                LAUNCHED();
            }
            if (with_obj) ++c->stats[0];
            else ++c->stats[1];
        }
    }
    for (int i = 0; i < G.count; ++i)
        G.cs[i]->work_level = (tape_seg >= 0) ? from_level : to_level;
    return LKS_OK;
}

// Copy a state of every context of the group: one launch over the instances on the table path
// (buffers by index, equal in every context), a memory copy otherwise.
template <class T>
lks_status group_copy(Group& G, int dst, int src) {
    if (G.table) {
        GCU(launch_t_copy<T>(*G.plan, dst, src, G.st));
        ++G.launches;
        return LKS_OK;
    }
    lks_ctx* c = G.cs[0];
    return copy_state(c, c->hbufs[dst], c->hbufs[src], G.st);
}

template <class T>
lks_status restore_level(Group& G, int seg) {
    // the contexts of a group follow one schedule: equal slots and levels
    lks_ctx* c0 = G.cs[0];
    const int lev = seg_start(c0, seg);
    if (c0->work_level == lev) return LKS_OK;
    if (seg != 0 && c0->slot_of[seg] < 0) return gfail(G, LKS_ERR_ARG, "schedule: no snapshot");
    const int src = seg == 0 ? (int)BUF_INIT : BUF_POOL + c0->slot_of[seg];
    lks_status s = group_copy<T>(G, BUF_S0 + c0->work, src);
    if (s != LKS_OK) return s;
    for (int i = 0; i < G.count; ++i) G.cs[i]->work_level = lev;
    return LKS_OK;
}

template <class T>
lks_status exec_forward_action(Group& G, const Act& a, bool with_obj) {
    lks_ctx* c0 = G.cs[0];
    switch (a.kind) {
        case A_RESTORE:
            return restore_level<T>(G, a.a);
        case A_ADVANCE:
            return run_steps<T>(G, seg_start(c0, a.a), seg_start(c0, a.b), with_obj, -1);
        case A_STORE:
            for (int i = 0; i < G.count; ++i) {
                lks_ctx* c = G.cs[i];
                if (c->free_slots.empty()) return fail(c, LKS_ERR_NOMEM, "schedule: out of slots");
                c->slot_of[a.a] = c->free_slots.back();
                c->free_slots.pop_back();
            }
            return group_copy<T>(G, BUF_POOL + c0->slot_of[a.a], BUF_S0 + c0->work);
        case A_FREE:
            for (int i = 0; i < G.count; ++i) {
                lks_ctx* c = G.cs[i];
                c->free_slots.push_back(c->slot_of[a.a]);
                c->slot_of[a.a] = -1;
            }
            return LKS_OK;
        case A_TAPE: {
            lks_status s = group_copy<T>(G, BUF_POOL, BUF_S0 + c0->work);
            if (s != LKS_OK) return s;
            return run_steps<T>(G, seg_start(c0, a.a), seg_end(c0, a.a), with_obj, a.a);
        }
        default:
            return gfail(G, LKS_ERR_ARG, "schedule: unexpected action");
    }
}

template <class T>
lks_status exec_adj(Group& G, int seg) {
    lks_ctx* c0 = G.cs[0];
    const int a = seg_start(c0, seg), b = seg_end(c0, seg), len = b - a;
    if (len <= 0) return LKS_OK;
    if (!G.table) {
        for (int n = b; n > a; --n) {
            lks_status s = adjoint_step<T>(c0, n, slot_ptr(c0, n - a), slot_ptr(c0, n - 1 - a));
            if (s != LKS_OK) return s;
        }
        return LKS_OK;
    }
    const int par0 = c0->lam_par;
    // the tape of this segment (levels 0..len) holds the transfer of step a + k in slot k, or the
    // transfers are formed again
    const bool kt = tape_transfers(G);
    auto fn = [&](int& nl, bool direct) -> cudaError_t {
        lks_ctx* timed = direct && G.count == 1 && c0->timing_stride > 0 ? c0 : nullptr;
        const int chunk = group_chunk(G, kt, true);
        for (int k1 = len; k1 >= 1; k1 -= chunk) {   // steps a + k1 down to a + k0
            const int n = std::min(chunk, k1), k0 = k1 - n + 1;
            cudaError_t e = cudaSuccess;
            if (!kt && (e = table_transfers<T>(G, k0, n, 0, nl)) != cudaSuccess) return e;
            StripRun r;
            r.taped = 1;
            r.tape = BUF_POOL;
            r.kslot = kt ? 0 : -k0;
            r.eslot = -k0;
            r.obj = 0;
            for (int k = k1; k >= k0; k -= r.n) {
                r.k0 = k;
                r.n = timed ? 1 : n;
                r.buf = par0 ^ ((len - k) & 1);
                const bool tm = timed && timing_begin(timed, a + k, 1);
                if ((e = launch_t_adj<T>(*G.plan, G.tile_adj, r, G.st)) != cudaSuccess) return e;
                if (tm) timing_end(timed, 1);
                ++nl;
            }
            if ((e = launch_t_sens<T>(*G.plan, k0, n, 0, G.st)) != cudaSuccess) return e;
            ++nl;
        }
        return cudaSuccess;
    };
    const auto key = std::make_tuple(2, kt ? 1 : 0, len, par0, 0, G.tile_adj);
    lks_status s = table_run(G, key, a, fn);
    if (s != LKS_OK) return s;
    for (int i = 0; i < G.count; ++i) G.cs[i]->lam_par = par0 ^ (len & 1);
    return LKS_OK;
}

// The status a run's four error words stand for.
lks_status word_status(const int* f) {
    if (f[1]) return LKS_ERR_ARG;
    if (f[3] & 8) return LKS_ERR_TIMEOUT;
    if (f[3]) return LKS_ERR_CUDA;
    return f[2] ? LKS_ERR_DIVERGED : LKS_OK;
}

lks_status run_status(lks_ctx* c, const int* f) {
    const lks_status s = word_status(f);
    switch (s) {
        case LKS_ERR_ARG: return fail(c, s, "transfer tap list overflow");
        case LKS_ERR_TIMEOUT: return fail(c, s, "a bounded wait ran out in a fused kernel");
        case LKS_ERR_CUDA: return fail(c, s, "fused step reported error %d", f[3]);
        case LKS_ERR_DIVERGED:
            return fail(c, s, "state diverged (non-finite or |u| >= 0.5)");
        default: return s;
    }
}

// A bounded wait that ran out in a launch over a group is recorded with the group's first context
// (Plan::err), but the run stopped half way for all of them: the record counts for each.  words: four
// error words per context.  True if there was one.
bool share_waits(int* words, int n) {
    int waited = 0;
    for (int k = 0; k < n; ++k) waited |= words[4 * k + 3] & 8;
    for (int k = 0; k < n; ++k) words[4 * k + 3] |= waited;
    return waited != 0;
}

// The error words of a group's finished run on the table kernels.
std::vector<int> result_words(const std::vector<RunResult>& res, bool& waited) {
    std::vector<int> w;
    for (const RunResult& r : res) w.insert(w.end(), r.flags, r.flags + 4);
    waited = share_waits(w.data(), (int)res.size());
    return w;
}

template <class T>
lks_status do_forward(Group& G, int N) {
    for (int i = 0; i < G.count; ++i) {
        lks_ctx* c = G.cs[i];
        c->n_fwd = N;
        plan_tape(N, c->pool_slots, c->K, c->M, c->S);
        c->acts.clear();
        gen_schedule(0, c->M, c->S, c->acts);
        c->slot_of.assign(c->M + 1, -1);
        c->free_slots.clear();
        for (int k = c->pool_slots - 1; k >= c->K + 1; --k) c->free_slots.push_back(k);
        c->stats[0] = c->stats[1] = 0;
        c->stats[2] = c->S;
        c->stats[3] = c->K;
        c->stats[4] = 0;
        c->work = 0;
        c->work_level = -1;
        c->last = nullptr;
        c->fwd_valid = false;
        if (G.table) continue;
        {
            lks_status s = transfer_join(c);
            if (s != LKS_OK) return s;
        }
        CU(cudaMemsetAsync(c->jstep, 0, (size_t)(c->cfg.max_steps + 2) * 8, G.st));
        CU(cudaMemsetAsync(c->flags, 0, 64, G.st));
    }
    if (G.table) {
        GCU(launch_t_begin<T>(*G.plan, false, G.st));
        ++G.launches;
    }
    const std::vector<Act>& acts = G.cs[0]->acts;
    size_t i = 0;
    for (; i < acts.size(); ++i) {
        lks_status s = exec_forward_action<T>(G, acts[i], true);
        if (s != LKS_OK) return s;
        if (acts[i].kind == A_TAPE) break;
    }
    if (G.table) {
        std::vector<RunResult> res(G.count);
        lks_ctx* c0 = G.cs[0];
        int last = 0;
        while (c0->hbufs[last] != c0->last) ++last;
        GCU(launch_t_end<T>(*G.plan, BUF_SEND, last, N, false, G.result, G.st));
        G.launches += 2;
        GCU(cudaMemcpyAsync(res.data(), G.result, sizeof(RunResult) * G.count,
                            cudaMemcpyDeviceToHost, G.st));
        GCU(cudaStreamSynchronize(G.st));
        bool waited;
        const std::vector<int> words = result_words(res, waited);
        lks_status worst = LKS_OK;
        for (int k = 0; k < G.count; ++k) {
            lks_ctx* c = G.cs[k];
            c->adj_begin = i + 1;
            const lks_status s = run_status(c, &words[4 * k]);
            if (s != LKS_OK) {
                if (waited) c->have_end = false;   // no end state: the run stopped half way
                if (worst == LKS_OK) worst = s;
                continue;
            }
            c->have_end = true;
            c->J = res[k].J;
            c->fwd_valid = true;
        }
        return worst;
    }
    std::vector<std::vector<double>> js(G.count);
    std::vector<int> fl(4 * (size_t)G.count);
    for (int k = 0; k < G.count; ++k) {
        lks_ctx* c = G.cs[k];
        lks_status st = transfer_settle(c);   // the adjoint may reuse the last step's transfer
        if (st != LKS_OK) return st;
        c->adj_begin = i + 1;
        js[k].assign(c->cfg.max_steps + 2, 0.0);
        CU(cudaMemcpyAsync(js[k].data(), c->jstep, js[k].size() * 8, cudaMemcpyDeviceToHost, G.st));
        launch_check_state<T>(c->g, (const V4<T>*)c->last, c->flags + 2, G.st);
        LAUNCHED();
        CU(cudaMemcpyAsync(c->s_end, c->last, c->snap_bytes, cudaMemcpyDeviceToDevice, G.st));
        CU(cudaMemcpyAsync(fl.data() + 4 * k, c->flags, 16, cudaMemcpyDeviceToHost, G.st));
    }
    GCU(cudaStreamSynchronize(G.st));
    lks_status worst = LKS_OK;
    for (int k = 0; k < G.count; ++k) {
        lks_ctx* c = G.cs[k];
        const lks_status s = run_status(c, fl.data() + 4 * k);
        if (s != LKS_OK) {
            if (worst == LKS_OK) worst = s;
            continue;
        }
        const int w0 = c->cfg.win_begin, w1 = std::min(c->cfg.win_end, N);
        const double h = 1.0 / (double)(c->cfg.win_end - c->cfg.win_begin + 1);
        c->have_end = true;
        double J = 0.0;
        for (int n = w0; n <= w1; ++n) J += h * js[k][n];   // J = h sum_n j_n in step order
        c->J = J;
        c->fwd_valid = true;
    }
    return worst;
}

template <class T>
lks_status do_adjoint(Group& G) {
    for (int i = 0; i < G.count; ++i) {
        lks_ctx* c = G.cs[i];
        c->lam_par = 0;
        if (G.table) continue;
        CU(cudaMemsetAsync(c->flags, 0, 64, G.st));
        if (c->adj_warm && c->have_lend)   // warm start: lambda^N from the last lambda^0
            CU(cudaMemcpyAsync(c->lam[0], c->l_end, c->snap_bytes, cudaMemcpyDeviceToDevice, G.st));
        else
            CU(cudaMemsetAsync(c->lam[0], 0, c->snap_bytes, G.st));
        if (c->u3) CU(cudaMemsetAsync(c->u3, 0, c->snap_bytes, G.st));
        if (c->d.nd > 0) CU(cudaMemsetAsync(c->gacc, 0, (size_t)c->d.nd * 8, G.st));
    }
    if (G.table) {
        GCU(launch_t_begin<T>(*G.plan, true, G.st));
        ++G.launches;
        for (int i = 0; i < G.count; ++i) {   // warm starts: lambda^N from the last lambda^0
            lks_ctx* c = G.cs[i];
            if (c->adj_warm && c->have_lend)
                CU(cudaMemcpyAsync(c->lam[0], c->l_end, c->snap_bytes, cudaMemcpyDeviceToDevice,
                                   G.st));
        }
    }
    lks_ctx* c0 = G.cs[0];
    for (size_t i = c0->adj_begin - 1; i < c0->acts.size(); ++i) {
        const Act& a = c0->acts[i];
        if (a.kind == A_TAPE && i == c0->adj_begin - 1) continue;  // recorded by the forward
        lks_status s = (a.kind == A_ADJ) ? exec_adj<T>(G, a.a) : exec_forward_action<T>(G, a, false);
        if (s != LKS_OK) return s;
    }
    // the tape of the last segment has been overwritten: a second adjoint needs a new forward
    if (G.table) {
        std::vector<RunResult> res(G.count);
        GCU(launch_t_end<T>(*G.plan, BUF_LEND, BUF_LAM0 + c0->lam_par, 0, true, G.result, G.st));
        G.launches += 2;
        GCU(cudaMemcpyAsync(res.data(), G.result, sizeof(RunResult) * G.count,
                            cudaMemcpyDeviceToHost, G.st));
        for (int k = 0; k < G.count; ++k) {
            G.cs[k]->fwd_valid = false;
            G.cs[k]->have_lend = true;
        }
        GCU(cudaStreamSynchronize(G.st));
        bool waited;
        const std::vector<int> words = result_words(res, waited);
        lks_status worst = LKS_OK;
        for (int k = 0; k < G.count; ++k) {
            if (waited) G.cs[k]->have_lend = false;   // the sweep stopped half way
            const lks_status s = run_status(G.cs[k], &words[4 * k]);
            if (s != LKS_OK && worst == LKS_OK) worst = s;
        }
        return worst;
    }
    std::vector<int> fl(4 * (size_t)G.count);
    for (int k = 0; k < G.count; ++k) {
        lks_ctx* c = G.cs[k];
        c->fwd_valid = false;
        {
            lks_status st = transfer_join(c);
            if (st != LKS_OK) return st;
        }
        CU(cudaMemcpyAsync(c->l_end, c->lam[c->lam_par], c->snap_bytes, cudaMemcpyDeviceToDevice,
                           G.st));
        c->have_lend = true;
        CU(cudaMemcpyAsync(fl.data() + 4 * k, c->flags, 16, cudaMemcpyDeviceToHost, G.st));
    }
    GCU(cudaStreamSynchronize(G.st));
    lks_status worst = LKS_OK;
    for (int k = 0; k < G.count; ++k) {
        lks_ctx* c = G.cs[k];
        const lks_status s = run_status(c, fl.data() + 4 * k);
        if (s != LKS_OK && worst == LKS_OK) worst = s;
    }
    return worst;
}

template <class T>
lks_status reset_initial(lks_ctx* c) {
    launch_fill_uniform<T>(c->g, st4<T>(c->s0), c->cfg.u_init, c->st);
    LAUNCHED();
    launch_apply_bc<T>(c->g, st4<T>(c->s0), c->st);
    LAUNCHED();
    return LKS_OK;
}

// Host record of a context's instance-table entry (valid once design and motion are set).
template <class T>
Inst<T> make_inst(const lks_ctx* c) {
    Inst<T> I;
    std::memset(&I, 0, sizeof(I));
    I.g = c->g;
    I.d = c->d;
    I.pos_b = (int2*)c->pos_b;
    I.pos_sc = (V4<T>*)c->pos_sc;
    I.motion = c->dmotion;
    for (int b = 0; b < BUF_POOL; ++b) I.bufs[b] = c->hbufs[b];
    I.pool = c->pool;
    I.snap = (long long)c->snap_bytes;
    I.kref = (const T*)c->kref;
    I.kprime = (const T*)c->kprime;
    I.kus = (V4<T>*)c->kus;
    I.kus_tape = (V4<T>*)c->ktape;
    I.e = (T*)c->etape;
    I.gacc = c->gacc;
    I.flags = c->flags;
    I.jpart = c->jpart;
    I.jparts = obj_parts(c->g.ocount);
    I.win_begin = c->cfg.win_begin;
    I.win_end = c->cfg.win_end;
    // the same FP64 expressions as the per-node source of the plain kernels, rounded once
    const double h = 1.0 / (double)(c->cfg.win_end - c->cfg.win_begin + 1);
    const Geom& g = c->g;
    I.A = (T)g.A;
    I.A9 = (T)(g.A / 9.0);
    I.bf[0] = (T)g.body[0];
    I.bf[1] = (T)g.body[1];
    I.src_r = g.okind == 0 ? (T)(-h / (3.0 * g.ocount)) : (T)0;
    I.src_x = g.okind == 0 ? (T)0 : (T)(-h * g.odir[0] / g.ocount);
    I.src_y = g.okind == 0 ? (T)0 : (T)(-h * g.odir[1] / g.ocount);
    for (int f = 0; f < 4; ++f) {
        I.bcf[f].r = (T)(g.bcv[f][3] - g.rho0);
        I.bcf[f].x = (T)g.bcv[f][0];
        I.bcf[f].y = (T)g.bcv[f][1];
        I.bcf[f].z = (T)0;
        I.bckeep[f] = g.bc[f] == BC_WALL || g.bc[f] == BC_INLET;
    }
    for (int q = 0; q < 4; ++q) {   // WALL > INLET > OUTLET, ties to the lower face
        auto prec = [&](int f) { return g.bc[f] == BC_WALL ? 3 : (g.bc[f] == BC_INLET ? 2 : 1); };
        const int fx = q & 1, fy = 2 + (q >> 1);
        I.corner[q] = prec(fy) > prec(fx) ? fy : fx;
    }
    return I;
}

// Work units of one instance per unit kind (lks_table.h).
void inst_units(const lks_ctx* c, int out[U_COUNT]) {
    const Geom& g = c->g;
    const bool body = c->d.nd > 0 && g.boxN > 0;
    out[U_DCOL] = body ? (int)((c->d.ncol + kUnitThreads - 1) / kUnitThreads) : 0;
    // footprint box in tiles of kBoxTileX x kBoxTileY nodes (the 2D transfer stages the design
    // nodes a tile reads in shared memory)
    out[U_BOX] = body ? ((g.bn[0] + kBoxTileX - 1) / kBoxTileX) *
                            ((g.bn[1] + kBoxTileY - 1) / kBoxTileY)
                      : 0;
    out[U_OBJ] = obj_parts(g.ocount);
    for (int k = 0; k < kStripCfgs; ++k)
        out[U_STRIP0 + k] = strip_count(g.n[0], kStripW, g.periodic[0]) *
                            ((g.n[1] + strip_rows(k) - 1) / strip_rows(k));
}

// Build a plan over contexts: the table and prefix arrays go to dinst / dpre (device, with
// room for cs.size() entries), the host plan gets the totals.  nbase: device words of the plan's
// owner: the step base, then the grid barrier's count.
template <class T>
cudaError_t build_plan(const std::vector<lks_ctx*>& cs, void* dinst, int* dpre, int* nbase,
                       cudaStream_t st, Plan& p) {
    const int B = (int)cs.size();
    std::vector<Inst<T>> tab(B);
    std::vector<int> pre((size_t)U_COUNT * (B + 1), 0);
    for (int i = 0; i < B; ++i) {
        tab[i] = make_inst<T>(cs[i]);
        int u[U_COUNT];
        inst_units(cs[i], u);
        for (int k = 0; k < U_COUNT; ++k)
            pre[(size_t)k * (B + 1) + i + 1] = pre[(size_t)k * (B + 1) + i] + u[k];
    }
    cudaError_t e =
        cudaMemcpyAsync(dinst, tab.data(), sizeof(Inst<T>) * B, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dpre, pre.data(), pre.size() * sizeof(int), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(nbase, 0, 2 * sizeof(int), st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);   // host vectors go out of scope
    if (e != cudaSuccess) return e;
    std::memset(&p, 0, sizeof(p));
    p.tab = dinst;
    p.pre = dpre;
    p.count = B;
    p.nbase = nbase;
    p.bar = nbase + 1;
    p.err = cs[0]->flags + 3;
    for (int k = 0; k < U_COUNT; ++k) p.total[k] = pre[(size_t)k * (B + 1) + B];
    return cudaGetLastError();
}

// The one-entry plan of a table context, and its strip height.
lks_status own_plan(lks_ctx* c) {
    std::vector<lks_ctx*> one(1, c);
    if (c->prec == LKS_FP64)
        CU(build_plan<double>(one, c->dinst, c->dpre, c->nbase, c->st, c->plan));
    else
        CU(build_plan<float>(one, c->dinst, c->dpre, c->nbase, c->st, c->plan));
    c->tile_fwd = c->tile_adj = default_strips(c->plan, (int)c->tsz);
    return LKS_OK;
}

// kappa_ref and kappa' from the stored gamma, through the filter chain when it is on (the
// [0,1] check of gamma sets flags[0]).
lks_status design_prep(lks_ctx* c) {
    const double* src = c->gamma;
    if (c->fR > 0.0) {
        launch_filter(c->d, c->fR, c->fbeta, c->feta, c->gamma, c->gbar, c->hp, c->fws, c->st);
        LAUNCHED();
        src = c->gbar;
    }
    if (c->prec == LKS_FP64)
        launch_design_prep<double>(c->d, src, c->cfg.kappa_max, c->cfg.q, (double*)c->kref,
                                   (double*)c->kref_t, (double*)c->kprime, c->flags, c->st);
    else
        launch_design_prep<float>(c->d, src, c->cfg.kappa_max, c->cfg.q, (float*)c->kref,
                                  (float*)c->kref_t, (float*)c->kprime, c->flags, c->st);
    LAUNCHED();
    return LKS_OK;
}

// dJ/dgamma of the last adjoint: the accumulator, or its pull-back through the filter chain.
const double* design_gradient(lks_ctx* c, cudaStream_t st) {
    if (c->fR <= 0.0) return c->gacc;
    launch_filter_T(c->d, c->fR, c->gacc, c->hp, c->fws, c->fq, c->gout, st);
    c->stats[4] += 2;
    return c->gout;
}

// Bytes of so many slots for a box of boxN nodes and ncol design columns, T bytes a number.
size_t tape_bytes(const TapeSlots& t, long long boxN, long long ncol, size_t T) {
    return align256((size_t)t.k * boxN * 4 * T) + align256((size_t)t.e * boxN * T) +
           align256((size_t)t.pos * ncol * 8) + align256((size_t)t.pos * ncol * 4 * T);
}

// The slots that fit p.bytes once the box is known (most boxes are a fraction of the grid, and the more
// slots): the least transfers, positions from a quarter of the rest, then e for those transfers, both for
// more steps, and positions from what is left.
TapeSlots tape_slots(const TapePlan& p, long long boxN, long long ncol, size_t T) {
    TapeSlots t;
    t.k = p.least;
    t.e = t.pos = 1;
    const long long slack = 4 * 256, kb = boxN * 4 * (long long)T, eb = boxN * (long long)T,
                    pb = ncol * (8 + 4 * (long long)T);
    long long left = (long long)p.bytes - (t.k * kb + t.e * eb + t.pos * pb) - slack;
    auto take = [&](int now, int most, long long each, long long room) -> int {
        const long long n = std::max(0LL, std::min((long long)(most - now), room / each));
        left -= n * each;
        return (int)n;
    };
    t.pos += take(t.pos, std::min(p.want, kMaxPosSlots), pb, left / 4);
    t.e += take(t.e, t.k, eb, left);
    const int n = take(t.k, p.want, kb + eb, left);
    t.k += n;
    t.e += n;
    t.pos += take(t.pos, std::min(p.want, kMaxPosSlots), pb, left);
    return t;
}

// After a new motion table: rows with cos/sin evaluated on the host go to the device (the
// instance-table kernels read them there), and a table context rebuilds its one-entry plan.
lks_status finish_motion(lks_ctx* c) {
    const int rows = c->cfg.max_steps + 1;
    std::vector<Motion> mr(rows);
    for (int n = 0; n < rows; ++n) mr[n] = motion_row(c, &c->motion[8 * (size_t)n]);
    CU(cudaMemcpyAsync(c->dmotion, mr.data(), sizeof(Motion) * rows, cudaMemcpyHostToDevice, c->st));
    CU(cudaStreamSynchronize(c->st));
    ++c->geo_gen;
    if (c->fused2d) {
        if (c->d.nd > 0) {
            const size_t T = c->tsz, box = (size_t)c->g.boxN, col = (size_t)c->d.ncol;
            c->slots = tape_slots(c->tape, c->g.boxN, c->d.ncol, T);
            c->ktape = c->tape_mem;
            c->etape = c->tape_mem + align256(c->slots.k * box * 4 * T);
            c->pos_b = (char*)c->etape + align256(c->slots.e * box * T);
            c->pos_sc = (char*)c->pos_b + align256(c->slots.pos * col * 8);
        }
        const lks_status s = own_plan(c);
        if (s != LKS_OK) return s;
    }
    c->have_motion = true;
    return LKS_OK;
}

template cudaError_t build_plan<float>(const std::vector<lks_ctx*>&, void*, int*, int*,
                                      cudaStream_t, Plan&);
template lks_status transfer_at<float>(lks_ctx*, int);
template lks_status transfer_at<double>(lks_ctx*, int);
template lks_status reset_initial<float>(lks_ctx*);
template lks_status reset_initial<double>(lks_ctx*);
template lks_status do_forward<float>(Group&, int);
template lks_status do_forward<double>(Group&, int);
template lks_status do_adjoint<float>(Group&);
template lks_status do_adjoint<double>(Group&);

}  // namespace eng
}  // namespace lks

extern "C" int lks_batch_statuses(const int* words, int n, int* status) {
    if (n < 1 || !words || !status) return -1;
    std::vector<int> w(words, words + 4 * (size_t)n);
    lks::eng::share_waits(w.data(), n);
    for (int k = 0; k < n; ++k) status[k] = (int)lks::eng::word_status(&w[4 * (size_t)k]);
    return n;
}
