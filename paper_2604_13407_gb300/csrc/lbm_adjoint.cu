// Checkpointed adjoint of n steps (host driver of the transposed-step kernels).
//
// J = (1/n) sum_{t=1..n} <W, A_t>, with A_t the stored populations after step t and W
// the weights of the objective.  Reverse-mode differentiation of the time loop:
//
//   lambda_n = W/n,  lambda_t = W/n + Step'(A_t)^T lambda_{t+1}  (t = n-1 .. 1),
//   lambda_0 = Step'(A_0)^T lambda_1,  dJ/dtheta = sum_t (dStep(A_t)/dtheta)^T lambda_{t+1}.
//
// Forward sweep: n steps, each from one buffer straight into another: the states at t = K, 2K, ... are
// written into their checkpoints, the others into scratch (the segment states, not yet in use), A_n
// into the context's buffer that n steps would leave it in (where that is A_0's own, n even, A_0 is
// copied to its checkpoint first).  The steps of the last segment write the segment's states and psi
// fields on the way, so that segment is never recomputed.  <W, A_n> is summed in FP64 there, <W, A_t>
// of the other states by the transposed steps (objective alone: every state in the forward sweep).
// Backward sweep, one segment of K steps at a time from the last: the states of the segment are
// recomputed from its checkpoint with the step kernels the context uses, each leaving the psi field of
// the state it reads in a buffer of its own (the two-pass step's psi pass writes it anyway; the
// one-pass steps write it on request), then the transposed step runs from the last state of the
// segment to the first.  The recompute of a segment runs on a second stream, overlapping the
// transposed steps of the segment after it, so segment states and psi fields come in two sets.  Device
// memory: ceil(n/K) checkpoints, 2 (K - 1) segment states, 2 K psi fields and the adjoint planes; it is
// kept for the next call with the same sizes.  Where two sets cannot be had the call takes one, and
// recomputes a segment after those transposed steps: less than the layout whose transposed step ran
// in two passes over single planes, so what fitted that still fits.
//
// 16-bit storage: a stored state is its nine planes of deviations plus, with a per-node
// reference density, that plane; the recompute repeats the forward steps' stochastic
// rounding (same step seeds).  The transposed step runs in FP32 on the decoded states and
// differentiates the FP32 step through the storage, whose rounding it takes as the
// identity: the gradient of the unrounded step along the trajectory the 16-bit run takes.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <string>
#include <vector>

#include "lbm_adjoint.h"

namespace lbm {

struct AdjointState {
    void *base = nullptr;
    size_t bytes = 0;
    size_t refused = SIZE_MAX;  // the smallest layout with two buffer sets that did not fit
    cudaStream_t side = nullptr;  // recomputes the next segment while the transposed steps run
    cudaEvent_t fork = nullptr, recomputed[2] = {nullptr, nullptr}, reversed[2] = {nullptr, nullptr};
};

void adjoint_free(AdjointState *a)
{
    if (!a) return;
    if (a->side) cudaStreamSynchronize(a->side);
    if (a->base) cudaFree(a->base);
    cudaEvent_t evs[] = {a->fork, a->recomputed[0], a->recomputed[1], a->reversed[0], a->reversed[1]};
    for (cudaEvent_t e : evs)
        if (e) cudaEventDestroy(e);
    if (a->side) cudaStreamDestroy(a->side);
    delete a;
}

namespace {

struct Carver {
    char *p;
    size_t used = 0;
    void *take(size_t bytes)
    {
        void *r = p ? p + used : nullptr;
        used += (bytes + 255) / 256 * 256;
        return r;
    }
};

struct Layout {
    std::vector<void *> ckpt, seg[2], psi[2];  // one or two sets of segment states and psi fields
    void *g[2], *dS[2], *dpsi[2], *rho[2], *psi_r[2];  // psi_r: FP64 only
    double *part;  // per-block partial sums of the transposed steps [blocks][kAdjSlots]
    double *red;   // their column sums (kAdjSlots)
    double *acc;
};

// Sizes of what a call keeps on the device.
struct Sizes {
    int64_t nseg = 0, K = 0;
    bool keep_first = false;  // A_0 needs a checkpoint of its own
    bool psi_planes = false;
    size_t state = 0, plane_r = 0, psi = 0, part = 0;
};

size_t carve(Carver &cv, Layout &L, const Sizes &z, int sets)
{
    L.ckpt.assign(z.nseg, nullptr);
    for (int64_t s = z.keep_first ? 0 : 1; s < z.nseg; ++s) L.ckpt[s] = cv.take(z.state);
    for (int q = 0; q < sets; ++q) {
        L.seg[q].resize(z.K > 0 ? z.K - 1 : 0);
        L.psi[q].resize(z.K);
        for (auto &b : L.seg[q]) b = cv.take(z.state);
        for (auto &b : L.psi[q]) b = cv.take(z.psi);
    }
    for (int s = 0; s < 2; ++s) {
        L.g[s] = cv.take(9 * z.plane_r);
        L.dS[s] = cv.take(2 * z.plane_r);
        L.dpsi[s] = cv.take(z.plane_r);
        L.rho[s] = cv.take(z.plane_r);
        L.psi_r[s] = z.psi_planes ? cv.take(z.plane_r) : nullptr;
    }
    L.part = static_cast<double *>(cv.take(z.part));
    L.red = static_cast<double *>(cv.take(kAdjSlots * sizeof(double)));
    L.acc = static_cast<double *>(cv.take(8 * sizeof(double)));
    return cv.used;
}

}  // namespace

#define ACK(call, what)                                                      \
    do {                                                                     \
        cudaError_t e_ = (call);                                             \
        if (e_ != cudaSuccess) {                                             \
            msg = std::string(what) + ": " + cudaGetErrorString(e_);         \
            return e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA; \
        }                                                                    \
    } while (0)

lbm_status adjoint_run(lbm_ctx *ctx, int64_t nsteps, int32_t K, int32_t objective, double *J, double *grad,
                       double *lambda0, std::string &msg)
{
    ContextView v = view_of(ctx);
    const lbm_params &p = *v.p;
    if (!v.L->adj_step) {
        msg = "no transposed step for this storage type";
        return LBM_ENOTSUP;
    }
    if (v.kp->wall_u || v.kp->q || v.kp->wall_rho) {
        msg = "the adjoint supports resting half-way walls with one virtual density only";
        return LBM_ENOTSUP;
    }
    if (p.force_mode == LBM_FORCE_FIELD) {
        msg = "the adjoint supports CONST and BUOYANT forces only";
        return LBM_ENOTSUP;
    }
    if (nsteps < 1 || K < 1 || (objective != LBM_OBJ_WALL_FORCE_Y && objective != LBM_OBJ_MEAN_JX)) {
        msg = "nsteps and checkpoint_every must be >= 1 and objective one of lbm_objective";
        return LBM_EINVAL;
    }
    if (v.n_fluid < 1) {
        msg = "no fluid node";
        return LBM_EINVAL;
    }
    cudaStream_t st = v.stream;
    const int64_t nseg = (nsteps + K - 1) / K;
    const int64_t Kseg = std::min<int64_t>(K, nsteps);
    // a stored state: the nine planes, then the per-node reference plane of 16-bit storage
    const size_t pop_bytes = (size_t)9 * v.plane * v.elem;
    const size_t ref_bytes = v.refp[0] ? (size_t)v.plane * sizeof(float) : 0;
    const size_t ref_at = (pop_bytes + 255) / 256 * 256;
    const size_t state_bytes = ref_bytes ? ref_at + ref_bytes : pop_bytes;
    auto ref_of = [&](const void *state) -> float * {
        return ref_bytes ? reinterpret_cast<float *>(const_cast<char *>(static_cast<const char *>(state)) + ref_at)
                         : nullptr;
    };
    const size_t real = v.elem == 8 ? 8 : 4;  // arithmetic type: FP64 for FP64 storage, FP32 otherwise
    const size_t plane_r = (size_t)v.plane * real;
    const size_t psi_bytes = (size_t)p.nx * p.ny * real;
    const size_t part_bytes = (size_t)v.L->adj_blocks(*v.kp) * kAdjSlots * sizeof(double);

    // grad == NULL and lambda0 == NULL: the objective alone (forward sweep only)
    const bool backward = grad != nullptr || lambda0 != nullptr;

    // Device memory, kept across calls: two buffer sets, so that a segment is recomputed beside the transposed
    // steps of the one after it; one where there is a single segment or the memory for two cannot be had.
    Sizes z;
    if (backward) {
        z.nseg = nseg, z.K = Kseg;
        z.keep_first = nsteps % 2 == 0;
        z.psi_planes = real == 8;
        z.state = state_bytes, z.plane_r = plane_r, z.psi = psi_bytes, z.part = part_bytes;
    }
    Layout L;
    int sets = nseg > 1 && backward ? 2 : 1;
    auto need = [&](int q) {
        Carver probe{nullptr};
        return carve(probe, L, z, q);
    };
    AdjointState *&as = *v.adj;
    if (!as) as = new AdjointState();
    if (sets == 2 && need(2) >= as->refused) sets = 1;
    while (as->bytes < need(sets)) {
        if (as->base) {
            cudaStreamSynchronize(st);
            cudaFree(as->base);
            as->base = nullptr;
            as->bytes = 0;
        }
        const size_t bytes = need(sets);
        cudaError_t e = cudaMalloc(&as->base, bytes);
        if (e == cudaSuccess) {
            as->bytes = bytes;
        } else {
            cudaGetLastError();
            as->base = nullptr;
            if (sets == 1) {
                msg = "adjoint: cudaMalloc of " + std::to_string(bytes >> 20) +
                      " MiB for checkpoints and segment states failed (lower checkpoint_every)";
                return LBM_ENOMEM;
            }
            as->refused = bytes;
            sets = 1;
        }
    }
    Carver cv{static_cast<char *>(as->base)};
    carve(cv, L, z, sets);
    if (sets == 2 && !as->side) {
        ACK(cudaStreamCreateWithFlags(&as->side, cudaStreamNonBlocking), "cudaStreamCreate");
        cudaEvent_t *evs[] = {&as->fork, &as->recomputed[0], &as->recomputed[1], &as->reversed[0], &as->reversed[1]};
        for (cudaEvent_t *e : evs) ACK(cudaEventCreateWithFlags(e, cudaEventDisableTiming), "cudaEventCreate");
    }

    const double inv_nfluid = 1.0 / double(v.n_fluid);
    const double w = 1.0 / double(nsteps);
    ACK(cudaMemsetAsync(L.acc, 0, 8 * sizeof(double), st), "memset");
    if (backward) ACK(cudaMemsetAsync(L.part, 0, part_bytes, st), "memset");

    // ---- forward sweep: checkpoints and the objective
    KParams kq = *v.kp;
    const int64_t step0 = *v.steps;  // the forward sweep's step t runs as the context's step step0 + t
    auto set_of = [&](int64_t s) { return sets == 2 ? (int)(s & 1) : 0; };  // buffer set of a segment
    const int last_q = set_of(nseg - 1);
    // One step of the context's kernel from one state buffer to another, leaving psi of the state it
    // reads in `psi` (null: where the context keeps it).
    auto step_to = [&](const void *src, const float *ref, void *dst, float *ref_dst, void *psi, int64_t t,
                       cudaStream_t on) -> lbm_status {
        KParams kp = *v.kp;
        kp.src = src, kp.ref_src = ref, kp.dst = dst, kp.ref_dst = ref_dst;
        kp.sr_seed = v.sr_seed(step0 + t);
        if (v.fused_pass) {
            kp.psi_out = psi;
            ACK(v.fused_pass(kp, on), "one-pass step kernel");
        } else {
            if (psi) kp.psi = psi;
            ACK(v.psi_pass(kp, on), "psi kernel");
            ACK(v.collide_pass(kp, on), "collide kernel");
        }
        return LBM_OK;
    };
    const void *first = nullptr;  // A_0 (during the backward sweep)
    const float *first_ref = nullptr;
    if (backward) {
        const int from = *v.cur, to = from ^ (int)(nsteps & 1);
        const void *src = v.pops[from];
        const float *src_ref = v.refp[from];
        if (to == from) {
            ACK(cudaMemcpyAsync(L.ckpt[0], src, pop_bytes, cudaMemcpyDeviceToDevice, st), "checkpoint copy");
            if (ref_bytes)
                ACK(cudaMemcpyAsync(ref_of(L.ckpt[0]), src_ref, ref_bytes, cudaMemcpyDeviceToDevice, st), "checkpoint copy");
            src = L.ckpt[0], src_ref = ref_of(src);
        }
        first = src, first_ref = src_ref;
        for (int64_t t = 0; t < nsteps; ++t) {
            const int64_t s = t / K, at = t - s * K;
            const bool last = s == nseg - 1;
            void *dst;
            float *dst_ref;
            if (t == nsteps - 1) {
                dst = v.pops[to], dst_ref = v.refp[to];
            } else {
                dst = (t + 1) % K == 0 ? L.ckpt[s + 1] : last ? L.seg[last_q][at] : L.seg[0][at & 1];
                dst_ref = ref_of(dst);
            }
            const lbm_status r = step_to(src, src_ref, dst, dst_ref, last ? L.psi[last_q][at] : nullptr, t, st);
            if (r != LBM_OK) return r;
            src = dst, src_ref = dst_ref;
        }
        *v.cur = to;
        *v.steps += nsteps;
        v.kp->sr_seed = v.sr_seed(step0 + nsteps - 1);  // as n calls of lbm_step leave it
        // <W, A_t> of t = 1 .. n-1 is summed by the transposed steps, which read those states anyway
        kq.src = src;
        kq.ref_src = src_ref;
        ACK(v.L->objective(kq, objective, inv_nfluid, L.acc, st), "objective kernel");
    } else {
        for (int64_t t = 0; t < nsteps; ++t) {
            lbm_status s = v.run_steps(ctx, 1);
            if (s != LBM_OK) {
                msg = "forward step failed";
                return s;
            }
            kq.src = v.pops[*v.cur];
            kq.ref_src = v.refp[*v.cur];
            ACK(v.L->objective(kq, objective, inv_nfluid, L.acc, st), "objective kernel");
        }
    }

    if (!backward) {
        double h0;
        ACK(cudaMemcpyAsync(&h0, L.acc, sizeof h0, cudaMemcpyDeviceToHost, st), "D2H");
        ACK(cudaStreamSynchronize(st), "objective");
        *J = h0 * w;
        return v.check_error(ctx, msg);
    }

    // ---- backward sweep
    AdjArgs aa{};
    aa.w_scale = w;
    aa.w_scale_f = float(w);
    aa.objective = objective;
    aa.inv_nfluid = inv_nfluid;
    aa.inv_nfluid_f = float(inv_nfluid);
    aa.part = L.part;
    int gi = 0;  // set of planes the last transposed step left; none before the first
    bool have_next = false;
    auto bind_in = [&]() {
        aa.g_in = L.g[gi], aa.dS_in = L.dS[gi], aa.dpsi_in = L.dpsi[gi], aa.rho_in = L.rho[gi], aa.psi_in = L.psi_r[gi];
    };
    // psi, the 16-bit reference plane and the stored state A_t of segment s, buffer set q
    auto state_at = [&](int64_t s, int q, int64_t t, const float **ref) -> const void * {
        if (t == 0) {
            *ref = first_ref;
            return first;
        }
        const void *p = t == s * K ? L.ckpt[s] : L.seg[q][t - s * K - 1];
        *ref = ref_of(p);
        return p;
    };
    // With two buffer sets segment s is recomputed on the side stream into set s & 1 while the
    // transposed steps of segment s + 1 run on the context stream from set (s + 1) & 1; events order a
    // set's reuse after the transposed steps that read it.  With one it is recomputed after them, on the
    // context stream.
    const cudaStream_t on = sets == 2 ? as->side : st;
    auto recompute = [&](int64_t s) -> lbm_status {
        const int q = set_of(s);
        const int64_t t0 = s * K, t1 = std::min<int64_t>((s + 1) * K, nsteps);
        if (sets == 2 && s + 2 < nseg) ACK(cudaStreamWaitEvent(as->side, as->reversed[q], 0), "event wait");
        for (int64_t t = t0; t < t1; ++t) {
            const float *ref;
            const void *src = state_at(s, q, t, &ref);
            if (t + 1 < t1) {
                void *dst = L.seg[q][t - t0];
                const lbm_status r = step_to(src, ref, dst, ref_of(dst), L.psi[q][t - t0], t, on);
                if (r != LBM_OK) return r;
            } else {
                KParams kp = *v.kp;
                kp.src = src, kp.ref_src = ref, kp.psi = L.psi[q][t - t0];
                ACK(v.psi_pass(kp, on), "psi kernel");
            }
        }
        if (sets == 2) ACK(cudaEventRecord(as->recomputed[q], on), "event record");
        return LBM_OK;
    };
    if (sets == 2) {
        ACK(cudaEventRecord(as->fork, st), "event record");
        ACK(cudaStreamWaitEvent(as->side, as->fork, 0), "event wait");
    }
    lbm_status rs;
    for (int64_t s = nseg - 1; s >= 0; --s) {
        const int q = set_of(s);
        const int64_t t0 = s * K, t1 = std::min<int64_t>((s + 1) * K, nsteps);
        if (sets == 2 && s > 0 && (rs = recompute(s - 1)) != LBM_OK) return rs;
        if (sets == 2 && s < nseg - 1) ACK(cudaStreamWaitEvent(st, as->recomputed[q], 0), "event wait");
        KParams kp = *v.kp;
        for (int64_t t = t1 - 1; t >= t0; --t) {
            kp.src = state_at(s, q, t, &kp.ref_src);
            kp.psi = L.psi[q][t - t0];
            if (have_next) bind_in();
            const int go = gi ^ 1;
            aa.g_out = L.g[go], aa.dS_out = L.dS[go], aa.dpsi_out = L.dpsi[go], aa.rho_out = L.rho[go], aa.psi_out = L.psi_r[go];
            aa.sum_J = t >= 1;  // <W, A_0> is not part of J
            ACK(v.L->adj_step(kp, aa, st), "transposed step");
            gi = go;
            have_next = true;
        }
        if (sets == 2) ACK(cudaEventRecord(as->reversed[q], st), "event record");
        if (sets == 1 && s > 0 && (rs = recompute(s - 1)) != LBM_OK) return rs;
    }

    bind_in();
    aa.tail = 1;
    void *const c = aa.c_out = L.g[gi ^ 1];  // (its own planes are the last ones read)
    ACK(v.L->adj_step(*v.kp, aa, st), "transposed step's tail");
    if (lambda0) {
        const size_t n = (size_t)p.nx * p.ny;
        double *dl = nullptr;
        ACK(cudaMalloc((void **)&dl, 9 * n * sizeof(double)), "cudaMalloc(lambda0)");
        cudaError_t e = v.L->adj_lambda(*v.kp, L.g[gi], c, dl, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(lambda0, dl, 9 * n * sizeof(double), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        cudaFree(dl);
        ACK(e, "lambda0");
    }
    ACK(v.L->adj_reduce(*v.kp, L.part, L.red, st), "adjoint reduction");
    double h[8], r[kAdjSlots];
    ACK(cudaMemcpyAsync(h, L.acc, sizeof h, cudaMemcpyDeviceToHost, st), "D2H");
    ACK(cudaMemcpyAsync(r, L.red, sizeof r, cudaMemcpyDeviceToHost, st), "D2H");
    ACK(cudaStreamSynchronize(st), "adjoint");
    *J = (h[0] + r[SLOT_J]) * w;
    if (grad) {
        grad[0] = r[SLOT_FX];
        grad[1] = r[SLOT_FY];
        grad[2] = r[SLOT_G1] + r[SLOT_G2];
        grad[3] = r[SLOT_T1] + r[SLOT_T2];
    }
    return v.check_error(ctx, msg);
}

}  // namespace lbm
