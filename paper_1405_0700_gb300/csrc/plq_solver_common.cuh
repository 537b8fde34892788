// Host-side helpers shared by the solver translation units: the launch of
// one hopping half-application inside a solve, reductions read back to the
// host, device solver states and the graph-captured loop of iterations.
#pragma once

#include <cstring>
#include <vector>

#include "plq_fields.cuh"

namespace plq {
namespace {

struct Solve {
    plq_ctx *c;
    cudaStream_t s;  // internal capture-capable stream
    int Vh;
    int n;           // right-hand sides
    long long N;     // elements of a half field: Vh * n
    double kappa;
    int P;   // inner storage precision
    int PX;  // inner solution accumulator precision
    double nu = 0.0;  // twisted mass: nu = 2 kappa mu (0 = Wilson)
    double hops = 0;
    LoopEnd loop;  // of the loop whose pass ends with the iteration being captured
};

// Twisted-mass terms of one hopping launch (all zero / one for Wilson).
struct Tw {
    double nu_x = 0.0, nu_h = 0.0, scale_h = 1.0;
};

Reduce reduce_of(plq_ctx *c, int fin) {
    Reduce r;
    r.partials = c->partials;
    r.ticket = c->ticket;
    r.sums = c->sums;
    r.st = c->state;
    r.fin = fin;
    return r;
}

plq_status hop(Solve &S, int prec, int out_par, void *out, const void *in, int epi, int dagger, const void *x,
               double a, int fin = FIN_NONE, const void *w = nullptr, bool freeze = false, Tw tw = Tw()) {
    plq_ctx *c = S.c;
    HopArgs h;
    h.in = in;
    h.out = out;
    h.x = x;
    h.w = w;
    h.a = a;
    h.gauge = c->gauge[prec].ptr;
    h.gblock = c->gauge[prec].block;
    h.out_parity = out_par;
    h.dagger = dagger;
    h.nrhs = S.n;
    h.lat = c->lat;
    h.red = reduce_of(c, fin);
    if (fin == FIN_NONE) h.red.st = nullptr;
    h.st = freeze ? c->state : nullptr;
    h.nu_x = tw.nu_x;
    h.nu_h = tw.nu_h;
    h.scale_h = tw.scale_h;
    apply_tune(c, prec, S.n, h);
    S.hops += 1;
    return launch_hop(h, prec, c->gauge[prec].reals, epi, S.s);
}

// The two half-applications of Mhat (dagger: Mhat^dagger = gamma5 Mhat(-mu) gamma5):
//   Mhat v = A v - kappa^2 H_eo A^{-1} H_oe v,  A = 1 + i nu gamma5.
Tw tw_first(const Solve &S, bool dag) {  // A^{-1} (or A(-mu)^{-1}) on H_oe v
    Tw t;
    t.nu_h = dag ? S.nu : -S.nu;
    t.scale_h = 1.0 / (1.0 + S.nu * S.nu);
    return t;
}
Tw tw_second(const Solve &S, bool dag) {  // A (or A(-mu)) on the source
    Tw t;
    t.nu_x = dag ? -S.nu : S.nu;
    return t;
}
Tw tw_diag(const Solve &S) {  // A on the xpay source of a full M application
    Tw t;
    t.nu_x = S.nu;
    return t;
}

plq_status read_sums(Solve &S, double *out, int count) {
    PLQ_CUDA(cudaMemcpyAsync(S.c->sums_host, S.c->sums, sizeof(double) * count, cudaMemcpyDeviceToHost, S.s));
    PLQ_CUDA(cudaStreamSynchronize(S.s));
    for (int k = 0; k < count; ++k) out[k] = S.c->sums_host[k];
    return PLQ_OK;
}

// per right-hand side |v|^2 of an FP64 half field
plq_status norm2_64(Solve &S, const void *v, double *out) {
    Reduce r = reduce_of(S.c, FIN_NONE);
    r.st = nullptr;
    PLQ_TRY(blas_norm2(S.N, S.n, v, PLQ_F64, r, S.s));
    return read_sums(S, out, S.n);
}

plq_status put_states(Solve &S, const std::vector<SolverState> &st) {
    std::memcpy(S.c->state_host, st.data(), sizeof(SolverState) * S.n);
    PLQ_CUDA(cudaMemcpyAsync(S.c->state, S.c->state_host, sizeof(SolverState) * S.n, cudaMemcpyHostToDevice, S.s));
    PLQ_CUDA(cudaStreamSynchronize(S.s));
    return PLQ_OK;
}

plq_status get_states(Solve &S, std::vector<SolverState> &st) {
    PLQ_CUDA(cudaMemcpyAsync(S.c->state_host, S.c->state, sizeof(SolverState) * S.n, cudaMemcpyDeviceToHost, S.s));
    PLQ_CUDA(cudaStreamSynchronize(S.s));
    std::memcpy(st.data(), S.c->state_host, sizeof(SolverState) * S.n);
    return PLQ_OK;
}

inline unsigned *loop_word(plq_ctx *c) { return c->ticket + 4; }

// Run `body` (one inner iteration) on the device until the state of every
// right-hand side says stop: the body is captured once into a while node of a
// graph, whose last launch ends the loop (loop_end: at the latest once maxit
// iterations are done).  The instantiated graph is kept in `cache` and reused
// while the key matches; the launches depend only on what the key records.
//
// Batches of 16 captured iterations with a poll of the host after each ran 8
// iterations too many per reliable-update cycle, launches that find everything
// frozen and leave: mixed BiCGstab on 20x12x28x36 (53 of its 80 iterations) 5.37
// -> 4.77 ms, mixed CG on 8^3x16 2.40 -> 2.18 ms, on 24^3x48 no change.  A pass
// of the loop costs a few us beside its launches; one to six iterations per pass:
// CG on 24^3x48 16.25, 16.11, 16.06, 16.08, 16.09 ms (1, 2, 3, 4, 6), CG on 8^3x16
// 2.31, 2.22, 2.18, 2.20, 2.19 ms, BiCGstab 4.84, 4.87, 4.86, 4.91, 4.93 ms.
constexpr int kLoopBody = 3;

template <class Body>
plq_status run_loop(Solve &S, Body body, std::vector<SolverState> &cur, Ctx::SolveGraph &cache, const unsigned long long *key) {
    if (!(cache.exec && std::memcmp(cache.key, key, sizeof(cache.key)) == 0)) {
        cudaGraph_t graph = nullptr, captured = nullptr;
        PLQ_CUDA(cudaGraphCreate(&graph, 0));
        cudaGraphNode_t node = nullptr;
        cudaGraphNodeParams np{};
        np.type = cudaGraphNodeTypeConditional;
        np.conditional.type = cudaGraphCondTypeWhile;
        np.conditional.size = 1;
        cudaError_t e = cudaGraphConditionalHandleCreate(&np.conditional.handle, graph, 1, cudaGraphCondAssignDefault);
        if (e == cudaSuccess) e = cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &np);
        plq_status st = PLQ_OK;
        if (e == cudaSuccess)
            e = cudaStreamBeginCaptureToGraph(S.s, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                              cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            const double hops0 = S.hops;
            for (int i = 0; i < kLoopBody && st == PLQ_OK; ++i) {
                if (i == kLoopBody - 1) S.loop = {np.conditional.handle, loop_word(S.c), kLoopBody};
                st = body();
            }
            S.loop = LoopEnd();
            S.hops = hops0;
            e = cudaStreamEndCapture(S.s, &captured);
        }
        cudaGraphExec_t exec = nullptr;
        if (st == PLQ_OK && e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        if (st != PLQ_OK) return st;
        if (e != cudaSuccess) return cuda_error(e, "solver iteration graph");
        if (cache.exec) cudaGraphExecDestroy(cache.exec);
        cache.exec = exec;
        std::memcpy(cache.key, key, sizeof(cache.key));
    }
    PLQ_CUDA(cudaGraphLaunch(cache.exec, S.s));
    PLQ_TRY(get_states(S, cur));
    for (int r = 0; r < S.n; ++r)
        if (!cur[r].stop) return set_error(PLQ_ERR_STATE, "inner iteration ended before right-hand side %d stopped", r);
    return PLQ_OK;
}

}  // namespace
}  // namespace plq
