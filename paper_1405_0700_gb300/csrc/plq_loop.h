// When the solvers' iteration loop on the device (the while node of a graph, see
// run_loop) ends: once every right-hand side has stopped, and in any case after the
// pass that completes `maxit` iterations.  The count does not depend on the
// reductions whose finalize step sets the stop flags, so the loop ends even where
// that step never runs (two solves that overlap on one context, which is not
// allowed, take each other's tickets); the host reports such an end as an error.  A
// sound solve never sees it: its right-hand sides stop by iteration
// maxit - (iterations before this loop).
//
// The header is plain C++ (usable by host compilers and nvcc alike).
#pragma once

#if defined(__CUDACC__)
#define PLQ_LOOP_HD __host__ __device__ __forceinline__
#else
#define PLQ_LOOP_HD inline
#endif

namespace plq {

// done: iterations of this loop, those of the pass that ends included.
PLQ_LOOP_HD bool loop_over(unsigned done, int maxit, bool all_stopped) {
    return all_stopped || maxit < 1 || done >= (unsigned)maxit;
}

}  // namespace plq
