// Device-side access to packed fields: complex arithmetic, spinor and link
// loads/stores in FP64, FP32 and FP16 storage, and block reductions.
#pragma once

#include "plq_internal.cuh"
#include "plq_loop.h"

namespace plq {

template <class R>
struct cx {
    R re, im;
};

template <class R>
__device__ __forceinline__ cx<R> cadd(cx<R> a, cx<R> b) { return {a.re + b.re, a.im + b.im}; }
template <class R>
__device__ __forceinline__ cx<R> csub(cx<R> a, cx<R> b) { return {a.re - b.re, a.im - b.im}; }
template <class R>
__device__ __forceinline__ cx<R> cscale(R s, cx<R> a) { return {s * a.re, s * a.im}; }
template <class R>
__device__ __forceinline__ cx<R> cconj(cx<R> a) { return {a.re, -a.im}; }

// a*b + c
template <class R>
__device__ __forceinline__ cx<R> cfma(cx<R> a, cx<R> b, cx<R> c) {
    c.re = fma(a.re, b.re, c.re);
    c.re = fma(-a.im, b.im, c.re);
    c.im = fma(a.re, b.im, c.im);
    c.im = fma(a.im, b.re, c.im);
    return c;
}
// conj(a)*b + c
template <class R>
__device__ __forceinline__ cx<R> cfma_conj(cx<R> a, cx<R> b, cx<R> c) {
    c.re = fma(a.re, b.re, c.re);
    c.re = fma(a.im, b.im, c.re);
    c.im = fma(a.re, b.im, c.im);
    c.im = fma(-a.im, b.re, c.im);
    return c;
}

// z * i^K for K = 0..3 (+1, +i, -1, -i): no multiplications.
template <int K, class R>
__device__ __forceinline__ cx<R> mul_ipow(cx<R> z) {
    if constexpr ((K & 3) == 0) return z;
    else if constexpr ((K & 3) == 1) return {-z.im, z.re};
    else if constexpr ((K & 3) == 2) return {-z.re, -z.im};
    else return {z.im, -z.re};
}

// ---------------------------------------------------------------- launches
// Kernels of a chain begin with chain_begin() and are launched by
// launch_chained (programmatic dependent launch): the next kernel's blocks start
// once this one's have all left, and wait for its memory, instead of being launched
// after it.  No kernel lets its dependents go earlier (griddepcontrol.
// launch_dependents): with that at the start of a kernel, the third kernel of a
// chain could be resident while the first still ran, and read-only loads (__ldg)
// are not kept coherent over a kernel's life; the waiting blocks also took the SMs
// unevenly (FP64 plq_schur_apply, 8^4 48.5 -> 19.9 us without, 16x8^2x16 51.3 ->
// 35.6; FP32 16^4 12-real 16.6 -> 11.7, 24^3x48 67.7 -> 65.2 us; with it behind the
// last site instead: 24^3x48 74.0 us).
__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_chained(bool chained, void (*kern)(P...), dim3 grid, dim3 block, cudaStream_t s, A &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

// ---------------------------------------------------------------- loads
// Read-only, L1-cacheable (neighbour spinors are reused by up to 8 sites).
__device__ __forceinline__ float4 ld_nc(const float4 *p) { return __ldg(p); }
__device__ __forceinline__ double2 ld_nc(const double2 *p) { return __ldg(p); }
__device__ __forceinline__ uint4 ld_nc(const uint4 *p) { return __ldg(p); }
__device__ __forceinline__ float ld_nc(const float *p) { return __ldg(p); }
// Streaming (evict-first): links are read exactly once per half-apply.
__device__ __forceinline__ float4 ld_stream(const float4 *p) { return __ldcs(p); }
__device__ __forceinline__ float2 ld_stream(const float2 *p) { return __ldcs(p); }
__device__ __forceinline__ double2 ld_stream(const double2 *p) { return __ldcs(p); }
__device__ __forceinline__ uint4 ld_stream(const uint4 *p) { return __ldcs(p); }
__device__ __forceinline__ uint2 ld_stream(const uint2 *p) { return __ldcs(p); }
__device__ __forceinline__ unsigned ld_stream(const unsigned *p) { return __ldcs(p); }

template <int P>
struct Real_;
template <>
struct Real_<PLQ_F64> {
    using T = double;
};
template <>
struct Real_<PLQ_F32> {
    using T = float;
};
template <>
struct Real_<PLQ_F16> {
    using T = float;
};
template <int P>
using RealOf = typename Real_<P>::T;

__device__ __forceinline__ float2 h2f(unsigned u) {
    __half2 h = *reinterpret_cast<__half2 *>(&u);
    return __half22float2(h);
}
__device__ __forceinline__ unsigned f2h(float a, float b) {
    __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<unsigned *>(&h);
}

// Packed half field: 12 complex components per site and rhs.
// `stride` = Vh * nrhs (elements of one plane); `e` = site * nrhs + rhs.
template <int P>
struct Spinor;

template <>
struct Spinor<PLQ_F64> {
    __device__ static void load(const void *base, size_t stride, size_t e, cx<double> v[12]) {
        const double2 *p = static_cast<const double2 *>(base) + e;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            double2 t = ld_nc(p + k * stride);
            v[k] = {t.x, t.y};
        }
    }
    __device__ static void store(void *base, size_t stride, size_t e, const cx<double> v[12]) {
        double2 *p = static_cast<double2 *>(base) + e;
#pragma unroll
        for (int k = 0; k < 12; ++k) __stcs(p + k * stride, make_double2(v[k].re, v[k].im));
    }
};

template <>
struct Spinor<PLQ_F32> {
    __device__ static void load(const void *base, size_t stride, size_t e, cx<float> v[12]) {
        const float4 *p = static_cast<const float4 *>(base) + e;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            float4 t = ld_nc(p + k * stride);
            v[2 * k] = {t.x, t.y};
            v[2 * k + 1] = {t.z, t.w};
        }
    }
    __device__ static void store(void *base, size_t stride, size_t e, const cx<float> v[12]) {
        float4 *p = static_cast<float4 *>(base) + e;
#pragma unroll
        for (int k = 0; k < 6; ++k)
            __stcs(p + k * stride, make_float4(v[2 * k].re, v[2 * k].im, v[2 * k + 1].re, v[2 * k + 1].im));
    }
};

template <>
struct Spinor<PLQ_F16> {
    // 3 planes of uint4 (8 halves), then stride floats of norms.
    __device__ static void load(const void *base, size_t stride, size_t e, cx<float> v[12]) {
        const uint4 *p = static_cast<const uint4 *>(base) + e;
        const float *nrm = reinterpret_cast<const float *>(static_cast<const uint4 *>(base) + 3 * stride);
        const float n = ld_nc(nrm + e);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            uint4 t = ld_nc(p + k * stride);
            float2 a = h2f(t.x), b = h2f(t.y), c = h2f(t.z), d = h2f(t.w);
            v[4 * k + 0] = {a.x * n, a.y * n};
            v[4 * k + 1] = {b.x * n, b.y * n};
            v[4 * k + 2] = {c.x * n, c.y * n};
            v[4 * k + 3] = {d.x * n, d.y * n};
        }
    }
    // The stored (normalised) components and the site norm separately: the
    // hopping kernel projects first and scales the 6 projected components
    // instead of the 12 loaded ones.
    __device__ static float load_unscaled(const void *base, size_t stride, size_t e, cx<float> v[12]) {
        const uint4 *p = static_cast<const uint4 *>(base) + e;
        const float *nrm = reinterpret_cast<const float *>(static_cast<const uint4 *>(base) + 3 * stride);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            uint4 t = ld_nc(p + k * stride);
            float2 a = h2f(t.x), b = h2f(t.y), c = h2f(t.z), d = h2f(t.w);
            v[4 * k + 0] = {a.x, a.y};
            v[4 * k + 1] = {b.x, b.y};
            v[4 * k + 2] = {c.x, c.y};
            v[4 * k + 3] = {d.x, d.y};
        }
        return ld_nc(nrm + e);
    }
    // Site norm of v, and its inverse (0 for a site stored as zero).
    __device__ static float site_norm(const cx<float> v[12], float &inv) {
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < 12; ++k) m = fmaxf(m, fmaxf(fabsf(v[k].re), fabsf(v[k].im)));
        // A site whose largest component is below the smallest normal float
        // (2^-126) is stored as zero: 1/m would overflow to infinity.  Such
        // sites occur at the edge of the support of the early Krylov vectors
        // of a point source, many orders of magnitude below the field's norm.
        constexpr float kMinNormal = 1.17549435e-38f;
        if (!(m >= kMinNormal)) m = 0.f;
        inv = m > 0.f ? 1.0f / m : 0.f;
        return m;
    }
    __device__ static uint4 halves(const cx<float> v[4], float inv) {
        uint4 t;
        t.x = f2h(v[0].re * inv, v[0].im * inv);
        t.y = f2h(v[1].re * inv, v[1].im * inv);
        t.z = f2h(v[2].re * inv, v[2].im * inv);
        t.w = f2h(v[3].re * inv, v[3].im * inv);
        return t;
    }
    __device__ static void store(void *base, size_t stride, size_t e, const cx<float> v[12]) {
        uint4 *p = static_cast<uint4 *>(base) + e;
        float inv;
        const float m = site_norm(v, inv);
#pragma unroll
        for (int k = 0; k < 3; ++k) __stcs(p + k * stride, halves(v + 4 * k, inv));
        __stcs(reinterpret_cast<float *>(static_cast<uint4 *>(base) + 3 * stride) + e, m);
    }
    // The same store written out.  The compiler (nvcc 13.0) schedules hop_kernel differently
    // around the two forms: 18-real links are faster with this one (32^3x64 77.1
    // against 79.7 us, plq_wilson_apply on 24^3x48 54.2 against 62.1 us), 12-real
    // ones with the other (83.9 against 76.7 us) but for the xpay epilogue
    // (plq_wilson_apply 59.3 against 61.4 us).
    __device__ static void store_flat(void *base, size_t stride, size_t e, const cx<float> v[12]) {
        uint4 *p = static_cast<uint4 *>(base) + e;
        float *nrm = reinterpret_cast<float *>(static_cast<uint4 *>(base) + 3 * stride);
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < 12; ++k) m = fmaxf(m, fmaxf(fabsf(v[k].re), fabsf(v[k].im)));
        constexpr float kMinNormal = 1.17549435e-38f;  // (see site_norm)
        if (!(m >= kMinNormal)) m = 0.f;
        const float inv = m > 0.f ? 1.0f / m : 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            uint4 t;
            t.x = f2h(v[4 * k + 0].re * inv, v[4 * k + 0].im * inv);
            t.y = f2h(v[4 * k + 1].re * inv, v[4 * k + 1].im * inv);
            t.z = f2h(v[4 * k + 2].re * inv, v[4 * k + 2].im * inv);
            t.w = f2h(v[4 * k + 3].re * inv, v[4 * k + 3].im * inv);
            __stcs(p + k * stride, t);
        }
        __stcs(nrm + e, m);
    }
    // One of the three planes (plane 0 with the norm).
    __device__ static void store_plane(void *base, size_t stride, size_t e, const cx<float> v[12], int k) {
        float inv;
        const float m = site_norm(v, inv);
        const cx<float> q[4] = {k == 0 ? v[0] : k == 1 ? v[4] : v[8], k == 0 ? v[1] : k == 1 ? v[5] : v[9],
                                k == 0 ? v[2] : k == 1 ? v[6] : v[10], k == 0 ? v[3] : k == 1 ? v[7] : v[11]};
        static_cast<uint4 *>(base)[k * stride + e] = halves(q, inv);
        if (k == 0) reinterpret_cast<float *>(static_cast<uint4 *>(base) + 3 * stride)[e] = m;
    }
};

// ---------------------------------------------------------------- links
// One (parity, mu) block of Vh links.  Complex element (row, col) = row*3 + col.
template <int P, int R>
struct Link;

template <class T>
__device__ __forceinline__ void reconstruct_row2(cx<T> u[3][3]) {
    // row2 = conj(row0 x row1): the third row of an SU(3) matrix.
    u[2][0] = cconj(csub(cfma(u[0][1], u[1][2], cx<T>{0, 0}), cfma(u[0][2], u[1][1], cx<T>{0, 0})));
    u[2][1] = cconj(csub(cfma(u[0][2], u[1][0], cx<T>{0, 0}), cfma(u[0][0], u[1][2], cx<T>{0, 0})));
    u[2][2] = cconj(csub(cfma(u[0][0], u[1][1], cx<T>{0, 0}), cfma(u[0][1], u[1][0], cx<T>{0, 0})));
}

template <int R>
struct Link<PLQ_F64, R> {
    __device__ static void load(const void *blk, int Vh, int i, cx<double> u[3][3]) {
        const double2 *p = static_cast<const double2 *>(blk) + i;
        constexpr int n = R / 2;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            double2 t = ld_stream(p + (size_t)k * Vh);
            u[k / 3][k % 3] = {t.x, t.y};
        }
        if constexpr (R == 12) reconstruct_row2(u);
    }
};

template <>
struct Link<PLQ_F32, 18> {
    __device__ static void load(const void *blk, int Vh, int i, cx<float> u[3][3]) {
        const float4 *p = static_cast<const float4 *>(blk) + i;
        cx<float> c[9];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float4 t = ld_stream(p + (size_t)k * Vh);
            c[2 * k] = {t.x, t.y};
            c[2 * k + 1] = {t.z, t.w};
        }
        float2 t = ld_stream(reinterpret_cast<const float2 *>(static_cast<const float4 *>(blk) + 4 * (size_t)Vh) + i);
        c[8] = {t.x, t.y};
#pragma unroll
        for (int k = 0; k < 9; ++k) u[k / 3][k % 3] = c[k];
    }
};

template <>
struct Link<PLQ_F32, 12> {
    __device__ static void load(const void *blk, int Vh, int i, cx<float> u[3][3]) {
        const float4 *p = static_cast<const float4 *>(blk) + i;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float4 t = ld_stream(p + (size_t)k * Vh);
            u[(2 * k) / 3][(2 * k) % 3] = {t.x, t.y};
            u[(2 * k + 1) / 3][(2 * k + 1) % 3] = {t.z, t.w};
        }
        reconstruct_row2(u);
    }
};

template <>
struct Link<PLQ_F16, 18> {
    // 2 planes of uint4 (complex 0..3, 4..7) + 1 plane of half2 (complex 8)
    __device__ static void load(const void *blk, int Vh, int i, cx<float> u[3][3]) {
        const uint4 *p = static_cast<const uint4 *>(blk) + i;
        cx<float> c[9];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            uint4 t = ld_stream(p + (size_t)k * Vh);
            float2 a = h2f(t.x), b = h2f(t.y), d = h2f(t.z), e = h2f(t.w);
            c[4 * k] = {a.x, a.y};
            c[4 * k + 1] = {b.x, b.y};
            c[4 * k + 2] = {d.x, d.y};
            c[4 * k + 3] = {e.x, e.y};
        }
        float2 t = h2f(ld_stream(reinterpret_cast<const unsigned *>(static_cast<const uint4 *>(blk) + 2 * (size_t)Vh) + i));
        c[8] = {t.x, t.y};
#pragma unroll
        for (int k = 0; k < 9; ++k) u[k / 3][k % 3] = c[k];
    }
};

template <>
struct Link<PLQ_F16, 12> {
    // 1 plane of uint4 (complex 0..3) + 1 plane of uint2 (complex 4, 5)
    __device__ static void load(const void *blk, int Vh, int i, cx<float> u[3][3]) {
        const uint4 *p = static_cast<const uint4 *>(blk) + i;
        uint4 t = ld_stream(p);
        uint2 q = ld_stream(reinterpret_cast<const uint2 *>(static_cast<const uint4 *>(blk) + (size_t)Vh) + i);
        float2 a = h2f(t.x), b = h2f(t.y), d = h2f(t.z), e = h2f(t.w), f = h2f(q.x), g = h2f(q.y);
        u[0][0] = {a.x, a.y};
        u[0][1] = {b.x, b.y};
        u[0][2] = {d.x, d.y};
        u[1][0] = {e.x, e.y};
        u[1][1] = {f.x, f.y};
        u[1][2] = {g.x, g.y};
        reconstruct_row2(u);
    }
};

// ---------------------------------------------------------------- reductions
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
    const double d = b.x * b.x + b.y * b.y;
    return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ bool finite2(double2 a) { return isfinite(a.x) && isfinite(a.y); }

// Finalize step of one right-hand side's reduction: update its solver
// scalars from the grid totals tot[0..NV).  The state is read, changed and
// written back as a whole: its fields are then one L2 round trip, not one for
// every field that a store to another might alias.
__device__ __forceinline__ void finalize_one(int fin, SolverState *state, const double *tot) {
    SolverState z = *state, *st = &z;
    // A frozen right-hand side contributed nothing to this reduction: its
    // scalars must not change (its last update of x and p has been made).
    if (st->stop) {
        if (fin == FIN_CG_ALPHA) state->xpend = 0;
        return;
    }
    switch (fin) {
    case FIN_CG_ALPHA:
        // an iteration that ends here (alpha not finite) updates neither x nor p
        st->xpend = 0;
        st->pAp = tot[0];
        st->alpha = st->rho / tot[0];
        st->alpha32 = (float)st->alpha;
        if (!isfinite(st->alpha)) { st->flags |= FLAG_NAN; st->stop = 1; }
        if (st->hist && st->iter < st->hist_cap) st->hist[3 * st->iter] = st->alpha;
        break;
    case FIN_CG_BETA:
        st->rho_new = tot[0];
        st->beta = tot[0] / st->rho;
        st->beta32 = (float)st->beta;
        st->rho = tot[0];
        st->xpend = 1;
        if (st->hist && st->iter < st->hist_cap) {
            st->hist[3 * st->iter + 1] = st->beta;
            st->hist[3 * st->iter + 2] = tot[0];
        }
        st->iter += 1;
        if (!isfinite(tot[0])) { st->flags |= FLAG_NAN; st->stop = 1; }
        else if (tot[0] <= st->stop_r2 || st->iter >= st->maxit) st->stop = 1;
        break;
    case FIN_BICG_ALPHA: {
        st->rv = make_double2(tot[0], tot[1]);
        const double m = fabs(tot[0]) + fabs(tot[1]);
        if (!(m > st->tiny)) { st->flags |= (isfinite(m) ? FLAG_BREAKDOWN : FLAG_NAN); st->stop = 1; break; }
        st->c_alpha = cdiv(st->c_rho, st->rv);
        st->c_alpha32 = make_float2((float)st->c_alpha.x, (float)st->c_alpha.y);
        break;
    }
    case FIN_BICG_OMEGA:
        st->ts = make_double2(tot[0], tot[1]);
        st->tt = tot[2];
        if (!(tot[2] > 0.0) || !finite2(st->ts)) {
            st->flags |= (isfinite(tot[2]) && finite2(st->ts) ? FLAG_BREAKDOWN : FLAG_NAN);
            st->stop = 1;
            break;
        }
        st->c_omega = make_double2(tot[0] / tot[2], tot[1] / tot[2]);
        st->c_omega32 = make_float2((float)st->c_omega.x, (float)st->c_omega.y);
        if (fabs(st->c_omega.x) + fabs(st->c_omega.y) == 0.0) { st->flags |= FLAG_BREAKDOWN; st->stop = 1; }
        break;
    case FIN_BICG_RHO: {
        const double2 rn = make_double2(tot[0], tot[1]);
        st->r2 = tot[2];
        st->iter += 1;
        if (!finite2(rn) || !isfinite(tot[2])) { st->flags |= FLAG_NAN; st->stop = 1; break; }
        if (tot[2] <= st->stop_r2 || st->iter >= st->maxit) { st->stop = 1; st->c_rho_new = rn; break; }
        if (!(fabs(rn.x) + fabs(rn.y) > 0.0)) { st->flags |= FLAG_BREAKDOWN; st->stop = 1; break; }
        st->c_beta = cmul(cdiv(rn, st->c_rho), cdiv(st->c_alpha, st->c_omega));
        st->c_beta32 = make_float2((float)st->c_beta.x, (float)st->c_beta.y);
        st->c_rho = rn;
        st->c_rho_new = rn;
        break;
    }
    default:
        break;
    }
    *state = z;
}

// Per-thread FP64 accumulator of NV sums for the RT right-hand sides a thread
// always handles: those of its right-hand-side column c (c*RT .. c*RT+RT-1).
// Kernels arrange their threads so that the column is fixed for the whole
// kernel: c = (linear thread index) mod ncols, with ncols = n / RT columns
// (2-D blocks of (n/RT) x sites, or 1-D blocks whose size is a multiple of n
// walking the elements with a stride that is too).  Contributions computed in
// the working precision (one site's 12 components) are added in FP64, and the
// combination over threads, warps and blocks below runs in a fixed order, so
// the sums are reproducible bit for bit for a given launch configuration.
template <int NV, int RT = 1, class V = double>
struct RedAcc {
    V v[NV][RT];
    __device__ __forceinline__ void add(int k, int t, double x) { v[k][t] += x; }
};

// A sum kept as an FP32 value and the FP32 sum of its rounding errors (Knuth's
// two-sum): 2^-47 relative, in six FP32 instructions and none of the FP64 pipe.
struct SumFF {
    float s, c;
    __device__ __forceinline__ void add(float x, float err) {
        const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
        c += __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b)) + err;
        s = t;
    }
};
__device__ __forceinline__ SumFF operator+(SumFF a, const SumFF &b) {
    a.add(b.s, b.c);
    return a;
}
__device__ __forceinline__ double sum_value(const SumFF &a) { return isfinite(a.c) ? (double)a.s + (double)a.c : (double)a.s; }
__device__ __forceinline__ double sum_value(double a) { return a; }
__device__ __forceinline__ SumFF shfl_xor(const SumFF &a, int h) {
    return {__shfl_xor_sync(0xffffffffu, a.s, h), __shfl_xor_sync(0xffffffffu, a.c, h)};
}
__device__ __forceinline__ double shfl_xor(double a, int h) { return __shfl_xor_sync(0xffffffffu, a, h); }

// Linear thread index and thread count of a (possibly 2-D) block.
__device__ __forceinline__ int ltid() { return threadIdx.y * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int lsize() { return blockDim.x * blockDim.y; }

template <int NV, int RT>
__device__ __forceinline__ void red_init(RedAcc<NV, RT> &acc) {
#pragma unroll
    for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int t = 0; t < RT; ++t) acc.v[k][t] = 0.0;
}

// Every one of n right-hand sides frozen.  A reducing kernel may then leave at
// once, without its ticket: states change only in the finalize step of a last
// block, after every block of that launch has read them here, so all blocks of
// a launch decide alike.
__device__ __forceinline__ bool all_frozen(const SolverState *st, int n) {
    bool f = true;
    for (int r = 0; r < n; ++r) f = f && st[r].stop;
    return f;
}
// The same, with what the finalize step does for frozen right-hand sides.
__device__ __forceinline__ bool frozen_exit(const SolverState *st, int n, const Reduce &red) {
    if (!all_frozen(st, n)) return false;
    if (red.fin == FIN_CG_ALPHA && red.st && blockIdx.x == 0)
        for (int r = ltid(); r < n; r += lsize()) red.st[r].xpend = 0;
    return true;
}

// The end of a pass of a loop, in its last launch (the states are final by then).  There and not in the finalize step: cudaGraphSetConditional is
// a call, and a call in the reducing and the operator kernels takes registers
// from them.
__device__ __forceinline__ void loop_end(const LoopEnd &loop, const SolverState *st, int n) {
    if (loop.cond == 0 || blockIdx.x != 0 || ltid() != 0) return;
    const unsigned done = atomicAdd(loop.done, loop.pass) + loop.pass;
    if (loop_over(done, st[0].maxit, all_frozen(st, n))) {
        *loop.done = 0;
        cudaGraphSetConditional(loop.cond, 0);
    }
}

// Block sums of the RedAcc values: total (value v, column c) goes to
// slot[(k*n + c*RT) + t], v = k*RT + t, valid for every thread after the
// closing barrier.  wv: kRedThreads * W doubles (W <= 4) or 32 * (warps) (W = 32).
//
// An FP64 warp instruction occupies this GPU's FP64 pipe for 15 cycles (2.1
// results per clock and SM), so what a reduction costs is its number of FP64
// warp instructions.  A shuffle tree in each of 8 warps takes 40 per value;
// here the threads store their values and one warp per value adds 8 of them
// per lane before a single tree: 13.  Wide sums (W = 32 values, one column)
// use recursive halving in each warp, 31 additions instead of 160.
constexpr int kRedThreads = 256;

template <int NV, int RT, class V = double>
__device__ __forceinline__ void block_sums(const V (&w)[NV * RT], int ncols, double *wv, double *slot) {
    constexpr int W = NV * RT;
    const int tid = ltid(), lane = tid & 31, warp = tid >> 5, nthr = lsize(), nw = (nthr + 31) >> 5;
    const int n = ncols * RT;
    if constexpr (W == 32) {  // one column, whole warps
        V x[W];
#pragma unroll
        for (int k = 0; k < W; ++k) x[k] = w[k];
#pragma unroll
        for (int h = 16; h >= 1; h >>= 1) {
            const bool up = (lane & h) != 0;
#pragma unroll
            for (int k = 0; k < h; ++k) {
                // lanes without bit h keep value k, the others value k + h
                const V give = up ? x[k] : x[k + h];
                const V keep = up ? x[k + h] : x[k];
                x[k] = keep + shfl_xor(give, h);
            }
        }
        wv[warp * 32 + lane] = sum_value(x[0]);  // lane l holds value l
        __syncthreads();
        if (tid < 32) {
            double s = 0.0;
            for (int q = 0; q < nw; ++q) s += wv[q * 32 + tid];
            slot[tid] = s;
        }
        __syncthreads();
    } else {
        // warps that add: the full ones, or the only one
        const int full = nthr >= 32 ? nthr >> 5 : 1, lanes = min(32, nthr);
        const int per = lanes / ncols;  // lanes per column
        const int c = lane % ncols, part = lane / ncols;
        for (int v0 = 0; v0 < W; v0 += full) {  // (a block of fewer warps than values goes round again)
            const int v = v0 + warp;
            const bool adds = warp < full && v < W;
            double s = 0.0;
            for (int base = 0; base < nthr; base += kRedThreads) {
                if (v0 > 0 || base > 0) __syncthreads();
                if (tid >= base && tid < base + kRedThreads) {
#pragma unroll
                    for (int k = 0; k < W; ++k) wv[k * kRedThreads + tid - base] = sum_value(w[k]);
                }
                __syncthreads();
                if (adds && part < per) {
                    int i = (c - base) % ncols;  // first thread of the round in column c
                    if (i < 0) i += ncols;
                    const int cnt = min(kRedThreads, nthr - base);
                    for (i += part * ncols; i < cnt; i += per * ncols) s += wv[v * kRedThreads + i];
                }
            }
            if (adds) {
                const unsigned mask = lanes >= 32 ? 0xffffffffu : ((1u << lanes) - 1u);
                int o = 1;
                while (2 * o < per) o *= 2;
                if (per > 1)
                    for (; o >= 1; o >>= 1) {
                        const double y = __shfl_down_sync(mask, s, o * ncols);
                        if (part < o && part + o < per) s += y;
                    }
                if (part == 0) {
                    const int k = v / RT;
                    slot[k * n + c * RT + (v - k * RT)] = s;
                }
            }
        }
        __syncthreads();
    }
}

// Combine the accumulators of the whole grid (ncols right-hand-side columns
// of RT right-hand sides each): each block writes its sums to red.partials,
// and the last block to finish (ticket counter) adds them, stores the totals
// in red.sums[k*n + r] and applies the finalize step to red.st[r].  The order
// is fixed for a launch configuration.  Every thread of every block must call it.
//
// Behind the last site this is a chain of barriers, fences and L2 round trips:
// one thread fences for its block (the barrier before it orders the other
// threads' stores), the partial sums of a slot lie side by side (the last
// block reads 256 blocks in one coalesced load per slot), and the loads of a
// slot group are in flight together.  Measured (with the early exit of
// all_frozen and the FP32 coefficients of SolverState): mixed BiCGstab on
// 20x12x28x36 8.10 -> 5.46 ms, EigCG on 16^3x32 303 -> 272 ms (its 32-value
// sums 234 -> 92 us), FP64 norm of a 24^3x48 half field 35 -> 25 us.
template <int NV, int RT, class V>
__device__ void grid_reduce(const Reduce &red, const RedAcc<NV, RT, V> &acc, int ncols) {
    constexpr int W = NV * RT;
    constexpr int kWords = W == 32 ? 32 * 32 : W * kRedThreads;
    __shared__ double wv[kWords];
    __shared__ double slot[kPartialSlots];
    __shared__ bool last;
    const int tid = ltid(), nthr = lsize();
    const int n = ncols * RT, slots = NV * n;
    V first[W];
#pragma unroll
    for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int t = 0; t < RT; ++t) first[k * RT + t] = acc.v[k][t];
    block_sums<NV, RT, V>(first, ncols, wv, slot);
    for (int t = tid; t < slots; t += nthr) red.partials[(size_t)t * kMaxReduceBlocks + blockIdx.x] = slot[t];
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        last = (atomicAdd(red.ticket, 1u) == gridDim.x - 1);
        if (last) __threadfence();
    }
    __syncthreads();
    if (!last) return;
    if (ncols == 1) {
        double w[W];
#pragma unroll
        for (int q = 0; q < W; ++q) w[q] = 0.0;
#pragma unroll 4
        for (int b = tid; b < (int)gridDim.x; b += nthr) {
#pragma unroll
            for (int q = 0; q < W; ++q) w[q] += __ldcg(red.partials + (size_t)q * kMaxReduceBlocks + b);
        }
        block_sums<W, 1>(w, 1, wv, slot);
    } else if constexpr (W <= 4) {
        for (int t0 = 0; t0 < slots; t0 += 4) {  // the loads of four slots in flight together
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            const double *p = red.partials + (size_t)t0 * kMaxReduceBlocks;
#pragma unroll 4
            for (int b = tid; b < (int)gridDim.x; b += nthr) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (t0 + q < slots) s[q] += __ldcg(p + (size_t)q * kMaxReduceBlocks + b);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (t0 + q >= slots) break;
                const double one[1] = {s[q]};
                block_sums<1, 1>(one, 1, wv, slot + t0 + q);
            }
        }
    }
    for (int t = tid; t < slots; t += nthr) red.sums[t] = slot[t];
    if (red.st) {
        for (int r = tid; r < n; r += nthr) {
            double tr[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) tr[k] = slot[k * n + r];
            finalize_one(red.fin, red.st + r, tr);
        }
    }
    if (tid == 0) *red.ticket = 0u;
}

// ---------------------------------------------------------------- geometry
// Coordinates of checkerboard site i of parity `par` (x = 2*(i mod Lx/2) + offset).
struct SiteGeom {
    int c[4];     // t, x, y, z
    int lex;      // lexicographic index
};

__device__ __forceinline__ SiteGeom site_geom(const Lattice &L, int par, int i) {
    SiteGeom g;
    unsigned xh, y, z;
    unsigned r = fd_divmod((unsigned)i, L.div_xh, &xh);
    r = fd_divmod(r, L.div_y, &y);
    const int t = (int)fd_divmod(r, L.div_z, &z);
    const int x = 2 * (int)xh + ((par + (int)y + (int)z + t) & 1);
    g.c[0] = t;
    g.c[1] = x;
    g.c[2] = (int)y;
    g.c[3] = (int)z;
    g.lex = ((t * L.L[3] + (int)z) * L.L[2] + (int)y) * L.L[1] + x;
    return g;
}

}  // namespace plq
