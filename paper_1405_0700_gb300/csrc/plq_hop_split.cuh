// Split hopping kernel: the eight directions of a site on eight warps.
//
// One thread per site walks the eight directions one after the other: eight
// L2 round trips in series, 8 us a launch on an 8^4 lattice whose 2048 sites
// occupy 16 of 152 SMs.  Here a block of eight warps owns 32 consecutive
// (site, right-hand side) elements; warp d loads the neighbour spinor and link
// of direction d for all of them (coalesced as in hop_kernel, one round trip),
// applies the link and leaves its contribution in shared memory; then the
// threads of the block, one 16-byte plane of an element each, add the eight
// contributions in direction order, apply the epilogue and store.
//
// FP64 storage runs this way at every size: either kernel is bound by the FP64
// pipe (a warp instruction takes 16 cycles of an SM), with 840 instructions per
// site here -- the signs of the reconstruction are those of additions -- and
// blocks of 32 sites spread them evenly where the 128-thread blocks of a one-wave
// grid leave a nearly empty second wave.  Two applications (plq_schur_apply),
// hop_kernel -> this: FP64 8^4 71 -> 25 us (chained 20), 12^3x16 70 -> 56 (51), 16^3x32
// 253 -> 226 (222), 24^3x32 745 -> 725 (719), 24^3x48 1110 -> 1079 us; one application 32^3x64 1628 ->
// 1619 us, 24^3x48 with 12 right-hand sides 6167 -> 6132 us; both parities in one
// launch (plq_wilson_apply) 16^3x32 236 -> 217 us.  Three blocks per SM
// with a few spilled registers beat two without (16^3x32 230, 24^3x48 1102 us).
//
// FP32 and FP16 storage are bound by memory or issue beyond small lattices and
// lose there to the reuse of loaded registers (FP32 16^3x32 22 -> 26 us, 24^3x48
// 87 -> 102 us).  As whole mixed CG solves: FP32 8^4 2.47 -> 2.00 ms, 8^3x16 2.80
// -> 2.40, 12^3x24 3.24 -> 3.47 ms; FP16 8^3x16 2.99 -> 2.71, 12^3x16 3.06 -> 3.10
// ms.  The line (split_default) lies between 4096 and 13824 elements.
#pragma once

namespace plq {

// One 16-byte plane of an element: 2 complex numbers in FP32 arithmetic, one in FP64.
template <class T>
struct Plane;
template <>
struct Plane<float> {
    static constexpr int N = 2, K = 6;  // complex numbers per plane, planes per element
    using V = float4;
    __device__ static V make(const cx<float> *v) { return make_float4(v[0].re, v[0].im, v[1].re, v[1].im); }
    __device__ static void get(V t, cx<float> *v) {
        v[0] = {t.x, t.y};
        v[1] = {t.z, t.w};
    }
};
template <>
struct Plane<double> {
    static constexpr int N = 1, K = 12;
    using V = double2;
    __device__ static V make(const cx<double> *v) { return make_double2(v[0].re, v[0].im); }
    __device__ static void get(V t, cx<double> *v) { v[0] = {t.x, t.y}; }
};

// Plane k of element e of a packed half field.
template <int P>
__device__ __forceinline__ void load_plane(const void *f, size_t stride, size_t e, int k, cx<RealOf<P>> *v) {
    using T = RealOf<P>;
    if constexpr (P == PLQ_F16) {
        const uint2 t = __ldg(reinterpret_cast<const uint2 *>(static_cast<const uint4 *>(f) + (size_t)(k >> 1) * stride + e) + (k & 1));
        const float n = ld_nc(reinterpret_cast<const float *>(static_cast<const uint4 *>(f) + 3 * stride) + e);
        const float2 a = h2f(t.x), b = h2f(t.y);
        v[0] = {a.x * n, a.y * n};
        v[1] = {b.x * n, b.y * n};
    } else {
        Plane<T>::get(ld_nc(static_cast<const typename Plane<T>::V *>(f) + (size_t)k * stride + e), v);
    }
}

// uh = U^(dagger) (upper two spin components of the projected neighbour)
template <int P, int R, int MU, bool BACK, bool DAG>
__device__ __forceinline__ void split_dir(const HopArgs &a, const SiteGeom &g, int i, int r, size_t stride,
                                          cx<RealOf<P>> uh[6]) {
    using T = RealOf<P>;
    constexpr int S = (DAG != BACK) ? +1 : -1;  // projector 1 + S gamma_mu
    const Lattice &L = a.lat;
    const int st = lex_stride(L, MU), cm = g.c[MU], Lm = L.L[MU];
    const bool wrap = BACK ? cm == 0 : cm == Lm - 1;
    const int step = BACK ? -st : st;
    const int j = PLQ_GUARD(a.kstatus, (g.lex + (wrap ? step * (1 - Lm) : step)) >> 1, L.Vh);
    cx<T> u[3][3], phi[12], h[6];
    T sc = load_for_projection<P>(a.in, stride, (size_t)j * a.nrhs + r, phi);
    Link<P, R>::load(static_cast<const char *>(a.gauge) + (size_t)((BACK ? 1 - a.out_parity : a.out_parity) * 4 + MU) * a.gblock,
                     L.Vh, BACK ? j : i, u);
    project<MU, S>(phi, h);
    const bool flip = MU == 0 && wrap && L.t_bc < 0;
    if (flip) sc = -sc;
    if (P == PLQ_F16 || (MU == 0 && flip)) {
#pragma unroll
        for (int k = 0; k < 6; ++k) h[k] = {sc * h[k].re, sc * h[k].im};
    }
    if constexpr (BACK) su3_dag_mul(u, h, uh);
    else su3_mul(u, h, uh);
}

// Output component 3*SPIN + col of an element: the sum over the directions of
// the upper components, or of their +-1, +-i multiples, in `part` (direction,
// component, element).  The phases are those of reconstruct(); they are taken
// here, where they are the signs of additions (a negated FP64 value that has
// to be stored costs an instruction of the FP64 pipe).
template <class T, bool DAG, int SPIN, int D>
__device__ __forceinline__ void add_direction(const cx<T> *part, int col, cx<T> &o) {
    using Q = Proj<(D >> 1)>;
    constexpr int S = (DAG != ((D & 1) != 0)) ? +1 : -1;
    constexpr int add = S > 0 ? 2 : 0;
    constexpr int row = SPIN < 2 ? SPIN : (Q::p0 == SPIN ? 0 : 1);
    constexpr int k = SPIN < 2 ? 0 : (row == 0 ? Q::k0 : Q::k1) + add;
    const cx<T> t = part[(D * 6 + 3 * row + col) * 32];
    if constexpr (D == 0) o = mul_ipow<(4 - (k & 3)) & 3>(t);
    else o = cadd(o, mul_ipow<(4 - (k & 3)) & 3>(t));
    if constexpr (D < 7) add_direction<T, DAG, SPIN, D + 1>(part, col, o);
}

template <class T, bool DAG, int C>
__device__ __forceinline__ void sum_component(const cx<T> *part, cx<T> &o) {
    add_direction<T, DAG, C / 3, 0>(part, C % 3, o);
}
template <class T, bool DAG, int K>
__device__ __forceinline__ void sum_plane(const cx<T> *part, cx<T> *o) {
    sum_component<T, DAG, K * Plane<T>::N>(part, o[0]);
    if constexpr (Plane<T>::N == 2) sum_component<T, DAG, 2 * K + 1>(part, o[1]);
}
template <class T, bool DAG>
__device__ __forceinline__ void sum_plane(int k, const cx<T> *part, cx<T> *o) {
    switch (k) {  // (one k per warp)
    case 0: sum_plane<T, DAG, 0>(part, o); break;
    case 1: sum_plane<T, DAG, 1>(part, o); break;
    case 2: sum_plane<T, DAG, 2>(part, o); break;
    case 3: sum_plane<T, DAG, 3>(part, o); break;
    case 4: sum_plane<T, DAG, 4>(part, o); break;
    case 5: sum_plane<T, DAG, 5>(part, o); break;
    default:
        if constexpr (Plane<T>::K == 12) {
            switch (k) {
            case 6: sum_plane<T, DAG, 6>(part, o); break;
            case 7: sum_plane<T, DAG, 7>(part, o); break;
            case 8: sum_plane<T, DAG, 8>(part, o); break;
            case 9: sum_plane<T, DAG, 9>(part, o); break;
            case 10: sum_plane<T, DAG, 10>(part, o); break;
            default: sum_plane<T, DAG, 11>(part, o); break;
            }
        }
    }
}

constexpr int kSplitThreads = 256;
constexpr long long kSplitElements = 8192;

// The reducing epilogues keep one right-hand side per thread: one in all.
inline bool split_fits(const HopArgs &a, int epi) { return a.nrhs == 1 || epi <= EPI_XPAY; }

// FP64 with a reduction: below the line the even spread of 32-site tiles wins, above
// it blocks walk several tiles and hop_kernel does.  FP64 solves of 45 iterations,
// hop_kernel / this for the reducing launches, CG and BiCGstab: 16^3x32 (65,536
// sites) 23.75 / 22.76 and 13.90 / 13.58 ms, 16^3x40 29.21 / 27.64 and 17.35 / 16.70,
// 16^3x48 35.18 / 33.50 and 20.36 / 19.65, 24^3x16 (110,592) 36.80 / 36.90 and 22.07 /
// 21.36, 20^3x32 (128,000) 42.60 / 42.64 and 25.86 / 27.05, 20^3x40 53.39 / 52.75 and
// 32.27 / 32.12, 24^3x24 (165,888) 54.79 / 55.04 and 31.69 / 33.36, 24^3x32 71.83 /
// 72.88 and 41.05 / 41.72, 28^3x24 84.06 / 87.34 and 49.99 / 54.00 ms.
constexpr int kSplitReduceSites = 120000;
template <int P>
bool split_default(const HopArgs &a, int epi) {
    if (P == PLQ_F64) return epi < EPI_XPAY_NORM || a.lat.Vh <= kSplitReduceSites;
    return (long long)a.lat.Vh * a.nrhs <= kSplitElements;
}

// Args: one launch, or the launches of both parities (blockIdx.y picks).
struct HopPair {
    HopArgs a[2];
};
template <int P, int R, int EPI, bool DAG, class Args>
__global__ void __launch_bounds__(kSplitThreads, P == PLQ_F64 || EPI >= EPI_XPAY_NORM ? 3 : 4) hop_split_kernel(const Args args) {
    const HopArgs &a = [&]() -> const HopArgs & {
        if constexpr (sizeof(Args) == sizeof(HopPair)) return args.a[blockIdx.y];
        else return args;
    }();
    if (chained<P>(a)) chain_begin();
    using T = RealOf<P>;
    using PL = Plane<T>;
    using V = typename PL::V;
    __shared__ __align__(16) cx<T> part[8 * 6 * 32];  // (direction, upper component, element)
    __shared__ cx<T> res[P == PLQ_F16 ? 12 * 32 : 1];  // FP16 storage: the element's output until its norm is known
    constexpr int NV = epi_sums(EPI);
    const int n = a.nrhs;
    if (a.st != nullptr && frozen_exit(a.st, n, a.red)) return;
    RedAcc<(NV > 0 ? NV : 1), 1> racc;
    red_init(racc);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t stride = (size_t)a.lat.Vh * n;
    const long long e_end = (long long)(a.site_end < 0 ? a.lat.Vh : a.site_end) * n;
    for (long long base = (long long)a.site_begin * n + 32LL * blockIdx.x; base < e_end; base += 32LL * gridDim.x) {
        if (base + lane < e_end) {
            const long long e = base + lane;
            const int i = n == 1 ? (int)e : (int)(e / n), r = n == 1 ? 0 : (int)(e - (long long)i * n);
            const SiteGeom g = site_geom(a.lat, a.out_parity, PLQ_GUARD(a.kstatus, i, a.lat.Vh));
            cx<T> v[6];
            switch (warp) {
            case 0: split_dir<P, R, 0, false, DAG>(a, g, i, r, stride, v); break;
            case 1: split_dir<P, R, 0, true, DAG>(a, g, i, r, stride, v); break;
            case 2: split_dir<P, R, 1, false, DAG>(a, g, i, r, stride, v); break;
            case 3: split_dir<P, R, 1, true, DAG>(a, g, i, r, stride, v); break;
            case 4: split_dir<P, R, 2, false, DAG>(a, g, i, r, stride, v); break;
            case 5: split_dir<P, R, 2, true, DAG>(a, g, i, r, stride, v); break;
            case 6: split_dir<P, R, 3, false, DAG>(a, g, i, r, stride, v); break;
            default: split_dir<P, R, 3, true, DAG>(a, g, i, r, stride, v); break;
            }
#pragma unroll
            for (int c = 0; c < 6; ++c) part[(warp * 6 + c) * 32 + lane] = v[c];
        }
        __syncthreads();
        // plane k of element base + lane, k = warp, warp + 8
#pragma unroll
        for (int k0 = 0; k0 < PL::K; k0 += 8) {
            const int k = k0 + warp;
            const long long e = base + lane;
            if (k >= PL::K || e >= e_end) break;
            if (EPI == EPI_PLAIN || n == 1 || a.st == nullptr || !a.st[e % n].stop) {
                cx<T> o[PL::N];
                sum_plane<T, DAG>(k, part + lane, o);
                const bool upper = k < PL::K / 2;  // gamma5 = diag(1, 1, -1, -1)
                if (a.twist_h) {
                    const T nu = upper ? hop_nu_h<T>(a) : -hop_nu_h<T>(a), s = hop_scale_h<T>(a);
#pragma unroll
                    for (int q = 0; q < PL::N; ++q)
                        o[q] = {s * (o[q].re - nu * o[q].im), s * (o[q].im + nu * o[q].re)};
                }
                if constexpr (EPI != EPI_PLAIN) {
                    cx<T> x[PL::N];
                    load_plane<P>(a.x, stride, (size_t)e, k, x);
                    if (a.twist_x) {
                        const T nu = upper ? hop_nu_x<T>(a) : -hop_nu_x<T>(a);
#pragma unroll
                        for (int q = 0; q < PL::N; ++q) x[q] = {x[q].re - nu * x[q].im, x[q].im + nu * x[q].re};
                    }
                    const T s = hop_a<T>(a);
#pragma unroll
                    for (int q = 0; q < PL::N; ++q) o[q] = {fma(s, o[q].re, x[q].re), fma(s, o[q].im, x[q].im)};
                    if constexpr (EPI == EPI_XPAY_RUPD) {  // (one right-hand side)
                        const T al = -hop_alpha<T>(a.st[0]);
                        load_plane<P>(a.w, stride, (size_t)e, k, x);
#pragma unroll
                        for (int q = 0; q < PL::N; ++q) o[q] = {fma(al, o[q].re, x[q].re), fma(al, o[q].im, x[q].im)};
                    }
                    // (FP64 sums go on in the thread's accumulators, whose additions the
                    // fused multiply-adds then are; FP32 ones are added in FP64)
                    constexpr bool go_on = NV > 0 && sizeof(T) == 8;
                    T s0 = go_on ? (T)racc.v[0][0] : T(0), s1 = go_on && NV > 1 ? (T)racc.v[NV > 1 ? 1 : 0][0] : T(0),
                      s2 = go_on && NV > 2 ? (T)racc.v[NV > 2 ? 2 : 0][0] : T(0);
                    if constexpr (EPI == EPI_XPAY_NORM || EPI == EPI_XPAY_RUPD) {
#pragma unroll
                        for (int q = 0; q < PL::N; ++q) s0 = fma(o[q].re, o[q].re, fma(o[q].im, o[q].im, s0));
                    } else if constexpr (EPI == EPI_XPAY_DOTW) {
                        cx<T> w[PL::N];
                        load_plane<P>(a.w, stride, (size_t)e, k, w);
#pragma unroll
                        for (int q = 0; q < PL::N; ++q) {  // <w, out>
                            s0 = fma(w[q].re, o[q].re, fma(w[q].im, o[q].im, s0));
                            s1 = fma(w[q].re, o[q].im, fma(-w[q].im, o[q].re, s1));
                        }
                    } else if constexpr (EPI == EPI_XPAY_TS) {
#pragma unroll
                        for (int q = 0; q < PL::N; ++q) {  // <out, x>, |out|^2
                            s0 = fma(o[q].re, x[q].re, fma(o[q].im, x[q].im, s0));
                            s1 = fma(o[q].re, x[q].im, fma(-o[q].im, x[q].re, s1));
                            s2 = fma(o[q].re, o[q].re, fma(o[q].im, o[q].im, s2));
                        }
                    }
                    const T sums[3] = {s0, s1, s2};
#pragma unroll
                    for (int q = 0; q < NV; ++q) racc.v[q][0] = go_on ? (double)sums[q] : racc.v[q][0] + (double)sums[q];
                }
                if constexpr (P == PLQ_F16) {
                    res[(2 * k) * 32 + lane] = o[0];
                    res[(2 * k + 1) * 32 + lane] = o[1];
                } else static_cast<V *>(a.out)[(size_t)PLQ_GUARD(a.kstatus, (long long)k * stride + e, (long long)PL::K * stride)] = PL::make(o);
            }
        }
        if constexpr (P == PLQ_F16) {
            // the site norm spans the planes: warp k < 3 stores 8 halves of each element
            __syncthreads();
            const long long e = base + lane;
            if (warp < 3 && e < e_end && (n == 1 || a.st == nullptr || !a.st[e % n].stop)) {
                cx<float> v[12];
#pragma unroll
                for (int k = 0; k < 12; ++k) v[k] = res[k * 32 + lane];
                Spinor<PLQ_F16>::store_plane(a.out, stride, (size_t)PLQ_GUARD(a.kstatus, e, (long long)stride), v, warp);
            }
        }
        __syncthreads();  // part is free again
    }
    if constexpr (NV > 0) grid_reduce(a.red, racc, 1);
}

template <int P, int R, int EPI, bool DAG, bool BOTH = false>
plq_status launch_split_t(const HopArgs &a, cudaStream_t s) {
    const int i_end = a.site_end < 0 ? a.lat.Vh : a.site_end;
    long long grid = ((long long)(i_end - a.site_begin) * a.nrhs + 31) / 32;
    if (grid <= 0) return PLQ_OK;
    // reducing launches: every block adds partial sums
    if (EPI >= EPI_XPAY_NORM && grid > kMaxReduceBlocks / 2) grid = kMaxReduceBlocks / 2;
    cudaError_t e;
    if constexpr (BOTH) {
        HopPair p{{a, a}};
        p.a[1].in = a.in2;
        p.a[1].x = a.x2;
        p.a[1].out = a.out2;
        p.a[1].out_parity = 1 - a.out_parity;
        e = launch_chained(chained<P>(a), hop_split_kernel<P, R, EPI, DAG, HopPair>, dim3((unsigned)grid, 2), dim3(kSplitThreads), s, p);
    } else {
        e = launch_chained(chained<P>(a), hop_split_kernel<P, R, EPI, DAG, HopArgs>, dim3((unsigned)grid),
                           dim3(kSplitThreads), s, a);
    }
    if (e != cudaSuccess) return cuda_error(e, "hop_split_kernel launch");
    return PLQ_OK;
}

template <int P, int R>
plq_status dispatch_split(const HopArgs &a, int epi, cudaStream_t s) {
    if (a.both && epi == EPI_XPAY && !a.dagger) return launch_split_t<P, R, EPI_XPAY, false, true>(a, s);
    switch (epi) {
    case EPI_PLAIN: return a.dagger ? launch_split_t<P, R, EPI_PLAIN, true>(a, s) : launch_split_t<P, R, EPI_PLAIN, false>(a, s);
    case EPI_XPAY: return a.dagger ? launch_split_t<P, R, EPI_XPAY, true>(a, s) : launch_split_t<P, R, EPI_XPAY, false>(a, s);
    case EPI_XPAY_NORM:
        return a.dagger ? launch_split_t<P, R, EPI_XPAY_NORM, true>(a, s) : launch_split_t<P, R, EPI_XPAY_NORM, false>(a, s);
    case EPI_XPAY_RUPD:
        if (!a.dagger) return set_error(PLQ_ERR_ARG, "the residual update belongs to the adjoint");
        return launch_split_t<P, R, EPI_XPAY_RUPD, true>(a, s);
    case EPI_XPAY_DOTW: return launch_split_t<P, R, EPI_XPAY_DOTW, false>(a, s);
    case EPI_XPAY_TS: return launch_split_t<P, R, EPI_XPAY_TS, false>(a, s);
    default: return set_error(PLQ_ERR_ARG, "bad epilogue %d", epi);
    }
}

}  // namespace plq
