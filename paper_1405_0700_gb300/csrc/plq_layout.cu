// Layout kernels: canonical AoS FP64 fields <-> packed even-odd SoA fields.
#include "plq_fields.cuh"

namespace plq {

namespace {

int grid_for(long long work, int block, int per_sm = 8) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long want = (work + block - 1) / block;
    long long cap = (long long)sms * per_sm;
    return (int)(want < cap ? want : cap);
}

// Checkerboard pair i holds the lexicographic sites 2i and 2i + 1: one of each
// parity, both with checkerboard index i.  The even site of the pair is 2i + odd.
__device__ __forceinline__ int pair_odd(const Lattice &L, int i) {
    unsigned xh, y, z;
    unsigned r = fd_divmod((unsigned)i, L.div_xh, &xh);
    r = fd_divmod(r, L.div_y, &y);
    const unsigned t = fd_divmod(r, L.div_z, &z);
    return (int)((y + z + t) & 1u);
}

// Canonical fields of nrhs right-hand sides stored back to back (each V sites
// x 12 complex, lexicographic) <-> packed full field (even half, odd half;
// element (plane k, site i, rhs r) at (k*Vh + i)*nrhs + r).
//
// A block moves `S` pairs of sites (2S consecutive lexicographic sites) of all
// right-hand sides through shared memory: the canonical side is read or written
// 16 bytes per thread along the site records (192 contiguous bytes per site,
// 384 S per right-hand side), the packed side by one (site, rhs) element per
// thread, consecutive elements side by side.  Straight from memory to memory, a
// warp writes 16-byte pieces of 32 records at a time: 24^3x48 took 145 us (FP64,
// 1 RHS) and 1914 us (12 RHS) to unpack, now 50 and 504 us, with 38 and 458 us
// for the bytes at the copy rate; FP32 1734 -> 444 us and FP16 1278 -> 329 us
// (12 RHS; 25 us per RHS of these are double -> float conversions).
//
// Packing reads the records, and reads of a record's pieces one after the other
// hit L1, so the direct form (pack_direct_kernel) stays the faster one except
// for FP64 storage with some counts of right-hand sides (pack_staged): FP64 1 / 3 RHS 48 /
// 141 us direct against 60 / 122 us on 24^3x48, FP16 1 / 3 / 12 RHS 35 / 98 / 383 against 56 /
// 107 / 400 us; on 28x22x14x6 FP64 with 3 RHS 10.9 against 12.9 us.
//
// In shared memory a site record takes 13 slots of 16 bytes and a right-hand
// side 2S * 13 + 1: both odd, so neighbouring sites and right-hand sides fall
// into different banks.
constexpr int kRec = 13;
constexpr int kLayoutThreads = 256;
__host__ __device__ constexpr int rhs_slots(int S) { return 2 * S * kRec + 1; }

// Pairs per block: up to 64, in 40 KB of shared memory (five blocks per SM).
int layout_pairs(int nrhs) {
    int S = 64;
    while (S > 4 && (size_t)nrhs * rhs_slots(S) * 16 > 40 * 1024) S /= 2;
    return S;
}

// Where two thirds of the block's threads hold an element in the packing phase (6, 11
// and 12 right-hand sides).  Direct / staged, 4 to 12 RHS on 16^3x32: 37.0 / 46.8, 47.2 /
// 57.5, 58.6 / 49.8, 67.2 / 80.1, 72.8 / 86.5, 78.9 / 100.3, 93.7 / 107.6, 105.9 / 86.3,
// 112.9 / 94.1 us; on 32^3x64 6 RHS 873 / 710, 8 RHS 1157 / 1293, 11 RHS 1612 / 1287, 12 RHS
// 1746 / 1414 us; on 28x22x14x6 6 RHS 20.4 / 19.6, 11 RHS 39.8 / 39.0 us.
bool pack_staged(int prec, int nrhs) {
    return prec == PLQ_F64 && nrhs >= 4 && 3 * 2 * layout_pairs(nrhs) * nrhs >= 2 * kLayoutThreads;
}

template <int P>
__global__ void pack_direct_kernel(Lattice L, int nrhs, char *out, const double *in, size_t half_bytes) {
    using T = RealOf<P>;
    const long long per_par = (long long)L.Vh * nrhs;
    const size_t V = 2 * (size_t)L.Vh;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < 2 * per_par;
         idx += (long long)gridDim.x * blockDim.x) {
        const int par = (int)(idx / per_par);
        const long long e = idx - par * per_par;
        const int i = (int)(e / nrhs);
        const int r = (int)(e - (long long)i * nrhs);
        const double2 *src = reinterpret_cast<const double2 *>(in) +
                             ((size_t)r * V + 2 * (size_t)i + (pair_odd(L, i) ^ par)) * 12;
        cx<T> v[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const double2 z = src[k];
            v[k] = {(T)z.x, (T)z.y};
        }
        Spinor<P>::store(out + par * half_bytes, (size_t)per_par, (size_t)e, v);
    }
}

__global__ void __launch_bounds__(kLayoutThreads) pack_staged_kernel(Lattice L, int nrhs, int S, char *out, const double *in,
                                                                     size_t half_bytes) {
    extern __shared__ double2 rec[];
    const size_t V = 2 * (size_t)L.Vh, per_par = (size_t)L.Vh * nrhs;
    const int i0 = blockIdx.x * S, np = min(S, L.Vh - i0);
    const int run = 2 * np * 12;  // 16-byte pieces of one right-hand side
    const double2 *src0 = reinterpret_cast<const double2 *>(in) + 2 * (size_t)i0 * 12;
#pragma unroll 8
    for (int q = threadIdx.x; q < run * nrhs; q += kLayoutThreads) {
        const int r = q / run, p = q - r * run;
        rec[r * rhs_slots(S) + p + p / 12] = __ldcs(src0 + (size_t)r * V * 12 + p);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < 2 * np * nrhs; q += kLayoutThreads) {
        const int par = q >= np * nrhs, e = q - par * np * nrhs;
        const int il = e / nrhs, r = e - il * nrhs;
        const double2 *src = rec + (size_t)r * rhs_slots(S) + (2 * il + (pair_odd(L, i0 + il) ^ par)) * kRec;
        cx<double> v[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) v[k] = {src[k].x, src[k].y};
        Spinor<PLQ_F64>::store(out + par * half_bytes, per_par, (size_t)i0 * nrhs + e, v);
    }
}

template <int P>
__global__ void __launch_bounds__(kLayoutThreads) unpack_spinor_kernel(Lattice L, int nrhs, int S, double *out, const char *in,
                                                                       size_t half_bytes) {
    extern __shared__ double2 rec[];
    using T = RealOf<P>;
    const size_t V = 2 * (size_t)L.Vh, per_par = (size_t)L.Vh * nrhs;
    const int i0 = blockIdx.x * S, np = min(S, L.Vh - i0);
    const int run = 2 * np * 12;
    for (int q = threadIdx.x; q < 2 * np * nrhs; q += kLayoutThreads) {
        const int par = q >= np * nrhs, e = q - par * np * nrhs;
        const int il = e / nrhs, r = e - il * nrhs;
        double2 *dst = rec + (size_t)r * rhs_slots(S) + (2 * il + (pair_odd(L, i0 + il) ^ par)) * kRec;
        cx<T> v[12];
        Spinor<P>::load(in + par * half_bytes, per_par, (size_t)i0 * nrhs + e, v);
#pragma unroll
        for (int k = 0; k < 12; ++k) dst[k] = make_double2((double)v[k].re, (double)v[k].im);
    }
    __syncthreads();
    double2 *dst0 = reinterpret_cast<double2 *>(out) + 2 * (size_t)i0 * 12;
#pragma unroll 8
    for (int q = threadIdx.x; q < run * nrhs; q += kLayoutThreads) {
        const int r = q / run, p = q - r * run;
        __stcs(dst0 + (size_t)r * V * 12 + p, rec[r * rhs_slots(S) + p + p / 12]);
    }
}

// Writes the packed form of one link (9 complex, row-major) at site i of a
// (parity, mu) block, for storage precision P and R reals.
template <int P, int R>
__device__ void store_link(char *blk, int Vh, int i, const double2 u[9]);

template <>
__device__ void store_link<PLQ_F64, 18>(char *blk, int Vh, int i, const double2 u[9]) {
    double2 *p = reinterpret_cast<double2 *>(blk) + i;
    for (int k = 0; k < 9; ++k) p[(size_t)k * Vh] = u[k];
}
template <>
__device__ void store_link<PLQ_F64, 12>(char *blk, int Vh, int i, const double2 u[9]) {
    double2 *p = reinterpret_cast<double2 *>(blk) + i;
    for (int k = 0; k < 6; ++k) p[(size_t)k * Vh] = u[k];
}
template <>
__device__ void store_link<PLQ_F32, 18>(char *blk, int Vh, int i, const double2 u[9]) {
    float4 *p = reinterpret_cast<float4 *>(blk) + i;
    for (int k = 0; k < 4; ++k)
        p[(size_t)k * Vh] = make_float4((float)u[2 * k].x, (float)u[2 * k].y, (float)u[2 * k + 1].x, (float)u[2 * k + 1].y);
    float2 *q = reinterpret_cast<float2 *>(reinterpret_cast<float4 *>(blk) + 4 * (size_t)Vh) + i;
    *q = make_float2((float)u[8].x, (float)u[8].y);
}
template <>
__device__ void store_link<PLQ_F32, 12>(char *blk, int Vh, int i, const double2 u[9]) {
    float4 *p = reinterpret_cast<float4 *>(blk) + i;
    for (int k = 0; k < 3; ++k)
        p[(size_t)k * Vh] = make_float4((float)u[2 * k].x, (float)u[2 * k].y, (float)u[2 * k + 1].x, (float)u[2 * k + 1].y);
}
template <>
__device__ void store_link<PLQ_F16, 18>(char *blk, int Vh, int i, const double2 u[9]) {
    uint4 *p = reinterpret_cast<uint4 *>(blk) + i;
    for (int k = 0; k < 2; ++k) {
        uint4 t;
        t.x = f2h((float)u[4 * k].x, (float)u[4 * k].y);
        t.y = f2h((float)u[4 * k + 1].x, (float)u[4 * k + 1].y);
        t.z = f2h((float)u[4 * k + 2].x, (float)u[4 * k + 2].y);
        t.w = f2h((float)u[4 * k + 3].x, (float)u[4 * k + 3].y);
        p[(size_t)k * Vh] = t;
    }
    unsigned *q = reinterpret_cast<unsigned *>(reinterpret_cast<uint4 *>(blk) + 2 * (size_t)Vh) + i;
    *q = f2h((float)u[8].x, (float)u[8].y);
}
template <>
__device__ void store_link<PLQ_F16, 12>(char *blk, int Vh, int i, const double2 u[9]) {
    uint4 *p = reinterpret_cast<uint4 *>(blk) + i;
    uint4 t;
    t.x = f2h((float)u[0].x, (float)u[0].y);
    t.y = f2h((float)u[1].x, (float)u[1].y);
    t.z = f2h((float)u[2].x, (float)u[2].y);
    t.w = f2h((float)u[3].x, (float)u[3].y);
    *p = t;
    uint2 *q = reinterpret_cast<uint2 *>(reinterpret_cast<uint4 *>(blk) + (size_t)Vh) + i;
    *q = make_uint2(f2h((float)u[4].x, (float)u[4].y), f2h((float)u[5].x, (float)u[5].y));
}

__device__ double2 dmul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }

// max deviation of u from SU(3): |u u^dagger - 1| and |row2 - conj(row0 x row1)|
__device__ double su3_defect(const double2 u[9]) {
    double d = 0.0;
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) {
            double re = 0, im = 0;
            for (int c = 0; c < 3; ++c) {  // u[a][c] * conj(u[b][c])
                re += u[3 * a + c].x * u[3 * b + c].x + u[3 * a + c].y * u[3 * b + c].y;
                im += u[3 * a + c].y * u[3 * b + c].x - u[3 * a + c].x * u[3 * b + c].y;
            }
            d = fmax(d, fabs(re - (a == b ? 1.0 : 0.0)));
            d = fmax(d, fabs(im));
        }
    for (int c = 0; c < 3; ++c) {
        const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
        double2 x = dmul(u[c1], u[3 + c2]), y = dmul(u[c2], u[3 + c1]);
        double2 r = make_double2(x.x - y.x, -(x.y - y.y));  // conj(row0 x row1)_c
        d = fmax(d, fabs(r.x - u[6 + c].x));
        d = fmax(d, fabs(r.y - u[6 + c].y));
    }
    return d;
}

// |d| > limit, or d is NaN, by the bit patterns (a comparison of doubles
// occupies the FP64 pipe).
__device__ __forceinline__ bool beyond(double d, double limit) {
    return (__double_as_longlong(d) & 0x7fffffffffffffffLL) > __double_as_longlong(limit);
}

// Whether u deviates from SU(3) by more than 1e-12 (su3_defect).  The full
// check is ~260 FP64 instructions per link at 2.1 per clock and SM: 1105 us for
// the FP32 links of 24^3x48, whose bytes take 76 us (now 367 us, FP64 storage
// 986 -> 330 us, FP16 1111 -> 369 us).  Links that pass the 48 of this
// test at a tenth of the limit need no more: with |r0|^2 - 1, |r1|^2 - 1,
// <r0, r1> and every component of r2 - conj(r0 x r1) within 1e-13, |r2|^2 - 1 is
// within 2 sqrt(6) 1e-13 + 3e-13 < 8e-13, and <r0, r2>, <r1, r2> within
// sqrt(6) 1e-13 < 3e-13.
__device__ __forceinline__ bool su3_bad(const double2 u[9]) {
    constexpr double near = 1e-13;
    double n0 = -1.0, n1 = -1.0, dr = 0.0, di = 0.0;
    bool far = false;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double2 a = u[c], b = u[3 + c];
        n0 = fma(a.x, a.x, fma(a.y, a.y, n0));
        n1 = fma(b.x, b.x, fma(b.y, b.y, n1));
        dr = fma(a.x, b.x, fma(a.y, b.y, dr));
        di = fma(a.y, b.x, fma(-a.x, b.y, di));
        const double2 p = u[(c + 1) % 3], q = u[3 + (c + 2) % 3], v = u[(c + 2) % 3], w = u[3 + (c + 1) % 3];
        double re = -u[6 + c].x, im = u[6 + c].y;  // conj(p q - v w) - r2
        re = fma(p.x, q.x, fma(-p.y, q.y, fma(-v.x, w.x, fma(v.y, w.y, re))));
        im = fma(p.x, q.y, fma(p.y, q.x, fma(-v.x, w.y, fma(-v.y, w.x, im))));
        far = far || beyond(re, near) || beyond(im, near);
    }
    far = far || beyond(n0, near) || beyond(n1, near) || beyond(dr, near) || beyond(di, near);
    return far && su3_defect(u) > 1e-12;
}

// Links, canonical (36 complex per site) -> 8 (parity, mu) blocks.  (Moving the
// records through shared memory as above gained nothing here: the SU(3) check
// and the conversions are FP64-pipe work, and without them 24^3x48 is at 125 us
// of the 86 us its bytes take.)
template <int P, int R>
__global__ void pack_gauge_kernel(Lattice L, char *out, const double *in, size_t block, unsigned *bad) {
    const long long total = 2LL * L.Vh;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int par = (int)(idx / L.Vh);
        const int i = (int)(idx - (long long)par * L.Vh);
        const SiteGeom g = site_geom(L, par, i);
        const double2 *src = reinterpret_cast<const double2 *>(in) + (size_t)g.lex * 36;
        for (int mu = 0; mu < 4; ++mu) {
            double2 u[9];
            for (int k = 0; k < 9; ++k) u[k] = src[9 * mu + k];
            if (R == 12 && su3_bad(u)) atomicOr(bad, 1u);
            store_link<P, R>(out + (size_t)(par * 4 + mu) * block, L.Vh, i, u);
        }
    }
}

}  // namespace

plq_status launch_pack_spinor(const Lattice &L, void *out, const double *in, int prec, int nrhs, cudaStream_t s) {
    const size_t half = spinor_site_bytes(prec) * L.Vh * nrhs;
    char *o = static_cast<char *>(out);
    if (pack_staged(prec, nrhs)) {
        const int S = layout_pairs(nrhs), grid = (L.Vh + S - 1) / S;
        pack_staged_kernel<<<grid, kLayoutThreads, (size_t)nrhs * rhs_slots(S) * sizeof(double2), s>>>(L, nrhs, S, o, in, half);
    } else {
        const int grid = grid_for(2LL * L.Vh * nrhs, 256);
        if (prec == PLQ_F64) pack_direct_kernel<PLQ_F64><<<grid, 256, 0, s>>>(L, nrhs, o, in, half);
        else if (prec == PLQ_F32) pack_direct_kernel<PLQ_F32><<<grid, 256, 0, s>>>(L, nrhs, o, in, half);
        else pack_direct_kernel<PLQ_F16><<<grid, 256, 0, s>>>(L, nrhs, o, in, half);
    }
    PLQ_CUDA(cudaGetLastError());
    return PLQ_OK;
}

plq_status launch_unpack_spinor(const Lattice &L, double *out, const void *in, int prec, int nrhs, cudaStream_t s) {
    const size_t half = spinor_site_bytes(prec) * L.Vh * nrhs;
    const int S = layout_pairs(nrhs), grid = (L.Vh + S - 1) / S;
    const size_t smem = (size_t)nrhs * rhs_slots(S) * sizeof(double2);
    const char *i = static_cast<const char *>(in);
    if (prec == PLQ_F64) unpack_spinor_kernel<PLQ_F64><<<grid, kLayoutThreads, smem, s>>>(L, nrhs, S, out, i, half);
    else if (prec == PLQ_F32) unpack_spinor_kernel<PLQ_F32><<<grid, kLayoutThreads, smem, s>>>(L, nrhs, S, out, i, half);
    else unpack_spinor_kernel<PLQ_F16><<<grid, kLayoutThreads, smem, s>>>(L, nrhs, S, out, i, half);
    PLQ_CUDA(cudaGetLastError());
    return PLQ_OK;
}

plq_status launch_pack_gauge(const Lattice &L, void *out, const double *in, int prec, int reals, size_t block,
                             unsigned *bad, cudaStream_t s) {
    const int tb = 128, grid = grid_for(2LL * L.Vh, tb);
    char *o = static_cast<char *>(out);
    if (prec == PLQ_F64) {
        if (reals == 12) pack_gauge_kernel<PLQ_F64, 12><<<grid, tb, 0, s>>>(L, o, in, block, bad);
        else pack_gauge_kernel<PLQ_F64, 18><<<grid, tb, 0, s>>>(L, o, in, block, bad);
    } else if (prec == PLQ_F32) {
        if (reals == 12) pack_gauge_kernel<PLQ_F32, 12><<<grid, tb, 0, s>>>(L, o, in, block, bad);
        else pack_gauge_kernel<PLQ_F32, 18><<<grid, tb, 0, s>>>(L, o, in, block, bad);
    } else {
        if (reals == 12) pack_gauge_kernel<PLQ_F16, 12><<<grid, tb, 0, s>>>(L, o, in, block, bad);
        else pack_gauge_kernel<PLQ_F16, 18><<<grid, tb, 0, s>>>(L, o, in, block, bad);
    }
    PLQ_CUDA(cudaGetLastError());
    return PLQ_OK;
}

}  // namespace plq
