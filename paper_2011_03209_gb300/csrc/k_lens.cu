// k_lens.cu -- filter (lens) kernels, "Mapper Interactive" §3 (filter
// function f: X -> R or R^2) and §4.1 (L2 norm, a chosen column; PCA;
// eccentricity), §5 (L-infinity norm). The density filter is a count pass of
// the DBSCAN kernels (capi.cu).
//
// The projection lens sums in double, k ascending, with explicitly rounded
// operations (never fused), so it is the exact IEEE result of the defining
// expression; the L2 lens rounds the exact sum of squares once. Rows are staged
// through shared memory so the loads stay coalesced while every thread walks
// its own row in order.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "dbscan.cuh"

namespace cg = cooperative_groups;

namespace mgb {

namespace {

constexpr int kRows = 128;    // rows per CTA (one thread per row)
constexpr int kChunk = 32;    // columns staged per step
constexpr int kMeanRows = 4096;   // rows per partial column sum

// (double)x from the bits, in integer instructions (the FP64 pipe of this chip,
// conversions included, issues two lanes a cycle and SM): for zeros and normal
// values; `plain` says whether x is one. Kernels ask once for a batch of
// values and convert the batches that hold another by the conversion.
__device__ __forceinline__ bool plain(float x)
{
    const unsigned t = __float_as_uint(x) & 0x7FFFFFFFu;
    return t == 0u || t - 0x00800000u < 0x7F000000u;
}

__device__ __forceinline__ double widen(float x)
{
    const unsigned b = __float_as_uint(x);
    const unsigned hi = ((b & 0x7FFFFFFFu) >> 3) + (896u << 20);
    return __hiloint2double((int)((b & 0x80000000u) | ((b & 0x7FFFFFFFu) ? hi : 0u)), (int)(b << 29));
}

// One CTA = 128 rows. Each warp loads whole 32-column row segments
// (coalesced); then each thread consumes its row's segment in order.
// MODE 0: sum x^2 then sqrt (L2). MODE 1: sum (x - mu) v (projection).
// MODE 3: two projections, sharing x - mu. Bound by the FP64 pipe (MODE 1: subtract,
// multiply, add per value). 500k x 128, two axes: 0.99 -> 0.63 ms.
template <int MODE>
__global__ void __launch_bounds__(kRows) lens_rows_kernel(const float* __restrict__ X, int64_t n,
                                                          int32_t d, int64_t ld,
                                                          const double* __restrict__ mu,
                                                          const double* __restrict__ v,
                                                          const double* __restrict__ v2,
                                                          double* __restrict__ f, int m, int j)
{
    __shared__ float tile[kRows][kChunk + 1];
    __shared__ double smu[kChunk], sv[kChunk], sv2[kChunk];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t row0 = (int64_t)blockIdx.x * kRows;
    double acc = 0.0, acc2 = 0.0;
    for (int32_t k0 = 0; k0 < d; k0 += kChunk) {
        const int kc = min(kChunk, d - k0);
        bool all_plain = true;
#pragma unroll 8
        for (int r = warp; r < kRows; r += kRows / 32) {
            const int64_t row = row0 + r;
            float x = 0.f;
            if (row < n && lane < kc) x = __ldg(X + row * ld + k0 + lane);
            tile[r][lane] = x;
            all_plain &= plain(x);
        }
        if (MODE >= 1 && tid < kc) {
            smu[tid] = mu[k0 + tid];
            if (MODE == 1 || MODE == 3) sv[tid] = v[k0 + tid];
            if (MODE == 3) sv2[tid] = v2[k0 + tid];
        }
        auto add = [&](int k, double x) {
            if (MODE == 0) {
                // x * x is exact in double (24-bit significands), so one
                // fused rounding equals the separate multiply and add
                acc = __fma_rn(x, x, acc);
            } else {
                const double t = __dsub_rn(x, smu[k]);
                acc = __dadd_rn(acc, __dmul_rn(t, sv[k]));
                if (MODE == 3) acc2 = __dadd_rn(acc2, __dmul_rn(t, sv2[k]));
            }
        };
        if (__syncthreads_and(all_plain)) {
#pragma unroll 8
            for (int k = 0; k < kc; ++k) add(k, widen(tile[tid][k]));
        } else {
            for (int k = 0; k < kc; ++k) add(k, (double)tile[tid][k]);
        }
        __syncthreads();
    }
    const int64_t row = row0 + tid;
    if (row >= n) return;
    f[row * m + j] = (MODE == 0) ? __dsqrt_rn(acc) : acc;
    if (MODE == 3) f[row * m + j + 1] = acc2;
}

// L2 lens from the exact sum of squares. A float x = m 2^(e-150) (m < 2^24)
// squares to m^2 2^(2e-300) exactly; the row's squares are added as integers
// and the exact sum is rounded to double once, then a correctly rounded sqrt.
// Per lane and 256-column chunk, with el the lane's largest exponent:
//   e >= el - 6:       (m << (e - el + 6))^2 into a 64-bit sum (unit 2^(2el-312))
//   el - 13 <= e < ..: (m << (e - el + 13))^2 into a second one (2^(2el-326))
// (one multiply-add each, at most 8 terms below 2^60); rarer small values
// and subnormals go to a 128-bit fixed-point sum whose unit is 2^(2emax-364)
// (emax: the row's largest exponent), where the two 64-bit sums also land at
// the end of each chunk. Bits of that sum below its unit are dropped: a
// relative change of at most d 2^-110, so the result is the exact sum rounded
// once up to that, within (d - 1) 2^-53 relative of a sequential double sum.
// A row holding a NaN (an Inf) gets NaN (Inf); d <= 32768 keeps the 128-bit
// sum below 2^127. One warp per row, 256 columns in registers at a time.
__device__ __forceinline__ void add128(unsigned long long& hi, unsigned long long& lo, unsigned long long bh,
                                       unsigned long long bl)
{
    const unsigned long long t = lo + bl;
    hi += bh + (t < lo ? 1ull : 0ull);
    lo = t;
}

// (hi, lo) += v 2^f, bits below 2^0 dropped (f < 64)
__device__ __forceinline__ void add128_shifted(unsigned long long& hi, unsigned long long& lo, unsigned long long v,
                                               int f)
{
    if (v == 0ull) return;
    if (f > 0) add128(hi, lo, v >> (64 - f), v << f);
    else if (f == 0) add128(hi, lo, 0ull, v);
    else if (f > -64) add128(hi, lo, 0ull, v >> -f);
}

__device__ __forceinline__ unsigned long long mad_wide(uint32_t a, unsigned long long acc)
{
    unsigned long long r;
    asm("mad.wide.u32 %0, %1, %1, %2;" : "=l"(r) : "r"(a), "l"(acc));
    return r;
}

constexpr int kL2Per = 8;                     // values per lane per 256-column chunk

// lane l of a row's lanes takes columns k0 + 8 l .. k0 + 8 l + 7 (two 16-byte
// loads when the row allows; the exact sum does not depend on the order)
__device__ __forceinline__ void l2_load(const float* __restrict__ x, int k0, int d, int lane, unsigned* v, bool vec)
{
    const int k = k0 + kL2Per * lane;
    if (vec && k + kL2Per <= d) {
        const uint4 a = __ldg(reinterpret_cast<const uint4*>(x + k));
        const uint4 b = __ldg(reinterpret_cast<const uint4*>(x + k + 4));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
        return;
    }
#pragma unroll
    for (int i = 0; i < kL2Per; ++i) v[i] = k + i < d ? __float_as_uint(__ldg(x + k + i)) : 0u;
}

// sqrt of (hi 2^64 + lo) 2^(2 emax - 364): the 128-bit value rounded once
// to double (its top 64 bits, a sticky bit for the rest), then sqrt
__device__ __forceinline__ double l2_finish(unsigned long long hi, unsigned long long lo, int emax, unsigned special)
{
    double val = 0.0;
    if (hi != 0ull || lo != 0ull) {
        const int lz = hi ? __clzll((long long)hi) : 64 + __clzll((long long)lo);
        unsigned long long top, rest;
        if (lz < 64) {
            top = lz ? (hi << lz) | (lo >> (64 - lz)) : hi;
            rest = lz ? lo << lz : lo;
        } else {
            top = lo << (lz - 64);
            rest = 0ull;
        }
        if (rest) top |= 1ull;
        val = ldexp(__ull2double_rn(top), 64 - lz + 2 * emax - 300 - 64);
    }
    if (special) val = (special & 2u) ? __longlong_as_double(0x7FF8000000000000ll)
                                      : __longlong_as_double(0x7FF0000000000000ll);
    return __dsqrt_rn(val);
}

// the largest biased exponent of the lane's values (254 for Inf/NaN, which
// are flagged separately), at least 1
__device__ __forceinline__ int lane_emax(const unsigned* v, int* raw)
{
    int el = 1;
#pragma unroll
    for (int t = 0; t < kL2Per; ++t) el = max(el, (int)((v[t] >> 23) & 0xFFu));
    *raw = el;
    return min(el, 254);
}

// G lanes take a row (8 columns each; G = 32 walks longer rows in chunks of
// 256), so a warp sums 32 / G rows at a time, `iters` (at most G) times over; lane
// i then holds the sum of the warp's row i, and the double conversions and
// square roots run side by side. Bound by integer instructions on long rows
// (2.2 TB/s at 1M x 256), by the chain of one row after another in a warp
// where there are few: with all lanes on one row and 32 rows a warp, 14k x 37
// took 61 us, now 11.
// SPLIT: the same pass also writes the rows for the pivot assignment, x - c
// rounded to BF16 (pitch dp, zero padded) and |x - c|^2 in FP32.
template <bool SPLIT, int G>
__global__ void __launch_bounds__(256) lens_l2_exact_kernel(const float* __restrict__ X, int64_t n, int32_t d,
                                                            int64_t ld, int iters, double* __restrict__ f, int m, int j,
                                                            const float* __restrict__ c, int dp,
                                                            __nv_bfloat16* __restrict__ xh, float* __restrict__ xn2)
{
    constexpr int kPar = 32 / G;                                   // rows at a time
    const int lane = threadIdx.x & 31;
    const int sub = lane & (G - 1), grp = lane / G;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const bool one_chunk = G < 32 || d <= 32 * kL2Per;             // (G < 32: d <= 8 G)
    const bool vec = ld % 4 == 0 && ((uintptr_t)X & 15) == 0;
    const int per_warp = kPar * iters;
    for (int64_t r0 = warp * per_warp; r0 < n; r0 += nwarp * per_warp) {
        unsigned long long my_hi = 0ull, my_lo = 0ull;
        int my_emax = 1;
        unsigned my_special = 0u;
        const int rows = n - r0 < per_warp ? (int)(n - r0) : per_warp;
        for (int i = 0; i < iters; ++i) {
            const bool live = i * kPar + grp < rows;
            const int64_t row = r0 + (live ? i * kPar + grp : 0);
            const float* x = X + row * ld;
            unsigned v[kL2Per];
            int emax = 1, raw_max = 0;
            for (int k0 = 0; k0 < d; k0 += G * kL2Per) {
                l2_load(x, k0, d, sub, v, vec);
                int raw;
                emax = max(emax, lane_emax(v, &raw));
                raw_max = max(raw_max, raw);
            }
            if (G == 32) {
                emax = __reduce_max_sync(0xffffffffu, emax);
            } else {
#pragma unroll
                for (int o = G / 2; o; o >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
            }
            unsigned special = 0u;                                 // 1: an Inf, 2: a NaN
            if (__any_sync(0xffffffffu, raw_max == 255)) {
                for (int k0 = 0; k0 < d; k0 += G * kL2Per) {
                    l2_load(x, k0, d, sub, v, vec);
#pragma unroll
                    for (int t = 0; t < kL2Per; ++t)
                        if (((v[t] >> 23) & 0xFFu) == 0xFFu) special |= (v[t] & 0x7FFFFFu) ? 2u : 1u;
                }
#pragma unroll
                for (int o = G / 2; o; o >>= 1) special |= __shfl_xor_sync(0xffffffffu, special, o);
            }
            unsigned long long hi = 0ull, lo = 0ull;
            float n2 = 0.f;
            for (int k0 = 0; k0 < d && !special; k0 += G * kL2Per) {
                if (!one_chunk) l2_load(x, k0, d, sub, v, vec);
                int raw;
                const int el = lane_emax(v, &raw);
                unsigned long long s1 = 0ull, s2 = 0ull;
#pragma unroll
                for (int t = 0; t < kL2Per; ++t) {
                    const int e = (int)((v[t] >> 23) & 0xFFu);
                    const int sh1 = e - el + 6;
                    if (e != 0 && sh1 >= 0) {
                        s1 = mad_wide(((v[t] | 0x800000u) & 0xFFFFFFu) << sh1, s1);
                    } else if (e != 0 && sh1 >= -7) {
                        s2 = mad_wide(((v[t] | 0x800000u) & 0xFFFFFFu) << (sh1 + 7), s2);
                    } else if (v[t] & 0x7FFFFFFFu) {
                        // small or subnormal: (m^2 << 64) >> 2 (emax - e) into the 128-bit sum
                        const unsigned mm = e ? ((v[t] | 0x800000u) & 0xFFFFFFu) : (v[t] & 0x7FFFFFu);
                        const int sh = 2 * (emax - (e ? e : 1));
                        const unsigned long long sq = (unsigned long long)mm * mm;
                        if (sh < 64) add128(hi, lo, sq >> sh, sh ? sq << (64 - sh) : 0ull);
                        else if (sh < 112) add128(hi, lo, 0ull, sq >> (sh - 64));
                    }
                }
                add128_shifted(hi, lo, s1, 52 - 2 * (emax - el));
                add128_shifted(hi, lo, s2, 38 - 2 * (emax - el));
                if constexpr (SPLIT) {
                    const int col0 = k0 + kL2Per * sub;
                    float a[kL2Per];
#pragma unroll
                    for (int t = 0; t < kL2Per; ++t) {
                        a[t] = col0 + t < d ? __uint_as_float(v[t]) - c[col0 + t] : 0.f;
                        n2 = fmaf(a[t], a[t], n2);
                    }
                    __nv_bfloat16* dst = xh + row * dp + col0;
                    if (live && col0 + kL2Per <= dp) {
                        uint32_t w[4];
#pragma unroll
                        for (int t = 0; t < kL2Per; t += 2) {
                            const __nv_bfloat162 h = __floats2bfloat162_rn(a[t], a[t + 1]);
                            w[t >> 1] = *reinterpret_cast<const uint32_t*>(&h);
                        }
                        *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
                    } else if (live) {
                        for (int t = 0; t < kL2Per && col0 + t < dp; ++t) dst[t] = __float2bfloat16_rn(a[t]);
                    }
                }
            }
            if constexpr (SPLIT) {
#pragma unroll
                for (int o = G / 2; o; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
                if (sub == 0 && live) xn2[row] = n2;
            }
#pragma unroll
            for (int o = G / 2; o; o >>= 1) {
                const unsigned long long oh = __shfl_xor_sync(0xffffffffu, hi, o);
                const unsigned long long ol = __shfl_xor_sync(0xffffffffu, lo, o);
                add128(hi, lo, oh, ol);
            }
            if (kPar > 1) {                                        // lane l: the sum of group l % kPar
                const int src = (lane & (kPar - 1)) * G;
                hi = __shfl_sync(0xffffffffu, hi, src);
                lo = __shfl_sync(0xffffffffu, lo, src);
                emax = __shfl_sync(0xffffffffu, emax, src);
                special = __shfl_sync(0xffffffffu, special, src);
            }
            if (lane / kPar == i) {
                my_hi = hi;
                my_lo = lo;
                my_emax = emax;
                my_special = special;
            }
        }
        if (lane < rows) f[(r0 + lane) * m + j] = l2_finish(my_hi, my_lo, my_emax, my_special);
    }
}

// Enough warps for the chip first (a row at a time each), then rows per warp.
template <bool SPLIT, int G>
cudaError_t launch_l2(const float* X, int64_t n, int32_t d, int64_t ld, double* f, int m, int j, const float* c, int dp,
                      void* xh, float* xn2, cudaStream_t s)
{
    constexpr int kPar = 32 / G;
    constexpr int64_t kWarps = 152 * 8 * 8;
    const int iters = (int)std::max<int64_t>(1, std::min<int64_t>(G, n / (kWarps * kPar)));
    const int blocks = (int)std::min<int64_t>(div_up(n, 8 * kPar * iters), 152 * 8);
    lens_l2_exact_kernel<SPLIT, G><<<blocks, 256, 0, s>>>(X, n, d, ld, iters, f, m, j, c, dp,
                                                          static_cast<__nv_bfloat16*>(xh), xn2);
    note_launch();
    return cudaGetLastError();
}

template <bool SPLIT>
cudaError_t launch_l2_by_width(const float* X, int64_t n, int32_t d, int64_t ld, double* f, int m, int j,
                               const float* c, int dp, void* xh, float* xn2, cudaStream_t s)
{
    if (d <= 4 * kL2Per) return launch_l2<SPLIT, 4>(X, n, d, ld, f, m, j, c, dp, xh, xn2, s);
    if (d <= 8 * kL2Per) return launch_l2<SPLIT, 8>(X, n, d, ld, f, m, j, c, dp, xh, xn2, s);
    if (d <= 16 * kL2Per) return launch_l2<SPLIT, 16>(X, n, d, ld, f, m, j, c, dp, xh, xn2, s);
    return launch_l2<SPLIT, 32>(X, n, d, ld, f, m, j, c, dp, xh, xn2, s);
}

// a + b = s + e exactly (FP32)
__device__ __forceinline__ float two_sum(float a, float b, float& e)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

// Column sums of a row block for the eccentricity, as col_partial_sum_kernel,
// but in FP32 expansions: (s, e, e2) with s + e + e2 the sum up to 2^-70 of its
// magnitude, so the FP64 pipe sees three conversions a column instead of an add
// a value, and the rows of a block split over the warps of a CTA (their sums
// added in order). A batch holding a value of magnitude above 2^100 or below
// 2^-80 (whose roundings might fall outside FP32) takes FP64 adds. *flag: set if
// a value is NaN or Inf. One CTA per (32 columns, row block).
constexpr int kEccWarps = 8;

__device__ __forceinline__ bool mid_range(float x)      // zero, or 2^-80 <= |x| < 2^100
{
    const unsigned t = __float_as_uint(x) & 0x7FFFFFFFu;
    return t == 0u || t - (47u << 23) < (180u << 23);
}

__global__ void __launch_bounds__(32 * kEccWarps) col_sum_exp_kernel(const float* __restrict__ X, int64_t n, int32_t d,
                                                                     int64_t ld, double* __restrict__ part, int* flag)
{
    __shared__ double s_sum[kEccWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = min((int)blockIdx.y * 32 + lane, d - 1);         // (lanes past d: the last column again)
    const int64_t r0 = (int64_t)blockIdx.x * kMeanRows;
    const int rows = (int)min((int64_t)kMeanRows, n - r0);
    const float* x = X + r0 * ld + c;
    float s = 0.f, e = 0.f, e2 = 0.f;
    double wide = 0.0;
    bool bad = false;
    for (int r = warp * 16; r < rows; r += kEccWarps * 16) {
        float v[16];
        bool mid = true;
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = r + i < rows ? __ldg(x + (int64_t)(r + i) * ld) : 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) mid &= mid_range(v[i]);
        if (__all_sync(0xffffffffu, mid)) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                float a, b;
                s = two_sum(s, v[i], a);
                e = two_sum(e, a, b);
                e2 = __fadd_rn(e2, b);
            }
        } else {
#pragma unroll 4
            for (int i = 0; i < 16; ++i) {
                wide += (double)v[i];
                bad |= !isfinite(v[i]);
            }
        }
    }
    s_sum[warp][lane] = wide + ((double)s + ((double)e + (double)e2));
    if (__syncthreads_or(bad) && flag && threadIdx.x == 0) atomicOr(flag, 1);
    if (warp == 0 && blockIdx.y * 32 + lane < d) {
        double t = 0.0;
        for (int w = 0; w < kEccWarps; ++w) t += s_sum[w][lane];
        part[(int64_t)blockIdx.x * d + c] = t;
    }
}

// Two columns at a time (each half rounded as the scalar instruction).
using f2 = unsigned long long;
__device__ __forceinline__ f2 f2_add(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_neg(f2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b)
{
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// a + b (a - b) = the result + e exactly
__device__ __forceinline__ f2 two_sum(f2 a, f2 b, f2& e)
{
    const f2 s = f2_add(a, b), bb = f2_sub(s, a);
    e = f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb));
    return s;
}
__device__ __forceinline__ f2 two_diff(f2 a, f2 b, f2& e)
{
    const f2 s = f2_sub(a, b), bb = f2_sub(s, a);
    e = f2_sub(f2_sub(a, f2_sub(s, bb)), f2_add(b, bb));
    return s;
}
// the same where |a| >= |b| or a = 0
__device__ __forceinline__ f2 fast_sum(f2 a, f2 b, f2& e)
{
    const f2 s = f2_add(a, b);
    e = f2_sub(b, f2_sub(s, a));
    return s;
}

// |x - mu|^2 of every row for the eccentricity. In FP64 that is a subtract and
// an FMA a value, which the FP64 pipe takes 0.84 ms for at 1M x 256; here two
// columns at a time take ~51 packed FP32 instructions, bound by the FP32 pipe. The
// mean's 53 bits are three floats, because what is cut from it shifts a whole
// column by a part of |mu|, however small x - mu is. t = x - mu as th + tl + t3 (to
// 2^-72 of |t| and |mu|):
//   x - m1 = y + a and a - m2 = v + b exactly; |y| >= |v| or y = 0 (x and m1 within
//   a factor of 2: a = 0 and y is a multiple of half an ulp of m1 or 0; else |y| is
//   half the larger of them or more), so y + v = th + c by the short sum; c + (b - m3)
//   likewise, up to 2^-24 of b, which is 2^-48 of |x| and |mu|.
// th^2 = p + pe and 2 th tl = q + qe exactly, qe + tl^2 + 2 th t3 in two FMAs, and a
// 32-column sum of them as an FP32 expansion of three terms a half, added to the
// row's FP64 sum. The roundings are below 2^-68 of a value's square, so a row's error
// is that of its d / 32 FP64 adds, against two FP64 roundings a value (largest
// relative error over 3000 rows, means 0 to 1e6: 1.1e-16 at 1 to 8 columns, 3.2e-16
// at 256; the FP64 form 4.7e-16 and 1.7e-15). A chunk where some |t| is not zero or
// in [2^-40, 2^55) is summed in FP64 instead (subtract and FMA, columns in order).
// One thread a row, as lens_rows_kernel. One column at a time, with two-sums
// throughout, the call of 1M x 256 took 990 us, now 900.
constexpr int kEccPitch = kChunk + 2;          // (a thread's pairs of columns: no bank conflicts)

__global__ void __launch_bounds__(kRows) ecc_rows_kernel(const float* __restrict__ X, int64_t n, int32_t d, int64_t ld,
                                                         const double* __restrict__ mu, double* __restrict__ f, int m,
                                                         int j)
{
    __shared__ __align__(16) float tile[kRows][kEccPitch];
    __shared__ double smu[kChunk];
    __shared__ __align__(16) float sm12[kChunk / 2][4];        // the mean's floats: m1 of two columns, m2 of two
    __shared__ __align__(8) float sm3[kChunk];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t row0 = (int64_t)blockIdx.x * kRows;
    const bool vec = ld % 4 == 0 && ((uintptr_t)X & 15) == 0;
    double acc = 0.0;
    for (int32_t k0 = 0; k0 < d; k0 += kChunk) {
        const int kc = min(kChunk, d - k0);
        if (vec && kc == kChunk) {
            // 16 bytes a lane: 8 lanes a row, 4 rows a warp at a time
#pragma unroll
            for (int i = 0; i < kRows / 16; ++i) {
                const int r = warp * 4 + (lane >> 3) + 16 * i, c4 = (lane & 7) * 4;
                const int64_t row = row0 + r;
                float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                if (row < n) x = __ldg(reinterpret_cast<const float4*>(X + row * ld + k0 + c4));
                *reinterpret_cast<float2*>(&tile[r][c4]) = make_float2(x.x, x.y);
                *reinterpret_cast<float2*>(&tile[r][c4 + 2]) = make_float2(x.z, x.w);
            }
        } else {
#pragma unroll 8
            for (int r = warp; r < kRows; r += kRows / 32) {
                const int64_t row = row0 + r;
                float x = 0.f;
                if (row < n && lane < kc) x = __ldg(X + row * ld + k0 + lane);
                tile[r][lane] = x;
            }
        }
        if (tid < kChunk) {                                        // (columns past d: x = mu = 0)
            const double mk = tid < kc ? mu[k0 + tid] : 0.0;
            const float m1 = (float)mk;
            const double rest = mk - (double)m1;                   // (exact)
            const float m2 = (float)rest;
            smu[tid] = mk;
            sm12[tid >> 1][tid & 1] = m1;
            sm12[tid >> 1][2 + (tid & 1)] = m2;
            sm3[tid] = (float)(rest - (double)m2);
        }
        __syncthreads();
        f2 s = 0ull, e = 0ull, e2 = 0ull;
        unsigned lo = ~0u, hi = 0u;                                // 2 |th| as bits: smallest (not 0) less 1, largest
        const int pairs = (kc + 1) / 2;
#pragma unroll 2
        for (int k = 0; k < pairs; ++k) {
            const ulonglong2 m12 = *reinterpret_cast<const ulonglong2*>(sm12[k]);
            const f2 m3 = *reinterpret_cast<const f2*>(&sm3[2 * k]);
            f2 a, b, c, t3, err;
            const f2 y = two_diff(*reinterpret_cast<const f2*>(&tile[tid][2 * k]), m12.x, a);
            const f2 v = two_diff(a, m12.y, b);
            const f2 th = fast_sum(y, v, c);
            const f2 tl = fast_sum(c, f2_sub(b, m3), t3);
            const f2 p = f2_mul(th, th), h2 = f2_add(th, th), q = f2_mul(h2, tl);
            const f2 pe = f2_fma(th, th, f2_neg(p));
            const f2 rest = f2_fma(h2, t3, f2_fma(tl, tl, f2_fma(h2, tl, f2_neg(q))));
            float th0, th1, s0, s1, p0, p1;
            f2_unpack(th, th0, th1);
            const unsigned b0 = __float_as_uint(th0) << 1, b1 = __float_as_uint(th1) << 1;
            hi = max(hi, max(b0, b1));
            lo = min(lo, min(b0 - 1u, b1 - 1u));
            // (both are sums of squares: the larger one first)
            f2_unpack(s, s0, s1);
            f2_unpack(p, p0, p1);
            s = fast_sum(f2_pack(fmaxf(s0, p0), fmaxf(s1, p1)), f2_pack(fminf(s0, p0), fminf(s1, p1)), err);
            e = two_sum(e, err, b);
            e2 = f2_add(e2, b);
            e = two_sum(e, pe, b);
            e2 = f2_add(e2, b);
            e = two_sum(e, q, b);
            e2 = f2_add(e2, f2_add(b, rest));
        }
        // 2^-40 and 2^55 as bits
        if (lo >= (87u << 24) - 1u && hi < (182u << 24)) {
            float s0, s1, e0, e1, l0, l1, err, b0, b1;
            f2_unpack(s, s0, s1);
            f2_unpack(e, e0, e1);
            f2_unpack(e2, l0, l1);
            const float sum = two_sum(s0, s1, err);
            const float low = two_sum(two_sum(e0, e1, b0), err, b1);
            acc += (double)sum + ((double)low + (double)__fadd_rn(__fadd_rn(l0, l1), __fadd_rn(b0, b1)));
        } else {
            for (int k = 0; k < kc; ++k) {
                const double t = __dsub_rn((double)tile[tid][k], smu[k]);
                acc = __fma_rn(t, t, acc);
            }
        }
        __syncthreads();
    }
    const int64_t row = row0 + tid;
    if (row < n) f[row * m + j] = acc;
}

// Mean of f[r * m + j] over the rows: per-block sums (rows strided over the
// threads, then a shuffle and shared-memory tree), then one block adds the
// block sums in a fixed order (the same result run to run).
constexpr int kMeanBlocks = 512;

__global__ void __launch_bounds__(256) col_lens_partial_kernel(const double* __restrict__ f, int64_t n, int m,
                                                               int j, double* __restrict__ part)
{
    __shared__ double ws[8];
    double s = 0.0;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
        s += f[r * m + j];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += ws[w];
        part[blockIdx.x] = t;
    }
}

// f = sqrt(q + V), V = (sum of the nb <= 512 block sums) / n, added up by every
// block in the same tree
__global__ void __launch_bounds__(256) ecc_finish_kernel(double* __restrict__ f, int64_t n, int m, int j,
                                                         const double* __restrict__ part, int nb)
{
    __shared__ double ws[8];
    double t = 0.0;
    for (int b = threadIdx.x; b < nb; b += 256) t += part[b];
    for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = t;
    __syncthreads();
    t = 0.0;
    for (int w = 0; w < 8; ++w) t += ws[w];
    const double V = t / (double)n;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
        f[r * m + j] = __dsqrt_rn(__dadd_rn(f[r * m + j], V));
}

__global__ void lens_coord_kernel(const float* __restrict__ X, int64_t n, int64_t ld, int32_t col,
                                  double* __restrict__ f, int m, int j)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) f[p * m + j] = (double)X[p * ld + col];
}

// L-infinity norm max_k |x_k|: one warp per row, lanes over columns, a
// NaN-propagating maximum (exact: no arithmetic, FP32 values widen exactly).
__global__ void __launch_bounds__(256) lens_linf_kernel(const float* __restrict__ X, int64_t n, int32_t d,
                                                        int64_t ld, double* __restrict__ f, int m, int j)
{
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = w0; r < n; r += nw) {
        const float* x = X + r * ld;
        float mx = 0.f;
        for (int k = lane; k < d; k += 32) {
            const float v = fabsf(__ldg(x + k));
            if (v > mx || v != v) mx = v;
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const float v = __shfl_xor_sync(0xffffffffu, mx, o);
            if (v > mx || v != v) mx = v;
        }
        if (lane == 0) f[r * m + j] = (double)mx;
    }
}

// One warp per row (grid-stride), lanes over columns, 16-byte loads when
// the rows allow them.
__global__ void __launch_bounds__(256) finite_kernel(const float* __restrict__ X, int64_t n, int32_t d, int64_t ld,
                                                     bool vec, int* flag)
{
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    bool bad = false;
    for (int64_t r = w0; r < n; r += nw) {
        const float* x = X + r * ld;
        if (vec) {
            const int d4 = d >> 2;
            for (int c = lane; c < d4; c += 32) {
                const float4 v = __ldg(reinterpret_cast<const float4*>(x) + c);
                bad |= !(isfinite(v.x) && isfinite(v.y) && isfinite(v.z) && isfinite(v.w));
            }
            for (int c = 4 * d4 + lane; c < d; c += 32) bad |= !isfinite(__ldg(x + c));
        } else {
            for (int c = lane; c < d; c += 32) bad |= !isfinite(__ldg(x + c));
        }
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
}

// --------------------------------------------------------------------- PCA
// Column means: partial FP64 sums per row block, rows in order, then a
// fixed-order reduce (deterministic run to run). One warp per (32 columns, row
// block): the sum is a chain of FP64 adds, so the next 32 rows are loaded
// while the current ones are added, and the columns spread over the SMs (the
// FP64 pipe takes 16 cycles for a warp's add). 1M x 256: 1.17 -> 0.54 ms.
constexpr int kMeanAhead = 32;

__global__ void __launch_bounds__(32) col_partial_sum_kernel(const float* __restrict__ X, int64_t n, int32_t d,
                                                             int64_t ld, double* __restrict__ part)
{
    const int c = min(blockIdx.y * 32 + (int)threadIdx.x, d - 1);  // (lanes past d: the last column again)
    const int64_t r0 = (int64_t)blockIdx.x * kMeanRows;
    const int64_t r1 = min(n, r0 + kMeanRows);
    const float* x = X + r0 * ld + c;
    const int rows = (int)(r1 - r0);
    float cur[kMeanAhead], nxt[kMeanAhead];
#pragma unroll
    for (int i = 0; i < kMeanAhead; ++i) cur[i] = i < rows ? __ldg(x + i * ld) : 0.f;
    double s = 0.0;
    for (int r = 0; r < rows; r += kMeanAhead) {
#pragma unroll
        for (int i = 0; i < kMeanAhead; ++i) {
            const int q = r + kMeanAhead + i;
            nxt[i] = q < rows ? __ldg(x + q * ld) : 0.f;
        }
        bool all_plain = true;
#pragma unroll
        for (int i = 0; i < kMeanAhead; ++i) all_plain &= plain(cur[i]);
        if (__all_sync(0xffffffffu, all_plain)) {                  // (rows past the end add 0)
#pragma unroll
            for (int i = 0; i < kMeanAhead; ++i) s += widen(cur[i]);
        } else {
#pragma unroll
            for (int i = 0; i < kMeanAhead; ++i) s += (double)cur[i];
        }
#pragma unroll
        for (int i = 0; i < kMeanAhead; ++i) cur[i] = nxt[i];
    }
    part[(int64_t)blockIdx.x * d + c] = s;
}

__global__ void __launch_bounds__(32) col_mean_kernel(const double* __restrict__ part, int nblk, int32_t d, int64_t n,
                                                      double* __restrict__ mu)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d) return;
    double s = 0.0;
#pragma unroll 16
    for (int b = 0; b < nblk; ++b) s += __ldg(part + (int64_t)b * d + c);
    mu[c] = s / (double)n;
}

// xc = (float)((double)x - mu), the centred rows of the covariance (n x d),
// without the FP64 pipe (three of its slots a value) for all but a few values:
// with mu = mh + ml + rest (FP32 parts), x - mh = s + e exactly (two-sum),
// t = e - ml and s + t = res + r2 exactly, so the true difference is
// res + r2 + delta, |delta| <= 2^-22 (|t| + |ml|); where that stays strictly
// inside half an ulp of res (by more than the 2^-53 of a rounding to double),
// res is the rounding. Otherwise, and for Inf, NaN, powers of two and small
// values, the FP64 expression itself decides.
// (not inlined: the compiler would predicate the FP64 instructions, and every
// value would pay for them)
__device__ __noinline__ float centred_fp64(float v, const double* mu)
{
    return (float)((double)v - *mu);
}

__global__ void __launch_bounds__(256) centre_rows_kernel(const float* __restrict__ X, int64_t n, int32_t d, int64_t ld,
                                                          const double* __restrict__ mu, float* __restrict__ xc)
{
    extern __shared__ float2 s_mu[];
    for (int k = threadIdx.x; k < d; k += blockDim.x) {
        const double m = mu[k];
        const float mh = (float)m;
        s_mu[k] = make_float2(mh, (float)(m - (double)mh));
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = w0; r < n; r += nw) {
        const float* x = X + r * ld;
        float* o = xc + r * d;
#pragma unroll 4
        for (int k = lane; k < d; k += 32) {
            const float v = __ldg(x + k);
            const float2 m = s_mu[k];
            const float s = __fsub_rn(v, m.x);
            const float bb = __fsub_rn(s, v);
            const float e = __fsub_rn(__fsub_rn(v, __fsub_rn(s, bb)), __fadd_rn(m.x, bb));
            const float t = __fsub_rn(e, m.y);
            float res = __fadd_rn(s, t);
            const float b2 = __fsub_rn(res, s);
            const float r2 = __fadd_rn(__fsub_rn(s, __fsub_rn(res, b2)), __fsub_rn(t, b2));
            const unsigned bits = __float_as_uint(res);
            const unsigned ex = bits & 0x7F800000u;
            // half an ulp of res, less a 2^-12 part of it
            const float half = __fmul_rn(__uint_as_float(ex), 5.9604645e-8f * (1.f - 0.000244140625f));
            const float off = __fmaf_rn(2.3841858e-7f, __fadd_rn(fabsf(t), fabsf(m.y)), fabsf(r2));
            if (!(off < half) || (bits & 0x7FFFFFu) == 0u || ex < (64u << 23) || ex == 0x7F800000u)
                res = centred_fp64(v, mu + k);
            o[k] = res;
        }
    }
}

// FP32 covariance tiles: CTA (tile, chunk) accumulates the 32 x 32 tile
// (ti, tj), tj >= ti, of sum_p xc_p xc_p^T over its row chunk, each entry an
// FMA chain over the chunk's rows in order. 64 threads with 4 x 4 entries each:
// the tiles are small so that a cloud of a hundred thousand rows x 64 columns
// still fills the SMs (49 chunks x 3 tiles at 100k x 64: 476 -> 89 us with the
// rows centred once, 26 us; 500k x 128: 1475 -> 390 + 370 us).
// The centred rows take at most kCentredBytes at a time, so that no second cloud
// stands beside a large one (600k x 256 held 658 MB of scratch), and
// 500k x 128 is still one block of large launches.
constexpr size_t kCentredBytes = size_t(256) << 20;
constexpr int kCovT = 32;
constexpr int kCovRows = 2048;
constexpr int kCovStep = 32;

__device__ __forceinline__ void cov_tile(int t, int ntile, int* ti, int* tj)
{
    int i = 0;
    while (t >= ntile - i) { t -= ntile - i; ++i; }
    *ti = i;
    *tj = i + t;
}

__global__ void __launch_bounds__(64) cov_partial_kernel(const float* __restrict__ xc, int64_t n, int32_t d,
                                                         float* __restrict__ part, int ntile)
{
    __shared__ __align__(16) float sa[kCovStep][kCovT], sb[kCovStep][kCovT];
    int ti, tj;
    cov_tile(blockIdx.x, ntile, &ti, &tj);
    const int chunk = blockIdx.y, tid = threadIdx.x;
    const int tx = tid & 7, ty = tid >> 3;
    const int lane = tid & 31, warp = tid >> 5;
    const int ca = ti * kCovT + lane, cb = tj * kCovT + lane;
    float acc[4][4] = {};
    const int64_t r0 = (int64_t)chunk * kCovRows, r1 = min(n, r0 + kCovRows);
    float ra[kCovStep / 2], rb[kCovStep / 2];               // the next step's rows warp, warp + 2, ..
    auto load = [&](int64_t r) {
#pragma unroll
        for (int i = 0; i < kCovStep / 2; ++i) {
            const int64_t row = r + warp + 2 * i;
            ra[i] = row < r1 && ca < d ? __ldg(xc + row * d + ca) : 0.f;
            rb[i] = row < r1 && cb < d ? __ldg(xc + row * d + cb) : 0.f;
        }
    };
    load(r0);
    for (int64_t r = r0; r < r1; r += kCovStep) {
#pragma unroll
        for (int i = 0; i < kCovStep / 2; ++i) {
            sa[warp + 2 * i][lane] = ra[i];
            sb[warp + 2 * i][lane] = rb[i];
        }
        __syncthreads();
        if (r + kCovStep < r1) load(r + kCovStep);
#pragma unroll 8
        for (int k = 0; k < kCovStep; ++k) {
            const float4 a4 = *reinterpret_cast<const float4*>(&sa[k][ty * 4]);
            const float4 b4 = *reinterpret_cast<const float4*>(&sb[k][tx * 4]);
            const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[i][q] = fmaf(a[i], b[q], acc[i][q]);
        }
        __syncthreads();
    }
    float* out = part + ((int64_t)chunk * gridDim.x + blockIdx.x) * kCovT * kCovT;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4*>(out + (ty * 4 + i) * kCovT + tx * 4) =
            make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
}

// One thread per entry: the chunks' partials added in order (a chain of FP64
// adds, the loads ahead of it).
__global__ void __launch_bounds__(128) cov_reduce_kernel(const float* __restrict__ part, int nchunk, int ntile,
                                                         int32_t d, int64_t n, double* __restrict__ C)
{
    const int e = blockIdx.y * blockDim.x + threadIdx.x;
    int ti, tj;
    cov_tile(blockIdx.x, ntile, &ti, &tj);
    const int i = ti * kCovT + e / kCovT, k = tj * kCovT + e % kCovT;
    if (i >= d || k >= d) return;
    const int64_t step = (int64_t)gridDim.x * kCovT * kCovT;
    const float* p = part + (int64_t)blockIdx.x * kCovT * kCovT + e;
    double s = 0.0;
#pragma unroll 16
    for (int c = 0; c < nchunk; ++c) s += (double)__ldg(p + c * step);
    s /= (double)n;
    C[(int64_t)i * d + k] = s;
    C[(int64_t)k * d + i] = s;
}

// Warp sums of NJ values per lane at once: out of p[j] on 32 lanes, the sum
// over the lanes of every p[j] in the order of a butterfly (16, 8, 4, 2, 1),
// returned on the lanes seg_lane<NJ>(j). A butterfly of every value by itself
// would spend 5 FP64 adds of a whole warp on each; here lanes that have no
// part in one value's next level carry another value's.
template <int NJ>
__device__ __forceinline__ double warp_sums(const double (&p)[NJ], int lane)
{
    double q[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) q[j] = p[j];
    int o = 16;
#pragma unroll
    for (int m = NJ; m > 1; m >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < m / 2; ++i) {
            const double a = q[2 * i], b = q[2 * i + 1];
            q[i] = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, o);
        }
    }
    double y = q[0];
    for (; o; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
    return y;
}

template <int NJ>
__device__ __forceinline__ int seg_lane(int j)
{
    int l = 0, o = 16;
#pragma unroll
    for (int m = NJ; m > 1; m >>= 1, o >>= 1, j >>= 1)
        if (j & 1) l |= o;
    return l;
}

// sum over the segments (columns 32 j ..) of their warp sums, in order
template <int NJ>
__device__ __forceinline__ double vec_sum(const double (&p)[NJ], int lane)
{
    const double y = warp_sums<NJ>(p, lane);
    double t = 0.0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) t += __shfl_sync(0xffffffffu, y, seg_lane<NJ>(j));
    return t;
}

// Power iteration (as power_iter_kernel, the same operations in the same
// order) for d <= 32 NJ <= 256 on a cluster of kPowCluster CTAs. An iteration
// is a d x d product and a few vector sums, bound by the FP64 pipe of the SMs
// taking part and by latency: each warp keeps two rows of C in registers, its
// products go to every CTA's shared memory, one cluster barrier, and the first
// warp of every CTA does the vector work for itself (lane l holds columns
// l + 32 j, as the products need them).
// 100k x 64, one axis: 3.52 -> 0.79 ms; 500k x 128, two axes: 1.47 -> 0.33 ms
// (one CTA of 1024 threads before).
constexpr int kPowCluster = 8;

template <int NJ>
__global__ void __launch_bounds__(512) power_iter_cluster_kernel(const double* __restrict__ C, int32_t d, int K,
                                                                 double* __restrict__ axes, int* status)
{
    extern __shared__ double s_axes[];                       // K x 32 NJ: the axes found so far
    __shared__ double s_w[2][32 * NJ], s_v[32 * NJ];
    __shared__ int s_stop;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int row = 2 * (rank * nwarp + warp);               // the warp's rows row, row + 1
    double c0[NJ], c1[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j;
        c0[j] = row < d && k < d ? C[(int64_t)row * d + k] : 0.0;
        c1[j] = row + 1 < d && k < d ? C[(int64_t)(row + 1) * d + k] : 0.0;
    }
    for (int k = threadIdx.x; k < 64 * NJ; k += blockDim.x) (&s_w[0][0])[k] = 0.0;
    cluster.sync();                                          // cleared before any CTA writes
    int not_conv = 0, buf = 0;
    for (int c = 0; c < K; ++c) {
        double v[NJ];
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const int k = lane + 32 * j;
            v[j] = k < d ? 1.0 + 0.25 * (double)((k * 7919) % 13) : 0.0;
        }
        for (int it = 0; it < 2000; ++it, buf ^= 1) {
            double p[2] = {0.0, 0.0};
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                p[0] = __fma_rn(c0[j], v[j], p[0]);
                p[1] = __fma_rn(c1[j], v[j], p[1]);
            }
            const double y = warp_sums<2>(p, lane);          // lane 0: row, lane 16: row + 1
            const double w0 = __shfl_sync(0xffffffffu, y, 0), w1 = __shfl_sync(0xffffffffu, y, 16);
            if (lane < kPowCluster) {
                double* dst = cluster.map_shared_rank(&s_w[buf][0], lane);
                if (row < d) dst[row] = w0;
                if (row + 1 < d) dst[row + 1] = w1;
            }
            cluster.sync();
            if (warp == 0) {
                double w[NJ], t[NJ];
#pragma unroll
                for (int j = 0; j < NJ; ++j) w[j] = s_w[buf][lane + 32 * j];
                for (int q = 0; q < c; ++q) {                // orthogonalise against earlier axes
                    const double* ax = s_axes + q * 32 * NJ;
#pragma unroll
                    for (int j = 0; j < NJ; ++j) t[j] = __dmul_rn(ax[lane + 32 * j], w[j]);
                    const double proj = vec_sum<NJ>(t, lane);
#pragma unroll
                    for (int j = 0; j < NJ; ++j) w[j] = __fma_rn(-proj, ax[lane + 32 * j], w[j]);
                }
#pragma unroll
                for (int j = 0; j < NJ; ++j) t[j] = __dmul_rn(w[j], w[j]);
                const double norm = sqrt(vec_sum<NJ>(t, lane));
                const double inv = norm > 0.0 ? 1.0 / norm : 0.0;
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const double nv = w[j] * inv;
                    const double dv = nv - v[j];
                    t[j] = __dmul_rn(dv, dv);
                    v[j] = nv;
                    s_v[lane + 32 * j] = nv;
                }
                const double diff = vec_sum<NJ>(t, lane);
                if (lane == 0) s_stop = diff < 1e-14;        // ||dv|| < 1e-7
            }
            __syncthreads();
            const int stop = s_stop;
            if (warp > 0) {
#pragma unroll
                for (int j = 0; j < NJ; ++j) v[j] = s_v[lane + 32 * j];
            }
            __syncthreads();
            if (stop) { buf ^= 1; break; }                   // (the same in every CTA)
            if (it == 1999) not_conv = 1;
        }
        // sign rule: the first entry of largest magnitude is positive
        if (warp == 0) {
            double best = -1.0, val = 0.0;
            int at = 0;
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const int k = lane + 32 * j;
                if (k < d && fabs(v[j]) > best) { best = fabs(v[j]); val = v[j]; at = k; }
            }
            for (int o = 16; o; o >>= 1) {
                const double ob = __shfl_xor_sync(0xffffffffu, best, o), ov = __shfl_xor_sync(0xffffffffu, val, o);
                const int oa = __shfl_xor_sync(0xffffffffu, at, o);
                if (ob > best || (ob == best && oa < at)) { best = ob; val = ov; at = oa; }
            }
            const double sign = val < 0.0 ? -1.0 : 1.0;
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const int k = lane + 32 * j;
                const double a = sign * v[j];
                s_axes[c * 32 * NJ + k] = k < d ? a : 0.0;
                if (rank == 0 && k < d) axes[(int64_t)c * d + k] = a;
            }
        }
        __syncthreads();
    }
    if (rank == 0 && threadIdx.x == 0) *status = not_conv;
    cluster.sync();                                          // no CTA leaves while another may write to it
}

// Power iteration for the top-K eigenvectors of C (d x d, FP64), one CTA.
// Each axis is orthogonalised against the earlier ones every step (deflation
// by projection), iterated until ||v_new - v|| < 1e-7 or 2000 steps, then
// signed so its entry of largest magnitude is positive (ties: lowest index).
__global__ void __launch_bounds__(1024) power_iter_kernel(const double* __restrict__ C, int32_t d,
                                                          int K, double* __restrict__ axes,
                                                          int* status)
{
    extern __shared__ double sm[];
    double* v = sm;           // d
    double* w = sm + d;       // d
    __shared__ double red[32];
    __shared__ double s_norm, s_diff;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    int not_conv = 0;
    for (int c = 0; c < K; ++c) {
        for (int k = tid; k < d; k += blockDim.x) v[k] = 1.0 + 0.25 * (double)((k * 7919) % 13);
        __syncthreads();
        for (int it = 0; it < 2000; ++it) {
            // w = C v
            for (int r = warp; r < d; r += nwarp) {
                double s = 0.0;
                for (int k = lane; k < d; k += 32) s += C[(int64_t)r * d + k] * v[k];
                for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) w[r] = s;
            }
            __syncthreads();
            // orthogonalise against earlier axes
            for (int q = 0; q < c; ++q) {
                double s = 0.0;
                for (int k = tid; k < d; k += blockDim.x) s += axes[q * d + k] * w[k];
                for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) red[warp] = s;
                __syncthreads();
                if (tid == 0) { double t = 0; for (int i = 0; i < nwarp; ++i) t += red[i]; s_norm = t; }
                __syncthreads();
                const double proj = s_norm;
                for (int k = tid; k < d; k += blockDim.x) w[k] -= proj * axes[q * d + k];
                __syncthreads();
            }
            double s = 0.0;
            for (int k = tid; k < d; k += blockDim.x) s += w[k] * w[k];
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) red[warp] = s;
            __syncthreads();
            if (tid == 0) { double t = 0; for (int i = 0; i < nwarp; ++i) t += red[i]; s_norm = sqrt(t); }
            __syncthreads();
            const double inv = s_norm > 0.0 ? 1.0 / s_norm : 0.0;
            double dd = 0.0;
            for (int k = tid; k < d; k += blockDim.x) {
                const double nv = w[k] * inv;
                dd += (nv - v[k]) * (nv - v[k]);
                v[k] = nv;
            }
            for (int o = 16; o; o >>= 1) dd += __shfl_xor_sync(0xffffffffu, dd, o);
            if (lane == 0) red[warp] = dd;
            __syncthreads();
            if (tid == 0) { double t = 0; for (int i = 0; i < nwarp; ++i) t += red[i]; s_diff = t; }
            __syncthreads();
            if (s_diff < 1e-14) break;           // ||dv|| < 1e-7
            if (it == 1999) not_conv = 1;
        }
        // sign rule
        if (tid == 0) {
            int arg = 0;
            for (int k = 1; k < d; ++k)
                if (fabs(v[k]) > fabs(v[arg])) arg = k;
            s_norm = v[arg] < 0.0 ? -1.0 : 1.0;
        }
        __syncthreads();
        for (int k = tid; k < d; k += blockDim.x) axes[c * d + k] = s_norm * v[k];
        __syncthreads();
    }
    if (tid == 0) *status = not_conv;
}

}  // namespace

cudaError_t lens_l2_split(const float* X, int64_t n, int32_t d, int64_t ld, double* f, int m, int j,
                          const float* c, int dp, void* xh, float* xn2, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    if (d > 32768) return cudaErrorInvalidValue;
    return launch_l2_by_width<true>(X, n, d, ld, f, m, j, c, dp, xh, xn2, s);
}

cudaError_t lens_l2(const float* X, int64_t n, int32_t d, int64_t ld, double* f, int m, int j,
                    cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    if (d <= 32768) return launch_l2_by_width<false>(X, n, d, ld, f, m, j, nullptr, 0, nullptr, nullptr, s);
    lens_rows_kernel<0><<<div_up(n, kRows), kRows, 0, s>>>(X, n, d, ld, nullptr, nullptr, nullptr, f, m, j);
    note_launch();
    return cudaGetLastError();
}

cudaError_t lens_project(const float* X, int64_t n, int32_t d, int64_t ld, const double* mu,
                         const double* v, double* f, int m, int j, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    { lens_rows_kernel<1><<<div_up(n, kRows), kRows, 0, s>>>(X, n, d, ld, mu, v, nullptr, f, m, j); note_launch(); }
    return cudaGetLastError();
}

cudaError_t lens_project2(const float* X, int64_t n, int32_t d, int64_t ld, const double* mu, const double* v0,
                          const double* v1, double* f, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    { lens_rows_kernel<3><<<div_up(n, kRows), kRows, 0, s>>>(X, n, d, ld, mu, v0, v1, f, 2, 0); note_launch(); }
    return cudaGetLastError();
}

cudaError_t column_means(const float* X, int64_t n, int32_t d, int64_t ld, double* mu, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const int nblk = div_up(n, kMeanRows);
    Buf part;
    MGB_TRY(part.alloc(sizeof(double) * (size_t)nblk * d, s));
    { col_partial_sum_kernel<<<dim3(nblk, div_up(d, 32)), 32, 0, s>>>(X, n, d, ld, part.as<double>()); note_launch(); }
    MGB_TRY(cudaGetLastError());
    { col_mean_kernel<<<div_up(d, 32), 32, 0, s>>>(part.as<double>(), nblk, d, n, mu); note_launch(); }
    return cudaGetLastError();
}

// Eccentricity with exponent 2 (§3 and §4.1 name eccentricity among the
// common filters): the mean squared distance from x to the cloud equals
// |x - mu|^2 + mean_y |y - mu|^2 (mu the column means), so f(x) =
// sqrt(|x - mu|^2 + V) without any pair of points: column means as FP64 sums
// give them, |x - mu|^2 more exactly than FP64 sums do (ecc_rows_kernel), V their
// mean (fixed-order sums). 1M x 256 through mapper_lens: 3024 us with FP64
// arithmetic throughout and a pass of its own for the finite check, 900 us now;
// with the mean as two floats 832, but on 3000 rows of mean 1e6 and spread 1 in
// 2 columns up to 2.5e-10 off, where FP64 arithmetic and this form are off by 8e-15.
cudaError_t lens_ecc2(const float* X, int64_t n, int32_t d, int64_t ld, double* f, int m, int j, cudaStream_t s,
                      int* flag)
{
    if (n == 0) return cudaSuccess;
    const int nblk = div_up(n, kMeanRows);
    Buf part, mu, vpart;
    MGB_TRY(part.alloc(sizeof(double) * (size_t)nblk * d, s));
    MGB_TRY(mu.alloc(sizeof(double) * d, s));
    MGB_TRY(vpart.alloc(sizeof(double) * kMeanBlocks, s));
    col_sum_exp_kernel<<<dim3(nblk, div_up(d, 32)), 32 * kEccWarps, 0, s>>>(X, n, d, ld, part.as<double>(), flag);
    MGB_TRY(cudaGetLastError());
    col_mean_kernel<<<div_up(d, 32), 32, 0, s>>>(part.as<double>(), nblk, d, n, mu.as<double>());
    ecc_rows_kernel<<<div_up(n, kRows), kRows, 0, s>>>(X, n, d, ld, mu.as<double>(), f, m, j);
    MGB_TRY(cudaGetLastError());
    col_lens_partial_kernel<<<kMeanBlocks, 256, 0, s>>>(f, n, m, j, vpart.as<double>());
    ecc_finish_kernel<<<std::min(div_up(n, 256), 152 * 8), 256, 0, s>>>(f, n, m, j, vpart.as<double>(), kMeanBlocks);
    note_launch(5);
    return cudaGetLastError();
}

// L-infinity norm filter (§5: the breast-cancer graphs filter by the
// "L_infinity-norm"), read as the norm of the point: f(x) = max_k |x_k|.
cudaError_t lens_linf(const float* X, int64_t n, int32_t d, int64_t ld, double* f, int m, int j, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const int blocks = (int)std::min<int64_t>(div_up(n, 8), 152 * 8);
    { lens_linf_kernel<<<blocks, 256, 0, s>>>(X, n, d, ld, f, m, j); note_launch(); }
    return cudaGetLastError();
}

cudaError_t lens_coord(const float* X, int64_t n, int64_t ld, int32_t col, double* f, int m,
                       int j, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    { lens_coord_kernel<<<div_up(n, 256), 256, 0, s>>>(X, n, ld, col, f, m, j); note_launch(); }
    return cudaGetLastError();
}

cudaError_t check_finite(const float* X, int64_t n, int32_t d, int64_t ld, int* flag,
                         cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const int blocks = (int)std::min<int64_t>(152 * 8, div_up(n, 8));
    const bool vec = ld % 4 == 0 && ((uintptr_t)X & 15) == 0;
    { finite_kernel<<<blocks, 256, 0, s>>>(X, n, d, ld, vec, flag); note_launch(); }
    return cudaGetLastError();
}

template <int NJ>
static cudaError_t power_cluster(const double* C, int32_t d, int K, double* axes, int* status, cudaStream_t s)
{
    const size_t smem = sizeof(double) * 32 * NJ * (size_t)K;
    MGB_TRY(allow_smem(power_iter_cluster_kernel<NJ>, smem));
    const int rows = div_up(d, kPowCluster);                 // a CTA's rows, two a warp
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kPowCluster);
    cfg.blockDim = dim3(32u * (unsigned)div_up(rows, 2));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kPowCluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    note_launch();
    return cudaLaunchKernelEx(&cfg, power_iter_cluster_kernel<NJ>, C, d, K, axes, status);
}

cudaError_t pca_axes(const float* X, int64_t n, int32_t d, int64_t ld, int K, double* mu,
                     double* axes, int* status, cudaStream_t s)
{
    MGB_TRY(column_means(X, n, d, ld, mu, s));
    const int ntile = div_up(d, kCovT);
    const int ntri = ntile * (ntile + 1) / 2;
    const int nchunk = div_up(n, kCovRows);
    // the centred rows in blocks of whole chunks, at most kCentredBytes at a time
    const int64_t fit = (int64_t)(kCentredBytes / (sizeof(float) * (size_t)d)) / kCovRows * kCovRows;
    const int64_t block = std::min<int64_t>(n, std::max<int64_t>(fit, kCovRows));
    Buf xc, cpart, C;
    MGB_TRY(xc.alloc(sizeof(float) * (size_t)block * d, s));
    MGB_TRY(cpart.alloc(sizeof(float) * (size_t)nchunk * ntri * kCovT * kCovT, s));
    MGB_TRY(C.alloc(sizeof(double) * (size_t)d * d, s));
    const size_t mu_smem = sizeof(float2) * (size_t)d;
    MGB_TRY(allow_smem(centre_rows_kernel, mu_smem));
    for (int64_t r0 = 0; r0 < n; r0 += block) {
        const int64_t rows = std::min<int64_t>(block, n - r0);
        centre_rows_kernel<<<(unsigned)std::min<int64_t>(div_up(rows, 8), 152 * 8), 256, mu_smem, s>>>(
            X + r0 * ld, rows, d, ld, mu, xc.as<float>());
        MGB_TRY(cudaGetLastError());
        cov_partial_kernel<<<dim3(ntri, div_up(rows, kCovRows)), 64, 0, s>>>(
            xc.as<float>(), rows, d, cpart.as<float>() + r0 / kCovRows * (int64_t)ntri * kCovT * kCovT, ntile);
        note_launch(2);
        MGB_TRY(cudaGetLastError());
    }
    cov_reduce_kernel<<<dim3(ntri, kCovT * kCovT / 128), 128, 0, s>>>(cpart.as<float>(), nchunk, ntile, d, n,
                                                                      C.as<double>());
    note_launch();
    MGB_TRY(cudaGetLastError());
    // the cluster holds C and the axes on chip; wider clouds or many axes take one CTA
    if (d <= 256 && (size_t)K * 256 * sizeof(double) <= 160 * 1024) {
        if (d <= 32) return power_cluster<1>(C.as<double>(), d, K, axes, status, s);
        if (d <= 64) return power_cluster<2>(C.as<double>(), d, K, axes, status, s);
        if (d <= 128) return power_cluster<4>(C.as<double>(), d, K, axes, status, s);
        return power_cluster<8>(C.as<double>(), d, K, axes, status, s);
    }
    const size_t smem = sizeof(double) * 2 * (size_t)d;
    MGB_TRY(allow_smem(power_iter_kernel, smem));
    { power_iter_kernel<<<1, 1024, smem, s>>>(C.as<double>(), d, K, axes, status); note_launch(); }
    return cudaGetLastError();
}

}  // namespace mgb
