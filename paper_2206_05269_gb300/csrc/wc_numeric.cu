// The paper's numeric MapReduce (Sec. 4.2): map each i in 1..n to a double
// term and reduce with +,
//   series 0: sum_{i=1}^{n} sqrt(i)
//   series 1: sum_{i=1}^{n} (-1)^(i+1) / i      (which tends to ln 2)
// The paper's kernel adds every term into one accumulator with an atomic.
// Here every term is the correctly rounded IEEE double, as a whole number of
// its last-place units, and the terms are added exactly in 128-bit integers;
// one rounding at the end gives the double nearest to the exact sum of the
// terms, whatever the grid.
//
// What bounds it, and why integers.  FP64 arithmetic runs at 1/32 of the
// 32-bit integer rate here (1.25 TFLOP/s nominal), and a square root or a
// division plus a compensated addition took 14-16 fp64 instructions a term:
// n = 1e8 took 2.97 ms (sqrt) and 2.60 ms (reciprocals), the FP64 pipe 86 %
// busy.  Over a short run x0, x0 + 1, ... both functions are, to 64 bits, a
// polynomial in the offset, so a run needs fp64 only at its start (the function
// value to 80 bits and its differences) and then three or four multi-word
// integer additions a term.  The shorter the runs, the more fp64: a quartic
// makes the runs of the small terms eight times as long as a cubic would
// (n = 1e8, both series: fp64 throughout 5.72 ms, cubics alone 0.212, now 0.173;
// n = 1e6 0.043 -> 0.034).  Large n is bound by the integer pipe: 0.66 ns per
// thousand terms.
#include <cuda_runtime.h>

#include <cstdint>

#include "wc_internal.h"

namespace wc {

constexpr int kSeriesThreads = 256;
constexpr int kSeriesBlocksPerSm = 6;  // 40 registers; a run's set-up spills a few (5 blocks: 0.181 ms, 8: 0.177)
constexpr int kRunMax4 = 256, kRunMax3 = 1024;  // terms a run, quartic and cubic

// Fixed point of the sums: sqrt(i) >= 1 is a whole number of 2^-52, a
// reciprocal of i < 2^53 a whole number of 2^-105.
constexpr int kUnitSqrt = 52, kUnitRecip = 106;

// Terms are numbered z: x = z for the square roots and x = z + 1 for the
// reciprocals, so that over z in [2^k, 2^(k+1)) every 1/x has one exponent (as
// every sqrt(x) has).  A run of m terms from there has m <= 2^k / 2^kShift4
// (quartic) or 2^k / 2^kShift3 (cubic).  With t = m / x0, the first omitted term
// of the series is at most 7/256 t^5 = 2^-70.2 of the root and t^5 = 2^-70 of
// the reciprocal for a quartic, 5/128 t^4 = 2^-68.7 and t^4 = 2^-68 for a cubic:
// at most 1/16 of the last of 64 bits.  z below kDirect is computed directly (its
// differences would need more than the words they have here).
template <int SERIES>
struct SeriesCfg {
    static constexpr int kShift4 = SERIES ? 14 : 13, kShift3 = SERIES ? 17 : 16;
    static constexpr unsigned long long kDirect = 1ull << (kShift4 + 3);
    static constexpr int kShort = 5;  // power-of-two intervals with runs shorter than kRunMax4
    static constexpr unsigned long long kLongRuns = kDirect << kShort;
    static constexpr int kCubic = kShift3 + 8;  // from 2^kCubic on a cubic serves kRunMax4 terms
    static_assert(kLongRuns >> kShift4 == kRunMax4, "short runs grow up to kRunMax4");
};

__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }

// The term z as a whole number of the series' units, from the fp64 function.
template <int SERIES>
__device__ __forceinline__ __int128 term_direct(unsigned long long z) {
    const double x = (double)(z + SERIES);
    const double v = SERIES ? 1.0 / x : sqrt(x);
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int e = (int)(b >> 52) - 1023;
    const __int128 t = (__int128)((b & ((1ull << 52) - 1)) | (1ull << 52)) << (SERIES ? e - 52 + kUnitRecip : e);
    return SERIES && (z & 1ull) ? -t : t;
}

// A value whose 64-bit mantissa lies within one unit of a rounding boundary
// of the 53-bit result: whether the term is above that boundary, exactly.
// M (odd) is the boundary in half-units of the 53-bit mantissa.
template <int SERIES>
__device__ __noinline__ bool above_boundary(unsigned long long x, int k, unsigned long long M) {
    if (SERIES) return ((unsigned __int128)1 << (54 + k)) > (unsigned __int128)M * x;
    return (unsigned __int128)x << (106 - 2 * (k >> 1)) > (unsigned __int128)M * M;
}

// Sum of the terms z0 .. z0 + m - 1 (one power-of-two interval 2^k.., m within
// the bound above), in the series' units, by a polynomial of degree ORDER.
//
// The function f scaled to [2^63, 2^64) is kept as a 64.32-bit number
// w2:w1.w0, its first difference d1 as e2:e1.e0, the others as 64-bit numbers
// of 2^-32 (d2, d3, d4): per term w +- d1, d1 - d2, d2 - d3, d3 - d4.  1024 is
// added to w once, so that the 53-bit mantissa rounded to nearest is w >> 11.
// Errors, in units of 2^-64 of the value: the start 2^-20; d1 is rounded to 2^-17
// and carries up to four (the quartic's reciprocal: two) fp64 roundings of a
// first difference that adds up to 2^49 (2^50) over a run, so 2^-2; d2 to d4
// are rounded to 2^-33 (over 256 terms of a quartic 2^-5); the omitted terms
// 2^-4: together well below 1 (largest found over the intervals: 0.19).  So only
// when w's low 11 bits are all zeros or all ones may the rounding be off, and
// those terms (1 in 1,024) are decided exactly.
// Not inlined: the callers' 128-bit sums would raise the loops' registers.
template <int SERIES, int ORDER>
__device__ __noinline__ __int128 run_sum(unsigned long long z0, int m) {
    const int k = 63 - __clzll((long long)z0);
    const unsigned long long x0 = z0 + SERIES;
    const double x = (double)x0;
    const int e = SERIES ? -(k + 1) : k >> 1;  // exponent of the value
    const double S = pow2d(63 - e);
    const double u = 1.0 / x;
    double y, dl, c1, c2, c3, c4 = 0.0;  // value, its remainder, |Taylor terms| of offset 1 (unscaled)
    if (SERIES) {
        y = u;
        dl = y * fma(-y, x, 1.0);
        c1 = ORDER == 4 ? fma(y, u, 2.0 * (y * dl)) : y * u;
        c2 = c1 * u;
        c3 = c2 * u;
        if (ORDER == 4) c4 = c3 * u;
    } else {
        y = sqrt(x);
        c1 = 0.5 * (y * u);  // 1 / (2 sqrt(x))
        dl = fma(-y, y, x) * c1;
        c2 = 0.25 * (c1 * u);
        c3 = 0.5 * (c2 * u);
        if (ORDER == 4) c4 = 0.625 * (c3 * u);
    }
    // |differences|
    const double a1 = c1 - (c2 - (c3 - c4)), a2 = 2.0 * c2 - (6.0 * c3 - 14.0 * c4), a3 = 6.0 * c3 - 36.0 * c4;
    const double S32 = S * 4294967296.0;
    const long long dli = __double2ll_rn(dl * S32);
    const unsigned long long f0 = __double2ull_rn(y * S) + 1024ull + (unsigned long long)(dli >> 32);
    const unsigned long long v1 = (unsigned long long)__double2ll_rn(a1 * (S * 65536.0));
    const unsigned long long d2i = (unsigned long long)__double2ll_rn(a2 * S32);
    const unsigned long long d3i = (unsigned long long)__double2ll_rn(a3 * S32);
    uint32_t w0 = (uint32_t)dli, w1 = (uint32_t)f0, w2 = (uint32_t)(f0 >> 32);
    uint32_t e0 = (uint32_t)(v1 << 16), e1 = (uint32_t)(v1 >> 16), e2 = (uint32_t)(v1 >> 48);
    uint32_t g0 = (uint32_t)d2i, g1 = (uint32_t)(d2i >> 32);
    uint32_t h0 = (uint32_t)d3i, h1 = (uint32_t)(d3i >> 32);
    const unsigned long long d4i = ORDER == 4 ? (unsigned long long)__double2ll_rn(24.0 * c4 * S32) : 0ull;
    const uint32_t i0 = (uint32_t)d4i, i1 = (uint32_t)(d4i >> 32);
    const uint32_t top0 = w2;
    uint32_t lo = 0, hi = 0;  // sums of w1 >> 11 and of w2 (mod 2^32), signed for the reciprocals
    auto term = [&](uint32_t j, bool minus) {
        uint32_t q = w1 >> 11;
        if (((w1 + 1u) & 0x7FEu) == 0u) {  // one unit from a rounding boundary
            const unsigned long long t = ((unsigned long long)w2 << 32) | w1, B = (t + 1ull) >> 11;
            const unsigned long long r = above_boundary<SERIES>(x0 + j, k, 2ull * B - 1ull) ? B : B - 1ull;
            q += (uint32_t)(r - (t >> 11));
        }
        lo = minus ? lo - q : lo + q;
        hi = minus ? hi - w2 : hi + w2;
    };
    auto advance = [&]() {
        if (SERIES)
            asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %4;\n\tsubc.u32 %2, %2, %5;"
                : "+r"(w0), "+r"(w1), "+r"(w2)
                : "r"(e0), "r"(e1), "r"(e2));
        else
            asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
                : "+r"(w0), "+r"(w1), "+r"(w2)
                : "r"(e0), "r"(e1), "r"(e2));
        asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %4;\n\tsubc.u32 %2, %2, 0;"
            : "+r"(e0), "+r"(e1), "+r"(e2)
            : "r"(g0), "r"(g1));
        asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, %3;" : "+r"(g0), "+r"(g1) : "r"(h0), "r"(h1));
        if (ORDER == 4)
            asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, %3;" : "+r"(h0), "+r"(h1) : "r"(i0), "r"(i1));
    };
    if constexpr (SERIES != 0) {
        // pairs (plus, minus): the sums of differences stay far inside 32 bits
        int j = 0;
#pragma unroll 2
        for (; j + 2 <= m; j += 2) {
            term((uint32_t)j, false);
            advance();
            term((uint32_t)j + 1u, true);
            advance();
        }
        long long mant = ((long long)(int32_t)hi << 21) + (int32_t)lo;
        if (j < m) {  // the odd last term
            lo = hi = 0;
            term((uint32_t)j, false);
            mant += (long long)(((unsigned long long)hi << 21) + lo);
        }
        const __int128 s = (__int128)mant << (kUnitRecip - 53 - k);
        return (z0 & 1ull) ? -s : s;
    } else {
#pragma unroll 4
        for (int j = 0; j < m; j++) {
            term((uint32_t)j, false);
            advance();
        }
        // the w2 of a run exceed the first by less than 2^18: their sum is known mod 2^32
        const unsigned long long base = (unsigned long long)top0 * (unsigned long long)m;
        const unsigned long long his = base + (uint32_t)(hi - (uint32_t)base);
        return ((__int128)his << (21 + e)) + ((__int128)lo << e);
    }
}

__device__ __forceinline__ __int128 shfl_down128(__int128 v, int o) {
    const unsigned long long l = __shfl_down_sync(0xFFFFFFFFu, (unsigned long long)v, o);
    const unsigned long long h = __shfl_down_sync(0xFFFFFFFFu, (unsigned long long)(v >> 64), o);
    return (__int128)(((unsigned __int128)h << 64) | l);
}

// Every thread's terms: a strided share of the directly computed ones; a
// strided share of the short runs (2^kShift4 of them in each power-of-two
// interval up to kLongRuns, as long as the bound allows: they cost mostly fp64,
// so they are spread over all SMs); and one contiguous piece of the rest in runs
// of about equal length, cut at powers of two.  A block's sum goes to part[b].
// Sums of n < 2^53 terms stay below 2^80 units of 2^-52 over all blocks and
// below 2^122 within one (blocks hold at most n / gridDim terms and grids of
// large n have hundreds of blocks).
template <int SERIES>
__global__ void __launch_bounds__(kSeriesThreads, kSeriesBlocksPerSm) k_series_part(unsigned long long n,
                                                                                    ulonglong2 *part) {
    using C = SeriesCfg<SERIES>;
    __shared__ unsigned long long sl[kSeriesThreads / 32], sh[kSeriesThreads / 32];
    const unsigned long long T = (unsigned long long)gridDim.x * kSeriesThreads;
    const unsigned long long t = (unsigned long long)blockIdx.x * kSeriesThreads + threadIdx.x;
    const unsigned long long zb = SERIES ? 0ull : 1ull, ze = n + zb;  // terms [zb, ze)
    __int128 acc = 0;
    for (unsigned long long z = zb + t; z < ze && z < C::kDirect; z += T) acc += term_direct<SERIES>(z);
    for (unsigned long long r = t; r < ((unsigned long long)C::kShort << C::kShift4); r += T) {
        const int k = C::kShift4 + 3 + (int)(r >> C::kShift4);
        const int m = 1 << (k - C::kShift4);
        const unsigned long long z0 = (1ull << k) + (r & ((1ull << C::kShift4) - 1ull)) * (unsigned long long)m;
        if (z0 >= ze) break;  // starts grow with r
        acc += run_sum<SERIES, 4>(z0, ze - z0 < (unsigned long long)m ? (int)(ze - z0) : m);
    }
    if (ze > C::kLongRuns) {
        const unsigned long long N = ze - C::kLongRuns, per = (N + T - 1) / T;
        unsigned long long z = C::kLongRuns + t * per;
        const unsigned long long end = z + per < ze ? z + per : ze;
        while (z < end) {
            const int k = 63 - __clzll((long long)z);
            const unsigned long long edge = 2ull << k, left = (end < edge ? end : edge) - z;
            const bool cubic = k >= C::kCubic;
            const uint32_t most = cubic ? (uint32_t)min((1ull << k) >> C::kShift3, (unsigned long long)kRunMax3) : kRunMax4;
            uint32_t len = most;
            if (left < 4ull * most) {  // the last few runs share what is left
                const uint32_t l = (uint32_t)left, runs = (l + most - 1) / most;
                len = (l + runs - 1) / runs;
            }
            acc += cubic ? run_sum<SERIES, 3>(z, (int)len) : run_sum<SERIES, 4>(z, (int)len);
            z += len;
        }
    }
    for (int o = 16; o; o >>= 1) acc += shfl_down128(acc, o);
    if ((threadIdx.x & 31) == 0) {
        sl[threadIdx.x >> 5] = (unsigned long long)acc;
        sh[threadIdx.x >> 5] = (unsigned long long)(acc >> 64);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kSeriesThreads / 32; w++) acc += (__int128)(((unsigned __int128)sh[w] << 64) | sl[w]);
        part[blockIdx.x] = make_ulonglong2((unsigned long long)acc, (unsigned long long)(acc >> 64));
    }
}

// The blocks' sums added in 192 bits (low words and signed high words apart)
// and rounded once, to nearest even: *out = sum * 2^-unit.
__global__ void __launch_bounds__(kSeriesThreads) k_series_final(const ulonglong2 *part, int nb, int unit, double *out) {
    __shared__ unsigned __int128 sl[kSeriesThreads / 32];
    __shared__ __int128 sh[kSeriesThreads / 32];
    grid_dependency_wait();
    __int128 lo = 0, hi = 0;  // lo: sums of low words (never negative)
    for (int k = threadIdx.x; k < nb; k += kSeriesThreads) {
        const ulonglong2 v = part[k];
        lo += (__int128)v.x;
        hi += (__int128)(long long)v.y;
    }
    for (int o = 16; o; o >>= 1) {
        lo += shfl_down128(lo, o);
        hi += shfl_down128(hi, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sl[threadIdx.x >> 5] = (unsigned __int128)lo;
        sh[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < kSeriesThreads / 32; w++) {
        lo += (__int128)sl[w];
        hi += sh[w];
    }
    // value = H * 2^64 + L
    __int128 H = hi + (__int128)(long long)(lo >> 64);
    unsigned long long L = (unsigned long long)lo;
    const bool neg = H < 0;
    if (neg) {
        L = ~L + 1ull;
        H = ~H + (L == 0ull ? 1 : 0);
    }
    unsigned long long a[3] = {(unsigned long long)((unsigned __int128)H >> 64), (unsigned long long)H, L};
    int top = 0;  // a[0]: most significant word
    while (top < 2 && a[top] == 0ull) top++;
    if (a[top] == 0ull) {
        *out = 0.0;
        return;
    }
    const int s = __clzll((long long)a[top]);
    const unsigned long long next = top < 2 ? a[top + 1] : 0ull;
    unsigned long long q = s ? (a[top] << s) | (next >> (64 - s)) : a[top];  // the leading 64 bits
    bool sticky = s ? (next << s) != 0ull : next != 0ull;
    if (top == 0) sticky = sticky || a[2] != 0ull;
    int e = 64 * (2 - top) - s - unit;  // value = q * 2^e
    const unsigned long long rest = q & 0x7FFull;
    q >>= 11;
    if (rest > 0x400ull || (rest == 0x400ull && (sticky || (q & 1ull)))) q++;
    const double v = ldexp((double)q, e + 11);
    *out = neg ? -v : v;
}

int series_blocks(unsigned long long n) {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // four terms a thread while all are computed directly; one wave of resident blocks at most
    unsigned long long want = (n + 4ull * kSeriesThreads - 1) / (4ull * kSeriesThreads);
    const unsigned long long cap = (unsigned long long)kSeriesBlocksPerSm * (unsigned long long)(sms > 0 ? sms : 1);
    if (want > cap) want = cap;
    return (int)(want ? want : 1);
}

cudaError_t launch_series(int series, unsigned long long n, ulonglong2 *part, int nb, double *d_out, cudaStream_t s) {
    if (series == 0) k_series_part<0><<<nb, kSeriesThreads, 0, s>>>(n, part);
    else k_series_part<1><<<nb, kSeriesThreads, 0, s>>>(n, part);
    launch_dependent(k_series_final, dim3(1), dim3(kSeriesThreads), 0, s, (const ulonglong2 *)part, nb,
                     series == 0 ? kUnitSqrt : kUnitRecip, d_out);
    return cudaGetLastError();
}

}  // namespace wc
