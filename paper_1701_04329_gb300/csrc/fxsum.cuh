// Sums of a few doubles formed exactly in 64-bit fixed point on the integer
// pipe, then rounded once.
//
// GB300 executes FP64 arithmetic at 2 FMA per clock per SM, 64 times below its
// FP32 / INT32 rate, so the FP64 stencil kernels are bound by the FP64 pipe,
// and most of their FP64 instructions are the additions of the neighbour sum
// of the (2D+1)-point operator (Eq. 5 and the relaxation of Sec. 3.1).  Here
// that sum is formed without FP64 instructions: every term's significand is
// aligned, as a 64-bit integer, to the largest exponent among the terms, with
// G guard bits below the 53-bit significand of the largest term and enough
// headroom above it for the total weight of the terms; the aligned integers
// are added exactly (two's complement) and the total is rounded once to
// nearest-even.  Besides that one rounding the only error is the truncation
// of bits lying more than 52 + G bits below the leading bit of the largest
// term: under one unit of 2^-G ulp(largest term) per unit of weight.
// Recursive FP64 summation rounds at every addition (up to half an ulp of each
// partial sum), so these sums are at least as accurate.  This is aligned
// (long-accumulator) summation in the manner of Kulisch & Miranker, cut to a
// 64-bit window.
//
// Range: the largest biased exponent E of the terms must lie in
// [kFxEmin, kFxEmax]; otherwise (every term zero or below 2^-959, a term near
// overflow, infinite or NaN) fx_sum returns false and the caller adds in FP64.
// Terms far below the largest one (zeros, subnormals) need no special case:
// their alignment shift exceeds the window and they contribute nothing.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define AFG_HD __host__ __device__ __forceinline__
#else
#define AFG_HD inline
#endif
#ifdef __CUDA_ARCH__
#define AFG_FX_UNROLL _Pragma("unroll")
#else
#define AFG_FX_UNROLL
#endif

namespace afg {

constexpr int kFxEmin = 64, kFxEmax = 2040;

AFG_HD uint64_t fx_bits(double x) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return b;
#endif
}

AFG_HD double fx_double(uint64_t b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    std::memcpy(&x, &b, 8);
    return x;
#endif
}

AFG_HD int fx_clz(uint64_t a) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)a);
#else
    return __builtin_clzll(a);
#endif
}

// Number of headroom bits for a total integer weight W (|sum| < W * 2^(63-h)).
constexpr int fx_headroom(int W) { return W <= 2 ? 1 : W <= 4 ? 2 : W <= 8 ? 3 : W <= 16 ? 4 : W <= 32 ? 5 : 6; }

// biased exponent field of x
AFG_HD int fx_exp(double x) { return (int)(fx_bits(x) >> 52) & 0x7FF; }

// Accumulator for terms of total |weight| at most W, aligned to E, the
// largest biased exponent among all terms (found by the caller first, with
// fx_exp).  add() the terms, then round().  Valid only when ok().
template <int W>
struct FxAcc {
    static constexpr int H = fx_headroom(W);
    static constexpr int G = 63 - H - 53;  // guard bits below the largest significand
    static_assert(G >= 4, "too many terms");
    int E;
    int64_t S;
    AFG_HD explicit FxAcc(int e) : E(e), S(0) {}
    AFG_HD bool ok() const { return E >= kFxEmin && E <= kFxEmax; }
    // S += w * x, w a small signed integer (sum of all |w| <= W)
    AFG_HD void add(double x, int w = 1) {
        const uint64_t b = fx_bits(x);
        // significand with its implicit bit (a zero or subnormal term gets a
        // spurious implicit bit, but its shift E - 0 >= 64 clears it)
        const uint64_t m = ((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << G;
        const int s = E - ((int)(b >> 52) & 0x7FF);
        int64_t a = (int64_t)(s < 64 ? m >> s : 0);
        const int64_t neg = (int64_t)b >> 63;  // 0 or -1
        a = (a ^ neg) - neg;
        S += a * w;
    }
    // nearest-even rounding of S * 2^(E - 1075 - G)
    AFG_HD double round() const {
        if (S == 0) return 0.0;
        const uint64_t sg = (uint64_t)S & 0x8000000000000000ull;
        const uint64_t A = S < 0 ? (uint64_t)(-S) : (uint64_t)S;
        const int p = 63 - fx_clz(A);  // leading bit; p <= 62
        const int r = p - 52;
        uint64_t M;
        if (r > 0)  // round to nearest, ties to even: add half - 1 + lsb, then shift
            M = (A + ((1ull << (r - 1)) - 1) + ((A >> r) & 1)) >> r;
        else
            M = A << (-r);
        // biased exponent p + E - 52 - G.  M carries the implicit bit, so
        // (exponent - 1) << 52 + M also takes the carry of a round-up to 2^53
        // into the exponent.
        return fx_double((((uint64_t)(p + E - 53 - G) << 52) + M) | sg);
    }
};

// x aligned to the exponent E of the largest of a set of values, in the fixed
// point of FxAcc<W>: x = result * 2^(E - 1075 - G), exactly where its own exponent
// is within G of E, and but for the truncated bits below that.
// x's own exponent must not exceed E.
template <int W>
AFG_HD int64_t fx_align(double x, int E) {
    const uint64_t b = fx_bits(x);
    const uint64_t m = ((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << FxAcc<W>::G;
    const int s = E - ((int)(b >> 52) & 0x7FF);
    const int64_t a = (int64_t)(m >> (s < 63 ? s : 63));  // m < 2^(53 + G) < 2^63
    const int64_t neg = (int64_t)b >> 63;
    return (a ^ neg) - neg;
}

// The extremes of a set of values' magnitudes, as their upper words (mx from 0,
// mn from 0xffffffff): the largest, and the smallest but for zeros less one.  A
// value whose upper word is zero counts as zero: it is below 2^-1042, far below
// the last guard bit of any exponent that is aligned to.
AFG_HD void fx_fold(double x, uint32_t &mx, uint32_t &mn) {
    const uint32_t m = (uint32_t)(fx_bits(x) >> 32) & 0x7fffffffu;
    mx = m > mx ? m : mx;
    mn = m - 1 < mn ? m - 1 : mn;
}

// The exponent to align the set to for sums of weight W: that of the largest
// value, where every other value's exponent lies within the G guard bits of it,
// so that no bit is lost and the sums are exact; else -1.
template <int W>
AFG_HD int fx_common_exponent(uint32_t mx, uint32_t mn) {
    const int E = (int)(mx >> 20);
    return E >= kFxEmin && E <= kFxEmax && E - (int)((mn + 1) >> 20) <= FxAcc<W>::G ? E : -1;
}

// S * 2^(E - 1075 - G), nearest even: FxAcc<W>::round with the leading bit moved
// to the top first, so that one path serves every size of S
template <int W>
AFG_HD double fx_round(int64_t S, int E) {
    const uint64_t A = S < 0 ? (uint64_t)(-S) : (uint64_t)S;
    if (A == 0) return 0.0;
    const int z = fx_clz(A);
    const uint64_t N = A << z, M = N >> 11;
    const uint32_t rem = (uint32_t)N & 0x7FF;
    const uint64_t up = rem + ((uint32_t)M & 1) > 0x400;
    return fx_double((((uint64_t)(10 - z + E - FxAcc<W>::G) << 52) + M + up) | ((uint64_t)S & 0x8000000000000000ull));
}

// a call: inlined, the compiler would run the conversion (64 cycles of the
// FP64 unit) for every value and select
#ifdef __CUDACC__
__host__ __device__ __noinline__
#endif
    static float
    fx_cast(double x) {
    return (float)x;
}

// (float)x, nearest even, without the FP64 unit while the result is a normal number
AFG_HD float fx_to_float(double x) {
    const uint64_t b = fx_bits(x);
    const int e = (int)(b >> 52) & 0x7FF;
    if (e < 897 || e > 1150) return fx_cast(x);
    const uint64_t u = (b & 0x7FFFFFFFFFFFFFFFull) - (896ull << 52);
    const uint32_t f = (uint32_t)((u + 0xFFFFFFFull + ((u >> 29) & 1)) >> 29) | ((uint32_t)(b >> 32) & 0x80000000u);
#ifdef __CUDA_ARCH__
    return __uint_as_float(f);
#else
    float r;
    std::memcpy(&r, &f, 4);
    return r;
#endif
}

#ifdef __CUDACC__
__host__ __device__ __noinline__
#endif
    static double
    fx_widen(float x) {
    return (double)x;
}

// (double)x without the FP64 unit for zeros and normal numbers
AFG_HD double fx_to_double(float x) {
    uint32_t b;
#ifdef __CUDA_ARCH__
    b = __float_as_uint(x);
#else
    std::memcpy(&b, &x, 4);
#endif
    const uint32_t a = b & 0x7FFFFFFFu, e = a >> 23;
    if (a == 0) return fx_double((uint64_t)b << 32);
    if (e == 0 || e == 255) return fx_widen(x);
    return fx_double((((uint64_t)a << 29) + (896ull << 52)) | ((uint64_t)(b & 0x80000000u) << 32));
}

// out = sum_k x[k] - C * c over x[0..K-1].  Returns false (out untouched)
// when the largest exponent is outside the handled range.
template <int K, int C = 0>
AFG_HD bool fx_sum(const double *x, double c, double &out) {
    int E = C ? fx_exp(c) : 0;
AFG_FX_UNROLL
    for (int k = 0; k < K; ++k) {
        const int e = fx_exp(x[k]);
        E = e > E ? e : E;
    }
    FxAcc<K + C> acc(E);
    if (!acc.ok()) return false;
AFG_FX_UNROLL
    for (int k = 0; k < K; ++k) acc.add(x[k]);
    if (C) acc.add(c, -C);
    out = acc.round();
    return true;
}

}  // namespace afg
