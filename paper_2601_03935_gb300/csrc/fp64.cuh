// FP64 elementary functions and conversions with few FP64 instructions.
//
// GB300 issues one FP64 warp instruction per 64 cycles and SM sub-partition (measured: 64
// cycles alone, 76 with every sub-partition busy, whatever the number of active lanes and
// independent chains); conversions between double, float and int cost the same, 32-bit and
// integer instructions 1 to 4 cycles.  FP64 time is therefore the number of FP64
// instructions, and CUDA's functions take (measured, in FP64 instructions): division 9,
// square root 9, exp 18, log 32, pow 90.  The functions here start from the hardware's
// approximate reciprocal (square root) or a table and finish with as few FP64 instructions
// as double precision needs; arguments outside their range take CUDA's function.
//
//   rcp_d      3   cubic iteration r + r (e + e^2), e = 1 - x r
//   div_d      6   a rcp(b) with one residual correction (Markstein 1990)
//   sqrt_d     5   x y (1 + e/2 + 3/8 e^2), y ~ x^(-1/2), e = 1 - x y^2 (the binomial series)
//   exp2n      8   2^(s c / EXP_N): table of 2^(j/EXP_N) and a degree-4 Taylor polynomial
//                  (table-driven reduction, Tang 1989)
//   log_d      19  table of reciprocals and logarithms, degree-7 Taylor polynomial of
//                  log(1 + r) (table-driven reduction, Tang 1990), summed with its rounding
//                  errors (fast two-sums, Dekker 1971)
//   pow_d      28  exp(p log x) with both words of the logarithm
//   widen / narrow: exact float -> double and round-to-nearest-even double -> float by
//                  integer instructions (0 FP64)
// Errors against 64-bit references are bounded in tests/test_gpu_fp64_math.py.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gsis {
namespace fp64 {

constexpr int EXP_N = 256;
constexpr int LOG_N = 256;
constexpr double LN2 = 0.693147180559945309417232121458176568;

// ---- tables, built by the compiler from the power series
struct Pair {
    double a, b;
};
struct ExpTable {
    double t[EXP_N];
};
struct LogTable {
    Pair t[LOG_N];          // 1 / m_j (rounded to 12 bits), log of its reciprocal
};
// sum of an (hi, lo) pair and x, renormalised (two-sum)
constexpr Pair pair_add(Pair s, double x) {
    const double t = s.a + x, v = t - s.a;
    const double lo = s.b + ((s.a - (t - v)) + (x - v));
    return Pair{t + lo, lo - ((t + lo) - t)};
}
constexpr ExpTable make_exp_table() {
    ExpTable T{};
    for (int j = 0; j < EXP_N; ++j) {
        // 2^(j/N) = exp(x), x = j ln2 / N < ln2: the series from its smallest term up
        const double x = (double)j / EXP_N * LN2;
        double term[24] = {};
        term[0] = 1.0;
        for (int k = 1; k < 24; ++k) term[k] = term[k - 1] * x / k;
        Pair s{0.0, 0.0};
        for (int k = 23; k >= 0; --k) s = pair_add(s, term[k]);
        T.t[j] = s.a + s.b;
    }
    return T;
}
constexpr LogTable make_log_table() {
    LogTable T{};
    for (int j = 0; j < LOG_N; ++j) {
        const double m = 1.0 + (j + 0.5) / LOG_N;
        const double c = (double)((int)(4096.0 / m + 0.5)) / 4096.0;
        // log(1 / c) = 2 atanh(z), z = (1 - c) / (1 + c)
        const double z = (1.0 - c) / (1.0 + c), z2 = z * z;
        double term[40] = {}, p = z;
        for (int k = 0; k < 40; ++k) {
            term[k] = 2.0 * p / (2 * k + 1);
            p *= z2;
        }
        Pair s{0.0, 0.0};
        for (int k = 39; k >= 0; --k) s = pair_add(s, term[k]);
        T.t[j] = Pair{c, s.a + s.b};
    }
    return T;
}
static __device__ const ExpTable g_exp_table = make_exp_table();
static __device__ const LogTable g_log_table = make_log_table();

// ---- conversions
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x), e = (u >> 23) & 0xffu;
    if (e - 1u < 254u)
        return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
    return (u << 1) == 0u ? __hiloint2double((int)u, 0) : (double)x;
}
__device__ __forceinline__ float narrow(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t e = (hi >> 20) & 0x7ffu;
    if (e - 897u < 253u) {          // results 2^-126 .. 2^127: normal, rounding cannot overflow
        uint32_t v = (((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29);
        const uint32_t rem = lo << 3;
        v += (rem > 0x80000000u) || (rem == 0x80000000u && (v & 1u));
        return __uint_as_float((hi & 0x80000000u) | v);
    }
    return ((hi << 1) | lo) == 0u ? __uint_as_float(hi) : (float)x;
}

// exponent field inside [lo, hi]: positive or negative normal numbers well inside the range
__device__ __forceinline__ bool moderate(double x) {
    return (((uint32_t)__double2hiint(x) >> 20) & 0x7ffu) - 64u < 1920u;
}

__device__ __forceinline__ double rcp_d(double x) {
    if (!moderate(x)) return 1.0 / x;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
// a / b to within an ulp; where b or the quotient is not moderate (a zero, infinity or NaN
// among them) as CUDA's division has it
__device__ __forceinline__ double div_d(double a, double b) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
    const double e = fma(-b, r, 1.0);
    r = fma(r, fma(e, e, e), r);
    const double q = a * r;
    if (!moderate(b) || !moderate(q)) return a / b;
    return fma(fma(-b, q, a), r, q);
}
__device__ __forceinline__ double sqrt_d(double x) {
    if (!moderate(x) || __double2hiint(x) < 0) return sqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double s = x * y, e = fma(-s, y, 1.0);
    return fma(s * e, fma(0.375, e, 0.5), s);
}

// 2^((s c + d) / EXP_N), |d| << 1: the scaled form of exp(a c) with s = a EXP_N / ln 2 (and a
// small correction d).  The product is reduced before it is rounded.
constexpr double EXP_SCALE = EXP_N / LN2;      // exp(x) = 2^(x EXP_SCALE / EXP_N)
template <bool CORR = false>
__device__ __forceinline__ double exp2n(double s, double c, double d = 0.0) {
    const double magic = 6755399441055744.0;   // 1.5 2^52: the integer part in the low word
    const double t = fma(s, c, magic);
    const int n = __double2loint(t);
    // |s c| <= 1000 EXP_N and no NaN: the high word is the magic number's with n's sign
    if (__double2hiint(t) != 0x43380000 + (n >> 31) || n > 1000 * EXP_N || n < -1000 * EXP_N)
        return exp2(s * c / EXP_N);
    double r = fma(s, c, magic - t);           // s c - n, |r| <= 1/2
    if constexpr (CORR) r += d;
    constexpr double l = LN2 / EXP_N;
    const double p = r * fma(r, fma(r, fma(r, l * l * l * l / 24.0, l * l * l / 6.0), l * l / 2.0), l);
    const double T = g_exp_table.t[n & (EXP_N - 1)];
    const double y = fma(T, p, T);
    return __hiloint2double(__double2hiint(y) + ((n >> 8) << 20), __double2loint(y));
}
static_assert(EXP_N == 256, "exp2n shifts by 8");
__device__ __forceinline__ double exp_d(double x) { return exp2n(EXP_SCALE, x); }

// log x = .a + .b for a moderate positive x, |.b| below an ulp of .a
__device__ __forceinline__ Pair log_pair(double x) {
    const int hi = __double2hiint(x);
    const int e = (hi >> 20) - 1023;
    const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
    const Pair t = g_log_table.t[(hi >> 12) & (LOG_N - 1)];
    const double r = fma(m, t.a, -1.0);        // |r| < 2^-8
    // e as a double: 2^52 + (e + 2^31) in the low word, minus the offset
    const double ed = __hiloint2double(0x43300000, (int)((uint32_t)e ^ 0x80000000u)) - 4503601774854144.0;
    const double r2 = r * r;
    double p = fma(r, 1.0 / 7.0, -1.0 / 6.0);
    p = fma(r, p, 0.2);
    p = fma(r, p, -0.25);
    p = fma(r, p, 1.0 / 3.0);
    p = fma(r, p, -0.5);
    const double tail = fma(r2, p, r);
    constexpr double LN2_HI = (double)(long long)(LN2 * 4294967296.0) / 4294967296.0;   // 32 bits: e LN2_HI is exact
    constexpr double LN2_LO = (LN2 - LN2_HI) + 2.3190468138462996e-17;                  // and the rounding of LN2
    const double s0 = ed * LN2_HI, s1 = s0 + t.b, s2 = s1 + tail;
    return Pair{s2, fma(ed, LN2_LO, (t.b - (s1 - s0)) + (tail - (s2 - s1)))};
}
static_assert(LOG_N == 256, "log_pair indexes by 8 mantissa bits");
__device__ __forceinline__ double log_d(double x) {
    if (!moderate(x) || __double2hiint(x) < 0) return log(x);
    const Pair l = log_pair(x);
    return l.a + l.b;
}
// x^p for x > 0
__device__ __forceinline__ double pow_d(double x, double p) {
    if (!moderate(x) || __double2hiint(x) < 0) return pow(x, p);
    const Pair l = log_pair(x);
    const double s = p * EXP_SCALE;
    return exp2n<true>(s, l.a, s * l.b);
}

}  // namespace fp64

// The same names for both compute types of a templated kernel.
__device__ __forceinline__ double rcp_r(double x) { return fp64::rcp_d(x); }
__device__ __forceinline__ float rcp_r(float x) { return 1.0f / x; }
__device__ __forceinline__ double sqrt_r(double x) { return fp64::sqrt_d(x); }
__device__ __forceinline__ float sqrt_r(float x) { return sqrtf(x); }
__device__ __forceinline__ double pow_r(double x, double p) { return fp64::pow_d(x, p); }
__device__ __forceinline__ float pow_r(float x, float p) { return powf(x, p); }
__device__ __forceinline__ double to_double(double x) { return x; }
__device__ __forceinline__ double to_double(float x) { return fp64::widen(x); }
template <typename R>
__device__ __forceinline__ R to_real(double x) {
    if constexpr (sizeof(R) == 8) return x;
    else return fp64::narrow(x);
}
// max(a, b) for a >= 0 and min(a, b) for a <= 0 (or -0), b any number: the bit patterns of
// doubles of one sign are ordered as integers, so neither needs an FP64 comparison
__device__ __forceinline__ double max_pos(double a, double b) {
    return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}
__device__ __forceinline__ double min_neg(double a, double b) {   // a starts at -0.0
    return __longlong_as_double((long long)max((unsigned long long)__double_as_longlong(a),
                                               (unsigned long long)__double_as_longlong(b)));
}
__device__ __forceinline__ float max_pos(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ float min_neg(float a, float b) { return fminf(a, b); }
// sign tests without an FP64 comparison (not for NaN)
__device__ __forceinline__ bool is_zero(double x) {
    return ((__double2hiint(x) << 1) | __double2loint(x)) == 0;
}
__device__ __forceinline__ bool is_zero(float x) { return x == 0.0f; }
__device__ __forceinline__ bool is_neg(double x) { return __double2hiint(x) < 0; }   // -0 counts as negative
__device__ __forceinline__ bool is_neg(float x) { return __float_as_int(x) < 0; }

}  // namespace gsis
