// mp_f64math.cuh - the FP64 arithmetic of a Pollock cell-step, shared by the
// rectilinear and the unstructured FP64 engines.  Every translation unit
// that includes it is compiled with -fmad=false: each multiply and add
// rounds on its own, in the order written, the operations of the plain
// double-precision statement of the method.
#pragma once

#include <math_constants.h>

#include "mp_f64_tables.h"

namespace mp {

// ---------------------------------------------------------------------------
// Exact tests and scalings on the bits of a double.  GB300 runs FP64 at 1/64
// of the FP32 rate and the FP64 kernel is bound by its FP64 pipe, so sign,
// zero and order tests with a known sign, frexp and ldexp are done as
// integer operations on the representation (the ALU pipe is idle); each
// gives exactly the IEEE result for the non-NaN operands the path produces.
// ---------------------------------------------------------------------------

// The representation of v, opaque to the optimiser (an empty asm): without
// it the compiler folds tests such as (bits << 1) == 0 back into FP64
// compares, which run on the FP64 pipe.
__device__ __forceinline__ long long bits(double v)
{
    long long b = __double_as_longlong(v);
    asm("" : "+l"(b));
    return b;
}
// v > 0
__device__ __forceinline__ bool gt0(double v) { return bits(v) > 0LL; }
// v < 0 (-0 is not)
__device__ __forceinline__ bool lt0(double v)
{
    return (unsigned long long)bits(v) > 0x8000000000000000ULL;
}
// v == 0 (either sign)
__device__ __forceinline__ bool eq0(double v) { return (bits(v) << 1) == 0LL; }
// a > b for b > 0
__device__ __forceinline__ bool gt_pos(double a, double b) { return bits(a) > bits(b); }
// |a| < b for b > 0
__device__ __forceinline__ bool abs_lt(double a, double b) { return (bits(a) & 0x7fffffffffffffffLL) < bits(b); }
__device__ __forceinline__ bool is_nan(double v)
{
    return (bits(v) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
}

// an integer key whose order is the IEEE order of non-NaN doubles (-0 and
// +0 share key 0): a >= b exactly when dkey(a) >= dkey(b)
__device__ __forceinline__ long long dkey(double v)
{
    const long long b = bits(v);
    return b >= 0LL ? b : -(b & 0x7fffffffffffffffLL);
}
// a >= b for non-NaN a, b
__device__ __forceinline__ bool ge_d(double a, double b) { return dkey(a) >= dkey(b); }

// The two 32-bit words of v, opaque to the optimiser like bits(): most tests
// below need one of them, or one three-input operation on both.
__device__ __forceinline__ void words(double v, unsigned& lo, unsigned& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "d"(v));
}
__device__ __forceinline__ unsigned hi_abs(unsigned hi) { return hi & 0x7fffffffu; }
// v == 0 (either sign) from its words
__device__ __forceinline__ bool zero_w(unsigned lo, unsigned hi) { return (lo | hi_abs(hi)) == 0u; }

// a key of times whose signed order is the IEEE order, -0 apart (below +0):
// a >= b exactly when tkey(a) >= tkey(b); three integer operations
__device__ __forceinline__ long long tkey(double v)
{
    unsigned lo, hi;
    words(v, lo, hi);
    const unsigned n = (unsigned)((int)hi >> 31);
    return (long long)(((unsigned long long)(hi ^ (n >> 1)) << 32) | (lo ^ n));
}
// the key of a bound that may be -0, to compare sums of times with (those
// are not -0)
__device__ __forceinline__ long long bound_key(double v) { return tkey(eq0(v) ? 0.0 : v); }

// f32_trunc from the words where 2^-126 <= |x| < 2^128 (elsewhere: some
// value): the exponent's low nine bits and the top 23 fraction bits come out
// of one funnel shift, the rebias is one addition
__device__ __forceinline__ float trunc_normal(unsigned lo, unsigned hi)
{
    const unsigned t = __funnelshift_l(lo, hi, 3) + 0x40000000u;   // - (896 mod 512) << 23
    return __uint_as_float(t | (hi & 0x80000000u));
}
// f32_trunc where |x| < 2^128 (below 2^-126: a signed zero)
__device__ __forceinline__ float trunc_small(unsigned lo, unsigned hi)
{
    const unsigned t = __funnelshift_l(lo, hi, 3) + 0x40000000u;
    return __uint_as_float((hi_abs(hi) < 0x38100000u ? 0u : t) | (hi & 0x80000000u));
}
// the same for x >= 0 (or -0: zero)
__device__ __forceinline__ float trunc_pos(unsigned lo, unsigned hi)
{
    const unsigned t = __funnelshift_l(lo, hi, 3) + 0x40000000u;
    return __uint_as_float((int)hi < 0x38100000 ? 0u : t);
}
// neither infinite nor NaN
__device__ __forceinline__ bool is_finite(double v)
{
    unsigned lo, hi;
    words(v, lo, hi);
    return hi_abs(hi) < 0x7ff00000u;
}

// -v (the sign bit flipped, as IEEE negation)
__device__ __forceinline__ double neg(double v)
{
    return __longlong_as_double(bits(v) ^ (long long)0x8000000000000000ULL);
}

// The helpers below compute every case and select (no branch): the FP64
// kernels' lanes then stay converged through them.

// frexp of a positive normal finite u: u = m 2^e with m in [1/2, 1)
__device__ __forceinline__ double frexp_normal(double u, int& e)
{
    const long long b = bits(u);
    e = (int)(b >> 52) - 1022;
    return __longlong_as_double((b & 0x000fffffffffffffLL) | 0x3fe0000000000000LL);
}

// (double)e for |e| < 2^30, exactly
__device__ __forceinline__ double i2d_exact(int e)
{
    const unsigned long long sgn = e < 0 ? 0x8000000000000000ULL : 0ULL;
    const unsigned a = (unsigned)(e < 0 ? -e : e);
    const int msb = 31 - __clz(a | 1u);
    const unsigned long long mant = ((unsigned long long)a << (52 - msb)) & 0x000fffffffffffffULL;
    const unsigned long long r = sgn | ((unsigned long long)(1023 + msb) << 52) | mant;
    return __longlong_as_double(a == 0u ? 0LL : (long long)r);
}

// 2^k as ldexp(1, k) gives it, k in [-2000, 2000]
__device__ __forceinline__ double pow2i(int k)
{
    const unsigned long long nrm = (unsigned long long)(k + 1023) << 52;        // -1022 <= k <= 1023
    const unsigned long long sub = 1ULL << ((unsigned)(k + 1074) & 63u);        // -1074 <= k < -1022
    unsigned long long r = k >= -1022 ? nrm : (k >= -1074 ? sub : 0ULL);
    r = k >= 1024 ? 0x7ff0000000000000ULL : r;
    return __longlong_as_double((long long)r);
}

// FP64 -> FP32 by truncating the significand on the ALU pipe (the FP64
// pipe, the binding unit of the FP64 kernels, is spared the conversion):
// relative error below 2^-23; magnitudes below the FP32 normal range give
// 0, above it (and infinities, NaN) give infinity, with the sign.
__device__ __forceinline__ float f32_trunc(double x)
{
    const long long b = bits(x);
    const unsigned s = (unsigned)((unsigned long long)b >> 63) << 31;
    const int e = (int)((b >> 52) & 0x7ff) - 1023;
    const unsigned nrm = s | ((unsigned)(e + 127) << 23) | (unsigned)((b >> 29) & 0x7fffff);
    return __uint_as_float(e < -126 ? s : (e > 127 ? (s | 0x7f800000u) : nrm));
}

// (float)u rounded to nearest even, for u >= 2^-126 (the values 1 + x
// takes in log1p are >= 2^-53), on the ALU pipe; above the FP32 range:
// infinity, as the conversion gives
__device__ __forceinline__ float f32_rn_pos(double u)
{
    const long long b = bits(u);
    const int e = (int)(b >> 52) - 1023;
    unsigned fb = ((unsigned)(e + 127) << 23) | (unsigned)((b >> 29) & 0x7fffff);
    const unsigned rem = (unsigned)(b & 0x1fffffff);
    fb += (rem > 0x10000000u || (rem == 0x10000000u && (fb & 1u))) ? 1u : 0u;
    return __uint_as_float(e > 127 ? 0x7f800000u : fb);
}

// (double)f for f >= 0 (zero, subnormal, normal, infinity: on the ALU pipe;
// a subnormal's fraction is normalised by its leading-zero count)
__device__ __forceinline__ double f2d_pos(float f)
{
    const unsigned fb = __float_as_uint(f);
    const unsigned fe = fb >> 23;
    const unsigned fm = fb & 0x7fffffu;
    const int sh = __clz(fm | 1u) - 8;   // brings a subnormal's leading 1 to bit 23
    const unsigned long long sub = ((unsigned long long)(897 - sh) << 52) |
                                   ((unsigned long long)((fm << sh) & 0x7fffffu) << 29);
    const unsigned long long nrm = ((unsigned long long)(fe + 896u) << 52) | ((unsigned long long)fm << 29);
    unsigned long long r = fe == 0u ? (fm == 0u ? 0ULL : sub) : nrm;
    r = fe == 255u ? 0x7ff0000000000000ULL : r;
    return __longlong_as_double((long long)r);
}

// (double)f for a normal f of either sign (no branch: the callers' values
// are normal by construction)
__device__ __forceinline__ double f2d_normal(float f)
{
    const unsigned fb = __float_as_uint(f);
    // sign | (exponent + 896) | top 20 fraction bits: an arithmetic shift by 3, the copies of the sign masked
    return __hiloint2double((int)((((unsigned)((int)fb >> 3)) & 0x8fffffffu) + 0x38000000u), (int)(fb << 29));
}
// the same for f > 0
__device__ __forceinline__ double f2d_normal_pos(float f)
{
    const unsigned fb = __float_as_uint(f);
    return __hiloint2double((int)((fb >> 3) + 0x38000000u), (int)(fb << 29));
}

// 1 / x rounded to nearest for normal x with a normal reciprocal: the
// hardware's approximation and one Newton step in fmas, which rounds
// correctly (P. W. Markstein, "Computation of elementary functions on the IBM
// RISC System/6000 processor", IBM J. Res. Dev. 34(1), 1990), compared with
// __frcp_rn over every significand (tests/cuda/f64_fast_check.cu); the
// general function takes 200 cycles of latency, this about 40
__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_rn_normal(float x)
{
    const float y = rcp_approx(x);
    return __fmaf_rn(y, __fmaf_rn(-x, y, 1.0f), y);
}

// d / v as d times 1 / v: the IEEE FP32 reciprocal y0 of the truncated v
// (relative error below 1.8e-7), then one third-order step
// y = y0 + y0 (e + e^2) with e = 1 - v y0 in one fma (rounded by less
// than 2^-75), which leaves e^3 < 2^-67 and the roundings, so 1 / v
// within about half an ulp and the quotient within about one (three fmas
// where two Newton steps take four).  |v| outside [2^-120, 2^121) (and 0,
// infinity, NaN) takes the IEEE division.
static __device__ __noinline__ double div_ieee(double a, double b) { return a / b; }

__device__ __forceinline__ double f64_div(double d, double v)
{
    unsigned lo, hi;
    words(v, lo, hi);
    if (hi_abs(hi) - 0x38700000u >= 0x0f100000u) return div_ieee(d, v);   // 2^-120 <= |v| < 2^121
    const double y0 = f2d_normal(rcp_rn_normal(trunc_normal(lo, hi)));   // |1 / v| in (2^-121, 2^120]: normal
    const double e0 = fma(-v, y0, 1.0);
    const double y1 = fma(y0, fma(e0, e0, e0), y0);
    return d * y1;
}

// ---------------------------------------------------------------------------
// log1p and expm1 by argument reduction, a table and a short series, with
// IEEE additions, multiplications and explicit fused multiply-adds in a
// fixed order (no implicit contraction: this file is built with
// -fmad=false), exact bit operations on the ALU pipe, one FP32 reciprocal
// and FP32 products, so that the FP64 path produces the same bits as any
// other evaluation of the same steps on the host.  Exit-axis choices near a
// tie then agree exactly, which library functions with different last-bit
// rounding cannot guarantee on ill-conditioned fields.  The method is
// Tang's table-driven one (P. T. P. Tang, "Table-driven implementation of
// the exponential function in IEEE floating-point arithmetic", ACM TOMS
// 15(2), 1989; "Table-driven implementation of the logarithm function in
// IEEE floating-point arithmetic", ACM TOMS 16(4), 1990), with tables and
// series lengths of this file's own choosing.  The tables
// (mp_f64_tables.h) hold correctly rounded constants.
//   log1p(x): u = 1 + x; u = m 2^e with m in [1/sqrt2, sqrt2); the bucket
//     of m (exponent and top 8 fraction bits) gives R ~ 1/m with 8
//     significant bits and -ln R = Lh + Ll.  For e in [-2, 3] (u in
//     [1/(4 sqrt2), 8 sqrt2): all but a few in ten thousand exit times,
//     also on strongly heterogeneous fields with wells) a
//     table row per (e, bucket) holds e ln2_hi + Lh (exact), e ln2_lo + Ll
//     rounded, R' = R 2^-e and R' - 1 (exact), and r = (1 + x) R' - 1 =
//     x R' + (R' - 1) is one fma on x itself, so the rounding of 1 + x never
//     enters; otherwise (out of line) r = m R - 1 exactly and the rounding
//     error c of 1 + x (two-sum) is added as c times the FP32 reciprocal of
//     u.  ln(1 + r) by its series to r^8 (|r| < 0.006), the factor of r^5
//     in FP32 on the truncated r; result (e ln2_hi + Lh) +
//     (ln(1 + r) + (e ln2_lo + Ll)).  u = +inf -> +inf, u = 0 -> -inf,
//     NaN -> NaN.
//   expm1(w): |w| limited to 800; k = nearest integer to w 256/ln2 in FP32
//     on the truncated w; j = k mod 256, m = (k - j) / 256;
//     r = w - k ln2_hi/256 (exact); expm1(r) by its series to r^5
//     (|r| < 0.0016), the factor of r^4 in FP32 on the truncated r.  For
//     m in [-2, 1] (|w| below about 2 ln2: all but a few in a thousand
//     motions, also on strongly heterogeneous fields with wells) expm1(w) =
//     A em + B in one fma, A = e^(k ln2_hi/256) and B = A - 1 rounded from
//     a table (the low part of k ln2/256 is in the table); otherwise (out
//     of line) r -= k ln2_lo/256, 2^(j/256) = Th + Tl, S = Th expm1(r) + Tl,
//     expm1(w) = (2^m Th - 1) + 2^m S ((Th + S) 2^(m-1023) 2^1023 when
//     2^m is not finite).  About 9 and 6 FP64 operations.
// ---------------------------------------------------------------------------

// ln(1 + r) by its series to r^8; the tail 1/5 - r/6 + r^2/7 - r^3/8 in
// FP32: it enters scaled by r^5, below 2.6e-10 of the result, so its FP32
// error stays below 0.15 ulp (and the FP64 pipe is spared three fmas)
__device__ __forceinline__ double log1p_series(double r)
{
    const double r2 = r * r;
    unsigned lo, hi;
    words(r, lo, hi);
    const float rf = trunc_small(lo, hi);
    float pf = __fmaf_rn(-0x1.0p-3f, rf, 0x1.24924ap-3f);   // -1/8, 1/7
    pf = __fmaf_rn(pf, rf, -0x1.555556p-3f);                // -1/6
    pf = __fmaf_rn(pf, rf, 0x1.99999ap-3f);                 // 1/5
    double q = fma(r, f2d_normal_pos(pf), -0.25);   // pf near 1/5: normal
    q = fma(q, r, 1.0 / 3.0);
    q = fma(q, r, -0.5);
    return fma(r2, q, r);
}

// log1p for exponents e outside the table rows (rare; out of line, and a
// side effect keeps the call from being evaluated speculatively):
// r = m R - 1 exactly and the two-sum error c of u = 1 + x as c / u
static __device__ __noinline__ double log1p_far(double x, double u, double m, int e, int key)
{
    asm volatile("");
    const double ln2_hi = 6.93147180369123816490e-01, ln2_lo = 1.90821492927058770002e-10;
    // (1 - (u - x)) when x > 1, else (x - (u - 1))
    const bool big = gt_pos(x, 1.0);
    const double c = (big ? 1.0 : x) - (u - (big ? x : 1.0));
    const double2 t0 = __ldg(reinterpret_cast<const double2*>(f64_log_tab) + 2 * key);       // R, Lh
    const double Ll = __ldg(reinterpret_cast<const double2*>(f64_log_tab) + 2 * key + 1).x;
    const double lg = log1p_series(fma(m, t0.x, -1.0));
    const double ru = f2d_pos(__frcp_rn(f32_rn_pos(u)));   // (double)(1.0f / (float)u)
    const double de = i2d_exact(e);
    return fma(de, ln2_hi, t0.y) + (fma(c, ru, lg) + fma(de, ln2_lo, Ll));
}

static __device__ __noinline__ double series_log1p(double x)
{
    asm volatile("");
    const double u = 1.0 + x;
    const long long ub = bits(u);
    const bool ok = ub > 0LL && ub < 0x7ff0000000000000LL;   // 0 < u < inf
    int e;
    double m = frexp_normal(ok ? u : 1.0, e);   // u >= 2^-53 when ok
    const bool below = bits(m) < bits(0.70710678118654752440);   // m in [1/2, 1/sqrt2): m * 2, exactly
    m = __longlong_as_double(bits(m) + (below ? (1LL << 52) : 0LL));
    e -= below ? 1 : 0;
    const int key = (int)(bits(m) >> 44) - F64_LOG_KEY0;
    const unsigned er = (unsigned)(e - F64_LOG_E0);
    double res;
    if (er < (unsigned)F64_LOG_NE) {
        // (e ln2_hi + Lh, RN(e ln2_lo + Ll)), (R 2^-e, R 2^-e - 1)
        const double2* row = reinterpret_cast<const double2*>(f64_log_e_tab) + 2 * (er * F64_LOG_N + key);
        const double2 hl = __ldg(row), rp = __ldg(row + 1);
        const double lg = log1p_series(fma(x, rp.x, rp.y));
        res = hl.x + (lg + hl.y);
    } else {
        res = log1p_far(x, u, m, e, key);
    }
    const long long special = eq0(u) ? (long long)0xfff0000000000000ULL
                                     : (ub == 0x7ff0000000000000LL ? 0x7ff0000000000000LL
                                                                   : (long long)0xfff8000000000000ULL);
    return __longlong_as_double(ok ? bits(res) : special);   // -inf, +inf, NaN
}

// The row of f64_log_e_tab for u = 1 + x from the words of u: the exponent
// and the top 8 fraction bits run through the rows of one exponent in order,
// 256 of them, and each exponent has 257 (the bucket holding sqrt2 is split),
// so the row is their sum plus one from sqrt2 on.  Rows outside the table (u
// outside [2^-2 / sqrt2, 2^3 sqrt2), zero, infinite, NaN) come out of range.
__device__ __forceinline__ unsigned log_row_f64(double u)
{
    unsigned lo, hi;
    words(u, lo, hi);
    const unsigned mh = hi & 0xfffffu;   // sqrt2's fraction: 0x6a09e 667f3bcd
    const unsigned up = (mh > 0x6a09eu || (mh == 0x6a09eu && lo >= 0x667f3bcdu)) ? 1u : 0u;
    return (hi >> 12) + (hi >> 20) + up - 262247u;
}

// log1p as series_log1p gives it, bit for bit.  Of u = 1 + x only the row is
// needed, so it is taken from u in FP32 (x truncated: within 5 ulp of the
// double's value wherever the row is in the table) except within 8 ulp of a
// row's edge, where the FP64 sum decides (one lane in two thousand; the
// branch is cheaper than that sum on every lane, the FP64 pipe being the
// binding unit).
__device__ __forceinline__ double fast_log1p(double x)
{
    unsigned lo, hi;
    words(x, lo, hi);
    // (|x| held below 2^126, whose rows are out of the table as well)
    hi = min(hi_abs(hi), 0x47d00000u) | (hi & 0x80000000u);
    const unsigned ub = __float_as_uint(1.0f + trunc_small(lo, hi));
    const unsigned mf = ub & 0x7fffffu;
    unsigned row = (ub >> 15) + (ub >> 23) + (mf >= 0x3504f3u ? 1u : 0u) - 31975u;
    if (((ub + 8u) & 0x7fffu) < 16u || mf - (0x3504f3u - 8u) < 16u) row = log_row_f64(1.0 + x);
    if (row >= (unsigned)(F64_LOG_NE * F64_LOG_N)) return series_log1p(x);
    // (e ln2_hi + Lh, RN(e ln2_lo + Ll)), (R 2^-e, R 2^-e - 1)
    const double2* t = reinterpret_cast<const double2*>(f64_log_e_tab) + 2 * row;
    const double2 hl = __ldg(t), rp = __ldg(t + 1);
    return hl.x + (log1p_series(fma(x, rp.x, rp.y)) + hl.y);
}

// e^r - 1 by its series to r^5 (the next term is below 1.5e-17 of the
// result); the factor of r^4, 1/24 + r/120, in FP32: scaled by r^4 (below
// 1.7e-10 of the result) its FP32 error stays below 0.1 ulp
__device__ __forceinline__ double expm1_series(double r)
{
    const double r2 = r * r;
    unsigned lo, hi;
    words(r, lo, hi);
    const float pf = __fmaf_rn(0x1.111112p-7f, trunc_small(lo, hi), 0x1.555556p-5f);   // 1/120, 1/24
    double p = fma(f2d_normal_pos(pf), r, 1.0 / 6.0);   // pf near 1/24: normal
    p = fma(p, r, 1.0 / 2.0);
    return fma(r2, p, r);
}

// expm1 for m outside [-2, 1] (rare; out of line, not evaluated
// speculatively): r -= k ln2_lo/256, S = Th em + Tl, (2^m Th - 1) + 2^m S,
// and (Th + S) 2^(m-1023) 2^1023 where 2^m overflows
static __device__ __noinline__ double expm1_far(double r, double dk, int j, int m)
{
    asm volatile("");
    const double ln2_lo = 1.90821492927058770002e-10;
    const double em = expm1_series(fma(dk, -(ln2_lo / 256.0), r));
    const double2 T = __ldg(reinterpret_cast<const double2*>(f64_exp_tab) + j);   // 2^(j/256)
    const double S = fma(T.x, em, T.y);
    if (m > 1023) return ((T.x + S) * pow2i(m - 1023 > 2000 ? 2000 : m - 1023)) * pow2i(1023);
    const double t = pow2i(m < -2000 ? -2000 : m);
    return fma(t, S, fma(t, T.x, -1.0));
}

__device__ __forceinline__ double series_expm1(double w)
{
    const double ln2_hi = 6.93147180369123816490e-01;
    const double wc = __longlong_as_double((abs_lt(w, 800.0) || is_nan(w))
                                               ? bits(w)
                                               : (lt0(w) ? (long long)0xc089000000000000ULL    // -800
                                                         : 0x4089000000000000LL));             // 800
    const float y = __fmul_rn(f32_trunc(wc), 0x1.715476p+8f);   // 256/ln2 in FP32
    const float sh = __fadd_rn(y, 12582912.0f);                  // rounds y to an integer
    const int k = (int)__float_as_uint(sh) - 0x4b400000;
    const int j = k & 255;
    const int m = (k - j) >> 8;
    const double dk = i2d_exact(k);
    // w - k ln2_hi/256, exact (the constant negated, not k: no separate
    // negation of k on the FP64 pipe)
    const double r = fma(dk, -(ln2_hi / 256.0), wc);
    // m in [-2, 1]: e^w - 1 = A em + B, A = e^(k ln2_hi/256) and B = A - 1
    // rounded, from the table, in one fma
    const unsigned mr = (unsigned)(m - F64_EXP_M0);
    if (mr < (unsigned)F64_EXP_NM) {
        const double2 ab = __ldg(reinterpret_cast<const double2*>(f64_exp_ab_tab) + mr * F64_EXP_N + j);
        return fma(ab.x, expm1_series(r), ab.y);
    }
    return expm1_far(r, dk, j, m);
}

// Exit time along one axis from the distance d to its reachable face at the
// particle velocity vp: t1 = d / vp by f64_div, z = A t1, t1 when z == 0,
// else log1p(z) * (1 / A).  (A z that is not used is replaced by one inside a
// row of log1p's table, so that it does not send the warp to the FP64 sum; so
// is that of a lane without use, whose result means nothing.)
__device__ __forceinline__ double f64_exit_time_d(double A, double iA, double d, double vp, bool use = true)
{
    const double t1 = f64_div(d, vp);
    const double z = A * t1;
    unsigned lo, hi;
    words(z, lo, hi);
    const bool lin = zero_w(lo, hi);
    const double te = fast_log1p(lin || !use ? 0.7 : z) * iA;
    return lin ? t1 : te;
}

// the reachable face (+1, -1, 0: none) from the words of vp and the signs of
// the face velocities (bits 1 and 2 of sg: v1 < 0, v2 > 0)
__device__ __forceinline__ int f64_face(unsigned vlo, unsigned vhi, unsigned sg)
{
    const bool down = (int)vhi < 0;
    const bool open = (sg & (down ? 2u : 4u)) != 0u && !zero_w(vlo, vhi);
    return open ? (down ? -1 : 1) : 0;
}

// the signed distance to that face (D - pp up, -pp down and otherwise)
__device__ __forceinline__ double f64_face_dist(int face, double D, double pp)
{
    return face > 0 ? D - pp : neg(pp);
}

// 0 <= pp <= D as unsigned words (a set sign is the largest; D > 0)
__device__ __forceinline__ bool f64_inside(double pp, double D)
{
    return (unsigned long long)bits(pp) <= (unsigned long long)bits(D);
}

// particle velocity at offset pp from face 1: v1 + A pp, one rounding
__device__ __forceinline__ double f64_vel(double v1, double A, double pp) { return fma(A, pp, v1); }

// analytic motion along one axis for a time dt, clamped to the cell (vp == 0
// or dt == 0 -> pp; w = A dt == 0 -> pp + vp dt in one fma; else pp +
// (vp * expm1(w)) * (1 / A), the last product and sum in one fma): the form
// for every w, out of line
static __device__ __noinline__ double f64_move(double A, double iA, double D, double vp, double pp, double dt)
{
    asm volatile("");
    const bool still = eq0(vp) || eq0(dt);
    const double w = A * dt;
    const bool lin = eq0(w);
    const double em = series_expm1(lin ? 0.5 : w);
    const double vem = vp * em;
    double pn = fma(lin ? vp : vem, lin ? dt : iA, pp);
    pn = lt0(pn) ? 0.0 : pn;
    pn = gt_pos(pn, D) ? D : pn;
    return still ? pp : pn;
}

// f64_move for |w| < 1.37 (all but a few in a thousand motions) and a result
// inside the cell, without a branch, so that the motions of the axes of one
// step interleave; `again` is set where f64_move has to give the result: w
// outside (the tables' rows end at 2 ln2), or a result that is clamped.
__device__ __forceinline__ double f64_move_fast(double A, double iA, double D, double vp, double pp, double dt,
                                                bool& again)
{
    const double ln2_hi = 6.93147180369123816490e-01;
    const double w = A * dt;
    unsigned lo, hi;
    words(w, lo, hi);
    const bool lin = zero_w(lo, hi);
    const bool out = hi_abs(hi) >= 0x3ff61000u;   // |w| >= 1.3789
    const float sh = __fadd_rn(__fmul_rn(trunc_small(lo, hi), 0x1.715476p+8f), 12582912.0f);
    const unsigned row = out ? 0u : __float_as_uint(sh) - 0x4b400000u - (unsigned)(F64_EXP_M0 * F64_EXP_N);
    // (double)k for |k| <= 512: the FP32 integer's top bits, 0 for k = 0
    const unsigned kb = __float_as_uint(__fadd_rn(sh, -12582912.0f));
    const double dk = __hiloint2double(
        kb == 0u ? 0 : (int)((((unsigned)((int)kb >> 3)) & 0x8fffffffu) + 0x38000000u), 0);
    const double2 ab = __ldg(reinterpret_cast<const double2*>(f64_exp_ab_tab) + row);
    const double r = fma(dk, -(ln2_hi / 256.0), w);
    const double vem = vp * fma(ab.x, expm1_series(r), ab.y);
    const double pn = fma(lin ? vp : vem, lin ? dt : iA, pp);
    unsigned vlo, vhi, tlo, thi;
    words(vp, vlo, vhi);
    words(dt, tlo, thi);
    const bool still = zero_w(vlo, vhi) || zero_w(tlo, thi);
    // outside [0, D] as unsigned numbers (a set sign is the largest)
    again = !still && (out || (unsigned long long)bits(pn) > (unsigned long long)bits(D));
    return still ? pp : pn;
}

// FP32 estimate of an exit time from an FP32 distance d and the truncated
// particle velocity vf.  Relative error: the truncation, the approximate
// reciprocal (1 ulp) and the products give below 1e-6 on t1 = d / vf and on
// z = A t1, and d from f32_face_dist below 6.2e-5; g(z) = ln(1 + z) / z is
// its series for |z| < 2^-7, else the hardware base-2 logarithm (absolute
// error at most 2^-22 on [1/2, 2], 1 ulp-scale outside) of u = fl(1 + z)
// over u - 1, in which the rounding of 1 + z cancels (Goldberg 1991), or for
// z < -1/2 of the velocity ratio u_exit / vp over z (the ratio, not 1 + z,
// carries the information there): below 4.6e-5, since |ln u| >= 0.0078
// wherever the logarithm is used.  In all below 1.2e-4, a quarter of the
// 2^-11 that the candidate margin of 2^-10 allows.
__device__ __forceinline__ float lg2_approx(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float f32_estimate(float d, float vf, float fA, float fue)
{
    const float iv = rcp_approx(vf);
    const float t1 = d * iv;
    const float z = fA * t1;
    // both forms, selected (no divergent branch)
    const bool near_m1 = z < -0.5f;
    const float u = 1.0f + z;
    const float L = lg2_approx(near_m1 ? fue * iv : u) * 0.693147181f;
    const float gl = L * rcp_approx(near_m1 ? z : u - 1.0f);
    const float gs = __fmaf_rn(z, __fmaf_rn(z, __fmaf_rn(z, __fmaf_rn(z, 0.2f, -0.25f), 1.0f / 3.0f), -0.5f), 1.0f);
    return t1 * (fabsf(z) < 0.0078125f ? gs : gl);
}

// velocities whose estimates are trusted: |vp| in [2^-100, 2^100) (FP32
// could not hold the quotients of others), from the high word
__device__ __forceinline__ bool vel_trusted(unsigned vhi) { return hi_abs(vhi) - 0x39b00000u < 0x0c800000u; }

// FP32 distance to the reachable face for the estimates without an FP64
// subtraction: -pp truncated, or D - pp from the truncated operands (error
// below 2^-23 D plus one FP32 rounding, so below 6.2e-5 relative while the
// distance is at least 2^-9 D); nearer the face (close is set; rare) the
// caller takes the truncated FP64 difference
__device__ __forceinline__ float f32_face_dist(int face, float Df, double pp, bool& close)
{
    unsigned lo, hi;
    words(pp, lo, hi);
    const float pf = trunc_pos(lo, hi);
    const float up = Df - pf;
    close = face > 0 && up < Df * 0x1.0p-9f;
    return face > 0 ? up : -pf;
}

// The exit axis's screening: axes whose exact exit time has to be formed.
// e: the estimates of the reachable axes (reach: bit a), infinity for the
// others; doubt: some reachable axis's estimate cannot be trusted.  Gives
// the leading axis (-1: none reachable) and the others that may still win:
// those within 2^-10 of it (the estimates are within 1.2e-4 of the exact
// times), or every reachable one when in doubt or nothing is finite.
__device__ __forceinline__ int screen(float e0, float e1, float e2, unsigned reach, bool doubt, unsigned& rest)
{
    const float em = fminf(fminf(e0, e1), e2);
    const float thr = em * (1.0f + 0.0009765625f);
    int a0 = e0 == em ? 0 : (e1 == em ? 1 : 2);
    rest = (e0 <= thr ? 1u : 0u) | (e1 <= thr ? 2u : 0u) | (e2 <= thr ? 4u : 0u);
    if (doubt || !(em < CUDART_INF_F)) {
        a0 = __ffs(reach) - 1;
        rest = reach;
    }
    rest &= ~(1u << (a0 & 31));
    return a0;
}

// ---------------------------------------------------------------------------
// quotients and conversions of the field records (once per cell; the same
// values as the IEEE operations, on fewer FP64 instructions)
// ---------------------------------------------------------------------------

// |D| in [2^-60, 2^60): divisors that the forms below take
__device__ __forceinline__ bool plain_divisor(double D)
{
    unsigned lo, hi;
    words(D, lo, hi);
    return hi_abs(hi) - 0x3c300000u < 0x07800000u;
}

// a / D from y = RN(1 / D), D a plain divisor: two corrections by the exact
// remainder, the first to within an ulp, the second to the rounded quotient
// (Markstein, as above); five instructions where the division takes about
// nine.  Magnitudes near the ends of the range take the division.
__device__ __forceinline__ double div_by(double a, double D, double y)
{
    unsigned lo, hi;
    words(a, lo, hi);
    if (zero_w(lo, hi)) return a;
    if (hi_abs(hi) - 0x0c700000u >= 0x67100000u) return a / D;   // 2^-824 <= |a| < 2^825
    const double q0 = a * y;
    const double q1 = fma(fma(-D, q0, a), y, q0);
    return fma(fma(-D, q1, a), y, q1);
}

// (float)x rounded to nearest even, on the ALU where the result is normal
__device__ __forceinline__ float f32_rn(double x)
{
    unsigned lo, hi;
    words(x, lo, hi);
    if (zero_w(lo, hi)) return __uint_as_float(hi);
    if (hi_abs(hi) - 0x38100000u >= 0x0fd00000u) return (float)x;   // 2^-126 <= |x| < 2^127
    const unsigned fb = __float_as_uint(trunc_normal(lo, hi)), rem = lo & 0x1fffffffu;
    return __uint_as_float(fb + ((rem > 0x10000000u || (rem == 0x10000000u && (fb & 1u))) ? 1u : 0u));
}

// (float)(v / D) from y = RN(1 / D), D a plain divisor: v y is within two ulp
// of the quotient, which decides the FP32 value unless it lies that close to
// the middle between two
__device__ __forceinline__ float quot_f32(double v, double D, double y)
{
    unsigned lo, hi;
    words(v, lo, hi);
    if (zero_w(lo, hi)) return __uint_as_float(hi);
    words(v * y, lo, hi);
    const unsigned rem = lo & 0x1fffffffu;
    if (hi_abs(hi) - 0x38100000u >= 0x0fd00000u || rem - 0x0ffffffcu < 9u) return (float)(v / D);
    return __uint_as_float(__float_as_uint(trunc_normal(lo, hi)) + (rem >> 28));
}

}  // namespace mp
