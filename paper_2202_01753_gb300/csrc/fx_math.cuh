// fx_math.cuh -- natural logarithm and exponential of doubles whose range
// reduction and polynomial run in 64-bit fixed-point integer arithmetic.
//
// GB300 executes 2 FP64 fused multiply-adds per clock per SM against 64+
// integer multiply-adds, and the double-precision integrands spend most of
// their FP64 work in log and exp.  These versions follow P. T. P. Tang's
// table-driven methods ("Table-driven implementation of the logarithm
// function in IEEE floating-point arithmetic", ACM TOMS 16(4), 1990; "...of
// the exponential function...", ACM TOMS 15(2), 1989) with 256-entry tables
// (fx_tables.h, generated by gen_fx_tables.py), applied twice -- a second
// 256-entry table step takes the reduced argument from below 2^-8 to below
// 2^-16, so that three series terms, formed with 32-bit multiplies, replace
// seven and the long chain of dependent 64-bit multiplies -- and evaluate
// everything in fixed-point integers: the logarithm uses no FP64 operation
// (its table points are the ones at or below the argument, so every quantity
// is non-negative; its parts are summed as a 128-bit fixed-point number and
// rounded to a double with integer operations), the exponential none either
// (n = round(y 256/ln 2) from y's significand by one high multiply;
// r = y - n ln2/256 is formed from the low 64 bits of its two terms and made
// non-negative).  fx_exp_neg_scaled multiplies the result by a 64-bit
// fixed-point factor before its single rounding (the FP64 kernels' Jacobian,
// kept as an integer product), which saves the FP64 multiply after it.
//
// Accuracy (tested against 60-digit references): fx_exp within 1 ulp
// (subnormal results within one unit of their last place);
// fx_log within 1 ulp plus 2^-58 absolute (the series is absolute-accurate,
// so for x within ~1e-3 of 1 the relative error grows as 2^-58 / |ln x|;
// every use in this library feeds an exponent or a difference, where the
// absolute error is what matters).  Outside the fast ranges (non-positive,
// subnormal, infinite or NaN x; y above ~708) they return CUDA's log/exp.
#pragma once

#include <cstdint>

#include "fx_tables.h"

namespace mc {
namespace fx {

// Rounds (-1)^neg (hi 2^64 + lo) / 2^64, a nonzero magnitude below 2^10
// (hi < 2^10), to a double (ties away from zero) with 64-bit integer
// operations: a value >= 1 from its Q54 window hi 2^54 + lo 2^-10 (the
// dropped bits are below a quarter of its last place), a value < 1 from lo.
__device__ __forceinline__ double q64_to_double(uint64_t hi, uint64_t lo, bool neg)
{
    const bool big = hi != 0;
    const uint64_t t = big ? ((hi << 54) | (lo >> 10)) : lo;
    const int p = 63 - __clzll((long long)t);  // leading bit of t
    int e = p - (big ? 54 : 64) + 1023;
    uint64_t m;
    if (p > 52) {
        const int sh = p - 52;
        m = (t >> sh) + ((t >> (sh - 1)) & 1ull);
        if (m >> 53) {  // rounding carried into a new leading bit
            m >>= 1;
            ++e;
        }
    } else {
        m = t << (52 - p);
    }
    const uint64_t bits = ((uint64_t)neg << 63) | (((uint64_t)e << 52) + m - (1ull << 52));
    return __longlong_as_double((long long)bits);
}

// The rare cases go to CUDA's functions through calls, so that their code is
// not inlined into every use (the sampling loop inlines the fast paths once
// per axis; inlined slow paths multiply its size and its instruction-fetch
// stalls).
static __device__ __noinline__ double log_slow(double x) { return log(x); }
static __device__ __noinline__ double exp_slow(double y) { return exp(y); }

// Constant of the series: round(2^32 / k).
__host__ __device__ constexpr uint32_t q32_inv(uint32_t k) { return (uint32_t)((((uint64_t)1 << 32) + k / 2) / k); }

// A logarithm table entry, one 16-byte load through the read-only cache.
__device__ __forceinline__ LogPair ld_pair(const LogPair* p)
{
#ifdef __CUDA_ARCH__
    const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(p));
    return LogPair{v.x, v.y};
#else
    return *p;
#endif
}

// ln x = e ln 2 + ln c_j + ln d_k + ln(1 + r2) for x = 2^e m, c_j = 1 + j/256
// the table point at or below m, r = (m - c_j)/c_j in [0, 2^-8), d_k =
// 1 + k/65536 the second table point at or below 1 + r and r2 = (r - k/65536)/d_k
// in [0, 2^-16): every quantity is non-negative.
// The mantissa's part, from its 52 fraction bits f: ln m in Q64 (< ln 2);
// load(t, i): entry i of table t (0: c_j, 1: d_k).
template <class Load>
__device__ __forceinline__ uint64_t fx_ln_mantissa_t(uint64_t f, Load load)
{
    const int j = (int)(f >> 44);
    // m - c_j is the mantissa's low 44 bits (Q52); r = (m - c_j)/c_j in Q64 (< 2^56)
    const LogPair cj = load(0, j);
    const uint64_t r = __umul64hi((f & 0xFFFFFFFFFFFull) << 13, cj.inv);
    // second step: k = the top 8 bits of r (r < 2^-8), r - k/65536 its low 48 bits
    // (Q64); r2 = (r - k/65536)/d_k in Q64 (< 2^48)
    const int k = (int)(r >> 48);
    const LogPair dk = load(1, k);
    const uint64_t R = __umul64hi((r & 0xFFFFFFFFFFFFull) << 16, dk.inv) >> 15;
    // ln(1 + r2) = r2 - r2^2/2 + r2^3/3 (+ r2^4/4 < 2^-66).  r2^2 from the top 32
    // bits of r2 (H = r2 in Q48; the dropped low bits move it by < 2^-62) and
    // r2^3 < 2^-48 from r2^2 and H, both with 32 x 32-bit products.
    const uint32_t H = (uint32_t)(R >> 16);
    const uint64_t sq = ((uint64_t)H * H) >> 32;                           // r2^2, Q64 (< 2^32)
    const uint32_t cube = (uint32_t)(((uint64_t)(uint32_t)sq * H) >> 48);  // r2^3, Q64 (< 2^16)
    const uint64_t l2 = R - (sq >> 1) + __umulhi(cube, q32_inv(3));        // ln(1 + r2), Q64
    return cj.ln + dk.ln + l2;
}

__device__ __forceinline__ uint64_t fx_ln_mantissa(uint64_t f)
{
    return fx_ln_mantissa_t(f, [](int t, int i) { return ld_pair(t ? &kLogD[i] : &kLogC[i]); });
}

__device__ __forceinline__ double fx_log(double x)
{
    const uint64_t u = (uint64_t)__double_as_longlong(x);
    if ((uint32_t)(u >> 32) - 0x00100000u >= 0x7FE00000u) return log_slow(x);  // not a positive normal number
    const int e = (int)(u >> 52) - 1023;
    const uint64_t f = u & 0xFFFFFFFFFFFFFull;
    const uint64_t U = fx_ln_mantissa(f);  // ln m, Q64 (< ln 2)
    // e ln 2 + ln m as sign and 128-bit magnitude in Q64; |e| < 2^11, so
    // |e| ln 2 is two 32 x 32-bit products (ln 2 = L1 2^32 + L0)
    const uint32_t ae = (uint32_t)(e < 0 ? -e : e);
    const uint64_t p0 = (uint64_t)ae * (uint32_t)kLn2Q64;
    const uint64_t p1 = (uint64_t)ae * (uint32_t)(kLn2Q64 >> 32);
    const uint64_t plo = p0 + (p1 << 32);
    const uint64_t phi = (p1 >> 32) + (plo < p0 ? 1ull : 0ull);
    uint64_t lo, hi;
    bool neg = false;
    if (e >= 0) {
        lo = plo + U;
        hi = phi + (lo < U ? 1ull : 0ull);
    } else {
        lo = plo - U;
        hi = phi - (plo < U ? 1ull : 0ull);
        neg = true;
        if ((int64_t)hi < 0) {  // ln m > |e| ln 2 by rounding (x just below 1): a tiny positive value
            lo = 0ull - lo;
            hi = ~hi + (lo == 0 ? 1ull : 0ull);
            neg = false;
        }
    }
    if ((hi | lo) == 0) return 0.0;
    return q64_to_double(hi, lo, neg);
}

// 2^(n/256) e^r for r = rq 2^-62 in [0, ln2/256], rounded once to a double;
// SCALED: times (jm / 2^63) 2^je, jm in [2^63, 2^64), before the rounding.
template <bool SCALED>
__device__ __forceinline__ double fx_exp_tail(int64_t n, uint64_t rq, uint64_t jm, int je)
{
    // e^r = e^(q/65536) e^b with q = floor(r 65536) (< 178) and b < 2^-16 (Q62 < 2^46):
    // e^b = 1 + b + b^2/2 + b^3/6 (+ b^4/24 < 2^-68), b^2 from the top 32 bits of b
    // (Hb = b in Q48) and b^3 from b^2 and Hb, with 32 x 32-bit products
    const uint32_t q = (uint32_t)(rq >> 46);
    const uint64_t B = rq & ((1ull << 46) - 1);
    const uint32_t Hb = (uint32_t)(B >> 14);
    const uint64_t sqb = ((uint64_t)Hb * Hb) >> 34;                      // b^2 in Q62 (< 2^30)
    const uint32_t cub = (uint32_t)((sqb * Hb) >> 48);                   // b^3 in Q62 (< 2^14)
    const uint64_t eb = (1ull << 62) + B + (sqb >> 1) + __umulhi(cub, q32_inv(6));  // e^b, Q62
    const uint64_t s = __umul64hi(__ldg(&kExpK16[q]) << 1, eb << 1);     // e^r, Q62
    // 2^(j/256) e^r in Q62, within [1, 2)
    const int j = (int)(n & 255);
    const int k = (int)(n >> 8);
    const uint64_t P = __umul64hi(__ldg(&kExp2[j]) << 1, s << 1);
    // assemble 2^k P / 2^62 (rounded to nearest, ties away): P normalised
    // into [2^62, 2^63), then a normal double (biased exponent eb >= 1) or,
    // for eb <= 0 (y below about -708.4), the subnormal round(P 2^-(11 - eb))
    // (a carry into 2^52 is the smallest normal; below 2^-1075 it is +0)
    uint64_t Pn = P;
    int be = k + 1023;  // biased exponent
    if constexpr (SCALED) {
        Pn = __umul64hi(P << 1, jm);  // Q62, a value in [1, 4)
        be += je;
        if (Pn >> 63) {
            Pn >>= 1;
            ++be;
        }
        if (be >= 2047) return __longlong_as_double(0x7FF0000000000000ll);  // overflow: +inf
    }
    if (Pn < ((uint64_t)1 << 62)) {
        Pn <<= 1;
        --be;
    }
    uint64_t bits;
    if (be >= 1) {
        bits = ((uint64_t)be << 52) + (((Pn + (1ull << 9)) >> 10) - (1ull << 52));
    } else {
        const int sh = 11 - be;
        bits = sh < 64 ? (Pn + (1ull << (sh - 1))) >> sh : 0ull;
    }
    return __longlong_as_double((long long)bits);
}

// exp of the double with bits u; SCALED: exp(y) (jm / 2^63) 2^je, jm in
// [2^63, 2^64), rounded once.  The scaled form keeps the unscaled one's
// special cases: where exp(y) alone rounds to +0 the result is +0 (as
// exp(y) * J would be), and exp(y)'s subnormal range is scaled exactly.
template <bool SCALED>
__device__ __forceinline__ double fx_exp_bits_t(uint64_t u, uint64_t jm, int je)
{
    const double y = __longlong_as_double((long long)u);
    const uint64_t ay = u & 0x7FFFFFFFFFFFFFFFull;
    const uint32_t ayh = (uint32_t)(ay >> 32);  // the thresholds below have zero low words
    if (ayh >= 0x40862000u) {  // |y| >= 708, infinite or NaN
        // y < -745.2 (down to -inf): exp(y) < 2^-1075 rounds to +0.  Integrands
        // with narrow peaks land here often, so it takes no FP64 work.  Down
        // from -708 the results are subnormal; they are assembled below with
        // integer rounding, so that these samples (a few percent of a narrow
        // peak's) do not send their warp through CUDA's exp with one or two
        // lanes on the FP64 pipe.  Overflow and NaN are CUDA's exp.
        if (!(u >> 63) || ay > 0x7FF0000000000000ull) {
            if constexpr (SCALED) return exp_slow(y) * ldexp((double)jm, je - 63);
            else return exp_slow(y);
        }
        if (ay > 0x408749999999999Aull) return 0.0;
    }
    if (ayh < 0x3C300000u) {  // |y| < 2^-60: exp(y) rounds to 1
        if constexpr (SCALED) return ldexp((double)jm, je - 63);
        else return 1.0;
    }
    // y = n ln2/256 + r, n = round(y 256/ln2) from y's significand M and
    // exponent E: |y| 256/ln2 = H 2^(E-1075) to 2^-52 relative, H =
    // floor(M K / 2^53) with K = 256/ln2 in Q53, rounded at bit 1075 - E (>= 43).
    // Near a tie n may be the other neighbour: |r| stays below ln2/256.
    const int E = (int)((u >> 52) & 0x7FF);
    const uint64_t M = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const uint64_t H = __umul64hi(M << 11, k256OverLn2Q53);
    const int sh1 = 1074 - E;  // the rounding bit's position minus one
    const int64_t na = (int64_t)(((sh1 < 64 ? H >> sh1 : 0ull) + 1ull) >> 1);
    int64_t n = (u >> 63) ? -na : na;
    // r = y - n ln2/256 in Q62 (|r| <= ln2/512 + tiny: |rq| < 2^54), so only the
    // low 64 bits of y in Q62 and of n ln2/256 matter: y's bits below 2^-62 are
    // dropped; n ln2/256 = (n C + 2^52) >> 53 with C = ln2/256 in Q115 =
    // Hi 2^64 + Lo, of which bits 53..116 are kept
    const int sh = E - 1013;  // y = M 2^(E-1075): Q62 needs a shift by E - 1013
    uint64_t Y = sh >= 0 ? M << sh : (sh > -64 ? M >> -sh : 0ull);
    if (u >> 63) Y = 0ull - Y;
    const uint64_t nu = (uint64_t)n;
    const uint64_t plo = nu * kLn2Over256Q115Lo;
    uint64_t phi = __umul64hi(nu, kLn2Over256Q115Lo) - (n < 0 ? kLn2Over256Q115Lo : 0ull);  // n Lo, signed
    const uint64_t plo2 = plo + (1ull << 52);
    phi += plo2 < plo ? 1ull : 0ull;
    const uint64_t L = ((phi + nu * kLn2Over256Q115Hi) << 11) | (plo2 >> 53);
    int64_t rq = (int64_t)(Y - L);
    if (rq < 0) {  // r in [0, ln2/256): n one lower
        --n;
        rq += (int64_t)kLn2Over256Q62;
    }
    return fx_exp_tail<SCALED>(n, (uint64_t)rq, jm, je);
}

__device__ __forceinline__ double fx_exp_bits(uint64_t u) { return fx_exp_bits_t<false>(u, 0, 0); }

__device__ __forceinline__ double fx_exp(double y) { return fx_exp_bits((uint64_t)__double_as_longlong(y)); }

// exp(-v) (jm / 2^63) 2^je (jm in [2^63, 2^64)), rounded once
__device__ __forceinline__ double fx_exp_neg_scaled(double v, uint64_t jm, int je)
{
    return fx_exp_bits_t<true>((uint64_t)__double_as_longlong(v) ^ 0x8000000000000000ull, jm, je);
}

// exp(-v), the sign flipped on the bits (no FP64 negation)
__device__ __forceinline__ double fx_exp_neg(double v)
{
    return fx_exp_bits((uint64_t)__double_as_longlong(v) ^ 0x8000000000000000ull);
}

// exp(-v) (NEG) or exp(v) of the non-negative fixed-point v = q 2^-fq (fq in
// 43..62, v < 2^(64 - fq)), times (jm / 2^63) 2^je, rounded once.  v < 746 is
// split at n ln2/256 with n = floor(v 256/ln2) by one 64-bit high multiply
// (one more for NEG, so that the remainder of -v is non-negative); the rest
// is the exponential's own tail.  No conversion to a double on the way in:
// the FP64 kernels' exponents are sums of fixed-point terms.
template <bool NEG>
__device__ __forceinline__ double fx_exp_fixed(uint64_t q, int fq, uint64_t jm, int je)
{
    if ((q >> fq) >= 746u) {
        if constexpr (NEG) return 0.0;  // exp(-v) rounds to +0
        else return __longlong_as_double(0x7FF0000000000000ll);
    }
    const uint64_t H = __umul64hi(q, k256OverLn2Q55);  // v 256/ln2, Q(fq - 9)
    uint32_t n = (uint32_t)(H >> (fq - 9));
    if constexpr (NEG) ++n;
    // n ln2/256 in Q62 (its low 64 bits) from ln2/256 in Q115 = Hi 2^64 + Lo
    const uint64_t p0 = (uint64_t)n * (uint32_t)kLn2Over256Q115Lo;
    const uint64_t p1 = (uint64_t)n * (uint32_t)(kLn2Over256Q115Lo >> 32) + (p0 >> 32);  // n Lo / 2^32
    const uint64_t top = (p1 >> 32) + (uint64_t)n * kLn2Over256Q115Hi;                  // n C in Q51
    const uint64_t L = (top << 11) + (((p1 & 0xFFFFFFFFull) + (1ull << 20)) >> 21);
    const uint64_t v = q << (62 - fq);
    int64_t m = NEG ? -(int64_t)n : (int64_t)n;
    int64_t rq = (int64_t)(NEG ? L - v : v - L);
    if (rq < 0) {  // n off by one at a multiple of ln2/256
        --m;
        rq += (int64_t)kLn2Over256Q62;
    }
    return fx_exp_tail<true>(m, (uint64_t)rq, jm, je);
}

// First approximation of 1/x, x in [1, 2): 23 bits suffice.
__device__ __forceinline__ float rcp_seed(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / x;
#endif
}

// The sum of n non-negative floats at p[0], p[stride], ... (as bits), to a
// double: 24-bit mantissas added as 128-bit integers, placed so that n of them
// at the largest exponent so far cannot overflow; nothing above 2^-100 of the
// largest is lost, and the sum is rounded at the end.  In double precision each
// addend is a conversion and an addition at 2 lanes per clock and SM: merging
// the partial histograms of 256 integrals of 1e5 calls, 49 parts each, took
// 110 us of an iteration there (the whole call 19.1 -> 17.8 ms, 64 integrals of
// 1e4-1e6 calls 3.70 -> 3.02 ms).  Infinities and NaN go that way still.
__device__ __forceinline__ double fx_sum_floats(const uint32_t* p, size_t stride, int n)
{
    using u128 = unsigned __int128;
    constexpr int kAhead = 8;  // loads in flight (16: the same)
    const int top = 40 - (n > 1 ? 64 - __clzll((long long)n - 1) : 0);
    u128 acc = 0;
    uint32_t E = 1;  // acc counts units of 2^(E - 150 - top - 64)
    bool plain = top < 8;
    for (int b = 0; b < n && !plain; b += kAhead) {
        uint32_t u[kAhead], mx = 0;
#pragma unroll
        for (int i = 0; i < kAhead; ++i) u[i] = b + i < n ? p[(size_t)(b + i) * stride] : 0u;
#pragma unroll
        for (int i = 0; i < kAhead; ++i) mx = u[i] > mx ? u[i] : mx;
        plain = mx >= 0x7F800000u;
        const uint32_t e = mx >> 23;
        if (e > E) {
            acc = e - E < 128u ? acc >> (e - E) : (u128)0;
            E = e;
        }
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            const uint32_t ei = u[i] >> 23 ? u[i] >> 23 : 1u, sh = E - ei;
            const uint64_t m = (uint64_t)(u[i] - ((ei - 1u) << 23)) << top;  // the implicit bit with it
            acc += sh < 128u ? (u128)m << 64 >> sh : (u128)0;  // (after an infinity or NaN: not used)
        }
    }
    if (plain) {
        double s = 0.0;
        for (int b = 0; b < n; ++b) {
            float f;
            memcpy(&f, &p[(size_t)b * stride], 4);
            s += (double)f;
        }
        return s;
    }
    const double unit = __longlong_as_double((long long)((int)E - 150 - top + 1023) << 52);  // of the upper word
    return (double)(uint64_t)(acc >> 64) * unit + (double)(uint64_t)acc * (unit * 5.421010862427522e-20);  // 2^-64
}

// 2^64 / x for x = m 2^-63 in [1, 2), by two Newton-Raphson steps y (2 - x y)
// in fixed point from a single-precision seed kept below 1/x, so that every
// residual is non-negative: relative error below 2^-60.  Returns a value in
// [2^63, 2^64): 1/x as Q64.
__device__ __forceinline__ uint64_t fx_recip(uint64_t m)
{
    const float xf = (float)(uint32_t)(m >> 40) * 1.1920928955078125e-07f;  // 24 bits, in [1, 2)
    // below 1/x by at most 2^-20: the argument was cut by < 2^-23, the seed and
    // the product are within 2^-22, and 2^-20.9 is taken off
    const uint32_t y0 = (uint32_t)(rcp_seed(xf) * 4294965148.0f);
    const uint64_t e0 = (1ull << 63) - __umul64hi(m, (uint64_t)y0 << 32);       // 1 - x y0, Q63 (< 2^43)
    const uint64_t y1 = ((uint64_t)y0 << 32) + (((uint64_t)y0 * (uint32_t)(e0 >> 11)) >> 20);  // Q64
    const uint64_t e1 = (1ull << 63) - __umul64hi(m, y1);                       // Q63 (< 2^24)
    const uint64_t y2 = y1 + (((y1 >> 32) * (uint64_t)(uint32_t)e1) >> 31);
    return y2 < (1ull << 63) ? (1ull << 63) : y2;  // x next to 2: the truncations may fall short of 1/2
}

__device__ __forceinline__ float rsqrt_seed(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / std::sqrt(x);
#endif
}

// sqrt(M 2^-64) as Q63 for M in [2^62, 2^64): s = M y from a single-precision
// seed y of the reciprocal root, then two steps s + (M - s^2) y / 2 (Newton's
// with y kept) in fixed point: relative error below 2^-58.
__device__ __forceinline__ uint64_t fx_sqrt(uint64_t M)
{
    const float xf = (float)(uint32_t)(M >> 40) * 5.9604644775390625e-08f;  // in [1/4, 1)
    const int64_t y = (int64_t)(uint32_t)fminf(rsqrt_seed(xf) * 2147483648.0f, 4294967040.0f);  // Q31
    uint64_t s = (M >> 32) * (uint64_t)y;                                   // Q63
    int64_t dl = (int64_t)((M >> 2) - __umul64hi(s, s));                    // M - s^2, Q62 (below 2^42)
    s += (uint64_t)(((dl >> 10) * y) >> 21);
    dl = (int64_t)((M >> 2) - __umul64hi(s, s));
    s += (uint64_t)((dl * y) >> 31);
    return s;
}

// cos(2 pi t) for the fraction of a turn t = a 2^-64: sign and magnitude, the
// magnitude as Q63 (up to 2^63).  The quadrant is a's top two bits (odd
// ones take the complement, cos(pi/2 - y) = sin y); within a quarter turn y
// = y_j + delta with y_j = (pi/2) j/256 from the table and delta in [0,
// pi/512): cos y = c_j cos(delta) - s_j sin(delta), the two series cut at
// delta^6/720 and delta^5/120 (next terms < 2^-63).  Absolute error < 2^-60.
__device__ __forceinline__ uint64_t fx_cos_turns(uint64_t a, bool* neg)
{
    const uint32_t quad = (uint32_t)(a >> 62);
    *neg = quad == 1u || quad == 2u;
    uint64_t x = a << 2;
    if (quad & 1u) x = ~x;
    const int j = (int)(x >> 56);
#ifdef __CUDA_ARCH__
    const ulonglong2 tv = __ldg(reinterpret_cast<const ulonglong2*>(&kCosSin[j]));
    const uint64_t c = tv.x, s = tv.y;
#else
    const uint64_t c = kCosSin[j].c, s = kCosSin[j].s;
#endif
    const uint64_t D = __umul64hi((x & 0xFFFFFFFFFFFFFFull) << 7, kHalfPiQ63);  // delta, Q70 (< 2^62.7)
    const uint64_t D2 = __umul64hi(D, D);                                        // delta^2, Q76 (< 2^61.4)
    const uint32_t h = (uint32_t)(D2 >> 32);                                     // Q44 (< 2^29.4)
    // 1 - cos delta = delta^2 (1/2 - delta^2 (1/24 - delta^2/720)), Q76
    const uint32_t k4 = 2863311531u - __umulhi(h, 23302u);                       // 1/24 - delta^2/720, Q36
    const uint32_t b = (uint32_t)(((uint64_t)h * k4) >> 29);                     // delta^2 k4, Q51 (< 2^32)
    const uint64_t u = (D2 >> 1) - (((uint64_t)h * b) >> 19);
    // sin delta = delta (1 - (delta^2/6 - delta^4/120)), Q70
    const uint64_t d4 = (uint64_t)h * h;                                         // delta^4, Q88
    const uint64_t e = __umul64hi(D2, 0x2AAAAAAAAAAAAAABull)                     // delta^2/6, Q76
                       - ((uint64_t)__umulhi((uint32_t)(d4 >> 28), 35791394u) << 16);  // delta^4/120: Q60 -> Q76
    const uint64_t sd = D - (__umul64hi(D, e << 4) >> 16);                       // e in Q80: D e in Q86 -> Q70
    const uint64_t cu = __umul64hi(c, u), ss = __umul64hi(s, sd);                // Q75, Q69
    const uint64_t r = c - (cu >> 12) - (ss >> 6);
    return r > (1ull << 63) ? 0ull : r;                                          // rounding below 0 next to a zero
}

// Single-precision cosine for the mixed-precision kernels: x = k pi/2 + r
// with k = rint(x 2/pi) and r = x - k pi/2 by a three-term Cody-Waite
// reduction with fused multiply-adds (pi/2 = F1 + F2 + F3; the products are
// exact inside the FMAs), |r| <= pi/4 (plus rounding); then cos x = cos r,
// -sin r, -cos r or sin r by k mod 4, with the Taylor series
// cos r = 1 - r^2/2! + ... + r^8/8! (next term < 2.5e-8) and
// sin r = r - r^3/3! + ... + r^9/9! (next term < 2.2e-9).  Error: a few
// units of 2^-24 for |x| < 2^22 (tested against CUDA's cosf).  Beyond 2^22,
// where a float argument is itself known only to about 0.5, the hardware
// approximation __cosf is used; no local-memory slow path is compiled in.
__device__ __forceinline__ float fx_cosf(float x)
{
    if (!(fabsf(x) < 4194304.0f)) return __cosf(x);
    const float k = rintf(x * kTwoOverPiF);
    float r = fmaf(-k, kHalfPiF1, x);
    r = fmaf(-k, kHalfPiF2, r);
    r = fmaf(-k, kHalfPiF3, r);
    const float r2 = r * r;
    float c = 1.0f / 40320.0f;
    c = fmaf(c, r2, -1.0f / 720.0f);
    c = fmaf(c, r2, 1.0f / 24.0f);
    c = fmaf(c, r2, -0.5f);
    c = fmaf(c, r2, 1.0f);
    float s = 1.0f / 362880.0f;
    s = fmaf(s, r2, -1.0f / 5040.0f);
    s = fmaf(s, r2, 1.0f / 120.0f);
    s = fmaf(s, r2, -1.0f / 6.0f);
    s = fmaf(s * r2, r, r);
    const int q = (int)k & 3;
    const float v = (q & 1) ? s : c;
    return (q == 1 || q == 2) ? -v : v;
}

}  // namespace fx
}  // namespace mc
