// mc_device.cuh -- device building blocks of the sampling kernel:
// counter-based random words, the exact sub-cube/bin position of a
// coordinate, the integrand families, and compensated single-precision sums.
#pragma once

#include <cstdint>

#include "fx_math.cuh"
#include "mc_internal.h"

namespace mc {

namespace fx {
// Reads the tables of an FP64 family's functions once, a load per 128-byte
// line, so that the samples' dependent lookups find them in L1 (called before
// the launch's wait, when the SM is idle).
__device__ __forceinline__ void warm_lines(const void* p, uint32_t bytes)
{
    if (threadIdx.x < bytes / 128u) {
        const uint32_t v = __ldg(static_cast<const uint32_t*>(p) + threadIdx.x * 32u);
        asm volatile("" ::"r"(v));
    }
}
template <int FAM> __device__ __forceinline__ void warm_tables()
{
    if constexpr (FAM == MCUBES_F_GAUSS || FAM == MCUBES_F_C0 || FAM == MCUBES_F_DISCONT || FAM == MCUBES_F_COSMO6) {
        warm_lines(kExpK16, sizeof kExpK16);
        warm_lines(kExp2, sizeof kExp2);
    }
    if constexpr (FAM == MCUBES_F_COSMO6) {
        warm_lines(kLogC, sizeof kLogC);
        warm_lines(kLogD, sizeof kLogD);
    }
    if constexpr (FAM == MCUBES_F_OSC) warm_lines(kCosSin, sizeof kCosSin);
}
}  // namespace fx

// Programmatic dependent launch (launch_dependent): a kernel's blocks may be
// placed, and run up to their wait, once every block of the kernel before it
// in the stream has called grid_dependents_launch or ended; the wait ends when
// that kernel has completed and its writes are visible.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependents_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Double-double numbers (value = hi + lo, |lo| <= ulp(hi)/2).  Grid edges are
// held in this form so that a narrow bin's width (a difference of two nearly
// equal edges, and a factor of the Jacobian) keeps full relative precision.
// ---------------------------------------------------------------------------
struct DD {
    double hi, lo;
};

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, "Parallel random numbers: as easy
// as 1, 2, 3", SC'11).  The round keys (key + r * Weyl increments) are
// precomputed on the host and read from the kernel's constant bank (single
// integrals) or formed from the integral's key (batches).
//
// The counter of a sample's block is (sample s, cube c, iteration it, block b),
// and the first three rounds mix those words only in part: with one word of
// the state multiplied per half and round, rounds 1-3 are products of it, of
// s (and b) and of c alone, and of one word of (c, s).  So they are taken
// apart: the products of (it, s, b) once per launch and segment for the first
// samples of a cube (philox_shared, kept in shared memory), that of c once
// per cube (PhiloxCube), that of (c, s) once per sample, and a block starts
// at round 4: 30 instructions instead of 40.
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;

__device__ __forceinline__ uint32_t round_key(const VsArgs& a, int r, int i) { return a.rk[r][i]; }

// Register view of one batch integral for the per-sample code (the family
// constants stay in shared memory).
struct BatchView {
    uint32_t d, nb, g, gmagic, key0, key1;
    uint32_t hist_d;  // axes with a histogram (d)
    double jac0;
    float phi_scale_f;
    double inv_p, inv_var_den;     // 1/p, 1/(p (p-1))
    float inv_p_f, inv_var_den_f;
    uint32_t want_abs;             // 0: a batch iteration does not use the sums of |cube mean|
    const uint32_t* cube_step;     // shared memory: [2][kDMax] digits of the cube step (cube_step_digit)
    const FamConsts& fam;
};

// The keys grow by Weyl increments from the integral's own key.
__device__ __forceinline__ uint32_t round_key(const BatchView& v, int r, int i)
{
    return i == 0 ? v.key0 + (uint32_t)r * 0x9E3779B9u : v.key1 + (uint32_t)r * 0xBB67AE85u;
}

// What rounds 1-3 make of (it, s, b) alone, the keys folded in.
template <class A>
__device__ __forceinline__ uint4 philox_shared(const A& a, uint32_t it, uint32_t s, uint32_t b)
{
    const uint32_t y1 = it * kPhiloxM1;
    const uint32_t z1 = __umulhi(s, kPhiloxM0) ^ b ^ round_key(a, 0, 1);
    const uint32_t x2 = __umulhi(z1, kPhiloxM1) ^ y1 ^ round_key(a, 1, 0);
    return make_uint4((z1 * kPhiloxM1) ^ round_key(a, 2, 0), __umulhi(x2, kPhiloxM0) ^ round_key(a, 2, 1),
                      (x2 * kPhiloxM0) ^ round_key(a, 3, 1), (s * kPhiloxM0) ^ round_key(a, 1, 1));
}

// What rounds 1 and 2 make of (it, c).
struct PhiloxCube {
    uint32_t h, l;
};
template <class A>
__device__ __forceinline__ PhiloxCube philox_cube(const A& a, uint32_t it, uint32_t c)
{
    const uint32_t x1 = __umulhi(it, kPhiloxM1) ^ c ^ round_key(a, 0, 0);
    return PhiloxCube{__umulhi(x1, kPhiloxM0), x1 * kPhiloxM0};
}

// The sample's word of rounds 2 and 3, from the cube's and the shared word w.
__device__ __forceinline__ PhiloxCube philox_sample(const PhiloxCube& pc, uint32_t w)
{
    const uint32_t z2 = pc.h ^ w;
    return PhiloxCube{__umulhi(z2, kPhiloxM1), z2 * kPhiloxM1};
}

// Rounds 4-10 of one block: u of the block (philox_shared), pc of the cube,
// ps of the sample.
template <class A>
__device__ __forceinline__ uint4 philox_block(const A& a, const uint4& u, const PhiloxCube& pc, const PhiloxCube& ps)
{
    uint4 x = make_uint4(ps.h ^ u.x, 0u, u.y ^ pc.l, 0u);
    {
        const uint32_t a0 = x.x * kPhiloxM0, h0 = __umulhi(x.x, kPhiloxM0);
        const uint32_t a1 = x.z * kPhiloxM1, h1 = __umulhi(x.z, kPhiloxM1);
        x = make_uint4(h1 ^ ps.l ^ round_key(a, 3, 0), a1, h0 ^ u.z, a0);
    }
#pragma unroll
    for (int r = 4; r < 10; ++r) {
        const uint32_t a0 = x.x * kPhiloxM0, h0 = __umulhi(x.x, kPhiloxM0);
        const uint32_t a1 = x.z * kPhiloxM1, h1 = __umulhi(x.z, kPhiloxM1);
        x = make_uint4(h1 ^ x.y ^ round_key(a, r, 0), a1, h0 ^ x.w ^ round_key(a, r, 1), a0);
    }
    return x;
}

// A launch's (segment's) random words: the shared parts of its first kPhiloxTab
// samples per cube in shared memory ([sample][block]), of later ones formed
// where they are used.
constexpr uint32_t kPhiloxTab = 4;
template <int NB4> struct SampleRng {
    uint32_t it;
    const uint4* tab;
    template <class A> __device__ uint4 shared_words(const A& a, uint32_t s, uint32_t b) const
    {
        return s < kPhiloxTab ? tab[s * NB4 + b] : philox_shared(a, it, s, b);
    }
};
template <int NB4, class A>
__device__ __forceinline__ void fill_philox_table(uint4* tab, const A& a, uint32_t it)
{
    if (threadIdx.x < kPhiloxTab * NB4) tab[threadIdx.x] = philox_shared(a, it, threadIdx.x / NB4, threadIdx.x % NB4);
}

// Digit of the cube step on axis j times nb; wrap: of the step that also takes
// the range's length off (both modulo the number of cubes).
__device__ __forceinline__ uint32_t cube_step_digit(const VsArgs& a, bool wrap, int j)
{
    return wrap ? a.cube_step[1][j] : a.cube_step[0][j];
}
__device__ __forceinline__ uint32_t cube_step_digit(const BatchView& v, bool wrap, int j)
{
    return v.cube_step[(wrap ? kDMax : 0) + j];
}

// ---------------------------------------------------------------------------
// Product of positive doubles in integer arithmetic (the FP64 kernels'
// Jacobian): the running value is m 2^(e - 63) with m in [2^63, 2^64); each
// factor's 53-bit significand is multiplied in as a 64 x 64 -> high-64
// product (truncated: < 2^-63 relative per factor) and renormalised by one
// bit; the result is rounded to a double once.  No FP64 instruction (GB300
// issues 2 per clock per SM, the integer multiplies run elsewhere).
// ---------------------------------------------------------------------------
struct IntProd {
    uint64_t m;
    int e;
};

__device__ __forceinline__ IntProd int_prod_of(double v)  // v > 0, finite
{
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const int E = (int)(b >> 52);
    const uint64_t mant = b & 0xFFFFFFFFFFFFFull;
    if (E) return IntProd{(mant | (1ull << 52)) << 11, E - 1023};
    const int s = __clzll((long long)mant);  // subnormal
    return IntProd{mant << s, -1074 + 63 - s};
}

__device__ __forceinline__ void int_prod_mul(IntProd& p, double v)
{
    const IntProd f = int_prod_of(v);
    const uint64_t H = __umul64hi(p.m, f.m);
    const uint64_t top = H >> 63;
    p.m = top ? H : H << 1;
    p.e += f.e + (int)top;
}

__device__ __forceinline__ IntProd int_prod_mul2(const IntProd& a, const IntProd& b)
{
    const uint64_t H = __umul64hi(a.m, b.m);
    const uint64_t top = H >> 63;
    return IntProd{top ? H : H << 1, a.e + b.e + (int)top};
}

// v 2^-f for v > 0
__device__ __forceinline__ IntProd int_prod_of_fixed(uint64_t v, int f)
{
    const int lz = __clzll((long long)v);
    return IntProd{v << lz, 63 - lz - f};
}

__device__ __forceinline__ IntProd int_prod_recip(const IntProd& p) { return IntProd{fx::fx_recip(p.m), -1 - p.e}; }

__device__ __forceinline__ double int_prod_value(const IntProd& p)
{
    // rounded to 53 bits (2^53 after a carry); m + 2^10 could wrap around
    const uint64_t r = (p.m >> 11) + ((p.m >> 10) & 1ull);
    const int E = p.e + 1023;
    if (E < 1 || E > 2046) return ldexp((double)r, p.e - 52);  // beyond the normal range: rare
    return __longlong_as_double((long long)(((uint64_t)E << 52) + r - (1ull << 52)));
}

// ---------------------------------------------------------------------------
// Grid edges as 128-bit integers.  The edges are kept in double-double (see
// above); the rebinning and the cells take differences and fractions of them
// in integers scaled by the right edge's exponent E (v -> v 2^(126 - E), so
// the right edge fills the word), where a dependent operation takes a few
// cycles against 66 for an FP64 one.
// ---------------------------------------------------------------------------
using u128 = unsigned __int128;

__device__ __forceinline__ int clz_u128(u128 v)  // v > 0
{
    const uint64_t hi = (uint64_t)(v >> 64);
    return hi ? __clzll((long long)hi) : 64 + __clzll((long long)(uint64_t)v);
}

__device__ __forceinline__ int exponent_of(double v) { return (int)(((uint64_t)__double_as_longlong(v) >> 52) & 0x7FF) - 1023; }

// |v| 2^(126 - E), |v| < 2^(E + 1)
__device__ __forceinline__ u128 scaled_u128(double v, int E)
{
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7FF);
    const uint64_t mant = (b & 0xFFFFFFFFFFFFFull) | (e ? 1ull << 52 : 0ull);
    const int sh = 74 - (E - ((e ? e : 1) - 1023));
    if (sh >= 0) return (u128)mant << sh;
    return sh > -64 ? (u128)(mant >> -sh) : (u128)0;
}

__device__ __forceinline__ u128 edge_u128(DD v, int E)
{
    const u128 h = scaled_u128(v.hi, E), l = scaled_u128(v.lo, E);
    return __double_as_longlong(v.lo) < 0 ? h - l : h + l;
}

// v 2^(E - 126) as a double-double: the high part rounded to 53 bits, the
// rest (of either sign) to 53 more; v > 0, v < 2^127
__device__ __forceinline__ DD edge_from_u128(u128 v, int E)
{
    const int z = clz_u128(v);
    const u128 n = v << z;
    const uint64_t mant = ((uint64_t)(n >> 75)) + ((uint64_t)(n >> 74) & 1ull);  // 2^52..2^53
    const uint64_t hb = ((uint64_t)(E - z + 1024) << 52) + (mant - (1ull << 52));
    const u128 back = (u128)mant << 75;  // 0 stands for 2^128 after a carry: the difference wraps right
    const bool neg = ((uint64_t)(n >> 74) & 1ull) != 0;
    const u128 mag = neg ? back - n : n - back;  // <= 2^74
    uint64_t lb = 0;
    if (mag != 0) {
        const int y = clz_u128(mag);
        const uint64_t m = (uint64_t)((mag << y) >> 75);  // 53 bits
        const int be = E + 1 - y - z + 1023;
        if (be >= 1) lb = ((uint64_t)neg << 63) | (((uint64_t)be << 52) + (m - (1ull << 52)));
    }
    return DD{__longlong_as_double((long long)hb), __longlong_as_double((long long)lb)};
}

// right - left > 0 as a 64-bit significand and exponent (m = 0: no width)
__device__ __forceinline__ IntProd edge_width(DD left, DD right)
{
    const int E = exponent_of(right.hi);
    const u128 w = edge_u128(right, E) - edge_u128(left, E);
    if (w == 0) return IntProd{0ull, 0};
    const int z = clz_u128(w);
    return IntProd{(uint64_t)((w << z) >> 64), E + 1 - z};
}

// ---------------------------------------------------------------------------
// Map cell of one axis in the box's coordinates, from the double-double edges
// (unit cube) at its two sides: (x left edge, x width / g) for the FP64
// kernels, (x left edge, nb * x width) in single precision for the mixed
// ones.  inv_g = 1 / g.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double2 map_cell_f64(DD left, DD right, double lo, double scale, double inv_g)
{
    const IntProd w = edge_width(left, right);
    const double wd = w.m ? int_prod_value(w) : 0.0;
    return make_double2(lo + scale * left.hi, scale * wd * inv_g);
}

// Map cell of the fixed-point form, in integers: (t at the left edge as an
// integer in units of 2^-f, rounded to nearest, and t width / g as a double).
__device__ __forceinline__ double2 map_cell_fix(DD left, DD right, const CellMap& m, int j)
{
    const int E = exponent_of(right.hi);
    const u128 lu = edge_u128(left, E);
    const u128 w = edge_u128(right, E) - lu;
    double width = 0.0;
    if (w != 0) {
        const int z = clz_u128(w);
        width = int_prod_value(int_prod_mul2(IntProd{(uint64_t)((w << z) >> 64), E + 1 - z},
                                             IntProd{m.bg_m[j], m.bg_e[j]}));
    }
    const int sh = 62 - E;  // the left edge (< 1) as Q64, rounded where that stays below 1
    uint64_t l64 = sh < 128 ? (uint64_t)(lu >> sh) : 0ull;
    if (sh <= 128 && l64 != ~0ull) l64 += (uint64_t)(lu >> (sh - 1)) & 1ull;
    const uint64_t t = __umul64hi(m.b[j], l64) + ((m.b[j] * l64) >> 63);
    return make_double2(__longlong_as_double(m.a[j] + (long long)t), width);
}

__device__ __forceinline__ float2 map_cell_f32(DD left, DD right, double lo, double scale, uint32_t nb)
{
    const IntProd w = edge_width(left, right);
    const double wd = w.m ? int_prod_value(w) : 0.0;
    const double xl = lo + scale * left.hi, xw = scale * wd;
    return make_float2((float)xl, (float)(xw * (double)nb));
}

__device__ __forceinline__ DD edge_right(const double* row, const double* row_lo, uint32_t k)
{
    return DD{row[k], row_lo[k]};
}

__device__ __forceinline__ DD edge_left(const double* row, const double* row_lo, uint32_t k)
{
    return k ? DD{row[k - 1], row_lo[k - 1]} : DD{0.0, 0.0};
}

// ---------------------------------------------------------------------------
// Exact position of one coordinate (Alg. 1 map step, Alg. 3 Get-Bin-ID).  The
// sample sits at y = (c + u)/g on this axis, c the sub-cube digit and
// u = (w + 1/2) / 2^32 the offset drawn from the random word w.  With
// A = nb (2w + 1) = a_hi 2^33 + a_lo and Q = nb c + a_hi:
//     nb y = (Q + a_lo 2^-33) / g,   k = floor(Q / g),
//     phi = nb y - k = (Q mod g + a_lo 2^-33) / g.
// Q < nb g <= 2^31, so floor(Q/g) is one high multiply by
// gmagic = floor((2^32-1)/g) and at most one correction.  With
// (Q + 1) gmagic = (Q + 1) 2^32 / g - (Q + 1) e / g, 1 <= e <= g, the high
// word of (Q + 1) gmagic is floor(Q/g) itself wherever nb g^2 <= 2^32: always
// for d >= 3, where g^3 < 2^32 and nb <= 1024.  There Q + 1 is kept (the
// cube's nb c carries the 1) and no correction is made (kExact).
// ---------------------------------------------------------------------------
template <bool kExact> struct BinPos {
    uint32_t k;    // bin index
    uint32_t r;    // Q mod g (kExact: plus 1)
    uint32_t ahi;  // bit 32 of a_lo (i.e. A >> 32 & 1)
    uint32_t alo;  // low 32 bits of a_lo
};

template <bool kExact>
__device__ __forceinline__ BinPos<kExact> bin_pos(uint32_t w, uint32_t nb_c, uint32_t nb, uint32_t g, uint32_t gmagic)
{
    const uint64_t A = (uint64_t)(2u * nb) * (uint64_t)w + (uint64_t)nb;
    const uint32_t hi = (uint32_t)(A >> 32);
    const uint32_t Q = nb_c + (hi >> 1);
    uint32_t q = __umulhi(Q, gmagic);
    uint32_t r = Q - q * g;
    if (!kExact && r >= g) { ++q; r -= g; }
    BinPos<kExact> b;
    b.k = q;
    b.r = r;
    b.ahi = hi & 1u;
    b.alo = (uint32_t)A;
    return b;
}

// r 2^33 + a_lo, the numerator of g phi 2^33
template <bool kExact> __device__ __forceinline__ uint64_t bin_numerator(const BinPos<kExact>& b)
{
    const uint32_t hi = kExact ? b.r + b.r + b.ahi - 2u : (b.r << 1) | b.ahi;
    return ((uint64_t)hi << 32) | (uint64_t)b.alo;  // < 2^63
}

// g phi = r + a_lo 2^-33 as a double, built from the integer numerator
// r 2^33 + a_lo with integer operations only (exact below 2^53, rounded to
// nearest above): no FP64 conversion or multiply in the sampling loop.  The
// numerator is never 0: its low 33 bits are those of A = nb (2w + 1), an odd
// multiple of nb < 2^33.
template <bool kExact> __device__ __forceinline__ double bin_gphi_f64(const BinPos<kExact>& b)
{
    const uint64_t num = bin_numerator(b);
    const int lz = __clzll((long long)num);
    uint64_t m;  // num with its leading one moved to bit 52 (bit 53 after a rounding carry)
    if (lz >= 11) {
        m = num << (lz - 11);
    } else {
        const int sh = 11 - lz;
        m = (num + (1ull << (sh - 1))) >> sh;
    }
    // value 2^(63 - lz - 33) (m / 2^52): biased exponent 1053 - lz, stored as
    // (exponent - 1) << 52 plus m, whose leading one adds the missing 1
    const uint64_t bits = ((uint64_t)(1052 - lz) << 52) + m;
    return __longlong_as_double((long long)bits);
}

// the same in single precision: (r + a_lo 2^-33) * scale, scale = 1/g for phi
// (kExact: r + 1 <= 2^11, so taking 1 off in single precision is exact)
template <bool kExact> __device__ __forceinline__ float bin_phi_f32(const BinPos<kExact>& b, float scale)
{
    const float base = kExact ? __uint2float_rn(b.r) + (b.ahi ? -0.5f : -1.0f)
                              : __uint2float_rn(b.r) + (b.ahi ? 0.5f : 0.0f);
    return __fmul_rn(__fmaf_rn(__uint2float_rn(b.alo), 1.16415321826934814453125e-10f /*2^-33*/, base), scale);
}

// ---------------------------------------------------------------------------
// Integrand families.  Each keeps a running state updated axis by axis, so
// the point x never has to be stored; constants come from FamConsts, whose
// layout per family is fixed by integrand_prepare (capi.cu):
//   CONST    c[0] = v
//   GAUSS    c[0] = A, c[1+j] = mu_j, c[13+j] = 1/(2 sig_j^2)
//   CORNER   c[j] = a_j
//   OSC      c[0] = 2 pi u, c[1+j] = a_j
//   PRODPEAK c[j] = c_j^-2, c[12+j] = w_j
//   C0       c[j] = c_j, c[12+j] = w_j
//   DISCONT  c[j] = c_j, c[12+j] = w_j
//   COSMO6   c[0..5] = a (c[2], c[3] = a_3 + 1, a_4 + 1), c[6] = mu, c[7] = 1/(2 s^2), c[8] = r, c[9] = 1/(2 t^2),
//            c[10] = 1/(2 pi s^2) (FP64: in the Jacobian's constant), c[11], c[12] = c[2], c[3] - 2 c7 mu,
//            c[13] = 2 c7 mu^2
// ---------------------------------------------------------------------------
template <typename R> struct RealOps;
template <> struct RealOps<double> {
    // fixed-point table-driven versions: a few FP64 operations instead of tens
    __device__ static double exp_(double v) { return fx::fx_exp(v); }
    __device__ static double expm_(double v) { return fx::fx_exp_neg(v); }   // exp(-v)
    __device__ static double log_(double v) { return fx::fx_log(v); }
    __device__ static double cos_(double v) { return cos(v); }
    __device__ static double rcp(double v) { return 1.0 / v; }
    __device__ static double par(const FamConsts& f, int i) { return f.c[i]; }
};
template <> struct RealOps<float> {
    __device__ static float exp_(float v) { return expf(v); }
    __device__ static float expm_(float v) { return expf(-v); }
    __device__ static float log_(float v) { return logf(v); }
    __device__ static float cos_(float v) { return fx::fx_cosf(v); }
    __device__ static float rcp(float v) { return 1.0f / v; }
    __device__ static float par(const FamConsts& f, int i) { return f.cf[i]; }
};

template <int FAM, typename R> struct Family;

template <typename R> struct Family<MCUBES_F_CONST, R> {
    struct S {};
    __device__ static void begin(S&) {}
    __device__ static void add(S&, int, R, const FamConsts&) {}
    __device__ static R end(const S&, uint32_t, const FamConsts& f) { return RealOps<R>::par(f, 0); }
};

template <typename R> struct Family<MCUBES_F_GAUSS, R> {
    struct S { R q; };
    __device__ static void begin(S& s) { s.q = R(0); }
    __device__ static void add(S& s, int j, R x, const FamConsts& f)
    {
        const R z = x - RealOps<R>::par(f, 1 + j);
        s.q += z * z * RealOps<R>::par(f, 13 + j);
    }
    __device__ static R end(const S& s, uint32_t, const FamConsts& f)
    {
        return RealOps<R>::par(f, 0) * RealOps<R>::expm_(s.q);
    }
};

template <typename R> struct Family<MCUBES_F_CORNER, R> {
    struct S { R t; };
    __device__ static void begin(S& s) { s.t = R(1); }
    __device__ static void add(S& s, int j, R x, const FamConsts& f) { s.t += RealOps<R>::par(f, j) * x; }
    __device__ static R end(const S& s, uint32_t d, const FamConsts&)
    {
        // t^-(d+1) by repeated squaring of 1/t
        R b = RealOps<R>::rcp(s.t), r = R(1);
        uint32_t e = d + 1;
        while (e) {
            if (e & 1u) r *= b;
            b *= b;
            e >>= 1;
        }
        return r;
    }
};

template <typename R> struct Family<MCUBES_F_OSC, R> {
    struct S { R t; };
    __device__ static void begin(S& s) { s.t = R(0); }
    __device__ static void add(S& s, int j, R x, const FamConsts& f) { s.t += RealOps<R>::par(f, 1 + j) * x; }
    __device__ static R end(const S& s, uint32_t, const FamConsts& f)
    {
        return RealOps<R>::cos_(RealOps<R>::par(f, 0) + s.t);
    }
};

template <typename R> struct Family<MCUBES_F_PRODPEAK, R> {
    struct S { R v; };
    __device__ static void begin(S& s) { s.v = R(1); }
    __device__ static void add(S& s, int j, R x, const FamConsts& f)
    {
        const R z = x - RealOps<R>::par(f, 12 + j);
        s.v *= RealOps<R>::rcp(RealOps<R>::par(f, j) + z * z);
    }
    __device__ static R end(const S& s, uint32_t, const FamConsts&) { return s.v; }
};

template <typename R> struct Family<MCUBES_F_C0, R> {
    struct S { R t; };
    __device__ static void begin(S& s) { s.t = R(0); }
    __device__ static void add(S& s, int j, R x, const FamConsts& f)
    {
        const R z = x - RealOps<R>::par(f, 12 + j);
        s.t += RealOps<R>::par(f, j) * (z < R(0) ? -z : z);
    }
    __device__ static R end(const S& s, uint32_t, const FamConsts&) { return RealOps<R>::expm_(s.t); }
};

template <typename R> struct Family<MCUBES_F_DISCONT, R> {
    struct S { R t; bool out; };
    __device__ static void begin(S& s) { s.t = R(0); s.out = false; }
    __device__ static void add(S& s, int j, R x, const FamConsts& f)
    {
        s.out |= !(x < RealOps<R>::par(f, 12 + j));
        s.t += RealOps<R>::par(f, j) * x;
    }
    __device__ static R end(const S& s, uint32_t, const FamConsts&)
    {
        return s.out ? R(0) : RealOps<R>::exp_(s.t);
    }
};

template <typename R> struct Family<MCUBES_F_COSMO6, R> {
    // f = c10 exp(-sum a_i L_i - L_3 - L_4 - (L_3-mu)^2 h - (L_4-mu)^2 h - (x_1+x_2-r)^2 ht)
    // with L_i = ln x_i (the 1/(x_3 x_4) of the lognormals folded into the
    // exponent, c2 = a_3 + 1 and c3 = a_4 + 1).  The add of axis j is unrolled
    // with j known, so each axis takes only its own terms.
    // In double precision the lognormal terms are expanded, h (L - mu)^2 =
    // h L^2 - 2 h mu L + h mu^2 (c11, c12: the linear coefficients; c13: the
    // two constants, added by the first FMA), each axis's quadratic taken
    // as L (h L + lin) by two FMAs, and c10 is part of the Jacobian's
    // constant: five FP64 instructions per sample fewer, on the pipe that
    // bounds these kernels; the Jacobian itself (an integer product) is
    // multiplied into the exponential's fixed-point result (end_scaled), one
    // FP64 multiply fewer.  Single precision keeps the factored form (its
    // rounding would not survive the expansion's cancellation).
    static constexpr bool kWide = sizeof(R) == 8;
    // a logarithm per axis: the FP64 sampling loop runs its axes as a loop
    // (one copy of the per-axis code) instead of unrolling them
    static constexpr bool kRolled = kWide;
    struct S { R e; R x12; };
    __device__ static void begin(S& s) { s.e = R(0); s.x12 = R(0); }
    __device__ static void add(S& s, int j, R x, const FamConsts& f)
    {
        const R L = RealOps<R>::log_(x);
        if constexpr (kWide) {
            if (j == 0) s.e = fma(f.c[0], L, f.c[13]);
            else if (j == 2 || j == 3) s.e = fma(L, fma(f.c[7], L, f.c[9 + j]), s.e);  // L (h L + lin) + e
            else s.e = fma(f.c[j], L, s.e);
        } else {
            s.e = j == 0 ? RealOps<R>::par(f, 0) * L : s.e + RealOps<R>::par(f, j) * L;
            if (j == 2 || j == 3) {
                const R z = L - RealOps<R>::par(f, 6);
                s.e += z * z * RealOps<R>::par(f, 7);
            }
        }
        if (j == 0) s.x12 = x;
        if (j == 1) s.x12 += x;
    }
    __device__ static R end(const S& s, uint32_t, const FamConsts& f)
    {
        const R z = s.x12 - RealOps<R>::par(f, 8);
        if constexpr (kWide) return RealOps<R>::expm_(s.e + z * z * f.c[9]);  // c10: in the Jacobian
        else return RealOps<R>::par(f, 10) * RealOps<R>::expm_(s.e + z * z * RealOps<R>::par(f, 9));
    }
    // f J in double precision, J = (jm / 2^63) 2^je the integer Jacobian
    __device__ static double end_scaled(const S& s, const FamConsts& f, uint64_t jm, int je)
    {
        const double z = s.x12 - f.c[8];
        return fx::fx_exp_neg_scaled(s.e + z * z * f.c[9], jm, je);
    }
};

// Interpolation tables (TABLE family): the point is clamped into the knot
// range, u = (x - lo) s with s = (n - 1)/(hi - lo), cell i = floor(u) (at
// most n - 2), t = u - i, and the value is (1 - t) v_i + t v_{i+1}
// (bilinear: the same on both axes).  The interpolant is continuous at the
// knots, so a point on a knot gives the same value from either cell.
template <typename R> struct TabOps;
template <> struct TabOps<double> {
    // Cell and fraction with one FP64 operation: u = x s - lo s by one FMA;
    // the floor of u (0 <= u < 2^31) and the fraction t = u - floor(u) are
    // taken from the bits of u's encoding (t normalised into a double with
    // integer operations), and the clamps are integer tests on those bits, so
    // no FP64 subtraction, conversion or compare is issued (GB300 runs 2 FP64
    // instructions per clock per SM against 64 integer ones).
    __device__ static void cell(double x, double s, double los, int n, int* i, double* t)
    {
        const double u = fma(x, s, -los);
        int64_t b = __double_as_longlong(u);
        if (b < 0) b = 0;                         // below the range (or -0): u = 0
        const int e = (int)((uint64_t)b >> 52) - 1023;
        if (e < 0) {                              // u < 1: cell 0, t = u
            *i = 0;
            *t = __longlong_as_double(b);
            return;
        }
        const int sh = 52 - e;
        const uint64_t M = ((uint64_t)b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
        const int k = e < 31 ? (int)(M >> sh) : n;  // u >= 2^31 > n - 1 (also inf, NaN)
        if (k > n - 2) {                          // floor(u) >= n - 1: at or above the last knot
            *i = n - 2;
            *t = 1.0;
            return;
        }
        *i = k;
        // t = F 2^-sh for the fraction bits F < 2^sh: exact, normalised here
        const uint64_t F = M & ((1ull << sh) - 1ull);
        const int q = 63 - __clzll((long long)F);  // leading bit of F (q < sh <= 52)
        const uint64_t tb = ((uint64_t)(q - sh + 1022) << 52) + (F << (52 - q));
        *t = F ? __longlong_as_double((long long)tb) : 0.0;
    }
    __device__ static double interp1(const TableDesc& T, double x)
    {
        int i;
        double t;
        cell(x, T.s0, T.los0, T.n0, &i, &t);
        const double v0 = __ldg(T.v + i), v1 = __ldg(T.v + i + 1);
        return fma(t, v1 - v0, v0);
    }
    __device__ static double interp2(const TableDesc& T, double x, double y)
    {
        int i, k;
        double t, s;
        cell(x, T.s0, T.los0, T.n0, &i, &t);
        cell(y, T.s1, T.los1, T.n1, &k, &s);
        const double* r0 = T.v + (size_t)i * T.n1 + k;
        const double* r1 = r0 + T.n1;
        const double v00 = __ldg(r0), v01 = __ldg(r0 + 1), v10 = __ldg(r1), v11 = __ldg(r1 + 1);
        const double a = fma(t, v10 - v00, v00), b = fma(t, v11 - v01, v01);
        return fma(s, b - a, a);
    }
};
template <> struct TabOps<float> {
    __device__ static void cell(float x, float lo, float hi, float s, int n, int* i, float* t)
    {
        const float u = (fminf(fmaxf(x, lo), hi) - lo) * s;
        const int k = min((int)u, n - 2);
        *i = k;
        *t = u - (float)k;
    }
    __device__ static float interp1(const TableDesc& T, float x)
    {
        int i;
        float t;
        cell(x, T.lo0f, T.hi0f, T.s0f, T.n0, &i, &t);
        return (1.0f - t) * __ldg(T.vf + i) + t * __ldg(T.vf + i + 1);
    }
    __device__ static float interp2(const TableDesc& T, float x, float y)
    {
        int i, k;
        float t, s;
        cell(x, T.lo0f, T.hi0f, T.s0f, T.n0, &i, &t);
        cell(y, T.lo1f, T.hi1f, T.s1f, T.n1, &k, &s);
        const float* r0 = T.vf + (size_t)i * T.n1 + k;
        const float* r1 = r0 + T.n1;
        return (1.0f - t) * (1.0f - s) * __ldg(r0) + t * (1.0f - s) * __ldg(r1) + (1.0f - t) * s * __ldg(r0 + 1) +
               t * s * __ldg(r1 + 1);
    }
};

template <typename R> struct Family<MCUBES_F_TABLE, R> {
    // the coordinates are kept (registers: every index below is a
    // compile-time constant) and the factors evaluated at the end
    struct S { R x[kDMax]; };
    __device__ static void begin(S& s)
    {
#pragma unroll
        for (int j = 0; j < kDMax; ++j) s.x[j] = R(0);
    }
    __device__ static void add(S& s, int j, R x, const FamParams&) { s.x[j] = x; }
    __device__ static R sel(const S& s, int a)
    {
        R v = s.x[0];
#pragma unroll
        for (int j = 1; j < kDMax; ++j)
            if (a == j) v = s.x[j];
        return v;
    }
    __device__ static R end(const S& s, uint32_t, const FamParams& f)
    {
        R prod = RealOps<R>::par(f, 0);
        for (int q = 0; q < f.nf; ++q) {
            const TableDesc& T = f.tabs[f.tid[q]];
            const R xa = sel(s, f.ta[q]);
            if (f.tb[q] < 0) prod *= TabOps<R>::interp1(T, xa);
            else prod *= TabOps<R>::interp2(T, xa, sel(s, f.tb[q]));
        }
        return prod;
    }
};

// ---------------------------------------------------------------------------
// Fixed-point form of the FP64 affine families.  The integrand reads each
// coordinate only through t_j = s_j (x_j - o_j) (plus, for DISCONT, a
// threshold on it), so the map cells hold t_j instead of x_j: the left edge
// as a 64-bit integer with f fraction bits and the width as a double, and a
// sample's t_j is one 64-bit high multiply (width significand x g phi's exact
// numerator), a shift and an addition.  The sums over the axes, the
// exponential, reciprocal or cosine and the Jacobian's product stay in
// integers and F = f J is rounded to a double once: no FP64 instruction
// before the moments and the histogram.  GB300 issues 2 FP64 instructions per
// clock per SM against 64 integer ones, and the double-precision form of
// these kernels kept that pipe 80% busy (its practical limit) on 47-100
// warp instructions per sample.  Adjusting passes of 9.65e6 samples at d = 6,
// before and with this form: GAUSS 779 -> 392 us, CORNER 676 -> 357, OSC (f_A)
// 781 -> 336, PRODPEAK 1224 -> 420, C0 879 -> 366, DISCONT 651 -> 360; what is
// left on the FP64 pipe is the histogram's additions.  t_j's error is about 2^-f
// absolute, f at least 57 (C0 and DISCONT 54, CORNER such that the sum is 2^56
// units or more; affine.cu keeps the ranges small enough for that, or the
// double-precision form is used): below the rounding of x itself.
// Scales: GAUSS t = (x - mu)/(sigma sqrt 2), sum of t^2; C0 t = c (x - w),
// sum of |t|; DISCONT, CORNER t = a (x - lo); OSC t = a x / (2 pi) in turns,
// whole turns dropped by the wrap-around; PRODPEAK t = c (x - w), f = prod
// c^2 / (1 + t^2).  Constant factors are part of the Jacobian's.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t abs_u64(int64_t t) { return t < 0 ? 0ull - (uint64_t)t : (uint64_t)t; }

// t^2 for |t| < 2^63 with f fraction bits: 2 f - 62 fraction bits
__device__ __forceinline__ uint64_t sq_fixed(int64_t t)
{
    const uint64_t a = abs_u64(t) << 1;
    return __umul64hi(a, a);
}

template <int FAM> struct FixFamily { static constexpr bool kHas = false; };

struct FixSum {
    uint64_t q;
};

template <> struct FixFamily<MCUBES_F_GAUSS> {
    static constexpr bool kHas = true;
    using S = FixSum;
    __device__ static void begin(S& s, const FamConsts& f) { s.q = f.fu[kDMax]; }
    __device__ static void add(S& s, int, int64_t t, const FamConsts&) { s.q += sq_fixed(t); }
    template <int D> __device__ static double end(const S& s, const FamConsts& f, const IntProd& jp)
    {
        return fx::fx_exp_fixed<true>(s.q, f.fq, jp.m, jp.e);
    }
};

template <> struct FixFamily<MCUBES_F_C0> {
    static constexpr bool kHas = true;
    using S = FixSum;
    __device__ static void begin(S& s, const FamConsts& f) { s.q = f.fu[kDMax]; }
    // |t|, or one less on the negative side: t is cut downwards, so both sides are short by half a unit on average
    __device__ static void add(S& s, int, int64_t t, const FamConsts&) { s.q += (uint64_t)(t ^ (t >> 63)); }
    template <int D> __device__ static double end(const S& s, const FamConsts& f, const IntProd& jp)
    {
        return fx::fx_exp_fixed<true>(s.q, f.fq, jp.m, jp.e);
    }
};

template <> struct FixFamily<MCUBES_F_DISCONT> {
    static constexpr bool kHas = true;
    struct S {
        uint64_t q;
        bool out;
    };
    __device__ static void begin(S& s, const FamConsts& f)
    {
        s.q = f.fu[kDMax];
        s.out = false;
    }
    __device__ static void add(S& s, int j, int64_t t, const FamConsts& f)
    {
        s.out |= (uint64_t)t >= f.fu[j];
        s.q += (uint64_t)t;
    }
    template <int D> __device__ static double end(const S& s, const FamConsts& f, const IntProd& jp)
    {
        return s.out ? 0.0 : fx::fx_exp_fixed<false>(s.q, f.fq, jp.m, jp.e);
    }
};

template <> struct FixFamily<MCUBES_F_CORNER> {
    static constexpr bool kHas = true;
    using S = FixSum;
    __device__ static void begin(S& s, const FamConsts& f) { s.q = f.fu[kDMax]; }
    __device__ static void add(S& s, int, int64_t t, const FamConsts&) { s.q += (uint64_t)t; }
    template <int D> __device__ static double end(const S& s, const FamConsts& f, const IntProd& jp)
    {
        // t^-(D+1) J by repeated squaring of 1/t
        IntProd b = int_prod_recip(int_prod_of_fixed(s.q, f.fq)), r = jp;
#pragma unroll
        for (uint32_t e = D + 1; e; e >>= 1) {
            if (e & 1u) r = int_prod_mul2(r, b);
            if (e > 1u) b = int_prod_mul2(b, b);
        }
        return int_prod_value(r);
    }
};

template <> struct FixFamily<MCUBES_F_OSC> {
    static constexpr bool kHas = true;
    using S = FixSum;
    __device__ static void begin(S& s, const FamConsts& f) { s.q = f.fu[kDMax]; }
    __device__ static void add(S& s, int, int64_t t, const FamConsts&) { s.q += (uint64_t)t; }
    template <int D> __device__ static double end(const S& s, const FamConsts& f, const IntProd& jp)
    {
        bool neg;
        const uint64_t v = fx::fx_cos_turns(s.q << (64 - f.fq), &neg);
        if (v == 0) return 0.0;
        const double F = int_prod_value(int_prod_mul2(jp, int_prod_of_fixed(v, 63)));
        return neg ? -F : F;
    }
};

template <> struct FixFamily<MCUBES_F_PRODPEAK> {
    static constexpr bool kHas = true;
    using S = IntProd;
    __device__ static void begin(S& s, const FamConsts&) { s = IntProd{1ull << 63, 0}; }
    __device__ static void add(S& s, int j, int64_t t, const FamConsts& f)
    {
        // the squares are cut, by half a last place on average: every other axis takes one back
        s = int_prod_mul2(s, int_prod_of_fixed((1ull << f.fq) + (uint64_t)(j & 1) + sq_fixed(t), f.fq));
    }
    template <int D> __device__ static double end(const S& s, const FamConsts&, const IntProd& jp)
    {
        return int_prod_value(int_prod_mul2(jp, int_prod_recip(s)));
    }
};

// TABLE: t_j in knots of the table dimension that reads axis j, so the cell is
// t's integer part and the fraction its low bits; the interpolants are formed
// in double as in the general form.  The values of up to four factors are
// fetched before the first is used (random 8-byte reads of tables larger than
// the caches: the fetches overlap instead of following one another).
// table6 at 1e8 calls: 9.50 -> 7.98 ms per pass (FP64 pipe 80% busy before, 46
// warp instructions per sample; now 38.7, and 5.0 TB/s from HBM, 74% of the
// measured copy rate).  128 registers, 16 warps per SM: 20 and 24 warps with
// spills measured 8.55 and 9.16 ms.
template <> struct FixFamily<MCUBES_F_TABLE> {
    static constexpr bool kHas = true;
    struct S {
        int64_t t[kDMax];
    };
    __device__ static void begin(S&, const FamParams&) {}
    __device__ static void add(S& s, int j, int64_t t, const FamParams&) { s.t[j] = t; }
    // cell i (at most n - 2) and fraction of the coordinate of axis a
    template <int D> __device__ static void cell(const S& s, const FamParams& f, int a, int n, int* i, double* frac)
    {
        int64_t t = s.t[0];
        int fb = f.ff[0];
#pragma unroll
        for (int j = 1; j < D; ++j)
            if (a == j) {
                t = s.t[j];
                fb = f.ff[j];
            }
        if (t < 0) t = 0;  // below the range
        const uint64_t u = (uint64_t)t;
        const int64_t k = (int64_t)(u >> fb);
        const uint64_t F = u & ((1ull << fb) - 1ull);
        // F 2^-fb, rounded to 53 bits
        const int lz = __clzll((long long)F);
        const uint64_t m = F << (lz & 63);
        const uint64_t r = (m >> 11) + ((m >> 10) & 1ull);
        const uint64_t bits = ((uint64_t)(1023 + 63 - lz - fb - 1) << 52) + r;
        const bool above = k > n - 2;  // at or above the last knot
        *i = above ? n - 2 : (int)k;
        *frac = above ? 1.0 : (F ? __longlong_as_double((long long)bits) : 0.0);
    }
    template <int D> __device__ static double end(const S& s, const FamParams& f, const IntProd& jp)
    {
        double prod = f.c[0];
#pragma unroll 1
        for (int q0 = 0; q0 < f.nf; q0 += 4) {
            double v[4][4], t[4], w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int q = q0 + u;
                if (q < f.nf) {
                    const TableDesc& T = f.tabs[f.tid[q]];
                    int i, k;
                    cell<D>(s, f, f.ta[q], T.n0, &i, &t[u]);
                    if (f.tb[q] < 0) {
                        const double* p = T.v + i;
                        v[u][0] = __ldg(p);
                        v[u][1] = __ldg(p + 1);
                    } else {
                        cell<D>(s, f, f.tb[q], T.n1, &k, &w[u]);
                        const double* p = T.v + (size_t)i * T.n1 + k;
                        v[u][0] = __ldg(p);
                        v[u][2] = __ldg(p + 1);
                        v[u][1] = __ldg(p + T.n1);
                        v[u][3] = __ldg(p + T.n1 + 1);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int q = q0 + u;
                if (q < f.nf) {
                    double a = fma(t[u], v[u][1] - v[u][0], v[u][0]);
                    if (f.tb[q] >= 0) {
                        const double b = fma(t[u], v[u][3] - v[u][2], v[u][2]);
                        a = fma(w[u], b - a, a);
                    }
                    prod *= a;
                }
            }
        }
        return prod * int_prod_value(jp);
    }
};

// ---------------------------------------------------------------------------
// Compensated single-precision accumulator (Knuth's TwoSum; the pair holds
// about 48 significant bits).  Used for the per-thread sums over cubes of the
// mixed-precision path, which must not issue FP64 work per sample.
// ---------------------------------------------------------------------------
struct DFloat {
    float hi, lo;
    __device__ void add(float v)
    {
        const float s = __fadd_rn(hi, v);
        const float bp = __fsub_rn(s, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(v, bp));
        hi = s;
        lo = __fadd_rn(lo, err);
    }
    __device__ double value() const { return (double)hi + (double)lo; }
};

}  // namespace mc
