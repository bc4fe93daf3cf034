// refine_dev.cuh -- device pieces of the per-iteration finalisation shared
// by the single-integral and the batched refinement launches: fixed-order
// sums, Weighted-Estimates with Check-Convergence (Alg. 2), and
// Adjust-Bin-Bounds of one axis (Alg. 2, Lepage 1978).
#pragma once

#include <cmath>

#include "mc_device.cuh"

namespace mc {
namespace refine_detail {

constexpr int kWarps = kRefineThreads / 32;
constexpr int kPerThread = (kNbMax + kRefineThreads - 1) / kRefineThreads;

// Deterministic block sum (each thread's value added in a fixed tree).
static __device__ __forceinline__ double block_sum(double v, double* scratch)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double w = lane < kWarps ? scratch[lane] : 0.0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) w += __shfl_down_sync(0xffffffffu, w, off);
        if (lane == 0) scratch[32] = w;
    }
    __syncthreads();
    const double out = scratch[32];
    __syncthreads();
    return out;
}

// ---------------------------------------------------------------------------
// Weighted-Estimates and the record of one iteration
// ---------------------------------------------------------------------------

// GB300's FP64 pipe takes one warp instruction per 16 cycles per SM whatever
// the number of active lanes, and a dependent FP64 instruction 66 cycles: the
// finalisation sums the partials on four warps and weighs on one.
constexpr int kRedThreads = 128;

// Sums of N values over the 32 lanes, the same in every lane.
template <int N>
static __device__ __forceinline__ void warp_sum(double (&v)[N])
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], off);
}

// Where one integral's iteration results live (a single context's DevState,
// or one entry of a batch's state array plus its history arrays).
struct IterRecord {
    uint32_t* it;
    int* done;
    int* error;
    int* n;
    int* converged;
    double* estimate;
    double* sigma;
    double* chi2_dof;
    double* hist_I;
    double* hist_V;
    int cap;
    double rel_tol, abs_tol;
};

// Weighted-Estimates (inverse-variance weights, chi^2 per degree of freedom)
// over n recorded iterations by one warp: lane l takes iterations l, l + 32,
// ...; its first one is (I, V), already in registers (an older one was read
// while the partials were summed).  The reciprocals of the variances are
// formed side by side: a dependent FP64 division takes ~450 cycles.
static __device__ __forceinline__ void weigh_warp(const double* hI, const double* hV, int n, double I, double V,
                                                  double* est, double* sigma, double* chi2_dof)
{
    const int lane = threadIdx.x & 31;
    const double inv_dof = n > 1 ? 1.0 / (double)(n - 1) : 0.0;  // off the dependent chain
    const bool mine = lane < n;
    const double w = mine && V != 0.0 ? 1.0 / V : 0.0;
    double s[2] = {w, w * I};
    bool exact = mine && V == 0.0;
    for (int i = lane + 32; i < n; i += 32) {
        const double Vi = hV[i];
        const double wi = Vi != 0.0 ? 1.0 / Vi : 0.0;
        exact |= Vi == 0.0;
        s[0] += wi;
        s[1] += wi * hI[i];
    }
    if (__any_sync(0xffffffffu, exact)) {  // iterations of zero variance are exact: their mean, sigma 0
        double e[2] = {0.0, 0.0};
        if (mine && V == 0.0) {
            e[0] = 1.0;
            e[1] = I;
        }
        for (int i = lane + 32; i < n; i += 32)
            if (hV[i] == 0.0) {
                e[0] += 1.0;
                e[1] += hI[i];
            }
        warp_sum<2>(e);
        *est = e[1] / e[0];
        *sigma = 0.0;
        *chi2_dof = 0.0;
        return;
    }
    warp_sum<2>(s);
    const double inv_sw = 1.0 / s[0];
    const double m = s[1] * inv_sw;
    double chi2 = 0.0;
    if (n > 1) {
        double c[1] = {mine ? (I - m) * (I - m) * w : 0.0};
        for (int i = lane + 32; i < n; i += 32) {
            const double z = hI[i] - m;
            c[0] += z * z * (1.0 / hV[i]);
        }
        warp_sum<1>(c);
        chi2 = c[0] * inv_dof;
    }
    *est = m;
    *sigma = sqrt(inv_sw);
    *chi2_dof = chi2;
}

// Reduces nparts block partials (3 doubles each, fixed order) into the
// iteration estimate I = sum means / m and variance sum vars / m^2, records
// them, weighs all iterations, tests convergence (Check-Convergence: n >= 2
// and sigma <= max(abs_tol, rel_tol |I|)) and advances the iteration.  With
// split > 1 the partials are (K, S1, S2) of cube slices, split consecutive
// ones per cube (sums of F - K over a slice of q = ceil(p/split) samples, the
// last slice shorter): each cube's slices are re-based on the first slice's
// shift and summed in order, then the cube's mean and the variance of that
// mean follow (UpdateVariance of Alg. 3).  Every thread of the block calls.
// The chain is FP64 latency: gauss4 at 1e4 calls, 608 partials, 9.9 us when
// every warp took part in each sum and the weighing met six block barriers,
// 5-6 us now, one barrier and three divisions deep.
static __device__ void finalize_iteration(const double* part, int nparts, double m, const IterRecord& r,
                                          int split = 1, double p = 0.0)
{
    __shared__ double sw[2][kRedThreads / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= kRedThreads / 32) {
        __syncthreads();
        return;
    }
    const int n = *r.n;
    double I = 0.0, V = 0.0;  // lane l of warp 0: iteration l, read ahead
    if (warp == 0 && lane < n) {
        I = r.hist_I[lane];
        V = r.hist_V[lane];
    }
    double s01[2] = {0.0, 0.0};
    if (split > 1) {
        // thread t merges cubes t, t + kRedThreads, ...: each slice re-based on
        // the cube's first shift and added in slice order, eight slices'
        // partials loaded ahead at a time; then the cube's mean and the variance
        // of that mean (UpdateVariance of Alg. 3) with the reciprocals formed once
        const int ncubes = nparts / split;
        // samples of a slice: q in the first k_full, then the rest, then none
        const double q = ceil(p / split);
        const int k_full = (int)(p / q);
        const double rest = p - q * k_full;
        const double inv_p = 1.0 / p, inv_var_den = inv_p / (p - 1.0);
        for (int cb = threadIdx.x; cb < ncubes; cb += kRedThreads) {
            const double* v = part + 3 * (size_t)cb * split;
            const double K0 = v[0];
            double S1 = 0.0, S2 = 0.0;
            for (int k0 = 0; k0 < split; k0 += 8) {
                double a0[8], a1[8], a2[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int k = min(k0 + u, split - 1);
                    a0[u] = v[3 * k];
                    a1[u] = v[3 * k + 1];
                    a2[u] = v[3 * k + 2];
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int k = k0 + u;
                    if (k < split) {
                        const double nk = k < k_full ? q : (k == k_full ? rest : 0.0);
                        const double dK = a0[u] - K0;
                        S2 += fma(dK, fma(nk, dK, 2.0 * a1[u]), a2[u]);
                        S1 += fma(nk, dK, a1[u]);
                    }
                }
            }
            s01[0] += K0 + S1 * inv_p;
            s01[1] += (S2 - S1 * S1 * inv_p) * inv_var_den;
        }
    } else {
        int b = threadIdx.x;
        for (; b + 3 * kRedThreads < nparts; b += 4 * kRedThreads) {
            double x[4], y[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                x[u] = part[3 * (size_t)(b + u * kRedThreads) + 0];
                y[u] = part[3 * (size_t)(b + u * kRedThreads) + 1];
            }
            s01[0] += (x[0] + x[1]) + (x[2] + x[3]);
            s01[1] += (y[0] + y[1]) + (y[2] + y[3]);
        }
        for (; b < nparts; b += kRedThreads) {
            s01[0] += part[3 * (size_t)b + 0];
            s01[1] += part[3 * (size_t)b + 1];
        }
    }
    warp_sum<2>(s01);
    if (lane == 0) {
        sw[0][warp] = s01[0];
        sw[1][warp] = s01[1];
    }
    __syncthreads();
    if (warp != 0) return;
    // lane 0 forms I, lane 1 V: one division for both
    const int h = lane & 1;
    const double tot = (sw[h][0] + sw[h][1]) + (sw[h][2] + sw[h][3]);
    const double iv = tot / (h ? m * m : m);
    const double In = __shfl_sync(0xffffffffu, iv, 0), Vn = __shfl_sync(0xffffffffu, iv, 1);
    const bool finite = isfinite(In) && isfinite(Vn);
    const int nn = n < r.cap ? n + 1 : n;
    if (n < r.cap) {
        if (lane == 0) {
            r.hist_I[n] = In;
            r.hist_V[n] = Vn;
            *r.n = nn;
        }
        if (lane == n) {
            I = In;
            V = Vn;
        }
    }
    if (!finite) {
        if (lane == 0) {
            *r.error = MCUBES_ENONFINITE;
            *r.done = 1;
        }
    } else {
        __syncwarp();  // the record is visible to the lanes (n >= 32: it is read back)
        double est, sig, chi2;
        weigh_warp(r.hist_I, r.hist_V, nn, I, V, &est, &sig, &chi2);
        const double tol = fmax(r.abs_tol, r.rel_tol * fabs(est));
        if (lane == 0) {
            *r.estimate = est;
            *r.sigma = sig;
            *r.chi2_dof = chi2;
            if (nn >= 2 && sig <= tol) {
                *r.converged = 1;
                *r.done = 1;
            }
        }
    }
    if (lane == 0) *r.it += 1;
}

// ---------------------------------------------------------------------------
// Adjust-Bin-Bounds
// ---------------------------------------------------------------------------

// Exact cumulative weights: each bin weight w in [0, 1] as an unsigned Q100
// integer (128 bits; bits below 2^-100 dropped), their prefix sums exact (at
// most nb 2^100 < 2^110), so the order of the additions does not matter and
// the quantile tests are exact integer comparisons.
static __device__ __forceinline__ u128 q100_of(double w)  // 0 <= w < 2^27
{
    const uint64_t b = (uint64_t)__double_as_longlong(w);
    const int E = (int)(b >> 52);
    if (E == 0) return 0;                             // zero (or below 2^-1022)
    const uint64_t M = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = E - 975;                           // w = (M << (E - 975)) 2^-100
    if (sh >= 0) return (u128)M << sh;                // sh < 75: below 2^128
    return sh > -53 ? (u128)(M >> -sh) : (u128)0;
}

static __device__ __forceinline__ u128 shfl_up_u128(u128 v, int off)
{
    const unsigned long long lo = __shfl_up_sync(0xffffffffu, (unsigned long long)v, off);
    const unsigned long long hi = __shfl_up_sync(0xffffffffu, (unsigned long long)(v >> 64), off);
    return ((u128)hi << 64) | (u128)lo;
}

// base plus the inclusive prefix sum over the block's threads of v (Q100),
// scanned by warp shuffles and then across warps; *total receives the last
// thread's.  Exact, so any order gives the same sums.  wtot is free again
// after the caller's next barrier.
static __device__ __forceinline__ u128 u128_scan(u128 v, u128 base, u128* wtot, u128* total)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    u128 incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const u128 o = shfl_up_u128(incl, off);
        if (lane >= off) incl += o;
    }
    if (lane == 31) wtot[warp] = incl;
    __syncthreads();
    // every warp scans the 16 warp totals for itself: no second barrier
    u128 x = lane < kWarps ? wtot[lane] : (u128)0;
#pragma unroll
    for (int off = 1; off < kWarps; off <<= 1) {
        const u128 o = shfl_up_u128(x, off);
        if (lane >= off) x += o;
    }
    const int src = warp > 0 ? warp - 1 : 0;
    const unsigned long long blo = __shfl_sync(0xffffffffu, (unsigned long long)x, src);
    const unsigned long long bhi = __shfl_sync(0xffffffffu, (unsigned long long)(x >> 64), src);
    u128 run = base + incl;
    if (warp > 0) run += ((u128)bhi << 64) | (u128)blo;
    if (t == kRefineThreads - 1) *total = run;
    return run;
}

// Three times the smoothed value of bin k: C_{k-1} + C_k + C_{k+1}; the ends
// 1.5 (C_0 + C_1) and 1.5 (C_{nb-2} + C_{nb-1}) (nb >= 2).
static __device__ __forceinline__ double smoothed3(const double* sC, int k, int nb)
{
    const bool end = k == 0 || k == nb - 1;
    const int i = k == 0 ? 0 : k - 1;  // the ends: the pair at that side, 1.5 times
    const double pair = sC[i] + sC[i + 1];
    return end ? 1.5 * pair : pair + sC[k + 1];
}

// q^alpha as Q100 for other exponents than 1 and 3/2 (out of line: a launch
// runs its code once per bin, from a cold instruction cache)
static __device__ __noinline__ u128 power_weight(double q, double alpha)
{
    return q100_of(fx::fx_exp(alpha * fx::fx_log(q)));
}

// Compressed weight ((r - 1)/ln r)^alpha of a bin, r = sm3 / total, as Q100,
// in integers: r = sm3 (1/total) rounded to a double's precision (subnormal
// ones included, so that the bins that count as empty are the same as in
// double arithmetic), |ln r| from the logarithm's own fixed-point parts, one
// fixed-point reciprocal, and for alpha = 3/2 a fixed-point square root.  The
// FP64 form of this (two divisions, a logarithm's rounding, a root) was ~75
// dependent FP64 instructions, 66 cycles each.
static __device__ __forceinline__ u128 compressed_weight(double sm3, const IntProd& inv_total, double alpha,
                                                         const fx::LogPair (*logs)[256])
{
    if (!(sm3 > 0.0)) return 0;
    IntProd r = int_prod_mul2(int_prod_of(sm3), inv_total);
    const int drop = r.e < -1022 ? 11 - 1022 - r.e : 11;  // bits below a double's last place
    if (drop > 64) return 0;                              // rounds to 0
    if (drop == 64) r = IntProd{1ull << 63, r.e + 1};     // rounds to the smallest subnormal
    else {
        const uint64_t up = r.m + (1ull << (drop - 1));
        r = up < r.m ? IntProd{1ull << 63, r.e + 1} : IntProd{up >> drop << drop, r.e};
    }
    if (r.e >= 0) return (u128)1 << 100;                  // r >= 1
    // |ln r| = -e ln 2 - ln m as a 128-bit Q64 magnitude
    const uint64_t U = fx::fx_ln_mantissa_t((r.m >> 11) & 0xFFFFFFFFFFFFFull, [&](int t, int i) { return logs[t][i]; });
    const u128 ln = (u128)(uint32_t)(-r.e) * fx::kLn2Q64 - U;
    const int z = clz_u128(ln);
    const IntProd L{(uint64_t)((ln << z) >> 64), 63 - z};
    const int sh = -1 - r.e;                              // r as Q64
    const uint64_t om = 0ull - (sh < 64 ? r.m >> sh : 0ull);  // 1 - r, Q64 (0: r below 2^-64)
    const IntProd q = int_prod_mul2(om ? int_prod_of_fixed(om, 64) : IntProd{~0ull, -1}, int_prod_recip(L));
    IntProd w = q;
    if (alpha == 1.5) {
        const int odd = (q.e + 1) & 1;                    // q = M 2^-64 4^h, M in [2^62, 2^64)
        const IntProd root{fx::fx_sqrt(q.m >> odd) << 1, (q.e + 1 + odd) / 2 - 1};
        w = int_prod_mul2(q, root);
    } else if (alpha != 1.0) {
        return power_weight(int_prod_value(q), alpha);
    }
    const int s = w.e + 37;                               // w 2^100 = m 2^(e + 37)
    return s >= 0 ? (u128)w.m << s : (s > -64 ? (u128)(w.m >> -s) : (u128)0);
}

// New right edge of bin i - 1 (1 <= i < nb): the first bin k whose cumulative
// weight reaches i/nb of the total W (nb C_k >= i W), at the fraction
// (i W - nb C_{k-1}) / (nb w_k) of its width; sX holds nb C_k.
static __device__ __forceinline__ DD rebin_edge(int i, int nb, u128 W, const u128* sX, const double* sB,
                                                const double* sBlo)
{
    const u128 T = (u128)(uint32_t)i * W;
    int lo = 0, hi = nb - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (sX[mid] >= T) hi = mid; else lo = mid + 1;
    }
    const int k = lo;
    const u128 before = k > 0 ? sX[k - 1] : (u128)0;  // < T
    const u128 den = sX[k] - before, num = T - before;
    const int z = clz_u128(den);
    const uint64_t rec = fx::fx_recip((uint64_t)((den << z) >> 64));
    const uint64_t frac = __umul64hi((uint64_t)((num << z) >> 64), rec);  // Q63
    const DD right{sB[k], sBlo[k]};
    const DD left = k > 0 ? DD{sB[k - 1], sBlo[k - 1]} : DD{0.0, 0.0};
    const int E = exponent_of(right.hi);
    const u128 l = edge_u128(left, E), w = edge_u128(right, E) - l;
    const u128 part = ((u128)(uint64_t)(w >> 64) * frac + __umul64hi((uint64_t)w, frac)) << 1;
    const u128 e = l + part;
    return e != 0 ? edge_from_u128(e, E) : DD{0.0, 0.0};
}

// Shared memory of one axis's rebinning (a block of kRefineThreads).
struct RebinShared {
    double C[kNbMax];               // the histogram row
    double B[kNbMax], Blo[kNbMax];  // edges: the old ones, then the new ones
    u128 X[kNbMax];                 // nb x the inclusive cumulative compressed weights, Q100
    u128 wtot[kWarps];
    u128 W[kPerThread];             // weight up to each round's last bin
    fx::LogPair logs[2][256];       // the logarithm's tables (load_log_tables)
    uint32_t emax[kWarps];
    uint32_t sum[3][kWarps];
    long long ends[4];              // C_0, C_1, C_{nb-2}, C_{nb-1} in the fixed-point scale
};

// The logarithm's tables into shared memory: a bin's two lookups depend on each
// other, ~700 cycles each from a cold cache.
static __device__ __forceinline__ void load_log_tables(RebinShared& s)
{
    const int t = threadIdx.x;
    static_assert(kRefineThreads == 512, "one entry per thread");
    s.logs[t >> 8][t & 255] = fx::ld_pair(t >= 256 ? &fx::kLogD[t & 255] : &fx::kLogC[t & 255]);
}

// Adjust-Bin-Bounds of one axis (Lepage 1978, as the paper's Alg. 2 cites):
// smooth the bin sums with their neighbours, normalise, compress with
// ((r - 1) / ln r)^alpha, then place the new right edges where the
// cumulative compressed weight reaches i / nb of its total, the weight of an
// old bin being spread evenly over it.  The smoothing keeps three times the
// neighbour mean (the normalisation removes the factor); the cumulative
// weight is exact in Q100 integers, the fraction within a bin is a 64-bit
// fixed-point quotient and the edge left + width * fraction is formed in
// 128-bit integers scaled by the old right edge, so the new bin widths keep
// full double precision.  All but the smoothing (two FP64 additions per bin)
// is integer work: GB300 issues 2 FP64 instructions per clock per SM and a
// dependent one takes 66 cycles, while the integer chain of a bin takes a few
// cycles per step, so one block per axis is enough (the FP64 form took
// 27,500 cycles spread over a cluster of four blocks per axis, five cluster
// barriers included; refine.cu has both sides' times).
// On entry s.C, s.B, s.Blo and s.logs hold the histogram, the edges and the
// logarithm's tables (written by this block, no barrier needed); true: s.B and
// s.Blo hold the new edges.  False: the grid stays (no information on the axis,
// or a non-finite sum, which is reported in *error and *done).
static __device__ bool rebin_block(RebinShared& s, int nb, double alpha, int* error, int* done)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    __syncthreads();
    // the total, as an integer: every C_k with 62 bits below the largest's
    // exponent; three 22-bit pieces are added by warp reductions
    uint64_t mant[kPerThread];
    int ex[kPerThread];
    uint32_t em = 0;
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
        const int k = t * kPerThread + i;
        const uint64_t b = k < nb ? (uint64_t)__double_as_longlong(s.C[k]) : 0ull;
        const uint32_t e = (uint32_t)(b >> 52) & 0x7FFu;
        mant[i] = ((b & 0xFFFFFFFFFFFFFull) | (e ? 1ull << 52 : 0ull)) << 9;
        ex[i] = e ? (int)e : 1;
        if (mant[i]) em = max(em, (uint32_t)ex[i]);  // 0: every bin is zero
    }
    em = __reduce_max_sync(0xffffffffu, em);
    if (lane == 0) s.emax[warp] = em;
    __syncthreads();
    em = __reduce_max_sync(0xffffffffu, lane < kWarps ? s.emax[lane] : 0u);
    if (em == 0) return false;  // no information on this axis: grid unchanged
    uint32_t p0 = 0, p1 = 0, p2 = 0;
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
        const int k = t * kPerThread + i;
        const int sh = (int)em - ex[i];
        const uint64_t c = sh < 64 ? mant[i] >> sh : 0ull;
        p0 += (uint32_t)c & 0x3FFFFFu;
        p1 += (uint32_t)(c >> 22) & 0x3FFFFFu;
        p2 += (uint32_t)(c >> 44);
        if (k == 0) s.ends[0] = (long long)c;
        if (k == 1) s.ends[1] = (long long)c;
        if (k == nb - 2) s.ends[2] = (long long)c;
        if (k == nb - 1) s.ends[3] = (long long)c;
    }
    p0 = __reduce_add_sync(0xffffffffu, p0);
    p1 = __reduce_add_sync(0xffffffffu, p1);
    p2 = __reduce_add_sync(0xffffffffu, p2);
    if (lane == 0) {
        s.sum[0][warp] = p0;
        s.sum[1][warp] = p1;
        s.sum[2][warp] = p2;
    }
    __syncthreads();
    p0 = __reduce_add_sync(0xffffffffu, lane < kWarps ? s.sum[0][lane] : 0u);
    p1 = __reduce_add_sync(0xffffffffu, lane < kWarps ? s.sum[1][lane] : 0u);
    p2 = __reduce_add_sync(0xffffffffu, lane < kWarps ? s.sum[2][lane] : 0u);
    // twice the sum of the smoothed3 values: 6 sum C - C_0 + C_1 + C_{nb-2} - C_{nb-1}
    const u128 sum = (u128)p0 + ((u128)p1 << 22) + ((u128)p2 << 44);
    const u128 t2 = 6 * sum + (u128)(__int128)(s.ends[1] - s.ends[0]) + (u128)(__int128)(s.ends[2] - s.ends[3]);
    const int z = clz_u128(t2);  // t2 > 0: 6 sum >= 6 (C_0 + C_{nb-1})
    const int eT = 127 - z + (int)em - 1085;  // C_k = c 2^(em - 1084)
    if (em == 0x7FFu || eT >= 1024) {
        if (t == 0) {
            *error = MCUBES_ENONFINITE;
            *done = 1;
        }
        return false;
    }
    const IntProd inv_total = int_prod_recip(IntProd{(uint64_t)((t2 << z) >> 64), eT});
    // one bin per thread and round (one round up to 512 bins); loops, not
    // unrolled: the code runs once or twice and its fetch counts
    u128 W = 0;
#pragma unroll 1
    for (int i = 0; i * kRefineThreads < nb; ++i) {
        const int k = t + i * kRefineThreads;
        const u128 w = k < nb ? compressed_weight(smoothed3(s.C, k, nb), inv_total, alpha, s.logs) : (u128)0;
        const u128 c = u128_scan(w, W, s.wtot, &s.W[i]);
        if (k < nb) s.X[k] = (u128)(uint32_t)nb * c;
        __syncthreads();
        W = s.W[i];
    }
    if (W == 0) {
        if (t == 0) {
            *error = MCUBES_ENONFINITE;
            *done = 1;
        }
        return false;
    }
    DD e{1.0, 0.0}, e0{1.0, 0.0};  // the last round's edge, and the one before it
#pragma unroll 1
    for (int i = 0; i * kRefineThreads < nb; ++i) {
        const int k = t + i * kRefineThreads;
        e0 = e;
        e = k < nb - 1 ? rebin_edge(k + 1, nb, W, s.X, s.B, s.Blo) : DD{1.0, 0.0};
    }
    static_assert(kPerThread <= 2, "two rounds at most");
    __syncthreads();  // every thread is done with the old edges
    const int last = nb > kRefineThreads ? t + kRefineThreads : t;
    if (last < nb) {
        s.B[last] = e.hi;
        s.Blo[last] = e.lo;
    }
    if (nb > kRefineThreads) {
        s.B[t] = e0.hi;
        s.Blo[t] = e0.lo;
    }
    __syncthreads();
    return true;
}

}  // namespace refine_detail
}  // namespace mc
