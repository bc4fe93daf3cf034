// vsample.cuh -- the sampling kernel (V-Sample / V-Sample-No-Adjust of
// Alg. 3 in the paper), instantiated once per integrand family by the
// vsample_<family>.cu translation units, and the device pieces it shares with
// the batched kernel (batch.cuh).
//
// Work layout.  A run of `lanes` consecutive threads of a warp owns one
// sub-cube; lane l of the run draws samples l, l + lanes, ... of it.  With
// lanes == 1 (the common case: p is 2 or 3 at 1e8-1e9 calls) a thread owns
// whole cubes and its cube moments need no communication; larger p spreads a
// cube over up to 32 lanes whose moments are merged by XOR shuffles.  Blocks
// walk the cube range with a grid stride.  The bin grid of all axes is staged
// in shared memory once per block as (left edge, nb * width) cells in the
// integration box's coordinates.  In adjusting iterations every sample adds
// F^2 to a per-block shared-memory histogram [d][nb], which the block adds
// to the pass's global histogram once at its end (one global reduction per
// non-empty bin; no per-sample global atomics).  Each block writes three
// double partials (sum of cube means, of their variances, of |means|) which
// the refinement launch reduces in fixed order.
#pragma once

#include <type_traits>

#include "mc_device.cuh"

namespace mc {

// The flat bin indices of a sample's axes are kept two per word, axis 2k in the
// low half of word k: as they are in double precision, as byte offsets into the
// histogram (4 times the index, below 2^16 as 12 x 1024 bins take 48 KB) in
// single precision.  An odd last axis leaves the top half kNoBin.
constexpr uint32_t kNoBin = 0xFFFFu;
template <class HT> constexpr uint32_t bin_unit() { return sizeof(HT) == 4 ? 4u : 1u; }

// Adds v to the bin at `idx` (bin_unit) of the shared-memory histogram at
// shared-window address `base` (a reduction: no value comes back, so nothing
// waits on it).
__device__ __forceinline__ void hist_add(uint32_t base, uint32_t idx, float v)
{
    asm volatile("red.shared.add.f32 [%0], %1;" ::"r"(base + idx), "f"(v));
}
__device__ __forceinline__ void hist_add(uint32_t base, uint32_t idx, double v)
{
    asm volatile("red.shared.add.f64 [%0], %1;" ::"r"(base + 8u * idx), "d"(v));
}

// Adds F2 to the sample's bin on every axis.  A shared-memory float addition
// is a compare-and-swap loop that repeats for the whole warp while lanes
// collide on one bin, so from three axes on the lanes start at different words
// and take the words in turn from there, NW = ceil(DC/2) words in all.  In
// double precision lane pair t (lanes 2t, 2t+1) starts at word (t mod NW), the
// odd lane of the pair with the two halves swapped, so each of the NW steps
// adds to 2 NW different axes' histograms, about 32 / (2 NW) lanes each,
// instead of two axes with 16 lanes each; in single precision lane l starts at
// word (l mod NW), no halves swapped (measured faster: corner8 17.57 -> 17.42
// ms, osc10 21.69 -> 21.00 ms per 1e9-call pass, against 17.65 and 21.33 with
// the swap).  The words are rotated by selects, a power of two at a time
// (static register indices).
template <int DC, int NB4, class HT>
__device__ __forceinline__ void hist_add_all(uint32_t hist_s, const uint32_t (&idx)[2 * NB4], HT F2)
{
    constexpr int NW = (DC + 1) / 2;
    constexpr bool kSwap = sizeof(HT) == 8;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t odd = kSwap ? (lane & 1u) : 0u;
    uint32_t w[NW];
#pragma unroll
    for (int t = 0; t < NW; ++t) w[t] = idx[t];
    if constexpr (NW >= 2) {
        const uint32_t rot = (kSwap ? (lane >> 1) : lane) % (uint32_t)NW;
#pragma unroll
        for (int sh = 1; sh < NW; sh <<= 1) {
            const bool on = (rot & (uint32_t)sh) != 0u;
            uint32_t u[NW];
#pragma unroll
            for (int t = 0; t < NW; ++t) u[t] = on ? w[(t + sh) % NW] : w[t];
#pragma unroll
            for (int t = 0; t < NW; ++t) w[t] = u[t];
        }
    }
#pragma unroll
    for (int t = 0; t < NW; ++t) {
        const uint32_t v = kSwap ? __funnelshift_l(w[t], w[t], odd << 4) : w[t];  // halves swapped on odd lanes
        const uint32_t lo = v & 0xFFFFu, hi = v >> 16;
        if (!(DC & 1) || !kSwap || lo != kNoBin) hist_add(hist_s, lo, F2);
        if (!(DC & 1) || hi != kNoBin) hist_add(hist_s, hi, F2);
    }
}

// The histogram adds of one sample: on all DC axes, or on axis 0 alone
// (m-Cubes1D, Sec. 3).
template <int DC, int NB4, class HT>
__device__ __forceinline__ void hist_add_one(uint32_t hist_s, const uint32_t (&idx)[2 * NB4], uint32_t hist_d, HT F2)
{
    if (hist_d == (uint32_t)DC) hist_add_all<DC, NB4, HT>(hist_s, idx, F2);
    else hist_add(hist_s, idx[0] & 0xFFFFu, F2);
}

// Packs axis j's bin into the index words.
template <int DC, class HT, int NW>
__device__ __forceinline__ void pack_bin(uint32_t (&idx)[NW], int j, uint32_t flat)
{
    const uint32_t v = flat * bin_unit<HT>();
    if (j & 1) idx[j >> 1] |= v << 16;
    else idx[j >> 1] = j == DC - 1 ? v | (kNoBin << 16) : v;
}

template <bool MIXED> struct Prec;
#ifndef MC_MIXED_CUBE_F64
#define MC_MIXED_CUBE_F64 0
#endif
// R: map and integrand; Cell: shared-memory map cell; H: histogram entry;
// S: a cube's shifted sums S1, S2 and its mean and variance.
template <> struct Prec<false> {
    using R = double;
    using Cell = double2;  // (x left edge, x width / g): x = left + (width/g)(g phi), J factor = (g nb)(width/g)
    using H = double;
    using S = double;
};
template <> struct Prec<true> {
    using R = float;
    using Cell = float2;   // (x left edge, nb * x width): x = left + (nb width)(phi/nb), J factor = nb width
    using H = float;
    using S = std::conditional_t<MC_MIXED_CUBE_F64 != 0, double, float>;
};

// Clears a block's histogram ([hist_d][nb]).
template <class HT>
__device__ __forceinline__ void clear_hist(HT* hist, uint32_t n)
{
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) hist[i] = HT(0);
}

// Stages the grid of all axes into shared-memory cells.  grid/grid_lo: [d][nb] double-double right
// edges (unit cube); lo/scale: the box's lower corner and hi - lo; g:
// sub-cubes per axis.
template <bool MIXED, bool FIX, class Arr>
__device__ __forceinline__ void stage_grid(typename Prec<MIXED>::Cell* cells, const double* grid,
                                           const double* grid_lo, const Arr& lo, const Arr& scale, const CellMap& cm,
                                           uint32_t d, uint32_t nb, uint32_t g)
{
    const double inv_g = 1.0 / (double)g;  // one division per thread, a multiply per cell
    for (uint32_t i = threadIdx.x; i < d * nb; i += blockDim.x) {
        const uint32_t j = i / nb, k = i - j * nb;
        const DD left = edge_left(grid + j * nb, grid_lo + j * nb, k);
        const DD right = edge_right(grid + j * nb, grid_lo + j * nb, k);
        if constexpr (MIXED) cells[i] = map_cell_f32(left, right, lo[j], scale[j], nb);
        else if constexpr (FIX) cells[i] = map_cell_fix(left, right, cm, (int)j);
        else cells[i] = map_cell_f64(left, right, lo[j], scale[j], inv_g);
    }
}

// The same staging from cells already built in global memory (by the
// refinement after each rebin, and at set-up): a copy, 16-byte words.
template <bool MIXED>
__device__ __forceinline__ void stage_cells(typename Prec<MIXED>::Cell* cells, const void* cells_g, uint32_t d,
                                            uint32_t nb)
{
    const uint32_t bytes = d * nb * (uint32_t)sizeof(typename Prec<MIXED>::Cell);
    const uint4* src = static_cast<const uint4*>(cells_g);
    uint4* dst = reinterpret_cast<uint4*>(cells);
    for (uint32_t i = threadIdx.x; i < bytes / 16; i += blockDim.x) dst[i] = src[i];
    if (threadIdx.x == 0 && (bytes & 15u))  // an odd number of 8-byte cells
        reinterpret_cast<uint2*>(cells)[bytes / 8 - 1] = static_cast<const uint2*>(cells_g)[bytes / 8 - 1];
}

// Whether a family runs its FP64 axes as a loop (Family::kRolled, default no).
template <class F, class = void> struct RolledAxes { static constexpr bool value = false; };
template <class F> struct RolledAxes<F, decltype((void)F::kRolled)> { static constexpr bool value = F::kRolled; };

// Only FP64 families with heavy per-axis work are rolled.  The mixed corner
// and oscillatory kernels, whose per-axis work is a few instructions with
// the axis's constants folded into constant-bank operands when unrolled,
// measured slower rolled (corner8 17.7 -> 21.1-23.1 ms, osc10 21.8 ->
// 26.6-30.2 ms per 1e9-call pass, blocks of 256 to 1024 threads).
template <int FAM, bool MIXED>
constexpr bool rolled_axes()
{
    if constexpr (MIXED) return false;
    else return RolledAxes<Family<FAM, double>>::value;
}

// sample_point for FP64 families with heavy per-axis work (a logarithm per
// axis): the same arithmetic with the axes as a loop that is not unrolled,
// so the per-axis code exists once instead of D times.  Unrolled, a six-axis
// sample is thousands of instructions, more than the SM's instruction
// caches keep close, and warps wait on instruction fetch.  In the loop the
// sub-cube digit of axis j is peeled off the cube index (one high multiply and
// one correction, as cube_digits; a second one cost cosmo6 0.9%),
// the Philox block of axes 4b..4b+3 is drawn at j = 4b and its words are
// rotated into place, and the flat bin indices are shifted into idx from the
// top, so that after the last axis axis j's index is field j (the layout
// sample_point leaves).  (Unrolled by two or three the loop measured slower:
// 9.55 and 9.69 ms against 8.80 ms per 1e8-call cosmo6 pass.)
template <int FAM, bool MIXED, int NB4, int D, class A>
__device__ __forceinline__ typename Prec<MIXED>::R
sample_point_rolled(const A& a, const typename Prec<MIXED>::Cell* cells, uint32_t c, uint32_t s,
                    const SampleRng<NB4>& rng, const PhiloxCube& pc, uint32_t (&idx)[2 * NB4])
{
    using R = typename Prec<MIXED>::R;
    using Fam = Family<FAM, R>;
    constexpr int NW = (D + 1) / 2;  // index words in use
    const uint32_t nb = a.nb;
    typename Fam::S fs;
    Fam::begin(fs);
    R jac = R(1);          // mixed: single-precision product of the widths
    IntProd jp{0, 0};      // FP64: the product in integer arithmetic, from jac0
    if constexpr (!MIXED) jp = int_prod_of(a.jac0);
    static_assert(D >= 3, "exact bin positions");
    uint32_t rest = c;
    uint4 r = make_uint4(0u, 0u, 0u, 0u);
    const PhiloxCube ps = philox_sample(pc, rng.shared_words(a, s, 0).w);
#pragma unroll
    for (int k = 0; k < 2 * NB4; ++k) idx[k] = 0u;
#pragma unroll 1
    for (int j = 0; j < D; ++j) {
        if ((j & 3) == 0) r = philox_block(a, rng.shared_words(a, s, (uint32_t)(j >> 2)), pc, ps);
        const uint32_t w = r.x;
        r = make_uint4(r.y, r.z, r.w, r.x);
        uint32_t q = __umulhi(rest, a.gmagic);
        uint32_t dig = rest - q * a.g;
        if (dig >= a.g) { ++q; dig -= a.g; }
        rest = q;
        const BinPos<true> bp = bin_pos<true>(w, dig * nb + 1u, nb, a.g, a.gmagic);
        const uint32_t flat = (uint32_t)j * nb + bp.k;
        const auto cell = cells[flat];
        R x;
        if constexpr (MIXED) {
            x = fmaf(cell.y, bin_phi_f32(bp, a.phi_scale_f), cell.x);   // (nb width)(phi/nb)
            jac *= cell.y;
        } else {
            x = fma(cell.y, bin_gphi_f64(bp), cell.x);                    // (width/g)(g phi)
            int_prod_mul(jp, cell.y);
        }
        Fam::add(fs, j, x, a.fam);
#pragma unroll
        for (int k = 0; k < NW - 1; ++k) idx[k] = __funnelshift_r(idx[k], idx[k + 1], 16);
        idx[NW - 1] = (idx[NW - 1] >> 16) | (flat << 16);
    }
    if constexpr (D & 1) {  // one field short of the top: move every field down once more
#pragma unroll
        for (int k = 0; k < NW - 1; ++k) idx[k] = __funnelshift_r(idx[k], idx[k + 1], 16);
        idx[NW - 1] = (idx[NW - 1] >> 16) | (kNoBin << 16);
    }
    if constexpr (!MIXED) return Fam::end_scaled(fs, a.fam, jp.m, jp.e);  // f J, rounded once
    else return Fam::end(fs, D, a.fam) * jac;
}

// The random words of a sample, four per Philox block.
template <int NB4, class A>
__device__ __forceinline__ void sample_words(const A& a, uint32_t s, const SampleRng<NB4>& rng, const PhiloxCube& pc,
                                             uint32_t (&w)[4 * NB4])
{
    PhiloxCube ps;
#pragma unroll
    for (int b = 0; b < NB4; ++b) {
        const uint4 u = rng.shared_words(a, s, (uint32_t)b);
        if (b == 0) ps = philox_sample(pc, u.w);
        const uint4 r = philox_block(a, u, pc, ps);
        w[4 * b + 0] = r.x;
        w[4 * b + 1] = r.y;
        w[4 * b + 2] = r.z;
        w[4 * b + 3] = r.w;
    }
}

// The same sample in the fixed-point form (FixFamily): the cell holds t at
// the left edge with f fraction bits and width / g as a double, of value M
// 2^(e - 63); g phi = num 2^-33, num < g 2^33 shifted to the top of 64 bits by
// fsg, so t = left + (M num 2^fsg) >> (64 + ftsh[j] - e).
template <int FAM, int NB4, int DC, class A>
__device__ __forceinline__ double sample_point_fix(const A& a, const double2* cells, uint32_t s,
                                                   const SampleRng<NB4>& rng, const PhiloxCube& pc,
                                                   const uint32_t (&nbc)[4 * NB4], uint32_t (&idx)[2 * NB4])
{
    using Fam = FixFamily<FAM>;
    const uint32_t nb = a.nb;
    uint32_t w[4 * NB4];
    sample_words<NB4>(a, s, rng, pc, w);
    typename Fam::S fs;
    Fam::begin(fs, a.fam);
    IntProd jp = int_prod_of(a.jac0);
#pragma unroll
    for (int j = 0; j < DC; ++j) {
        const auto bp = bin_pos<(DC >= 3)>(w[j], nbc[j], nb, a.g, a.gmagic);
        const uint32_t flat = (uint32_t)j * nb + bp.k;
        const double2 cell = cells[flat];
        const IntProd wd = int_prod_of(cell.y);
        const uint64_t num = bin_numerator(bp) << a.fam.fsg;
        const uint64_t H = __umul64hi(wd.m, num);
        const uint32_t sh = (uint32_t)(a.fam.ftsh[j] - wd.e);  // >= 0; beyond 63 for the narrowest bins
        const int64_t t = __double_as_longlong(cell.x) + (int64_t)(sh < 64u ? H >> sh : 0ull);
        jp = int_prod_mul2(jp, wd);
        Fam::add(fs, j, t, a.fam);
        pack_bin<DC, double>(idx, j, flat);
    }
    return Fam::template end<DC>(fs, a.fam, jp);
}

// One sample: random words -> exact bin position -> map -> integrand.
// Returns F = f(x) * J and leaves the flat histogram index of every axis in
// idx (16 bits each, two per word).  A provides d, nb, g, gmagic, jac0 ((g nb)^d), phi_scale_f
// (1/(g nb)), hist_d and fam, and round_key(a, r, i) its Philox keys.
template <int FAM, bool MIXED, int NB4, int DC, bool FIX, class A>
__device__ __forceinline__ typename Prec<MIXED>::R
sample_point(const A& a, const typename Prec<MIXED>::Cell* cells, uint32_t c, uint32_t s, const SampleRng<NB4>& rng,
             const PhiloxCube& pc, const uint32_t (&nbc)[4 * NB4], uint32_t (&idx)[2 * NB4])
{
    using R = typename Prec<MIXED>::R;
    using Fam = Family<FAM, R>;
    if constexpr (FIX) {
        return sample_point_fix<FAM, NB4, DC>(a, cells, s, rng, pc, nbc, idx);
    } else if constexpr (rolled_axes<FAM, MIXED>()) {
        return sample_point_rolled<FAM, MIXED, NB4, DC>(a, cells, c, s, rng, pc, idx);
    } else {
    constexpr uint32_t d = DC;
    const uint32_t nb = a.nb;
    uint32_t w[4 * NB4];
    sample_words<NB4>(a, s, rng, pc, w);
    typename Fam::S fs;
    Fam::begin(fs);
    R jac = R(1);                          // mixed: single-precision product of the widths
    IntProd jp{0, 0};                      // FP64: the product in integer arithmetic, from jac0
    if constexpr (!MIXED) jp = int_prod_of(a.jac0);
#pragma unroll
    for (int j = 0; j < DC; ++j) {
        {
            const auto bp = bin_pos<(DC >= 3)>(w[j], nbc[j], nb, a.g, a.gmagic);
            const uint32_t flat = (uint32_t)j * nb + bp.k;
            const auto cell = cells[flat];
            R x;
            if constexpr (MIXED) {
                const float phin = bin_phi_f32(bp, a.phi_scale_f);   // phi / nb
                x = fmaf(cell.y, phin, cell.x);
            } else {
                x = fma(cell.y, bin_gphi_f64(bp), cell.x);            // (width/g)(g phi)
            }
            if constexpr (MIXED) jac *= cell.y;
            else int_prod_mul(jp, cell.y);
            Fam::add(fs, j, x, a.fam);
            pack_bin<DC, typename Prec<MIXED>::H>(idx, j, flat);
        }
    }
    if constexpr (!MIXED) jac = int_prod_value(jp);
    return Fam::end(fs, d, a.fam) * jac;
    }
}

// Per-thread sums over the cubes a thread finishes: double, or a compensated
// single-precision pair in the mixed path (no FP64 work per cube).
struct CubeSums {
    double I = 0.0, V = 0.0, A = 0.0;
    DFloat fI{0.f, 0.f}, fV{0.f, 0.f}, fA{0.f, 0.f};
    __device__ double vI() const { return I + fI.value(); }
    __device__ double vV() const { return V + fV.value(); }
    __device__ double vA() const { return A + fA.value(); }
};

// x mod n with inv = floor((2^64 - 1)/n) from the host (a 64-bit division is
// ~100 dependent instructions, most of a small launch's set-up); n = 0: 0.
__device__ __forceinline__ uint64_t mod_by(uint64_t x, uint64_t n, uint64_t inv)
{
    if (n == 0) return 0;
    uint64_t r = x - __umul64hi(x, inv) * n;  // the quotient is short by 2 at most
    if (r >= n) r -= n;
    if (r >= n) r -= n;
    return r;
}

// nb times the digit of cube c on every axis (axis 0 fastest), plus 1 where bin
// positions are exact (bin_pos).
// One correction is enough: with gmagic = (2^32 - e)/g, 1 <= e <= g, the high
// word of rest gmagic is below rest/g by rest e/(g 2^32) < 1 at most.
template <int NB4, int DC, class A>
__device__ __forceinline__ void cube_digits(const A& a, uint32_t c, uint32_t (&nbc)[4 * NB4])
{
    uint32_t rest = c;
#pragma unroll
    for (int j = 0; j < DC; ++j) {
        uint32_t q = __umulhi(rest, a.gmagic);
        uint32_t r = rest - q * a.g;
        if (r >= a.g) { ++q; r -= a.g; }
        nbc[j] = r * a.nb + (DC >= 3 ? 1u : 0u);
        rest = q;
    }
}

// Adds the cube step's digits to a cube's, with carries (the last one drops:
// cube indices are taken modulo g^d): four instructions per axis against ten
// for splitting the new index by divisions.
template <int NB4, int DC, class A>
__device__ __forceinline__ void advance_digits(const A& a, bool wrap, uint32_t (&nbc)[4 * NB4])
{
    const uint32_t nb = a.nb, ng = nb * a.g, top = ng + (DC >= 3 ? 1u : 0u);
    uint32_t carry = 0;
#pragma unroll
    for (int j = 0; j < DC; ++j) {
        const uint32_t t = nbc[j] + cube_step_digit(a, wrap, j) + carry;  // < 2 ng <= 2^32
        const bool over = t >= top;
        nbc[j] = over ? t - ng : t;
        carry = over ? nb : 0u;
    }
}

// The digits of a segment's cube step into shared memory (cube_step_digits on
// the device, 32-bit: one thread, D high multiplies each).
template <class A>
__device__ __forceinline__ void cube_step_digits32(uint32_t step, uint32_t n, uint32_t m, uint32_t d, const A& a,
                                                   uint32_t* out)
{
    uint32_t u[2] = {step, step + (m - n)};
#pragma unroll 1
    for (uint32_t j = 0; j < d; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t q = __umulhi(u[h], a.gmagic);
            uint32_t rem = u[h] - q * a.g;
            if (rem >= a.g) { ++q; rem -= a.g; }
            out[h * kDMax + j] = rem * a.nb;
            u[h] = q;
        }
}

// Samples cubes [cube_lo, cube_lo + ncubes) of one integral.  The block takes
// groups of (blockDim / lanes) logical cube indices: group0, group0 + gstride,
// ...; logical index i is cube cube_lo + (i * perm_k mod ncubes), a bijection
// of the range (gcd(perm_k, ncubes) = 1) that gives the lanes of a warp
// cubes with unrelated digits on every axis, so that their samples spread
// over all bins instead of crowding the same few (fewer shared-memory atomic
// conflicts and bank conflicts).  From group to group a thread's cube moves by
// one fixed step (or that step less ncubes), whose digits cube_step_digit(a)
// gives.  Besides what sample_point reads, A provides inv_p = 1/p and
// inv_var_den = 1/(p (p-1)) (inv_p_f, inv_var_den_f in single precision) and
// want_abs (whether the sums of |cube mean| are needed: they are reported by
// the sampling-pass calls, not used by an iteration).
template <int FAM, bool MIXED, bool ADJ, int NB4, int DC, bool FIX, class A>
__device__ __forceinline__ void sample_cubes(const A& a, const typename Prec<MIXED>::Cell* cells,
                                             typename Prec<MIXED>::H* hist, uint64_t cube_lo, uint64_t ncubes,
                                             uint64_t perm_k, uint64_t perm_inv, uint64_t group0, uint64_t gstride,
                                             const SampleRng<NB4>& rng, uint32_t lanes, uint32_t p, CubeSums& acc)
{
    using R = typename Prec<MIXED>::R;
    using HT = typename Prec<MIXED>::H;
    constexpr bool kRolled = !FIX && rolled_axes<FAM, MIXED>();  // peels its digits itself
    const uint32_t hist_d = a.hist_d;  // axes with a histogram: d, or 1 (m-Cubes1D, Sec. 3)
    const uint32_t hist_s = (uint32_t)__cvta_generic_to_shared(hist);
    const uint32_t L = lanes;
    const uint32_t seg_lane = threadIdx.x & (L - 1u);
    const uint32_t cubes_per_group = blockDim.x / L;
    // 1/p and 1/(p (p-1)), rounded once on the host: a division here would be
    // recomputed inside the cube loop when registers run short
    using RS = typename Prec<MIXED>::S;  // per-cube shifted sums and moments
    RS inv_p, inv_var_den;
    if constexpr (sizeof(RS) == 4) {
        inv_p = a.inv_p_f;
        inv_var_den = a.inv_var_den_f;
    } else {
        inv_p = a.inv_p;
        inv_var_den = a.inv_var_den;
    }
    const uint64_t first = group0 * cubes_per_group + threadIdx.x / L;
    const uint64_t stride = gstride * cubes_per_group;
    // physical offset of `first`, and its step from group to group (below 2^32, as the cube counter)
    uint32_t off = (uint32_t)mod_by(mod_by(first, ncubes, perm_inv) * perm_k, ncubes, perm_inv);
    const uint32_t step = (uint32_t)mod_by(mod_by(stride, ncubes, perm_inv) * perm_k, ncubes, perm_inv);
    uint32_t nbc[4 * NB4];
    if constexpr (!kRolled) cube_digits<NB4, DC>(a, (uint32_t)cube_lo + off, nbc);
    auto advance = [&] {  // to this thread's cube of the next group
        off += step;
        const bool wrap = off < step || off >= (uint32_t)ncubes;
        if (wrap) off -= (uint32_t)ncubes;
        if constexpr (!kRolled) advance_digits<NB4, DC>(a, wrap, nbc);
    };
    if (L == 1u && p == 2u) {
        // two samples per cube, one thread each (every 1e8-call geometry)
        for (uint64_t ci = first; ci < ncubes; ci += stride) {
            const uint32_t c = (uint32_t)cube_lo + off;
            const PhiloxCube pc = philox_cube(a, rng.it, c);
            R K = R(0), F = R(0);
            // Both samples unrolled in single precision (corner8 14.85 -> 14.54 ms
            // a pass); in double precision within 1% either way, so a loop.
            // Against the loop, passes of 8e6-3.4e7 samples: corner 0.93-1.00 of
            // its time, gauss 0.90-0.99 up to d = 9 and 1.00-1.02 beyond, osc
            // 0.93-1.04 adjusting and 0.95-1.10 without (slower from d = 6 on,
            // where it spills); batches 0.97-1.03.
#pragma unroll (MIXED ? 2 : 1)
            for (uint32_t s = 0; s < 2u; ++s) {
                uint32_t idx[2 * NB4];
                K = F;
                F = sample_point<FAM, MIXED, NB4, DC, FIX>(a, cells, c, s, rng, pc, nbc, idx);
                if constexpr (ADJ) hist_add_one<DC, NB4>(hist_s, idx, hist_d, (HT)(F * F));
            }
            advance();
            // UpdateVariance (Alg. 3): cube mean and the variance of that mean;
            // S1 = z, S2 = z^2 and the variance (z^2 - z^2/2)/2 is exactly z^2/4:
            // the z^2 are summed and the sum scaled once after the loop (exact)
            const RS S1 = (RS)F - (RS)K;
            const RS mean = (RS)K + S1 * RS(0.5);
            if constexpr (sizeof(RS) == 4) {
                acc.fI.add(mean);
                acc.fV.add(S1 * S1);
                if (a.want_abs) acc.fA.add(fabsf(mean));
            } else {
                acc.I += mean;
                acc.V = fma(S1, S1, acc.V);  // one FMA for the z^2
                if (a.want_abs) acc.A += fabs(mean);
            }
        }
        acc.V *= 0.25;
        acc.fV.hi *= 0.25f;
        acc.fV.lo *= 0.25f;
        return;
    }
    for (uint64_t base = group0 * cubes_per_group; base < ncubes; base += stride) {
        const bool valid = base + threadIdx.x / L < ncubes;
        const uint32_t c = (uint32_t)cube_lo + off;
        // this lane's samples of the cube, shifted by its first value
        R K = R(0);
        RS S1 = RS(0), S2 = RS(0);
        uint32_t n = 0;
        if (valid) {
            const PhiloxCube pc = philox_cube(a, rng.it, c);
            for (uint32_t s = seg_lane; s < p; s += L) {
                uint32_t idx[2 * NB4];
                const R F = sample_point<FAM, MIXED, NB4, DC, FIX>(a, cells, c, s, rng, pc, nbc, idx);
                if (n == 0) {
                    K = F;  // the shift: its own term is zero
                } else if (n == 1) {
                    S1 = (RS)F - (RS)K;  // S2 = S1^2 is formed when needed
                } else {
                    if (n == 2) S2 = S1 * S1;
                    const RS z = (RS)F - (RS)K;
                    S1 += z;
                    S2 += z * z;
                }
                ++n;
                if constexpr (ADJ) {
                    hist_add_one<DC, NB4>(hist_s, idx, hist_d, (HT)(F * F));
                }
            }
        }
        advance();
        if (L == 1u) {
            if (valid) {  // UpdateVariance (Alg. 3): cube mean and the variance of that mean
                const RS mean = (RS)K + S1 * inv_p;
                const RS var = (S2 - S1 * S1 * inv_p) * inv_var_den;
                if constexpr (sizeof(RS) == 4) {
                    acc.fI.add(mean);
                    acc.fV.add(var);
                    if (a.want_abs) acc.fA.add(fabsf(mean));
                } else {
                    acc.I += mean;
                    acc.V += var;
                    if (a.want_abs) acc.A += fabs(mean);
                }
            }
        } else {
            if (n == 2) S2 = S1 * S1;
            // the cube's lanes re-base their sums on the shift of its first lane
            // (S1 += n dK, S2 += dK (2 S1 + n dK), dK = K_l - K_0; a lane without
            // samples adds nothing) and add them with XOR shuffles: no division
            const double K0 = __shfl_sync(0xffffffffu, (double)K, (int)((threadIdx.x & 31u) & ~(L - 1u)));
            const double dK = (double)K - K0, cnt = (double)n;
            double s1 = (double)S1, s2 = (double)S2;
            s2 = fma(dK, fma(cnt, dK, 2.0 * s1), s2);
            s1 = fma(cnt, dK, s1);
            for (uint32_t o = 1; o < L; o <<= 1) {
                s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            }
            if (valid && seg_lane == 0) {
                const double mean = K0 + s1 * a.inv_p;
                acc.I += mean;
                acc.V += (s2 - s1 * s1 * a.inv_p) * a.inv_var_den;
                if (a.want_abs) acc.A += fabs(mean);
            }
        }
    }
}

// Cube-split sampling, for geometries with few cubes and many samples each
// (e.g. 64 cubes of 16384 samples): `split` blocks share one cube, block k
// drawing samples [k q, min(p, (k+1) q)), q = ceil(p / split), spread over
// its threads.  Every thread keeps sums of its samples shifted by its first
// value K_t; they are re-based on thread 0's shift K (S1 += n dK,
// S2 += dK (2 S1 + n dK), dK = K_t - K: no division) and summed in a fixed
// order; the block writes (K, S1, S2) to out[0..2] and the refinement
// combines a cube's blocks the same way.
template <int FAM, bool MIXED, bool ADJ, int NB4, int DC, bool FIX, class A>
__device__ __forceinline__ void sample_cube_slice(const A& a, const typename Prec<MIXED>::Cell* cells,
                                                  typename Prec<MIXED>::H* hist, uint64_t cube, uint32_t k,
                                                  uint32_t split, const SampleRng<NB4>& rng, uint32_t p,
                                                  double (*red)[kVsThreadsMax / 32], double* out)
{
    using R = typename Prec<MIXED>::R;
    using HT = typename Prec<MIXED>::H;
    const uint32_t hist_d = a.hist_d;
    const uint32_t q = (p + split - 1) / split;
    const uint32_t s_lo = k * q, s_hi = min(p, s_lo + q);
    const uint32_t hist_s = (uint32_t)__cvta_generic_to_shared(hist);
    const uint32_t c = (uint32_t)cube;
    uint32_t nbc[4 * NB4];
    cube_digits<NB4, DC>(a, c, nbc);
    const PhiloxCube pc = philox_cube(a, rng.it, c);
    R K = R(0), S1 = R(0), S2 = R(0);
    uint32_t n = 0;
    for (uint32_t s = s_lo + threadIdx.x; s < s_hi; s += blockDim.x) {
        uint32_t idx[2 * NB4];
        const R F = sample_point<FAM, MIXED, NB4, DC, FIX>(a, cells, c, s, rng, pc, nbc, idx);
        if (n == 0) {
            K = F;  // the shift: its own term is zero
        } else {
            const R z = F - K;
            S1 += z;
            S2 += z * z;
        }
        ++n;
        if constexpr (ADJ) {
            hist_add_one<DC, NB4>(hist_s, idx, hist_d, (HT)(F * F));
        }
    }
    // re-base on thread 0's shift (every thread has a sample: q >= blockDim;
    // a thread without one adds nothing)
    __syncthreads();
    if (threadIdx.x == 0) red[0][0] = (double)K;
    __syncthreads();
    const double K0 = red[0][0];
    __syncthreads();
    const double dK = (double)K - K0, cnt = (double)n;
    double s1 = (double)S1, s2 = (double)S2;
    s2 = fma(dK, fma(cnt, dK, 2.0 * s1), s2);
    s1 = fma(cnt, dK, s1);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        s1 += __shfl_down_sync(0xffffffffu, s1, off);
        s2 += __shfl_down_sync(0xffffffffu, s2, off);
    }
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[1][warp] = s1;
        red[2][warp] = s2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double b1 = 0.0, b2 = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            b1 += red[1][w];
            b2 += red[2][w];
        }
        out[0] = K0;
        out[1] = b1;
        out[2] = b2;
    }
}

// Fixed-order block sum of the per-thread sums; out[2] (the sum of |cube
// mean|) only where it is wanted.  A block's FP64 additions take the SM's
// pipe 16 cycles each whatever the number of active lanes, and 32 resident
// warps with three five-step shuffle trees spent ~8000 cycles here: lanes
// 0-15 and 16-31 first swap halves and then sum one quantity each, five
// additions for both, and the warps' sums are added the same way.
template <bool MIXED, int NW>
__device__ __forceinline__ void block_write_sums(const CubeSums& acc, bool want_abs, double (*red)[NW], double* out)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool up = lane >= 16;
    const double vI = MIXED ? acc.vI() : acc.I, vV = MIXED ? acc.vV() : acc.V;
    double v = (up ? vV : vI) + __shfl_xor_sync(0xffffffffu, up ? vI : vV, 16);
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((lane & 15) == 0) red[up][warp] = v;
    if (want_abs) {
        double a = MIXED ? acc.vA() : acc.A;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        if (lane == 0) red[2][warp] = a;
    }
    __syncthreads();
    if (warp != 0) return;
    if (!want_abs && lane == 0) out[2] = 0.0;
    const int nw = (int)(blockDim.x >> 5);
    const int w = lane & 15;
    v = w < nw ? red[up][w] : 0.0;
    if (nw > 16 && w + 16 < nw) v += red[up][w + 16];
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((lane & 15) == 0) out[up] = v;
    if (want_abs) {
        double a = lane < nw ? red[2][lane] : 0.0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        if (lane == 0) out[2] = a;
    }
}

// Resident blocks per SM the register allocation is bounded for: three (80
// registers, 24 warps) — measured against two: osc10 mixed +10% despite 132
// bytes of spills, cosmo6 FP64 +4% and gauss3 FP64 +9% with none — except
// for the table integrands in FP64, whose spills and larger table footprint
// in L1/L2 cost a third (two blocks; table6 at three: 16.6 ms per 1e8 calls
// against 10.0 ms).  Four blocks (64 registers) for the mixed kernels up to
// d = 8 measured slower too (corner8: 23.3 ms per 1e9 calls against 21.3);
// for d <= 4 four blocks fit in 64 registers without spills (gauss3 in
// cube-split mode lives on resident warps).  That is the single-integral
// kernels, of which mixed ones spill from d = 6 on (up to 180 bytes) and FP64
// table ones at d = 11 and 12.  The batched kernels hold two to four copies of
// the sample and spill under the same bounds, up to 750 bytes in single and
// 1.1 KB in double precision; batches of 16 and 64 integrals of one class, every
// family and d, still take 0.35-0.99 of the time that one copy of the earlier
// sampling loop without spills took.
template <int FAM, bool MIXED, int NB4>
constexpr int vsample_min_blocks() { return (FAM == MCUBES_F_TABLE && !MIXED) ? 2 : (NB4 == 1 ? 4 : 3); }

// The same for the single-integral kernel, whose block size can differ
// (vsample_threads): blocks that fill the register file at its size.
template <int FAM, bool MIXED, int D>
constexpr int vsample_kernel_min_blocks()
{
    return vsample_threads(FAM, MIXED, D) == kVsThreads ? vsample_min_blocks<FAM, MIXED, (D + 3) / 4>()
                                                        : 1024 / vsample_threads(FAM, MIXED, D);
}

__device__ __forceinline__ int2 ld_volatile_int2(const void* p)
{
    int2 v;
    asm volatile("ld.volatile.global.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}

// One instantiation per dimension D: with the axis count a compile-time
// constant every per-axis loop is unrolled without guards and the families'
// dimension-dependent code (the corner family's power) folds (corner8: 21.4
// -> 17.7 ms per 1e9-call launch against a runtime count).
template <int FAM, bool MIXED, bool ADJ, int D, bool FIX>
__global__ void __launch_bounds__(vsample_threads(FAM, MIXED, D), vsample_kernel_min_blocks<FAM, MIXED, D>())
vsample_kernel(const __grid_constant__ VsArgs a)
{
    constexpr int NB4 = (D + 3) / 4;  // Philox blocks per sample
    if constexpr (FAM == MCUBES_F_COSMO6 && D != 6) {
        return;  // six axes only: never launched
    } else {
    using Cell = typename Prec<MIXED>::Cell;
    using HT = typename Prec<MIXED>::H;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[3][kVsThreadsMax / 32];
    __shared__ uint4 philox_tab[kPhiloxTab * NB4];  // with red at most 960 bytes (mcubes_setup allows 1 KB)

    constexpr uint32_t d = D;
    const uint32_t nb = a.nb;
    // single precision: the histogram first, its address a constant of the
    // additions (corner8 15.32 -> 14.82 ms per 1e9-call pass with the bins kept
    // as byte offsets); double precision: the cells first
    HT* hist = reinterpret_cast<HT*>(smem + (MIXED ? 0u : cell_bytes(false) * d * nb));
    Cell* cells = reinterpret_cast<Cell*>(smem + (MIXED && ADJ ? hist_smem_bytes(true, a.hist_d * nb) : 0u));
    if constexpr (ADJ) clear_hist(hist, a.hist_d * nb);
    if constexpr (!MIXED) fx::warm_tables<FAM>();
    grid_dependency_wait();  // the refinement before this pass (launch_dependent)
    uint32_t it = a.it_fixed;
    if (a.st != nullptr) {
        // iteration index and flag by one load
        const int2 v = ld_volatile_int2(&a.st->it);
        const int done = v.y;
        if (blockIdx.x == 0 && threadIdx.x == 0) a.st->active = done ? 0 : 1;
        if (done) return;
        it = (uint32_t)v.x;
    }

    fill_philox_table<NB4>(philox_tab, a, it);
    const SampleRng<NB4> rng{it, philox_tab};
    if (a.cells_g) stage_cells<MIXED>(cells, a.cells_g, d, nb);
    else stage_grid<MIXED, FIX>(cells, a.grid, a.grid_lo, a.lo, a.scale, a.cm, d, nb, a.g);
    __syncthreads();

    if (a.split > 1) {
        sample_cube_slice<FAM, MIXED, ADJ, NB4, D, FIX>(a, cells, hist, a.cube_begin + blockIdx.x / a.split,
                                                blockIdx.x % a.split, a.split, rng, a.p, red,
                                                a.part + 3 * (size_t)blockIdx.x);
    } else {
        CubeSums acc;
        sample_cubes<FAM, MIXED, ADJ, NB4, D, FIX>(a, cells, hist, a.cube_begin, a.cube_end - a.cube_begin, a.perm_k, a.perm_inv,
                                           blockIdx.x, gridDim.x, rng, a.lanes, a.p, acc);
        grid_dependents_launch();  // the refinement's blocks may take their places
        block_write_sums<MIXED>(acc, a.want_abs != 0, red, a.part + 3 * (size_t)blockIdx.x);
    }
    if constexpr (ADJ) {
        // (every warp has passed a barrier since its last histogram addition)
        // the block's histogram goes into the pass's accumulator once: one
        // global reduction per non-empty bin (no per-sample global atomics)
        for (uint32_t i = threadIdx.x; i < a.hist_d * nb; i += blockDim.x) {
            const double v = (double)hist[i];
            if (v != 0.0) atomicAdd(a.hist_acc + i, v);
        }
    }
    }
}

template <int FAM, bool MIXED, bool ADJ, bool FIX>
inline auto vsample_kernel_d(int d)
{
    using K = void (*)(VsArgs);
    switch (d) {
    case 1: return (K)vsample_kernel<FAM, MIXED, ADJ, 1, FIX>;
    case 2: return (K)vsample_kernel<FAM, MIXED, ADJ, 2, FIX>;
    case 3: return (K)vsample_kernel<FAM, MIXED, ADJ, 3, FIX>;
    case 4: return (K)vsample_kernel<FAM, MIXED, ADJ, 4, FIX>;
    case 5: return (K)vsample_kernel<FAM, MIXED, ADJ, 5, FIX>;
    case 6: return (K)vsample_kernel<FAM, MIXED, ADJ, 6, FIX>;
    case 7: return (K)vsample_kernel<FAM, MIXED, ADJ, 7, FIX>;
    case 8: return (K)vsample_kernel<FAM, MIXED, ADJ, 8, FIX>;
    case 9: return (K)vsample_kernel<FAM, MIXED, ADJ, 9, FIX>;
    case 10: return (K)vsample_kernel<FAM, MIXED, ADJ, 10, FIX>;
    case 11: return (K)vsample_kernel<FAM, MIXED, ADJ, 11, FIX>;
    default: return (K)vsample_kernel<FAM, MIXED, ADJ, 12, FIX>;  // d is checked to be 1..12
    }
}

// The kernel of a launch; fix: its fixed-point form (families that have one).
template <int FAM>
inline auto vsample_kernel_ptr(bool mixed, bool adjust, bool fix, int d)
{
    if (mixed) return adjust ? vsample_kernel_d<FAM, true, true, false>(d) : vsample_kernel_d<FAM, true, false, false>(d);
    if constexpr (FixFamily<FAM>::kHas)
        if (fix) return adjust ? vsample_kernel_d<FAM, false, true, true>(d) : vsample_kernel_d<FAM, false, false, true>(d);
    return adjust ? vsample_kernel_d<FAM, false, true, false>(d) : vsample_kernel_d<FAM, false, false, false>(d);
}

template <int FAM>
cudaError_t launch_vsample_family(bool mixed, bool adjust, const VsArgs& args, int grid, size_t smem,
                                  cudaStream_t s)
{
    VsArgs a = args;
    const uint64_t n = a.cube_end - a.cube_begin;
    if (n > 0 && a.split == 1) {  // the cube step of this launch's groups
        const uint64_t group = (uint64_t)grid * (vsample_threads(FAM, mixed, (int)a.d) / a.lanes);
        uint64_t m = 1;
        for (uint32_t j = 0; j < a.d; ++j) m *= a.g;
        cube_step_digits((group % n) * a.perm_k % n, n, m, a.d, a.g, a.nb, a.cube_step[0], a.cube_step[1]);
    }
    auto k = vsample_kernel_ptr<FAM>(mixed, adjust, a.fam.fix != 0, (int)a.d);
    cudaError_t e = raise_smem_limit((const void*)k, smem);
    if (e != cudaSuccess) return e;
    return launch_dependent(k, grid, vsample_threads(FAM, mixed, (int)a.d), smem, s, a);
}

template <int FAM>
cudaError_t occupancy_family(bool mixed, bool adjust, bool fix, int d, size_t smem, int* blocks)
{
    auto k = vsample_kernel_ptr<FAM>(mixed, adjust, fix, d);
    cudaError_t e = raise_smem_limit((const void*)k, smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, k, vsample_threads(FAM, mixed, d), smem);
}

}  // namespace mc

#define MC_INSTANTIATE_FAMILY(FAM, NAME)                                                          \
    namespace mc {                                                                                \
    cudaError_t launch_vsample_##NAME(bool mixed, bool adjust, const VsArgs& a, int grid,         \
                                      size_t smem, cudaStream_t s)                                \
    {                                                                                             \
        return launch_vsample_family<FAM>(mixed, adjust, a, grid, smem, s);                       \
    }                                                                                             \
    cudaError_t occupancy_##NAME(bool mixed, bool adjust, bool fix, int d, size_t smem, int* blocks) \
    {                                                                                             \
        return occupancy_family<FAM>(mixed, adjust, fix, d, smem, blocks);                             \
    }                                                                                             \
    }
