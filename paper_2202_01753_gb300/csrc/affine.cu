// affine.cu -- host side of the fixed-point form of the FP64 affine families
// (FixFamily in mc_device.cuh): which integrands take it, and its constants.
// Scales and offsets are double-double, formed with error-free sums and
// FMA-based products, so that the fixed-point coordinates carry the rounding
// of the caller's parameters and nothing else.
#include <algorithm>
#include <cmath>

#include "fx_tables.h"
#include "mc_internal.h"

namespace mc {
namespace {

struct HD {
    double h = 0.0, l = 0.0;
};

HD two_sum(double a, double b)
{
    const double s = a + b, bb = s - a;
    return HD{s, (a - (s - bb)) + (b - bb)};
}
HD renorm(double h, double l)
{
    const double s = h + l;
    return HD{s, l - (s - h)};
}
HD add(HD a, HD b)
{
    const HD t = two_sum(a.h, b.h);
    return renorm(t.h, t.l + (a.l + b.l));
}
HD mul(HD a, HD b)
{
    const double p = a.h * b.h;
    return renorm(p, std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
HD div(HD a, HD b)
{
    const double q = a.h / b.h;
    const HD p = mul(HD{q, 0.0}, b);
    const HD r = add(a, HD{-p.h, -p.l});
    return renorm(q, (r.h + r.l) / b.h);
}

// 1 / (sqrt(2) v): s0 = 1 / (sqrt(2) v) in double, corrected by the residual of 2 (s0 v)^2 = 1
HD rsqrt2(double v)
{
    const double s0 = 1.0 / (std::sqrt(2.0) * v);
    const HD y = mul(HD{s0, 0.0}, HD{v, 0.0});
    HD r = mul(y, y);
    r = add(HD{1.0, 0.0}, HD{-2.0 * r.h, -2.0 * r.l});
    return renorm(s0, 0.5 * s0 * (r.h + r.l));
}

// Smallest b with v < 2^b (v > 0)
int bits_above(double v)
{
    int e;
    std::frexp(v, &e);
    return e;
}

long long to_fixed(HD v, int f)  // v 2^f rounded, |v| 2^f < 2^63
{
    const double h = std::ldexp(v.h, f), t = std::trunc(h);
    return (long long)t + std::llround((h - t) + std::ldexp(v.l, f));
}

}  // namespace

// The fixed-point form applies where every axis really is scaled (positive
// coefficients of a sane size) and the running quantity's unit is small enough
// for results no less exact than the double-precision form's: negative
// coefficients, flat axes, and wide or far boxes keep that form.  A sample's t
// is its cell's left edge rounded to nearest plus a product cut downwards; the
// running sums start with the half units that their terms lose on average, so
// that what is left of an estimate's error is below a double's last place
// (tests/test_affine_host.py; without them, 12 axes of |t| or of a corner
// family's slopes 300 put the mean off by 5-9e-16 relative).  An axis's whole
// range of t is below 2^(63 - f), so that a cell of any width has a product
// shift of at least 0.  Rules per family:
//   GAUSS    sum of the largest t^2 < 2^12 (unit of the exponent 2^-52), an axis's range < 2^6
//   C0       sum of the largest |t| < 2^9 (2^-54)
//   DISCONT  the same, and a cut inside the box at t >= 2^55 units (the threshold
//            and a sample's t are within three: less than the last place of
//            x, where the double-precision form puts it)
//   CORNER   largest sum < 2^12, and 1 + a.lo >= 2^56 units: the power d + 1
//            multiplies the sum's relative error (from 1, sums below 128)
//   PRODPEAK 1 + t^2 < 2^12 and the range < 2^6 per axis
//   OSC      at most 2^6 turns per axis
//   TABLE    every axis read by one table dimension at most
void affine_prepare(int id, const double* params, int d, const double* lo, const double* scale, long long g, int nb,
                    const TableDesc* tabs, FamParams* fp, CellMap* cm, double* jac0)
{
    fp->fix = 0;
    HD s[kDMax], a[kDMax], b[kDMax];
    HD fac{1.0, 0.0};      // f's constant factor
    double tmax[kDMax], sum = 0.0, sum2 = 0.0, most = 0.0, bmax = 0.0;
    HD start{0.0, 0.0};
    // TABLE: the table dimension that reads each axis (at most one)
    int knots[kDMax] = {0};
    HD tab_lo[kDMax], tab_s[kDMax];
    if (id == MCUBES_F_TABLE) {
        if (!tabs) return;
        for (int q = 0; q < fp->nf; ++q) {
            const TableDesc& T = tabs[fp->tid[q]];
            for (int h = 0; h < T.ndim; ++h) {
                const int j = h ? fp->tb[q] : fp->ta[q];
                if (knots[j]) return;  // read twice: two scales
                knots[j] = h ? T.n1 : T.n0;
                tab_lo[j] = HD{h ? T.lo1 : T.lo0, 0.0};
                tab_s[j] = div(HD{(double)(knots[j] - 1), 0.0}, h ? two_sum(T.hi1, -T.lo1) : two_sum(T.hi0, -T.lo0));
            }
        }
    }
    for (int j = 0; j < d; ++j) {
        double off = lo[j];  // a = s (lo - off')
        switch (id) {
        case MCUBES_F_GAUSS: s[j] = rsqrt2(std::fabs(params[1 + d + j])); break;
        case MCUBES_F_OSC: s[j] = mul(HD{params[1 + j], 0.0}, HD{fx::kInv2PiHi, fx::kInv2PiLo}); break;
        case MCUBES_F_CORNER:
        case MCUBES_F_DISCONT:
        case MCUBES_F_C0: s[j] = HD{params[j], 0.0}; break;
        case MCUBES_F_PRODPEAK: s[j] = HD{std::fabs(params[j]), 0.0}; break;
        case MCUBES_F_TABLE: s[j] = knots[j] ? tab_s[j] : div(HD{1.0, 0.0}, HD{scale[j], 0.0}); break;
        default: return;
        }
        if (!(s[j].h > 0x1p-40) || !(s[j].h < 0x1p40) || !(scale[j] > 0x1p-40) || !(scale[j] < 0x1p40)) return;
        b[j] = mul(s[j], HD{scale[j], 0.0});
        HD x0{0.0, 0.0};  // lo - o_j
        if (id == MCUBES_F_GAUSS) x0 = two_sum(off, -params[1 + j]);
        else if (id == MCUBES_F_OSC) x0 = HD{off, 0.0};
        else if (id == MCUBES_F_TABLE) x0 = knots[j] ? two_sum(off, -tab_lo[j].h) : HD{0.0, 0.0};
        else if (id == MCUBES_F_C0 || id == MCUBES_F_PRODPEAK) x0 = two_sum(off, -params[d + j]);
        if (!(std::fabs(x0.h) < 0x1p40)) return;
        a[j] = mul(s[j], x0);
        tmax[j] = std::max(std::fabs(a[j].h), std::fabs(a[j].h + b[j].h)) * (1.0 + 0x1p-40);
        sum += tmax[j];
        sum2 += tmax[j] * tmax[j];
        most = std::max(most, tmax[j]);
        bmax = std::max(bmax, b[j].h * (1.0 + 0x1p-40));
        if (id == MCUBES_F_CORNER) start = add(start, mul(s[j], HD{off, 0.0}));
        if (id == MCUBES_F_DISCONT && off != 0.0) return;  // exp(c.lo) would need an exponential of its own
        if (id == MCUBES_F_PRODPEAK) fac = mul(fac, mul(HD{params[j], 0.0}, HD{params[j], 0.0}));
    }
    int f = 0, fq = 0, fj[kDMax] = {0};
    uint64_t fu[kDMax + 1] = {0};
    switch (id) {
    case MCUBES_F_GAUSS: {
        if (!(params[0] > 0.0)) return;
        fac = HD{params[0], 0.0};
        int qb = std::max(2, bits_above(sum2));  // sum of t^2 < 2^qb, |t| < 2^(qb / 2)
        qb += qb & 1;
        f = std::min((126 - qb) / 2, 63 - bits_above(bmax));
        fq = 2 * f - 62;
        if (fq < 52) return;
        fu[kDMax] = (uint64_t)(d + 1) / 2;  // the d squares are cut, by half a last place each on average
        break;
    }
    case MCUBES_F_C0:
    case MCUBES_F_DISCONT: {
        const int qb = std::max(1, bits_above(std::max(sum, bmax)));
        if (qb > 9) return;
        f = fq = 63 - qb;
        fu[kDMax] = (uint64_t)d / 2;  // the d terms are cut, by half a unit each on average
        if (id == MCUBES_F_DISCONT) {
            if (!(sum < 700.0)) return;  // exp could overflow: the double-precision form reports it
            for (int j = 0; j < d; ++j) {  // x < w_j: t < c_j w_j (lo = 0)
                const double w = params[d + j];
                const HD t = mul(s[j], HD{w, 0.0});
                if (!(w > 0.0)) fu[j] = 0;                   // always out
                else if (w >= scale[j]) fu[j] = ~0ull;       // always in
                else if (std::ldexp(t.h, f) < 0x1p55) return;  // an axis flat beside the others: a cut as coarse as f
                else fu[j] = (uint64_t)to_fixed(t, f);
            }
        }
        break;
    }
    case MCUBES_F_CORNER: {
        start = add(start, HD{1.0, 0.0});
        const int qb = std::max(1, bits_above((start.h + sum) * (1.0 + 0x1p-40)));
        f = fq = 63 - qb;
        if (qb > 12 || !(std::ldexp(start.h, f) >= 0x1p56)) return;
        fu[kDMax] = (uint64_t)to_fixed(add(start, HD{std::ldexp(0.5 * d, -f), 0.0}), f);  // the terms are cut as C0's
        break;
    }
    case MCUBES_F_OSC: {
        const int tb = std::max(1, bits_above(bmax));
        if (tb > 6) return;
        f = fq = 63 - tb;
        const double u = params[0] - std::floor(params[0]);  // whole turns dropped
        fu[kDMax] = (uint64_t)std::llround(std::ldexp(u, f));
        break;
    }
    case MCUBES_F_PRODPEAK: {
        int qb = std::max(2, bits_above(1.0 + most * most));
        qb += qb & 1;
        f = std::min((126 - qb) / 2, 63 - bits_above(bmax));
        fq = 2 * f - 62;
        if (fq < 52) return;
        break;
    }
    case MCUBES_F_TABLE:
        // cell and fraction to f = 63 - (bits of the axis's range in knots): finer than u = x s - lo s in
        // double wherever the box is not much wider than the table
        for (int j = 0; j < d; ++j) {
            const int tb = std::max(1, bits_above(std::max(tmax[j], b[j].h * (1.0 + 0x1p-40))));
            fj[j] = std::min(62, 63 - tb);
            if (knots[j] && fj[j] < 53 - bits_above((double)knots[j]) + 2) return;
            if (fj[j] < 32) return;
        }
        break;
    default: return;
    }
    if (id != MCUBES_F_TABLE) std::fill(fj, fj + d, f);
    // J f0 = prod (nb scale_j) f0 = jac0 prod W_j with W_j = (b_j / g) (unit width), as the cells hold it
    HD j0 = fac, bg[kDMax];
    for (int j = 0; j < d; ++j) {
        bg[j] = div(b[j], HD{(double)g, 0.0});
        j0 = mul(j0, div(mul(HD{(double)nb, 0.0}, HD{scale[j], 0.0}), bg[j]));
    }
    if (!std::isnormal(j0.h) || !(j0.h > 0.0)) return;
    int lg = 0;  // ceil(log2 g)
    while ((1ll << lg) < g) ++lg;
    if (lg > 31) return;
    for (int j = 0; j < d; ++j) {
        if (id == MCUBES_F_OSC) a[j] = add(a[j], HD{-std::nearbyint(a[j].h), 0.0});
        cm->a[j] = to_fixed(a[j], fj[j]);
        cm->b[j] = (uint64_t)to_fixed(b[j], fj[j]);
        int e;  // b / g = m 2^(e - 63), m in [2^63, 2^64): rounded to 61 bits
        (void)std::frexp(bg[j].h, &e);
        const uint64_t v = (uint64_t)to_fixed(bg[j], 61 - e);  // 2^60..2^61
        const int z = __builtin_clzll(v);
        cm->bg_m[j] = v << z;
        cm->bg_e[j] = e + 2 - z;  // v 2^(e - 61) = m 2^(e - 61 - z)
    }
    cm->on = 1;
    fp->fix = 1;
    fp->fsg = 31 - lg;
    // t = M 2^(e - 63) num 2^-33 with M num 2^fsg = H 2^64: H 2^(e - 32 - fsg), moved to f fraction bits
    for (int j = 0; j < d; ++j) {
        fp->ftsh[j] = 32 + fp->fsg - fj[j];
        fp->ff[j] = fj[j];
    }
    fp->fq = fq;
    std::copy(fu, fu + kDMax + 1, fp->fu);
    *jac0 = j0.h + j0.l;
}

}  // namespace mc
