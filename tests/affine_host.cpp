// Host build of the FP64 affine families: affine_prepare (csrc/affine.cu) and
// the sampling code of both forms (csrc/vsample.cuh) with plain C++ stand-ins for
// the device intrinsics, against the same sums in long double from the exact
// rational position of each sample.
//
// Reads lines "<op> <family> <d> <nb> <g> <n> <power> <axis> <offset> params[np] lo[d] hi[d]"
// (np by family); edges ((k + 1) / nb)^power.  Ops:
//   fix   prints whether the fixed-point form is taken, and its fraction bits
//   mean  over n samples in random cubes: prints fix and the relative error of
//         the mean of F in the form taken and in the double-precision form
//   cut   DISCONT: for each of n samples, axis's cut is put offset units of the
//         last place above or below the sample's x; prints how many samples fall on
//         the wrong side in the form that affine_prepare then takes
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include <sstream>
#include <string>
#include <vector>
#include "mc_internal.h"
using std::max;
using std::min;
struct Idx { unsigned x, y, z; };
static Idx threadIdx_, blockIdx_, blockDim_, gridDim_;
#define threadIdx threadIdx_
#define blockIdx blockIdx_
#define blockDim blockDim_
#define gridDim gridDim_
#undef __shared__
#define __shared__
#define __noinline__
#undef __launch_bounds__
#define __launch_bounds__(...)
static inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
template <class T> static inline T __ldg(const T* p) { return *p; }
static inline long long __double_as_longlong(double d) { long long x; std::memcpy(&x, &d, 8); return x; }
static inline double __longlong_as_double(long long x) { double d; std::memcpy(&d, &x, 8); return d; }
static inline float __uint2float_rn(uint32_t u) { return (float)u; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, uint32_t s) { s &= 31; return s ? (hi << s) | (lo >> (32 - s)) : hi; }
static inline uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t s) { s &= 31; return s ? (lo >> s) | (hi << (32 - s)) : lo; }
static inline void __syncthreads() {}
static inline size_t __cvta_generic_to_shared(const void* p) { return (size_t)p; }
template <class T> static inline T __shfl_sync(unsigned, T v, int) { return v; }
template <class T> static inline T __shfl_xor_sync(unsigned, T v, int) { return v; }
template <class T> static inline T __shfl_down_sync(unsigned, T v, int) { return v; }
static inline void atomicAdd(double* p, double v) { *p += v; }
static inline double __ddiv_rn(double a, double b) { return a / b; }
#include "vsample.cuh"
#include "affine.cu"

using namespace mc;
typedef long double LD;

struct Prob {
    int fam, d, nb, g;
    std::vector<double> par, lo, hi;
    VsArgs a;
    std::vector<double> edges;
    std::vector<double2> fixed, dbl;

    bool prepare()
    {
        std::memset(&a, 0, sizeof a);
        a.d = d; a.nb = nb; a.g = g; a.gmagic = 0xFFFFFFFFu / (uint32_t)g;
        for (int r = 0; r < 10; ++r) { a.rk[r][0] = 12345u + r * 0x9E3779B9u; a.rk[r][1] = 678u + r * 0xBB67AE85u; }
        FamParams& f = a.fam;
        const double* p = par.data();
        for (int j = 0; j < d; ++j) {
            a.lo[j] = lo[j];
            a.scale[j] = hi[j] - lo[j];
            switch (fam) {
            case MCUBES_F_GAUSS: f.c[0] = p[0]; f.c[1 + j] = p[1 + j]; f.c[13 + j] = 1.0 / (2.0 * p[1 + d + j] * p[1 + d + j]); break;
            case MCUBES_F_OSC: f.c[0] = 2.0 * M_PI * p[0]; f.c[1 + j] = p[1 + j]; break;
            case MCUBES_F_PRODPEAK: f.c[j] = 1.0 / (p[j] * p[j]); f.c[12 + j] = p[d + j]; break;
            case MCUBES_F_CORNER: f.c[j] = p[j]; break;
            default: f.c[j] = p[j]; f.c[12 + j] = p[d + j];
            }
        }
        a.jac0 = std::pow((double)nb * g, d);
        double jac0 = a.jac0;
        affine_prepare(fam, p, d, a.lo, a.scale, g, nb, nullptr, &f, &a.cm, &jac0);
        fixed.assign((size_t)d * nb, double2{0, 0});
        dbl = fixed;
        for (int j = 0; j < d; ++j)
            for (int k = 0; k < nb; ++k) {
                const DD l{k ? edges[k - 1] : 0.0, 0.0}, r{edges[k], 0.0};
                dbl[(size_t)j * nb + k] = map_cell_f64(l, r, a.lo[j], a.scale[j], 1.0 / g);
                if (f.fix) fixed[(size_t)j * nb + k] = map_cell_fix(l, r, a.cm, j);
            }
        if (f.fix) std::swap(jac0, a.jac0);
        jac_dbl = f.fix ? jac0 : a.jac0;
        return f.fix != 0;
    }
    double jac_dbl;
};

// One sample: F in the form taken and in the double-precision form, and the exact x and Jacobian
struct Out { double fix, dbl; LD x[kDMax], jac; };
template <int FAM, int D> Out sample(const Prob& P, uint32_t c, uint32_t s)
{
    constexpr int NB4 = (D + 3) / 4;
    Out o;
    const VsArgs& a = P.a;
    const SampleRng<NB4> rng{3u, nullptr};
    const PhiloxCube pc = philox_cube(a, 3u, c);
    uint32_t nbc[4 * NB4], idx[2 * NB4], w[4 * NB4];
    cube_digits<NB4, D>(a, c, nbc);
    s += kPhiloxTab;
    VsArgs b = a;
    b.jac0 = P.jac_dbl;
    o.dbl = sample_point<FAM, false, NB4, D, false>(b, P.dbl.data(), c, s, rng, pc, nbc, idx);
    o.fix = a.fam.fix ? sample_point<FAM, false, NB4, D, true>(a, P.fixed.data(), c, s, rng, pc, nbc, idx) : o.dbl;
    sample_words<NB4>(a, s, rng, pc, w);
    o.jac = 1;
    uint32_t rest = c;
    for (int j = 0; j < D; ++j) {
        const uint64_t digit = rest % (uint32_t)P.g;
        rest /= (uint32_t)P.g;
        const unsigned __int128 num = (unsigned __int128)((digit << 33) + 2ull * w[j] + 1) * (unsigned)P.nb, den = (unsigned __int128)P.g << 33;
        const int k = (int)(num / den);
        const LD phi = (LD)(uint64_t)(num % den) / (LD)(uint64_t)den;
        const LD l = k ? P.edges[k - 1] : 0.0, r = P.edges[k];
        o.x[j] = (LD)a.lo[j] + (LD)a.scale[j] * (l + (r - l) * phi);
        o.jac *= (LD)P.nb * (LD)a.scale[j] * (r - l);
    }
    return o;
}

static LD exact(const Prob& P, const Out& o)
{
    const int d = P.d;
    const double* p = P.par.data();
    LD t = 0, f = 1;
    for (int j = 0; j < d; ++j) {
        const LD x = o.x[j];
        switch (P.fam) {
        case MCUBES_F_GAUSS: { const LD z = (x - p[1 + j]) / p[1 + d + j]; t += z * z / 2; break; }
        case MCUBES_F_OSC: t += (LD)p[1 + j] * x; break;
        case MCUBES_F_PRODPEAK: { const LD z = x - p[d + j]; f /= 1 / ((LD)p[j] * p[j]) + z * z; break; }
        case MCUBES_F_CORNER: t += (LD)p[j] * x; break;
        case MCUBES_F_C0: t += (LD)p[j] * std::fabs(x - (LD)p[d + j]); break;
        default: t += (LD)p[j] * x; if (!(x < (LD)p[d + j])) f = 0;
        }
    }
    switch (P.fam) {
    case MCUBES_F_GAUSS: f = (LD)p[0] * std::exp(-t); break;
    case MCUBES_F_OSC: f = std::cos(2 * std::acos((LD)-1) * (LD)p[0] + t); break;
    case MCUBES_F_PRODPEAK: break;
    case MCUBES_F_CORNER: f = std::pow(1 + t, (LD)-(d + 1)); break;
    case MCUBES_F_C0: f = std::exp(-t); break;
    default: f *= std::exp(t);
    }
    return f * o.jac;
}

template <int FAM> Out sample_d(const Prob& P, uint32_t c, uint32_t s)
{
    switch (P.d) {
    case 1: return sample<FAM, 1>(P, c, s);
    case 2: return sample<FAM, 2>(P, c, s);
    case 3: return sample<FAM, 3>(P, c, s);
    case 6: return sample<FAM, 6>(P, c, s);
    case 11: return sample<FAM, 11>(P, c, s);
    default: return sample<FAM, 12>(P, c, s);
    }
}
static Out sample_f(const Prob& P, uint32_t c, uint32_t s)
{
    switch (P.fam) {
    case MCUBES_F_GAUSS: return sample_d<MCUBES_F_GAUSS>(P, c, s);
    case MCUBES_F_OSC: return sample_d<MCUBES_F_OSC>(P, c, s);
    case MCUBES_F_PRODPEAK: return sample_d<MCUBES_F_PRODPEAK>(P, c, s);
    case MCUBES_F_CORNER: return sample_d<MCUBES_F_CORNER>(P, c, s);
    case MCUBES_F_C0: return sample_d<MCUBES_F_C0>(P, c, s);
    default: return sample_d<MCUBES_F_DISCONT>(P, c, s);
    }
}

int main()
{
    char buf[8192];
    while (std::fgets(buf, sizeof buf, stdin)) {
        std::istringstream in(buf);
        std::string op;
        Prob P;
        int n, axis;
        double power, offset;
        if (!(in >> op >> P.fam >> P.d >> P.nb >> P.g >> n >> power >> axis >> offset)) continue;
        auto read = [&](std::vector<double>& v, int k) {
            v.resize(k);
            for (double& x : v) {
                std::string t;
                in >> t;
                x = std::strtod(t.c_str(), nullptr);
            }
        };
        const int d = P.d;
        read(P.par, P.fam == MCUBES_F_GAUSS ? 1 + 2 * d : P.fam == MCUBES_F_OSC ? 1 + d : P.fam == MCUBES_F_CORNER ? d : 2 * d);
        read(P.lo, d);
        read(P.hi, d);
        for (int k = 0; k < P.nb; ++k) P.edges.push_back(k + 1 == P.nb ? 1.0 : std::pow((k + 1.0) / P.nb, power));
        const bool fix = P.prepare();
        uint64_t m = 1;
        for (int j = 0; j < d; ++j) m *= P.g;
        std::mt19937_64 rng(7);
        if (op == "fix") {
            std::printf("%d %d\n", (int)fix, P.a.fam.fq);
        } else if (op == "mean") {
            LD sum = 0, ef = 0, ed = 0;
            for (int i = 0; i < n; ++i) {
                const Out o = sample_f(P, (uint32_t)(rng() % m), (uint32_t)i);
                const LD F = exact(P, o);
                sum += std::fabs(F);
                ef += (LD)o.fix - F;
                ed += (LD)o.dbl - F;
            }
            std::printf("%d %.6e %.6e\n", (int)fix, (double)(ef / sum), (double)(ed / sum));
        } else if (op == "cut") {
            int wrong = 0, taken = 0;
            for (int i = 0; i < n; ++i) {
                const uint32_t c = (uint32_t)(rng() % m);
                const LD x = sample_f(P, c, (uint32_t)i).x[axis];
                const double xd = (double)x, ulp = std::nextafter(xd, 1e300) - xd;
                P.par[d + axis] = xd + ((i & 1) ? offset : -offset) * ulp;
                taken += P.prepare();
                const double F = sample_f(P, c, (uint32_t)i).fix;
                wrong += (F != 0.0) != (x < (LD)P.par[d + axis]);
            }
            std::printf("%d %d\n", taken, wrong);
        }
    }
    return 0;
}
