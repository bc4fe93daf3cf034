// Host build of the fixed-point functions of the FP64 kernels' affine families
// (csrc/fx_math.cuh: fx_exp_fixed, fx_recip, fx_cos_turns) with plain C++
// stand-ins for the device intrinsics.  Reads lines "<op> <u64> [<int>]" and
// prints: e/E exp(-q 2^-fq)/exp(q 2^-fq) as a hex double, r the reciprocal of
// a normalised 64-bit value, c the signed magnitude of cos(2 pi a 2^-64).
#include <cstdint>
#include <cstring>
#include <cmath>
#include <cstdio>
#define __device__
#define __forceinline__ inline
#define __noinline__
#define __host__
static inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
template <class T> static inline T __ldg(const T* p) { return *p; }
static inline long long __double_as_longlong(double d) { long long x; std::memcpy(&x, &d, 8); return x; }
static inline double __longlong_as_double(long long x) { double d; std::memcpy(&d, &x, 8); return d; }
using std::log; using std::exp; using std::ldexp;
#include "fx_math.cuh"
int main()
{
    char line[256], op;
    while (std::fgets(line, sizeof line, stdin)) {
        unsigned long long u;
        int f = 0;
        bool neg = false;
        if (std::sscanf(line, "%c %llu %d", &op, &u, &f) < 2) continue;
        if (op == 'e') std::printf("%a\n", mc::fx::fx_exp_fixed<true>(u, f, 1ull << 63, 0));
        else if (op == 'E') std::printf("%a\n", mc::fx::fx_exp_fixed<false>(u, f, 1ull << 63, 0));
        else if (op == 'r') std::printf("%llu\n", (unsigned long long)mc::fx::fx_recip(u));
        else if (op == 'c') {
            const uint64_t v = mc::fx::fx_cos_turns(u, &neg);
            std::printf("%s%llu\n", neg ? "-" : "", (unsigned long long)v);
        }
    }
    return 0;
}
