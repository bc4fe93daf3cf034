// Host build of fx_sum_floats (csrc/fx_math.cuh) with plain C++ stand-ins for
// the device intrinsics.  Reads lines "<stride> <n> <bits> ..." (n * stride
// values in all) and prints the sum of every stride-th float as a hex double.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <iostream>
#include <vector>
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
using std::log; using std::exp; using std::ldexp; using std::memcpy;
#include "fx_math.cuh"
int main()
{
    size_t stride;
    int n;
    while (std::cin >> stride >> n) {
        std::vector<uint32_t> v(stride * n);
        for (auto& x : v) std::cin >> x;
        std::printf("%a\n", mc::fx::fx_sum_floats(v.data(), stride, n));
    }
    return 0;
}
