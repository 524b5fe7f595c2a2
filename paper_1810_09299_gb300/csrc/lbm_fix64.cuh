// lbm_fix64.cuh -- sums of doubles in 64-bit integers, for the FP64 kernels
// (this chip's FP64 pipe takes 1.6 operations per SM and cycle).
#pragma once

#include <stdint.h>

namespace axilbm {

// ---------------------------------------------------------------- block fixed point
// Sums of doubles in 64-bit integers: the values of one sum are brought to the
// largest exponent E of the block (E the exponent field, x = m 2^(E - 1075 - K),
// K extra bits below the last place of the largest value), added exactly, and
// the result is rounded once to a double.  An addition costs two integer
// instructions of the ~100 per SM and cycle instead of one of the 1.6 FP64
// operations, a conversion into the block 0.27 and out of it 0.31 cycles per
// node and SM against 0.62 for an FP64 operation, and both run beside the FP64
// pipe.  The rounding is at most that of the FP64 sums it replaces: the bits a
// smaller value loses lie K bits below the largest one's last place.
// E is at least kMinE (values below 2^-959 lose their low bits, as subnormal
// numbers do); from kBadE on (2^1007, infinities, NaN) the results are NaN.
constexpr int kMinE = 64, kBadE = 2030;

__device__ __forceinline__ int exp64(double x) { return (int)(((uint32_t)__double2hiint(x) >> 20) & 0x7ffu); }
__device__ __forceinline__ double nan64() { return __longlong_as_double(0x7ff8000000000000ll); }

// x in the block of exponent E >= exp64(x), truncated towards zero.
template <int K>
__device__ __forceinline__ long long fix64(double x, int E) {
    const int hi = __double2hiint(x);
    const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
    const unsigned long long m = (((unsigned long long)mh << 32) | (uint32_t)__double2loint(x)) << K;
    const long long v = (long long)(m >> min(E - exp64(x), 63)), sg = (long long)(hi >> 31);
    return (v ^ sg) - sg;
}
// v 2^(E - 1075 - K) as a double (rounded to nearest, ties away from zero).
template <int K>
__device__ __forceinline__ double unfix64(long long v, int E) {
    const long long sg = v >> 63;
    unsigned long long a = (unsigned long long)((v ^ sg) - sg);
    const int n = __clzll((long long)a);
    a <<= n & 63;
    unsigned long long b = (a >> 11) + ((a >> 10) & 1ull) + ((unsigned long long)(uint32_t)(E + 10 - K - n) << 52);
    b |= (unsigned long long)sg << 63;
    return v == 0 ? 0.0 : __longlong_as_double((long long)b);
}
template <int N>
__device__ __forceinline__ int block_exp(const double* x) {
    int e = kMinE << 20;
#pragma unroll
    for (int i = 0; i < N; ++i) e = max(e, __double2hiint(x[i]) & 0x7fffffff);
    return e >> 20;
}

constexpr int kPopK = 6;  // populations: sums of at most 16 largest values stay below 2^63

// f_0 + .. + f_8 (Eq. 16's sum), rounded once.
__device__ __forceinline__ double sum64(const double* f) {
    const int E = block_exp<9>(f);
    long long t = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) t += fix64<kPopK>(f[i], E);
    const double r = unfix64<kPopK>(t, E);
    return E >= kBadE ? nan64() : r;
}

}  // namespace axilbm
