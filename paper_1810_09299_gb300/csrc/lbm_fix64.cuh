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
// operations, a conversion into the block 0.21 cycles per node and SM against
// 0.62 for an FP64 operation, and they run beside the FP64 pipe.  The rounding is
// at most that of the FP64 sums it replaces: the bits a smaller value loses lie K
// bits below the largest one's last place.
// E is at least kMinE (values below 2^-959 lose their low bits, as subnormal
// numbers do); from kBadE on (2^1007, infinities, NaN) the results are NaN.
constexpr int kMinE = 64, kBadE = 2030;

__device__ __forceinline__ int exp64(double x) { return (int)(((uint32_t)__double2hiint(x) >> 20) & 0x7ffu); }
__device__ __forceinline__ int abs_hi(double x) { return __double2hiint(x) & 0x7fffffff; }
#ifdef __CUDACC__
// shifts whose amounts may exceed 63 (PTX: all bits leave, or the sign fills)
__device__ __forceinline__ unsigned long long shr64u(unsigned long long v, int s) {
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}
__device__ __forceinline__ long long shr64(long long v, int s) {
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}
__device__ __forceinline__ unsigned long long shl64u(unsigned long long v, int s) {
    unsigned long long r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}
// places from the leading non-sign bit to bit 63 (31); -1 for 0 and -1
__device__ __forceinline__ int lead_shift64(long long v) {
    int r;
    asm("bfind.shiftamt.s64 %0, %1;" : "=r"(r) : "l"(v));
    return r;
}
__device__ __forceinline__ int lead_shift32(int v) {
    int r;
    asm("bfind.shiftamt.s32 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}
// 1 / x and 1 / sqrt(x) within 1 ulp and 2^-22.9 (the PTX ISA's bounds)
__device__ __forceinline__ float rcp_start(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt_start(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
#endif  // a host compiler includes this file after its own definitions of these and of CUDA's intrinsics
__device__ __forceinline__ double nan64() { return __longlong_as_double(0x7ff8000000000000ll); }

// x in the block of exponent E >= exp64(x), truncated towards zero.
template <int K>
__device__ __forceinline__ long long fix64(double x, int E) {
    const int hi = __double2hiint(x);
    const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
    const unsigned long long m = (((unsigned long long)mh << 32) | (uint32_t)__double2loint(x)) << K;
    const long long v = (long long)shr64u(m, E - exp64(x)), sg = (long long)(hi >> 31);
    return (v ^ sg) - sg;
}
// m 2^e as a double, rounded to nearest, for |m| < 2^63 and a result within the
// normal numbers (or m = 0): -1000 <= e <= 900 does.  The FP64 pipe's conversion takes
// 0.53 cycles per node and SM, a normalisation and packing in integers 0.3, but
// the integer pipes have more to do.
__device__ __forceinline__ double double_cvt(long long m, int e) {
    const double d = __ll2double_rn(m);
    const int hi = __double2hiint(d);
    return __hiloint2double(hi == 0 ? 0 : hi + (e << 20), __double2loint(d));
}
// v 2^(E - 1075 - K) as a double, kMinE <= E < kBadE.
template <int K>
__device__ __forceinline__ double unfix64(long long v, int E) {
    return double_cvt(v, E - 1075 - K);
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

// ---------------------------------------------------------------- numbers of 62 bits
// x = m 2^e with |m| < 2^62 in integer registers, for products and sums that
// would wait for the FP64 pipe.  Cycles per node and SM (measured): a product
// 0.15, a sum 0.09, norm29 0.08, norm 0.19, sf_of 0.15, against 0.62 for an FP64
// operation of either kind.  A product keeps all but 1 bit of normalised operands (|m| >= 2^61) and
// is exact to about 2^-58 of itself; a sum is exact to the last place of its
// larger operand.  A factor that may have cancelled (a sum) is normalised
// first; zero carries a large negative exponent, so that it never shifts the
// other operand of a sum.
struct Sf {
    long long m;
    int e;
};
constexpr int kZeroE = -(1 << 17);

// a b 2^-62, |a|, |b| < 2^62 (-2^62 too), within 10 units: the bits below the high
// words of the mixed products (up to 8 units), the low words' product (4) and their last
// bits (1 each, either way) are left out, about 5 units on average, and 4 are added back
// (to a zero, too: one that must stay zero is the caller's, or has the exponent
// kZeroE).  High-word multiplications (30.6 per SM and cycle) rather than signed wide
// ones (12).
__device__ __forceinline__ long long mul62(long long a, long long b) {
    const int ah = (int)(a >> 32) * 2, bh = (int)(b >> 32) * 2;
    const int al = (int)((uint32_t)a >> 1), bl = (int)((uint32_t)b >> 1);
    const int mixed = __mulhi(ah, bl) + __mulhi(bh, al) + 1;
    const long long high = ((long long)__mulhi(ah, bh) << 32) | (uint32_t)(ah * bh);
    return high + (long long)mixed * 4;
}
__device__ __forceinline__ Sf operator*(Sf a, Sf b) { return Sf{mul62(a.m, b.m), a.e + b.e + 62}; }
__device__ __forceinline__ Sf operator+(Sf a, Sf b) {
    const int e = max(a.e, b.e) + 1;
    return Sf{shr64(a.m, e - a.e) + shr64(b.m, e - b.e), e};
}
__device__ __forceinline__ Sf operator-(Sf a, Sf b) {
    const int e = max(a.e, b.e) + 1;
    return Sf{shr64(a.m, e - a.e) - shr64(b.m, e - b.e), e};
}
// a and b as integers of one unit 2^e, each below 2^61, for several sums of them
struct Two {
    long long a, b;
    int e;
};
__device__ __forceinline__ Two align(Sf a, Sf b) {
    const int e = max(a.e, b.e) + 1;
    return Two{shr64(a.m, e - a.e), shr64(b.m, e - b.e), e};
}
__device__ __forceinline__ Sf scale2(Sf a, int n) { return Sf{a.m, a.e + n}; }  // a 2^n
__device__ __forceinline__ Sf neg(Sf a) { return Sf{-a.m, a.e}; }
// The same value with 2^61 <= |m| < 2^62 (zero: see above).
__device__ __forceinline__ Sf norm(Sf a) {
    const int sh = lead_shift64(a.m);
    return Sf{(long long)shl64u((unsigned long long)a.m, sh - 2), sh < 0 ? kZeroE : a.e - (sh - 2)};
}
// The same by at most 29 places, from the high word alone: enough for a factor
// that is a sum, since bits further down carry the sum's own rounding.
__device__ __forceinline__ Sf norm29(Sf a) {
    const int n = (int)min((uint32_t)lead_shift32((int)(a.m >> 32)), 31u) - 2;
    return Sf{a.m << n, a.e - n};
}
// An ordinary double (zero and subnormal numbers count as numbers near 2^-1022;
// infinities and NaN: the caller replaces the result).
__device__ __forceinline__ Sf sf_of(double x) {
    const int hi = __double2hiint(x);
    const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
    const long long v = (long long)((((unsigned long long)mh << 32) | (uint32_t)__double2loint(x)) << 9);
    const long long sg = (long long)(hi >> 31);
    return Sf{(v ^ sg) - sg, exp64(x) - 1084};
}
// The same with zero as zero: a number near -2^-1022 would become -1 in any larger unit.
__device__ __forceinline__ Sf sf_of_or_zero(double x) {
    const Sf a = sf_of(x);
    return Sf{exp64(x) == 0 ? 0ll : a.m, a.e};
}
// m 2^e as a double for any e: below the normal numbers zero, above them NaN.
__device__ __forceinline__ double double_of(Sf a) {
    const double d = double_cvt(a.m, a.e);
    return a.e < -1000 ? 0.0 : (a.e > 900 ? nan64() : d);
}
// The leading 64 bits of |a|, a != 0: bit 63 set.
__device__ __forceinline__ unsigned long long lead64(long long a, int& n) {
    const long long sg = a >> 63;
    const unsigned long long u = (unsigned long long)((a ^ sg) - sg);
    n = __clzll((long long)u);
    return shl64u(u, n);
}
// 1 / a, within 2^-59.9 of itself, also from a start one ulp off; bad is raised for
// zero.  x = |a| scaled to [1/2, 1); y0 = 1 / x from the FP32 approximation as an integer
// of 31 bits, e = 1 - x y0 to 62 places (below 2^-22), y0 (1 + e + e^2).  An FP64 Newton
// step took three operations of the FP64 pipe and two conversions.
__device__ __forceinline__ Sf rcp(Sf a, bool& bad) {
    int n;
    const unsigned long long u = lead64(a.m, n);  // x 2^64
    const uint32_t uh = (uint32_t)(u >> 32), ul = (uint32_t)u;
    const uint32_t y0 = min(__float2uint_rn(rcp_start(__uint2float_rn(uh)) * 0x1p62f), 0x7fffffffu);  // y 2^30
    const long long e = (long long)((1ull << 62) - ((unsigned long long)uh * y0 + __umulhi(ul, y0)));
    const int es = (int)(e >> 10);
    const unsigned long long t = (unsigned long long)(e + (__mulhi(es, es) >> 10)) << 20;
    const long long d = (((long long)__mulhi((int)(t >> 32), (int)y0) << 32) | (uint32_t)((uint32_t)(t >> 32) * y0)) +
                        __umulhi((uint32_t)t, y0);
    const unsigned long long y = ((unsigned long long)y0 << 32) + (unsigned long long)(d >> 18);  // y 2^62
    bad = bad || a.m == 0;
    const long long m = (long long)((y - 1) >> 1), sg = a.m >> 63;  // below 2^62 for x = 1/2, too
    return Sf{(m ^ sg) - sg, n - a.e - 125};
}
// sqrt(a), a >= 0, within 2^-58.8 of itself, also from a start one ulp off.  v = a
// scaled by an even power of two to [1/4, 1); r0 = 1 / sqrt(v) from the FP32
// approximation, e = 1 - v r0^2, s = v r0 (1 + e / 2 + 3 e^2 / 8).
__device__ __forceinline__ Sf root(Sf a) {
    int n;
    unsigned long long v = lead64(a.m, n);
    const int ex = 64 - n + a.e, odd = ex & 1;  // a = (v 2^-64) 2^ex
    v >>= odd;
    const uint32_t vh = (uint32_t)(v >> 32), vl = (uint32_t)v;
    const uint32_t r0 = min(__float2uint_rn(rsqrt_start(__uint2float_rn(vh)) * 0x1p46f), 0x7fffffffu);  // 2^30 / sqrt(v)
    const unsigned long long w = (unsigned long long)r0 * r0;          // 2^60 / v
    const uint32_t wh = (uint32_t)(w >> 32), wl = (uint32_t)w;
    const unsigned long long vw = (unsigned long long)vh * wh + __umulhi(vh, wl) + __umulhi(vl, wh);
    const long long e = (long long)((1ull << 60) - vw);
    const int es = (int)(e >> 8);
    const long long t = (e >> 1) + ((__mulhi(es, es) * 3) >> 15);
    const long long s0 = (long long)((unsigned long long)vh * r0 + __umulhi(vl, r0));  // sqrt(v) 2^62
    // (s0 passes 2^62 where v is just below 1 and r0 above 1 / sqrt(v): halved for the product)
    const long long s = min(s0 + (mul62(s0 >> 1, t << 23) >> 20), (1ll << 62) - 1);
    return a.m == 0 ? Sf{0ll, kZeroE} : Sf{s, ((ex + odd) >> 1) - 62};
}
// v / 3 and v / 9, within 1.5 units: v times 2^64 / 3 (or 9), words H and L, without the
// low words' product and plus Up for what the high words leave out (0 stays 0)
template <uint32_t H, uint32_t L, uint32_t Up>
__device__ __forceinline__ long long mul_const(long long v) {
    const int h = (int)(v >> 32);
    const int mixed = (int)__umulhi((uint32_t)v, H) + __mulhi(h, (int)L) + (int)min((uint32_t)v, Up);
    return (((long long)__mulhi(h, (int)H) << 32) | (uint32_t)(h * (int)H)) + mixed;
}
template <uint32_t Up = 1>
__device__ __forceinline__ long long third64(long long v) { return mul_const<0x55555555u, 0x55555555u, Up>(v); }
template <uint32_t Up = 1>
__device__ __forceinline__ long long ninth64(long long v) { return mul_const<0x1c71c71cu, 0x71c71c72u, Up>(v); }
// v times the double nearest 1/9 (5.6e-17 below it), for the weights of the phase
// field: the conserved sum of f takes this factor every step.  With 1/9 itself it
// drifts by 4e-15 instead of 1.1e-13 over 2000 steps, but the oracle and the
// general kernels hold the weights as doubles, and on the 64 x 128 static drop runs
// with and without that drift part by 2e-12 (phi) and 1e-11 (p) in that time.
__device__ __forceinline__ long long ninth_double(long long v) { return mul_const<0x1c71c71cu, 0x71c71c00u, 2>(v); }

}  // namespace axilbm
