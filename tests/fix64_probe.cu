// The 62-bit numbers of lbm_fix64.cuh one operation at a time, for test_fix64.py: a kernel (nvcc), or a loop on the
// host (any other compiler), where the FP32 starts of rcp and root are 1 / x and 1 / sqrt(x) rounded to nearest and
// moved by fix64_start_ulps ulps.
#include <stdint.h>
#ifndef __CUDACC__
#include <math.h>
#include <string.h>
#define __device__
#define __forceinline__ inline
template <class T>
T max(T a, T b) { return a < b ? b : a; }
template <class T>
T min(T a, T b) { return b < a ? b : a; }
inline int64_t bits_of(double x) { int64_t b; memcpy(&b, &x, 8); return b; }
inline double __longlong_as_double(long long b) { double x; memcpy(&x, &b, 8); return x; }
inline int __double2hiint(double x) { return (int)(bits_of(x) >> 32); }
inline int __double2loint(double x) { return (int)bits_of(x); }
inline double __hiloint2double(int hi, int lo) { return __longlong_as_double((long long)hi << 32 | (uint32_t)lo); }
inline double __ll2double_rn(long long v) { return (double)v; }
inline int __mulhi(int a, int b) { return (int)(((long long)a * b) >> 32); }
inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
inline int __clzll(long long v) { return v == 0 ? 64 : __builtin_clzll((unsigned long long)v); }
inline float __uint2float_rn(unsigned v) { return (float)v; }
inline unsigned __float2uint_rn(float v) { return (unsigned)llrint((double)v); }
static int start_ulps = 0;
extern "C" void fix64_start_ulps(int n) { start_ulps = n; }
inline float moved(double x) {
    float y = (float)x;
    for (int i = 0; i < start_ulps; ++i) y = nextafterf(y, INFINITY);
    for (int i = 0; i > start_ulps; --i) y = nextafterf(y, 0.0f);
    return y;
}
namespace axilbm {
inline unsigned long long shr64u(unsigned long long v, int s) { return (uint32_t)s > 63u ? 0 : v >> s; }
inline unsigned long long shl64u(unsigned long long v, int s) { return (uint32_t)s > 63u ? 0 : v << s; }
inline long long shr64(long long v, int s) { return v >> ((uint32_t)s > 63u ? 63 : s); }
inline int lead_shift64(long long v) { const long long u = v ^ (v >> 63); return u == 0 ? -1 : __clzll(u); }
inline int lead_shift32(int v) { const int u = v ^ (v >> 31); return u == 0 ? -1 : __builtin_clz((unsigned)u); }
inline float rcp_start(float x) { return moved(1.0 / x); }
inline float rsqrt_start(float x) { return moved(1.0 / sqrt((double)x)); }
}  // namespace axilbm
#endif
#include "../paper_1810_09299_gb300/csrc/lbm_fix64.cuh"

using namespace axilbm;

__device__ inline Sf fix64_op(int op, Sf a, Sf b) {
    bool bad = false;
    switch (op) {
        case 0: return a * b;
        case 1: return rcp(a, bad);
        case 2: return root(a);
        case 3: return Sf{third64(a.m), a.e};
        default: return Sf{ninth64(a.m), a.e};
    }
}
#ifdef __CUDACC__
__global__ void fix64_kernel(int op, int64_t n, const int64_t* am, const int* ae, const int64_t* bm, const int* be,
                             int64_t* rm, int* re) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Sf r = fix64_op(op, Sf{(long long)am[i], ae[i]}, Sf{(long long)bm[i], be[i]});
    rm[i] = r.m;
    re[i] = r.e;
}
#endif
// n operations on arrays of this memory (the device's with nvcc)
extern "C" int fix64_run(int op, int64_t n, const int64_t* am, const int* ae, const int64_t* bm, const int* be, int64_t* rm,
                         int* re) {
#ifdef __CUDACC__
    fix64_kernel<<<(unsigned)((n + 255) / 256), 256>>>(op, n, am, ae, bm, be, rm, re);
    return (int)cudaDeviceSynchronize();
#else
    for (int64_t i = 0; i < n; ++i) {
        const Sf r = fix64_op(op, Sf{(long long)am[i], ae[i]}, Sf{(long long)bm[i], be[i]});
        rm[i] = r.m;
        re[i] = r.e;
    }
    return 0;
#endif
}
