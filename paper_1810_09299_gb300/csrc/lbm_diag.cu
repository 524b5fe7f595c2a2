// lbm_diag.cu -- FP64 diagnostics of one case (deterministic reductions) and the initial phase-field shapes of the paper's tests (Sec. 3).
#include <cuda_runtime.h>
#include <math.h>

#include <mutex>

#include "../../include/lbm.h"
#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace axilbm {

namespace {

constexpr int kDiagBlocks = kDiagPartials / kDiagRecord;  // 2 x 152 SMs; fixed so the summation order is fixed
constexpr int kDiagThreads = 256;

// Quantities: 0 mass, 1 kinetic, 2 z-moment, 3 p in liquid, 4 weight in liquid,
// 5 p in gas, 6 weight in gas (sums); 7 max |u|^2, 8 phi_min, 9 phi_max
// (extrema); 10 non-finite count (sum).  A partial record holds them in this order.
constexpr int kSums = 7;

// The bits of x below 2^(L - 1075), in units of 2^(e - 1075).
__device__ __forceinline__ unsigned long long bits_below(double x, int L, int& e) {
    const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
    const unsigned long long m =
        ((unsigned long long)(((uint32_t)hi & 0xfffffu) | (ex ? 0x100000u : 0u)) << 32) | (uint32_t)__double2loint(x);
    e = max(ex, 1);  // subnormal numbers share the exponent of the smallest normal ones
    const int n = L - e;
    return n >= 53 ? m : n <= 0 ? 0ull : m & ((1ull << n) - 1);
}
// The warp's sum of the bits of v[0 .. count) below 2^(L - 1075), in units of 2^(E - 1139), E
// the exponent field of the largest value that has any; what lies below one unit is left out.
__device__ __forceinline__ __int128 warp_window_sum(const double* v, int count, int stride, int L, int& E) {
    const int lane = threadIdx.x & 31;
    int top = 1, e;
    for (int i = lane; i < count; i += 32)
        if (bits_below(v[(size_t)i * stride], L, e) != 0) top = max(top, e);
    E = (int)__reduce_max_sync(0xffffffffu, (unsigned)top);
    __int128 acc = 0;
    for (int i = lane; i < count; i += 32) {
        const double x = v[(size_t)i * stride];
        const unsigned long long m = bits_below(x, L, e);
        const int sh = E - e;
        const unsigned __int128 y = sh < 128 ? ((unsigned __int128)m << 64) >> sh : (unsigned __int128)0;
        acc += __double2hiint(x) < 0 ? -(__int128)y : (__int128)y;
    }
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)acc, off);
        const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(acc >> 64), off);
        acc += ((__int128)hi << 64) | lo;
    }
    return acc;
}
// The rest of a sum whose largest values cancelled: window after window below the first
// one (sum acc, exponent E), each in four exact parts that are added up with compensation.
__device__ __noinline__ double warp_cancelled_sum(const double* v, int count, int stride, __int128 acc, int E) {
    double s = 0.0, c = 0.0;
    for (;;) {
        const bool neg = acc < 0;
        const unsigned __int128 a = neg ? -(unsigned __int128)acc : (unsigned __int128)acc;
        for (int k = 96; k >= 0; k -= 32) {
            const double part = scalbn((double)(uint32_t)(a >> k), E - 1139 + k), x = neg ? -part : part, t = s + x;
            c += fabs(s) >= fabs(x) ? (s - t) + x : (x - t) + s;
            s = t;
        }
        if (E <= 65) return s + c;  // (the unit is below the smallest number)
        int next;
        acc = warp_window_sum(v, count, stride, E - 64, next);
        E = next;
    }
}
// The sum of v[0 .. count) (stride `stride`, count <= 512) into every lane of the
// calling warp: the values as 128-bit integers in units of 2^-64 of the last place of
// the largest one, rounded once.  A value may lose what lies below a unit; where so much
// cancels that this could count (the sum is below 2^74 units, of which at most 512 are
// lost), the bits below are added as well.  Compensated (Neumaier) sums in FP64
// took most of diag_final_kernel's 19.5 us: some 100 dependent operations of a pipe
// that takes a warp instruction every 20 cycles; this takes 8.  Values of 2^1007 and
// more, infinities and NaN are summed plainly.
__device__ __forceinline__ double warp_exact_sum(const double* v, int count, int stride) {
    const int lane = threadIdx.x & 31;
    int top = 0;
    for (int i = lane; i < count; i += 32) top = max(top, __double2hiint(v[(size_t)i * stride]) & 0x7fffffff);
    int E = max((int)(__reduce_max_sync(0xffffffffu, (unsigned)top) >> 20), 1);
    if (E >= 2030) {
        double acc = 0.0;
        for (int i = lane; i < count; i += 32) acc += v[(size_t)i * stride];
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        return acc;
    }
    const __int128 acc = warp_window_sum(v, count, stride, 4096, E);
    // one rounding: |acc| below 2^126 with its leading bit brought to bit 62 of
    // 64, the bits below folded into the last one
    const bool neg = acc < 0;
    unsigned __int128 a = neg ? -(unsigned __int128)acc : (unsigned __int128)acc;
    const unsigned long long ah = (unsigned long long)(a >> 64), al = (unsigned long long)a;
    if (ah < 1024 && E > 65) return warp_cancelled_sum(v, count, stride, acc, E);
    if ((ah | al) == 0) return 0.0;
    const int lead = ah ? 127 - __clzll((long long)ah) : 63 - __clzll((long long)al);
    const int down = lead - 62;
    unsigned long long r;
    if (down > 0) {
        r = (unsigned long long)(a >> down);
        if ((a & (((unsigned __int128)1 << down) - 1)) != 0) r |= 1ull;
    } else {
        r = (unsigned long long)(a << -down);
    }
    const double d = scalbn(__ull2double_rn(r), E - 1075 - 64 + down);
    return neg ? -d : d;
}

// The plain sum of v[0 .. count) (stride as above) into lane 0: each lane adds
// its share in a fixed order, then a fixed pairwise shuffle tree.  Used inside
// a block, where a thread holds few nodes: pairwise summation of the block's
// values keeps the error near log2(values) rounding units.
__device__ __forceinline__ double warp_sum(const double* v, int count, int stride) {
    const int lane = threadIdx.x & 31;
    double acc = 0.0;
    for (int i = lane; i < count; i += 32) acc += v[(size_t)i * stride];
    for (int off = 16; off > 0; off >>= 1) {
        const double o = __shfl_down_sync(0xffffffffu, acc, off);
        if (lane + off < 32) acc += o;
    }
    return acc;
}

// The extrema and the count the same way: max |u|^2, min phi, max phi, count.
__device__ __forceinline__ void warp_extrema(const double* uu, const double* lo, const double* hi,
                                             const double* bad, int count, int stride, double out[4]) {
    const int lane = threadIdx.x & 31;
    double m = 0.0, mn = INFINITY, mx = -INFINITY, nb = 0.0;
    for (int i = lane; i < count; i += 32) {
        m = fmax(m, uu[(size_t)i * stride]);
        mn = fmin(mn, lo[(size_t)i * stride]);
        mx = fmax(mx, hi[(size_t)i * stride]);
        nb += bad[(size_t)i * stride];
    }
    for (int off = 16; off > 0; off >>= 1) {
        m = fmax(m, __shfl_down_sync(0xffffffffu, m, off));
        mn = fmin(mn, __shfl_down_sync(0xffffffffu, mn, off));
        mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, off));
        const double o = __shfl_down_sync(0xffffffffu, nb, off);
        if (lane + off < 32) nb += o;
    }
    out[0] = m;
    out[1] = mn;
    out[2] = mx;
    out[3] = nb;
}

// A double as an integer of the same order (and back): extrema and thresholds are
// compared beside the FP64 pipe.
__device__ __forceinline__ long long ordered(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double unordered(long long b) {
    return __longlong_as_double(b ^ ((b >> 63) & 0x7fffffffffffffffll));
}
// phi of these bits: of a finite phi, b > kLiquid where phi > 0.99 and b < kGas
// where phi < 0.01 (negative ones have negative bits)
constexpr long long kLiquid = 0x3fefae147ae147aell, kGas = 0x3f847ae147ae147bll;

// The kernels of a record and of the drops follow each other and the fields kernel
// with overlapping launches (pdl_wait); what they read of one another's is not
// marked __restrict__, so that no load of it moves above the wait.  A record right
// after a step of the 64 x 128 drop (FP64): 78 -> 71 us; its drops 30 -> 26 us.
//
// One partial record per block.  Rows k = blockIdx.x, blockIdx.x + gridDim.x,
// ...; of these each thread takes the columns j = threadIdx.x + 256 i, so it
// holds only a few nodes and sums them plainly, a column's before they are
// weighted with its r: 7 FP64 operations per node instead of some 25
// (256 x 1024: 20.9 -> 13.7 us, a whole record 77 -> 51 us in FP32); the block's 256 values
// of each quantity are then summed pairwise by one warp per quantity (warps
// 0-6 the sums, warp 7 the extrema and the count).  The records of the blocks
// are combined exactly by diag_final_kernel.
__global__ void __launch_bounds__(kDiagThreads) diag_partial_kernel(const double* F, int nz, int nr, double* partials) {
    static_assert(kDiagThreads == 32 * (kSums + 1), "one warp per sum plus one");
    pdl_trigger();
    pdl_wait();
    const int64_t n = (int64_t)nz * nr;
    double acc[kSums] = {};
    long long uu_max = 0, pmin = ordered(INFINITY), pmax = ordered(-INFINITY);
    int bad = 0;
    for (int j = threadIdx.x; j < nr; j += blockDim.x) {
        double phi_s = 0.0, uu_s = 0.0, z_s = 0.0, p_liq = 0.0, p_gas = 0.0, z = blockIdx.x + 0.5;
        int n_liq = 0, n_gas = 0;
        for (int k = blockIdx.x; k < nz; k += gridDim.x, z += (double)gridDim.x) {
            const int64_t o = (int64_t)k * nr + j;
            const double phi = F[o], rho = F[n + o], uz = F[2 * n + o], ur = F[3 * n + o], p = F[4 * n + o];
            if (max(max(abs_hi(phi), abs_hi(p)), max(abs_hi(uz), abs_hi(ur))) >= 0x7ff00000) {
                ++bad;
                continue;
            }
            const double uu = uz * uz + ur * ur;
            phi_s += phi;
            uu_s += rho * uu;
            z_s += z * phi;
            const long long b = __double_as_longlong(phi);
            if (b > kLiquid) p_liq += p, ++n_liq;  // phi > 0.99
            if (b < kGas) p_gas += p, ++n_gas;     // phi < 0.01
            uu_max = max(uu_max, __double_as_longlong(uu));
            pmin = min(pmin, ordered(phi));
            pmax = max(pmax, ordered(phi));
        }
        const double r = j + 0.5;
        acc[0] += r * phi_s;
        acc[1] += 0.5 * r * uu_s;
        acc[2] += r * z_s;
        acc[3] += r * p_liq;
        acc[4] += r * n_liq;
        acc[5] += r * p_gas;
        acc[6] += r * n_gas;
    }
    __shared__ double sh[kSums + 4][kDiagThreads];
    for (int q = 0; q < kSums; ++q) sh[q][threadIdx.x] = acc[q];
    sh[kSums][threadIdx.x] = __longlong_as_double(uu_max);
    sh[kSums + 1][threadIdx.x] = unordered(pmin);
    sh[kSums + 2][threadIdx.x] = unordered(pmax);
    sh[kSums + 3][threadIdx.x] = bad;
    __syncthreads();
    const int w = threadIdx.x >> 5;
    double* out = partials + (size_t)blockIdx.x * kDiagRecord;
    if (w < kSums) {
        const double t = warp_sum(sh[w], kDiagThreads, 1);
        if ((threadIdx.x & 31) == 0) out[w] = t;
    } else {
        double e[4];
        warp_extrema(sh[kSums], sh[kSums + 1], sh[kSums + 2], sh[kSums + 3], kDiagThreads, 1, e);
        if ((threadIdx.x & 31) == 0)
            for (int q = 0; q < 4; ++q) out[kSums + q] = e[q];
    }
}

// Contribution of the axis link (k, k+1) to the length of the phi > 1/2 set on
// the axis row (linear crossing); the last link wraps when z is periodic and
// is half a cell at a wall.
__device__ __forceinline__ double axis_link(const double* F, int k, int nz, int nr, int zper) {
    const double a = F[(int64_t)k * nr] - 0.5;
    int kn = k + 1;
    if (kn >= nz) {
        if (!zper) return a > 0 ? 0.5 : 0.0;
        kn = 0;
    }
    const double b = F[(int64_t)kn * nr] - 0.5;
    if (a > 0 && b > 0) return 1.0;
    if (a > 0 && b <= 0) return a / (a - b);
    if (a <= 0 && b > 0) return b / (b - a);
    return 0.0;
}

// Final combination and the interface lengths, one block of kFinalThreads:
// warps 0-6 combine one sum each over the partial records (exact, see
// warp_exact_sum) and warp 7 the extrema and the count, every one in a fixed
// order, so the result is deterministic.  A case of fewer rows than blocks has
// records only for its rows.
constexpr int kFinalThreads = 256;
static_assert(kFinalThreads == 32 * (kSums + 1), "one warp per sum plus one");
__global__ void __launch_bounds__(kFinalThreads) diag_final_kernel(const double* F, int nz, int nr,
                                                                   int zper, double step,
                                                                   const double* partials, double* out, const int* status,
                                                                   int* status_out) {
    __shared__ double sres[kSums + 4];
    __shared__ double slen[kFinalThreads / 32];
    __shared__ double s_dp[2], s_umax;
    __shared__ int sjmin;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const int records = min(nz, kDiagBlocks);
    if (t == 0) sjmin = nr;
    pdl_wait();
    // axis half-length: per-thread sums over k = t, t + T, ..., then a shuffle tree
    double len = 0.0;
    for (int k = t; k < nz; k += kFinalThreads) len += axis_link(F, k, nz, nr, zper);
    for (int off = 16; off > 0; off >>= 1) len += __shfl_down_sync(0xffffffffu, len, off);
    if (lane == 0) slen[w] = len;
    if (w < kSums) {
        const double r = warp_exact_sum(partials + w, records, kDiagRecord);
        if (lane == 0) sres[w] = r;
    } else {
        double e[4];
        const double* x = partials + kSums;
        warp_extrema(x, x + 1, x + 2, x + 3, records, kDiagRecord, e);
        if (lane == 0)
            for (int q = 0; q < 4; ++q) sres[kSums + q] = e[q];
    }
    __syncthreads();
    const double mass = sres[0];
    const double zc = sres[2] / mass;
    // radial crossing on the row nearest the centroid: the first outward crossing
    int kc = (int)floor(zc);
    kc = kc < 0 ? 0 : (kc >= nz ? nz - 1 : kc);
    // the record's other divisions and its root, a warp each
    if (lane == 0) {
        if (w == 1) s_dp[0] = sres[4] > 0 ? sres[3] / sres[4] : 0.0;
        if (w == 2) s_dp[1] = sres[6] > 0 ? sres[5] / sres[6] : 0.0;
        if (w == 3) s_umax = sqrt(sres[kSums]);  // |u|max from the largest |u|^2
    }
    for (int j = t; j + 1 < nr; j += kFinalThreads) {
        const double a = F[(int64_t)kc * nr + j] - 0.5, b = F[(int64_t)kc * nr + j + 1] - 0.5;
        if (a > 0 && b <= 0) {
            atomicMin(&sjmin, j);
            break;
        }
    }
    __syncthreads();
    if (t != 0) return;
    double rc = 0.0;
    if (sjmin + 1 < nr) {
        const double a = F[(int64_t)kc * nr + sjmin] - 0.5, b = F[(int64_t)kc * nr + sjmin + 1] - 0.5;
        rc = (sjmin + 0.5) + a / (a - b);
    }
    double axis = 0.0;
    for (int i = 0; i < kFinalThreads / 32; ++i) axis += slen[i];
    if (!zper && F[0] - 0.5 > 0) axis += 0.5;
    out[0] = step;
    out[1] = mass;
    out[2] = sres[1];
    out[3] = zc;
    out[4] = s_dp[0] - s_dp[1];
    out[5] = s_umax;
    out[6] = sres[kSums + 1];
    out[7] = sres[kSums + 2];
    out[8] = 0.5 * axis;
    out[9] = rc;
    out[10] = sres[kSums + 3];
    if (status_out) *status_out = *status;
}

// ---------------------------------------------------------------- drops on the axis
// The liquid bodies a breaking thread forms (Sec. 3.3), read off the axis row
// j = 0: every maximal run of axis nodes with phi > 1/2 is one drop.  The rows
// of the case are split between the drops at one row inside each gas gap (the
// row of least r-weighted phi of the gap, first on ties), so every row belongs
// to exactly one drop and a drop's volume is 2 pi sum r phi over its rows.
// Its ends are the linearly interpolated phi = 1/2 crossings on the axis (a
// wall plane where the run reaches a z wall).  In a periodic case the rows
// wrap; with no gap at all the whole axis is one unbroken body.
//
// Output (FP64): out[0] = number of drops, out[1] = min phi on the axis row,
// out[2] = row of that minimum + 1/2 (its z), then for each of the first
// min(number, max_drops) drops in z order (z_start, z_end, volume, radius of
// the sphere of that volume); z_end < z_start for a drop that wraps a periodic
// boundary.  rows: scratch of 2 nz doubles.
//
// Two kernels.  axis_rows_kernel, one warp per row of the case: rows[k] = sum_j
// r_j phi(k, j), lanes along r and a fixed shuffle tree, and the axis row copied
// to rows[nz + k].  axis_drops_kernel, one block: both arrays in shared memory
// (global for nz > kAxisRows), the runs found by a block scan over contiguous
// chunks of the axis row, then one warp per drop for its two cuts and its sum.
// What bounds it is latency: one block and one thread walking the rows one by
// one took 225 us on a 600 x 200 case and 650 us on a 1024 x 256 one; these two
// take about 12 and 15.
constexpr int kAxisThreads = 256;
constexpr int kAxisRows = 2816;  // rows whose two doubles fit 44 KB of shared memory

__global__ void __launch_bounds__(kAxisThreads) axis_rows_kernel(const double* F, int nz, int nr, double* rows) {
    const int k = blockIdx.x * (kAxisThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    pdl_trigger();
    pdl_wait();
    if (k >= nz) return;
    const double* P = F + (int64_t)k * nr;
    double s = 0.0;
    for (int j = lane; j < nr; j += 32) s += (j + 0.5) * P[j];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if (lane == 0) {
        rows[k] = s;
        rows[nz + k] = P[0];
    }
}

// The first row of least weight of the gap of scan indices [a, b), a < b, in
// row k0 + i of the scan (a row is replaced only by a strictly lighter one, so a
// NaN at a keeps the cut there); the whole warp calls it.
__device__ __forceinline__ int lightest_row(const double* rows, int nz, int k0, int a, int b) {
    const auto at = [&](int i) { return rows[k0 + i < nz ? k0 + i : k0 + i - nz]; };
    const double first = at(a);
    if (!(first == first)) return a;
    const int lane = threadIdx.x & 31;
    double v = INFINITY;
    int c = a;
    for (int i = a + lane; i < b; i += 32) {
        const double x = at(i);
        if (x < v) v = x, c = i;
    }
    for (int off = 16; off > 0; off >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, v, off);
        const int oc = __shfl_xor_sync(0xffffffffu, c, off);
        if (ov < v || (ov == v && oc < c)) v = ov, c = oc;
    }
    return v < first ? c : a;
}

// Sum of the rows of scan indices [a, b) (lanes, then a fixed tree); valid in lane 0.
__device__ __forceinline__ double sum_rows(const double* rows, int nz, int k0, int a, int b) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (int i = a + lane; i < b; i += 32) s += rows[k0 + i < nz ? k0 + i : k0 + i - nz];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    return s;
}

__global__ void __launch_bounds__(kAxisThreads) axis_drops_kernel(const double* rows_g, int nz, int zper,
                                                                  int max_drops, double* out,
                                                                  const int* status, int* status_out) {
    constexpr int kWarps = kAxisThreads / 32;
    __shared__ double sbuf[2 * kAxisRows];
    __shared__ double s_min[kWarps];
    __shared__ int s_kmin[kWarps], s_gas[kWarps], s_last[kWarps], s_cnt[kWarps];
    __shared__ int s_a[kMaxAxisDrops + 1], s_b[kMaxAxisDrops + 1];  // runs of the first drops, scan indices
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    pdl_wait();
    if (t == 0) *status_out = *status;
    const bool fits = nz <= kAxisRows;
    for (int i = t; fits && i < 2 * nz; i += kAxisThreads) sbuf[i] = rows_g[i];
    __syncthreads();
    const double* rows = fits ? sbuf : rows_g;
    const double* axis = rows + nz;
    const int chunk = (nz + kAxisThreads - 1) / kAxisThreads;
    // the least phi of the axis row (the first such row) and the first gas row
    double vmin = INFINITY;
    int kmin = 0, gas = nz;
    for (int i = t * chunk; i < min((t + 1) * chunk, nz); ++i) {
        const double v = axis[i];
        if (v < vmin) vmin = v, kmin = i;
        if (gas == nz && !(v > 0.5)) gas = i;
    }
    for (int off = 16; off > 0; off >>= 1) {
        const double ov = __shfl_down_sync(0xffffffffu, vmin, off);
        const int ok = __shfl_down_sync(0xffffffffu, kmin, off), og = __shfl_down_sync(0xffffffffu, gas, off);
        if (ov < vmin || (ov == vmin && ok < kmin)) vmin = ov, kmin = ok;
        gas = min(gas, og);
    }
    if (lane == 0) s_min[w] = vmin, s_kmin[w] = kmin, s_gas[w] = gas;
    __syncthreads();
    gas = nz;
    for (int i = 0; i < kWarps; ++i) gas = min(gas, s_gas[i]);
    if (t == 0) {
        for (int i = 1; i < kWarps; ++i)
            if (s_min[i] < vmin) vmin = s_min[i], kmin = s_kmin[i];
        out[1] = vmin;
        out[2] = kmin + 0.5;
    }
    const double two_pi = 6.283185307179586;
    const auto put = [&](int drop, int field, double v) { out[3 + 4 * drop + field] = v; };
    const auto put_volume = [&](int drop, double v) {
        put(drop, 2, two_pi * v);
        put(drop, 3, cbrt(3.0 * two_pi * v / (4.0 * M_PI)));
    };
    if (gas == nz) {  // liquid along the whole axis: one unbroken body
        if (w == 0) {
            const double vol = sum_rows(rows, nz, 0, 0, nz);
            if (lane == 0) {
                out[0] = 1.0;
                if (max_drops > 0) {
                    put(0, 0, 0.0);
                    put(0, 1, (double)nz);
                    put_volume(0, vol);
                }
            }
        }
        return;
    }
    // The scan starts at row 0, or in a periodic case at the first row of the
    // gas gap that the first gas row lies in, so that the rows before it
    // (cyclically) end the last drop.
    int k0 = 0;
    if (zper) {
        if (gas > 0) {
            k0 = gas;
        } else {  // row 0 is gas: its gap starts after the last liquid row
            int last = -1;
            for (int i = t * chunk; i < min((t + 1) * chunk, nz); ++i)
                if (axis[i] > 0.5) last = i;
            for (int off = 16; off > 0; off >>= 1) last = max(last, __shfl_down_sync(0xffffffffu, last, off));
            if (lane == 0) s_last[w] = last;
            __syncthreads();
            last = -1;
            for (int i = 0; i < kWarps; ++i) last = max(last, s_last[i]);
            if (last < 0) {  // gas along the whole axis: no drop
                if (t == 0) out[0] = 0.0;
                return;
            }
            k0 = last + 1 < nz ? last + 1 : 0;
        }
    }
    const auto liquid = [&](int i) { return axis[k0 + i < nz ? k0 + i : k0 + i - nz] > 0.5; };
    // runs of liquid in scan order: each thread counts the starts of its chunk
    // of scan indices, then numbers them from the block's exclusive sum
    const int i0 = min(t * chunk, nz), i1 = min(i0 + chunk, nz);
    int count = 0;
    bool prev = i0 > 0 && i0 < nz && liquid(i0 - 1);
    for (int i = i0; i < i1; ++i) {
        const bool l = liquid(i);
        count += l && !prev;
        prev = l;
    }
    int incl = count;
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += o;
    }
    if (lane == 31) s_cnt[w] = incl;
    __syncthreads();
    int d = incl - count, ndrops = 0;
    for (int i = 0; i < kWarps; ++i) {
        if (i < w) d += s_cnt[i];
        ndrops += s_cnt[i];
    }
    prev = i0 > 0 && i0 < nz && liquid(i0 - 1);
    for (int i = i0; i < i1; ++i) {
        const bool l = liquid(i);
        if (l && !prev) {
            if (d <= kMaxAxisDrops) s_a[d] = i;
            ++d;
        }
        if (l && (i + 1 == nz || !liquid(i + 1)) && d - 1 <= kMaxAxisDrops) s_b[d - 1] = i;
        prev = l;
    }
    __syncthreads();
    if (t == 0) out[0] = (double)ndrops;
    // z of the phi = 1/2 crossing between the rows of scan indices i and i + 1
    const auto crossing = [&](int i) {
        const int k = k0 + i < nz ? k0 + i : k0 + i - nz, kn = k + 1 < nz ? k + 1 : 0;
        const double a = axis[k], b = axis[kn];
        const double z = (k + 0.5) + (0.5 - a) / (b - a);
        return z >= nz ? z - nz : z;
    };
    // One warp per drop: the rows from the lightest row of the gap before it to
    // the one before the lightest row of the gap after it; at walls the whole
    // gap; in a periodic case the first gap's rows before its cut end the last
    // drop.
    for (int q = w; q < min(ndrops, max_drops); q += kWarps) {
        const bool last = q + 1 == ndrops;
        int lo = 0, hi = nz;
        if (q > 0) lo = lightest_row(rows, nz, k0, s_b[q - 1] + 1, s_a[q]);
        else if (zper) lo = lightest_row(rows, nz, k0, 0, s_a[0]);
        if (!last) hi = lightest_row(rows, nz, k0, s_b[q] + 1, s_a[q + 1]);
        double vol = sum_rows(rows, nz, k0, lo, hi);
        if (last && zper) vol += sum_rows(rows, nz, k0, 0, lightest_row(rows, nz, k0, 0, s_a[0]));
        if (lane == 0) {
            put(q, 0, !zper && s_a[q] == 0 ? 0.0 : crossing(s_a[q] == 0 ? nz - 1 : s_a[q] - 1));
            put(q, 1, !zper && s_b[q] + 1 == nz ? (double)nz : crossing(s_b[q]));
            put_volume(q, vol);
        }
    }
}

// ---------------------------------------------------------------- shapes
struct ShapeArgs {
    double a[8];
};

__global__ void shape_kernel(int shape, ShapeArgs A, int nz, int nr, double* __restrict__ phi) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (j >= nr || k >= nz) return;
    const double z = k + 0.5, r = j + 0.5;
    double v = 0.0;
    switch (shape) {
        case 0: {  // flat: {z_i, W, axis}
            const double x = (A.a[2] == 0.0) ? z : r;
            v = 0.5 + 0.5 * tanh(2.0 * (A.a[0] - x) / A.a[1]);
            break;
        }
        case 1:
        case 5: {  // sphere / bubble: {z_c, R, W}
            const double d = sqrt((z - A.a[0]) * (z - A.a[0]) + r * r);
            v = 0.5 + 0.5 * tanh(2.0 * (A.a[1] - d) / A.a[2]);
            if (shape == 5) v = 1.0 - v;
            break;
        }
        case 2: {  // ellipsoid: {z_c, R_z, R_r, W}
            const double Re = cbrt(A.a[2] * A.a[2] * A.a[1]);
            const double q = sqrt((z - A.a[0]) * (z - A.a[0]) / (A.a[1] * A.a[1]) + r * r / (A.a[2] * A.a[2]));
            v = 0.5 + 0.5 * tanh(2.0 * Re * (1.0 - q) / A.a[3]);
            break;
        }
        case 3: {  // P2 drop: {z_c, R0, eps, W}
            const double d = sqrt((z - A.a[0]) * (z - A.a[0]) + r * r);
            const double c = (z - A.a[0]) / fmax(d, 1e-300);
            const double Rs = A.a[1] * (1.0 + A.a[2] * 0.5 * (3.0 * c * c - 1.0));
            v = 0.5 + 0.5 * tanh(2.0 * (Rs - d) / A.a[3]);
            break;
        }
        case 4: {  // thread: {R, amp, lambda, theta, W}
            const double d = A.a[1] * cos(2.0 * M_PI * z / A.a[2] + A.a[3]);
            v = 0.5 + 0.5 * tanh(2.0 * (A.a[0] + d - r) / A.a[4]);
            break;
        }
        default:
            v = 0.0;
    }
    phi[(int64_t)k * nr + j] = v;
}

}  // namespace

int diag_partials_size() { return kDiagPartials; }

cudaError_t launch_diag(const double* fields, int nz, int nr, int zper, double step, double* partials, double* out,
                        const int* status, int* status_out, cudaStream_t st) {
    launch_pdl(diag_partial_kernel, nz < kDiagBlocks ? nz : kDiagBlocks, dim3(kDiagThreads), st, fields, nz, nr, partials);
    launch_pdl(diag_final_kernel, 1, dim3(kFinalThreads), st, fields, nz, nr, zper, step, partials, out, status, status_out);
    return cudaGetLastError();
}

cudaError_t launch_axis_drops(const double* fields, int nz, int nr, int zper, int max_drops, double* rows, double* out,
                              const int* status, int* status_out, cudaStream_t st) {
    constexpr int per = kAxisThreads / 32;
    launch_pdl(axis_rows_kernel, (nz + per - 1) / per, dim3(kAxisThreads), st, fields, nz, nr, rows);
    launch_pdl(axis_drops_kernel, 1, dim3(kAxisThreads), st, rows, nz, zper, max_drops, out, status, status_out);
    return cudaGetLastError();
}

cudaError_t launch_shape(int shape, const double* args, int nargs, int nz, int nr, double* phi0, cudaStream_t st) {
    ShapeArgs A{};
    for (int i = 0; i < nargs && i < 8; ++i) A.a[i] = args[i];
    dim3 grid((nr + 127) / 128, nz);
    shape_kernel<<<grid, 128, 0, st>>>(shape, A, nz, nr, phi0);
    return cudaGetLastError();
}

}  // namespace axilbm

// ---------------------------------------------------------------- bounded-wait self-test
namespace {
// An mbarrier expecting two arrivals gets one, so its phase never completes:
// the bounded wait must give up after `tries` polls and raise the status word.
__global__ void selftest_wait_kernel(int tries, int* status) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) axilbm::mbar_init(&bar, 2);
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(axilbm::smem_addr(&bar)) : "memory");
    axilbm::mbar_wait_bounded(&bar, 0, status, tries);
}
}  // namespace

extern "C" int lbm_selftest_bounded_wait(int32_t tries, void* stream, int32_t* device_status_word) {
    if (tries < 1 || !device_status_word) return LBM_ERR_INVALID_ARG;
    selftest_wait_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(tries, device_status_word);
    if (cudaGetLastError() != cudaSuccess) return LBM_ERR_CUDA;
    int st = 0;
    if (cudaMemcpyAsync(&st, device_status_word, sizeof(int), cudaMemcpyDeviceToHost, (cudaStream_t)stream) !=
            cudaSuccess ||
        cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ERR_CUDA;
    }
    return st != 0 ? LBM_ERR_TIMEOUT : LBM_OK;
}

// ---------------------------------------------------------------- FP64 pipe rate
// Throughput probe of the FP64 pipe (no paper counterpart): every thread runs
// kChains independent chains of dependent FP64 fused multiply-adds, enough
// independent work per warp to keep the pipe busy, and writes one sum so the
// work is not removed.  The rate is the FMA count over the CUDA-event time of
// the launch.
namespace {
constexpr int kFmaChains = 8;
__global__ void __launch_bounds__(256) dfma_rate_kernel(int iters, double a, double b, double* out) {
    double x[kFmaChains];
#pragma unroll
    for (int c = 0; c < kFmaChains; ++c) x[c] = (double)(threadIdx.x + c) * 1e-3;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int c = 0; c < kFmaChains; ++c) x[c] = fma(x[c], a, b);
    }
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < kFmaChains; ++c) s += x[c];
    out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}
}  // namespace

extern "C" int lbm_measure_fp64_rate(int32_t iters, void* stream, double* fma_per_second) {
    if (iters < 1 || !fma_per_second) return LBM_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ERR_CUDA;
    }
    const int blocks = 4 * sms, threads = 256;
    double* out = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = LBM_OK;
    if (cudaMalloc(&out, (size_t)blocks * threads * sizeof(double)) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ERR_OOM;
    }
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) rc = LBM_ERR_CUDA;
    // one warm-up launch, then the timed one
    for (int rep = 0; rep < 2 && rc == LBM_OK; ++rep) {
        if (rep == 1 && cudaEventRecord(e0, st) != cudaSuccess) rc = LBM_ERR_CUDA;
        dfma_rate_kernel<<<blocks, threads, 0, st>>>(iters, 0.999999, 1e-7, out);
        if (cudaGetLastError() != cudaSuccess) rc = LBM_ERR_CUDA;
        if (rep == 1 && rc == LBM_OK && cudaEventRecord(e1, st) != cudaSuccess) rc = LBM_ERR_CUDA;
    }
    float ms = 0.0f;
    if (rc == LBM_OK && (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess))
        rc = LBM_ERR_CUDA;
    if (rc == LBM_OK) *fma_per_second = (double)blocks * threads * kFmaChains * (double)iters / (ms * 1e-3);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(out);
    if (rc != LBM_OK) cudaGetLastError();
    return rc;
}

// ---------------------------------------------------------------- allocation-free reduction
// lbm_diag_reduce_noalloc: the diagnostics reduction for callers that cannot
// allocate device memory when they need the numbers (for example a caller
// whose device memory is entirely held by its own pool, or a monitoring loop
// that must not pay for an allocation).  Its only scratch, the per-block
// partial sums, is a fixed static device array of this module.
namespace {

constexpr int kScratchDoubles = axilbm::kDiagPartials;  // 304 blocks x 11 doubles = 26,752 bytes
constexpr int64_t kNoAllocMaxNodes = 2147483647;       // nz * nr must fit a signed 32-bit count
constexpr int kMaxDevices = 64;

// Every GPU that loads the library holds this array until the process exits.
static __device__ __align__(256) double g_diag_scratch[kScratchDoubles];

std::mutex g_scratch_mutex;
double* g_scratch_addr[kMaxDevices] = {};  // device address of g_diag_scratch, per device

}  // namespace

extern "C" int lbm_diag_reduce_noalloc(const double* d_fields, int32_t nz, int32_t nr, int32_t z_periodic,
                                       double step, double* d_out, void* stream) {
    if (!d_fields || !d_out || nz < 1 || nr < 1 || (z_periodic != 0 && z_periodic != 1))
        return LBM_ERR_INVALID_ARG;
    if ((int64_t)nz * nr > kNoAllocMaxNodes) return LBM_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ERR_CUDA;
    }
    if (dev < 0 || dev >= kMaxDevices) return LBM_ERR_INVALID_ARG;
    double* scratch = nullptr;
    {
        // one-time set-up on this device (current device): the host-side name
        // g_diag_scratch is not a device address, so look the address up
        std::lock_guard<std::mutex> lock(g_scratch_mutex);
        if (!g_scratch_addr[dev]) {
            void* p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_diag_scratch);
            if (e != cudaSuccess || !p) {
                cudaGetLastError();
                return LBM_ERR_CUDA;
            }
            g_scratch_addr[dev] = (double*)p;
        }
        scratch = g_scratch_addr[dev];
    }
    // Every partial slot is overwritten by the first kernel before the second
    // reads it, so nothing from an earlier call needs clearing.
    cudaError_t e = axilbm::launch_diag(d_fields, nz, nr, z_periodic, step, scratch, d_out, nullptr, nullptr,
                                         (cudaStream_t)stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return LBM_ERR_CUDA;
    }
    return LBM_OK;
}
