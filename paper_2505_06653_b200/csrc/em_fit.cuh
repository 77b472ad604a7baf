// All iterations of a fit in one CTA, over samples whose sums in the order of x are at hand: what both ways share (em_sorted.cu: one sample per weight;
// em_cells_fit.cu: the distinct normalised weights of bf16 data).
//
// An iteration is a chain of latencies, so it is kept short: what lies below a threshold is one sum, and a region is the difference of
// two such sums.  The sums of large parts of the samples are kept in two doubles each, so that their difference is as good as
// adding the region up; the rest is rounded once to a double.  For the squared error a region that is light beside this rest (2^-8, so that
// its level is good to 2^-45), or stands beside sums that are not finite, is added up by itself; the absolute error, which only goes to the
// log, is known to the rounding of these differences, 2^-53 of the weight in each (with one double for a sum over all parts it was off by 30
// times as much).  The weights of the medians are integers.
//
// When an iteration leaves every level unchanged the remaining ones would repeat it bit for bit: their entries of the error log
// are filled in and the loop ends.
#pragma once

#include "em_sorted.cuh"

namespace bof4 {

constexpr int kFitThreads = 32 * kLevels;  // those that form the running sums

// This thread's asynchronous copies have arrived.
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Asynchronous copy of `bytes` (rounded up to 16) to shared memory, by all threads of the CTA.
__device__ __forceinline__ void copy_in(void* to, const void* from, int bytes)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(to);
    for (int k = threadIdx.x; k < (bytes + 15) / 16; k += blockDim.x)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a + 16u * k), "l"(static_cast<const char*>(from) + 16 * k) : "memory");
}

// A table in shared memory that is complete: made behind the barrier that its writers pass.  Holds its address in that space,
// which the compiler does not find out for pointers in the sources.
template <class T>
struct SharedTable {
    uint32_t base;
    __device__ __forceinline__ explicit SharedTable(const T* p)
    {
        asm volatile("mov.u32 %0, %1;" : "=r"(base) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
    }
    __device__ __forceinline__ T operator[](int i) const
    {
        const uint32_t a = base + (uint32_t)i * (uint32_t)sizeof(T);
        T v;
        if constexpr (sizeof(T) == 16) asm("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a));
        else if constexpr (sizeof(T) == 8) asm("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(a));
        else if constexpr (sizeof(T) == 4) asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
        else asm("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
        return v;
    }
};

// A sum in two doubles, high + low with |low| at most half a unit of high.
struct TwoSum {
    double h, l;
};
__device__ __forceinline__ TwoSum two_add(const TwoSum& a, const TwoSum& b)
{
    const double s = a.h + b.h, t = s - a.h;
    const double e = ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l);
    const double h = s + e;
    return TwoSum{h, e - (h - s)};
}
__device__ __forceinline__ TwoSum two_shfl_up(const TwoSum& a, int off)
{
    return TwoSum{__shfl_up_sync(kFull, a.h, off), __shfl_up_sync(kFull, a.l, off)};
}

__device__ __forceinline__ unsigned long long shfl_up(unsigned long long v, int off) { return __shfl_up_sync(kFull, v, off); }
__device__ __forceinline__ unsigned long long shfl(unsigned long long v, int from) { return __shfl_sync(kFull, v, from); }
// {s, sx} in two doubles each, of which the low ones take up what the high ones are rounded by (they are not made small again
// after an addition: a few units of the high ones at most, and three operations of eleven less).
struct TwoPair {
    TwoSum s, x;
};
__device__ __forceinline__ TwoSum two_gather(const TwoSum& a, const TwoSum& b)
{
    const double s = a.h + b.h, t = s - a.h;
    return TwoSum{s, ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l)};
}
__device__ __forceinline__ TwoPair operator+(const TwoPair& a, const TwoPair& b) { return TwoPair{two_gather(a.s, b.s), two_gather(a.x, b.x)}; }
__device__ __forceinline__ TwoPair shfl_up(const TwoPair& v, int off) { return TwoPair{two_shfl_up(v.s, off), two_shfl_up(v.x, off)}; }
__device__ __forceinline__ TwoSum two_shfl(const TwoSum& a, int from) { return TwoSum{__shfl_sync(kFull, a.h, from), __shfl_sync(kFull, a.l, from)}; }
__device__ __forceinline__ TwoPair shfl(const TwoPair& v, int from) { return TwoPair{two_shfl(v.s, from), two_shfl(v.x, from)}; }

// put(k, sum of part(0) ... part(k - 1)), k = 0 ... n <= PER * kFitThreads, by the CTA's first kFitThreads threads or its next ones (`has`;
// the others only pass the barrier).  All parts have been read before anything is put, so a sum may take the place of its part.
// (The cells' parts come from shared memory, see copy_in: a thread's are neighbours, and the lines that they share do not stay in the
// L1 that those tables leave: read from global memory, 11 us more.)
template <int PER, class T, class Part, class Put>
__device__ __forceinline__ void running_sums(bool has, int n, Part part, Put put)
{
    __shared__ T s_warp[kLevels];
    const int tid = threadIdx.x & (kFitThreads - 1), lane = tid & 31, warp = tid >> 5;
    T v[PER], t{};
    auto scan = [&](T& u, int width) {  // inclusive, over the first `width` lanes of the warp
#pragma unroll
        for (int off = 1; off < width; off <<= 1) {
            const T w = shfl_up(u, off);
            if (lane >= off) u = w + u;
        }
    };
    if (has) {
#pragma unroll
        for (int k = 0; k < PER; ++k) v[k] = tid * PER + k < n ? part(tid * PER + k) : T{};
        t = v[0];
#pragma unroll
        for (int k = 1; k < PER; ++k) t = t + v[k];
        scan(t, 32);
        if (lane == 31) s_warp[warp] = t;
    }
    __syncthreads();
    if (!has) return;
    T w{};
    if (lane < warp) w = s_warp[lane];
    scan(w, kLevels);
    T run = shfl_up(t, 1);
    if (lane == 0) run = T{};
    run = shfl(w, kLevels - 1) + run;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (tid * PER + k <= n) put(tid * PER + k, run);
        run = run + v[k];
    }
    if (tid == kFitThreads - 1 && n == kFitThreads * PER) put(n, run);
}

// {s, sx} of what lies below a point, in two doubles each.
struct Below {
    double2 high, low;
};

// The absolute error is added up half region by half region, each the difference of two such sums.  Lane l has what lies below level l,
// lane 16 + l what lies below the threshold above it (lane 31: everything): a lane's half ends there and begins at the point of the
// lane that `lower_end_of` says.
__device__ __forceinline__ int lower_end_of(int lane) { return lane < kLevels ? lane + kLevels - 1 : lane - kLevels; }

// The points of level l: the thresholds on either side and the level itself, within them whatever the levels are.
struct FitPoints {
    float lo, mid, hi;
};
__device__ __forceinline__ FitPoints points_of(int l, float left, float lv, float right)
{
    const float inf = __int_as_float(0x7f800000);
    FitPoints p;
    p.lo = l ? __fmul_rn(__fadd_rn(left, lv), 0.5f) : -inf;
    p.hi = l < kLevels - 1 ? __fmul_rn(__fadd_rn(lv, right), 0.5f) : inf;
    p.mid = fminf(fmaxf(lv, p.lo), p.hi);
    return p;
}

// What the samples of a lane's half add to the error of level lv (levels that do not ascend have regions without samples).
__device__ __forceinline__ double half_error(int lane, const FitPoints& p, float lv, const Below& begin, const Below& end)
{
    if (p.lo > p.hi) return 0.0;
    const bool first = lane == 0;  // nothing lies in front of it
    auto part = [&](double b, double e) { return e - (first ? 0.0 : b); };
    const double s = part(begin.high.x, end.high.x) + part(begin.low.x, end.low.x);
    const double x = part(begin.high.y, end.high.y) + part(begin.low.y, end.low.y);
    return lane < kLevels ? (double)lv * s - x : x - (double)lv * s;
}

// The last warp of a fit of squared errors.  Iteration by iteration, beside the others' next one: the error, and whether the levels have
// stopped to move (`stop`: the iteration behind whose barrier all leave).  w2: the sum of squares of all samples.
__device__ __forceinline__ void squared_errors(const SortFit& F, double w2, const float (&level)[2][kLevels], const double2 (&below)[2][3][kLevels + 1], int& stop)
{
    const int lane = threadIdx.x & 31, l = lane & (kLevels - 1);
    float before = __int_as_float(0x7fc00001);
    double err = 0.0;
    int iter = 0;
    for (; iter < F.iters; ++iter) {
        const int set = iter & 1;
        __syncthreads();
        if (stop <= iter) break;
        const float lv = level[set][l];
        const double2 h0 = below[set][0][l], h1 = below[set][0][l + 1], l0 = below[set][1][l], l1 = below[set][1][l + 1];
        const double2 r0 = below[set][2][l], r1 = below[set][2][l + 1];
        const double s0 = ((h1.x - h0.x) + (l1.x - l0.x)) + (r1.x - r0.x);
        const double s1 = ((h1.y - h0.y) + (l1.y - l0.y)) + (r1.y - r0.y);
        const double o = (double)lv;
        err = o * (2.0 * s1 - o * s0);
#pragma unroll
        for (int off = 8; off; off >>= 1) err += __shfl_xor_sync(kFull, err, off);
        err = fmax(w2 - err, 0.0) / (double)F.n_total;
        if (lane == 0 && F.err_log) F.err_log[iter] = err;
        if (__all_sync(kFull, __float_as_uint(lv) == __float_as_uint(before)) && lane == 0) stop = iter + 1;
        before = lv;
    }
    err = __shfl_sync(kFull, err, 0);
    if (F.err_log)
        for (int k = iter + lane; k < F.iters; k += 32) F.err_log[k] = err;
}

// Whether the difference of two sums {s, sx}, s0 and s1, is too rough to be a region's: not finite, negative, or small beside all that lies
// in front (2^-50) or beside what was rounded, the `rest` of either sum (2^-8).  What is compared with it is what the region is known to
// hold: its weight, s0, and of sum |weight x|, which s1 may cancel, the upper rest if the points have different parts in front of them.
// (From 2^-3 on, all regions go the long way where one group of bins holds all the data: 2^20 weights 53 us an iteration, 16 this way.)  By
// the upper halves of the doubles, whose exponents begin at bit 20, and without branches: these were 1 % of a fit over bf16 data.
__device__ __forceinline__ bool too_rough(double s0, double s1, double2 rest0, double2 rest1, double front0, double front1)
{
    auto top = [](double d) { return __double2hiint(d) & 0x7fffffff; };
    const int t0 = __double2hiint(s0), t1 = top(s1), held = front0 != front1 ? max(t1, top(rest1.y)) : t1;
    const int least0 = max(max(top(rest0.x), top(rest1.x)) - (8 << 20), top(front1) - (50 << 20));
    return (t0 < max(least0, 0)) | (held < top(rest0.y) - (8 << 20)) | (max(t0, t1) >= 0x7ff00000);
}

}  // namespace bof4
