// All iterations of a fit in one CTA, over samples whose sums in the order of x are at hand: what both ways share (em_sorted.cu: one sample per weight;
// em_cells_fit.cu: the distinct normalised weights of bf16 data).
//
// An iteration is a chain of latencies, so it is kept short: what lies below a threshold is one sum, and a region is the difference of
// two such sums.  For the squared error the sums of large parts of the samples are kept in two doubles each, so that their
// difference is as good as adding the region up; the rest is rounded once to a double.  A region that is very light beside its
// neighbours, or stands beside sums that are not finite, is added up by itself.  The weights of the medians are integers.
//
// When an iteration leaves every level unchanged the remaining ones would repeat it bit for bit: their entries of the error log
// are filled in and the loop ends.
#pragma once

#include "em_sorted.cuh"

namespace bof4 {

constexpr int kFitThreads = 32 * kLevels;  // those that form the running sums

// This thread's asynchronous copies have arrived.
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

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
struct PairSum {
    double s, sx;
};
__device__ __forceinline__ PairSum operator+(const PairSum& a, const PairSum& b) { return PairSum{a.s + b.s, a.sx + b.sx}; }
__device__ __forceinline__ PairSum shfl_up(const PairSum& v, int off) { return PairSum{__shfl_up_sync(kFull, v.s, off), __shfl_up_sync(kFull, v.sx, off)}; }
__device__ __forceinline__ PairSum shfl(const PairSum& v, int from) { return PairSum{__shfl_sync(kFull, v.s, from), __shfl_sync(kFull, v.sx, from)}; }

// The same for values of any type with a sum.
template <int PER, class T, class Part, class Put>
__device__ __forceinline__ void running_sums(int n, Part part, Put put)
{
    __shared__ T s_warp[kLevels];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool has = warp < kLevels;
    T v[PER], t{};
#pragma unroll
    for (int k = 0; k < PER; ++k) v[k] = has && tid * PER + k < n ? part(tid * PER + k) : T{};
#pragma unroll
    for (int k = 0; k < PER; ++k) t = t + v[k];
    auto scan = [&](T& u) {  // inclusive, over the warp
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const T w = shfl_up(u, off);
            if (lane >= off) u = w + u;
        }
    };
    scan(t);
    if (lane == 31 && has) s_warp[warp] = t;
    __syncthreads();
    T w{};
    if (lane < warp && lane < kLevels) w = s_warp[lane];
    scan(w);
    T run = shfl_up(t, 1);
    if (lane == 0) run = T{};
    run = shfl(w, 31) + run;
    if (!has) return;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (tid * PER + k <= n) put(tid * PER + k, run);
        run = run + v[k];
    }
    if (tid == kFitThreads - 1 && n == kFitThreads * PER) put(n, run);
}

// Whether the difference of two sums {s, sx}, s0 and s1, is too rough to be a region's: small beside what was rounded (2^-20 of it; `rest`: what
// was in the two sums) or beside all that lies in front (2^-50), negative, or not finite.  By the upper halves of the
// doubles, whose exponents begin at bit 20.
__device__ __forceinline__ bool too_rough(double s0, double s1, double2 rest0, double2 rest1, double front)
{
    auto top = [](double d) { return __double2hiint(d) & 0x7fffffff; };
    const int least0 = max(max(top(rest0.x), top(rest1.x)) - (20 << 20), top(front) - (50 << 20)), least1 = max(top(rest0.y), top(rest1.y)) - (20 << 20);
    const int t0 = __double2hiint(s0), t1 = top(s1);
    return t0 < max(least0, 0) || t1 < least1 || max(t0, t1) >= 0x7ff00000;
}

}  // namespace bof4
