// Codebook fit over ordered samples (see em_sorted.cuh): one sample per weight, the ordering passes,
// the sums per bin and the iterations.
//
// Launches of a fit, whatever its number of iterations: samples (one per 64 tensors), two ordering
// passes of eight bits (count and scatter each, least significant digit first, stable), first samples and sums
// of the bins in two steps, full order where a bin is crowded, iterations.  Nothing depends on the order in which CTAs run:
// the samples' order, the order of every sum and hence the result are reproducible.
#include <type_traits>

#include "em_fit.cuh"

namespace bof4 {

constexpr int kSortThreads = 1024;
constexpr int kSortPerThread = 8;
constexpr int kSortTile = kSortThreads * kSortPerThread;

size_t sorted_layout(void* base, int64_t n, SortWs* W)
{
    char* p = static_cast<char*>(base);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* q = p ? p + off : nullptr;
        off += align_up(bytes, 256);
        return q;
    };
    const size_t chunks = (size_t)((n + kSortChunk - 1) / kSortChunk) + 1;
    SortWs L;
    L.n_items = reinterpret_cast<uint32_t*>(take(256));
    L.w2 = reinterpret_cast<double*>(take(kSortParts * 8));
    L.counts = reinterpret_cast<uint32_t*>(take((size_t)kSortGrid * 256 * 4));
    L.start = reinterpret_cast<uint32_t*>(take((size_t)(kSortBins + 1) * 4));
    L.first = reinterpret_cast<uint32_t*>(take((size_t)(kSortGroups + 1) * 4));
    L.off = reinterpret_cast<uint16_t*>(take((size_t)kSortBins * 2));
    L.pre = reinterpret_cast<SortSums*>(take((size_t)kSortBins * sizeof(SortSums)));
    L.bin = reinterpret_cast<SortSums*>(take((size_t)kSortBins * sizeof(SortSums)));
    L.group = reinterpret_cast<SortSums*>(take((size_t)kSortGroups * sizeof(SortSums)));
    L.lead = reinterpret_cast<SortSums*>(take(chunks * sizeof(SortSums)));
    L.trail = reinterpret_cast<SortSums*>(take(chunks * sizeof(SortSums)));
    L.a = reinterpret_cast<float2*>(take((size_t)n * 8));
    L.b = reinterpret_cast<float2*>(take((size_t)n * 8));
    L.before = nullptr;
    if (W) *W = L;
    return off;
}

// ---------------------------------------------------------------- samples, one per weight

// Every lane owns 16 consecutive weights; x = RN(w / m) and |m| (1 for the normalised-domain metrics) go
// to the sample array in the order of the weights.  Bound by its stores (8 bytes per weight).  Every CTA leaves its sum of
// squares and its largest constant in slots of its own; the first launch of a fit writes all slots, and the head.
__device__ __forceinline__ void st_256(void* p, const Raw8& r)
{
    asm volatile("st.global.v8.u32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(r.u[0]), "r"(r.u[1]), "r"(r.u[2]), "r"(r.u[3]),
                 "r"(r.u[4]), "r"(r.u[5]), "r"(r.u[6]), "r"(r.u[7])
                 : "memory");
}
template <class DT, int I, bool SIGNED>
__global__ void __launch_bounds__(512, 2)
sort_samples_kernel(const EmTensors T, const uint32_t first, const uint32_t n, float2* __restrict__ items,
                    uint32_t* __restrict__ head, double* __restrict__ w2, uint32_t* __restrict__ tops)
{
    if (!after_previous()) return;
    constexpr int NT = 512;
    __shared__ WideScratch s_wide;
    __shared__ uint32_t s_item0[kEmMaxTensors];
    __shared__ double s_sum[NT / 32];
    __shared__ uint32_t s_max[NT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        uint32_t at = first;
        for (int t = 0; t < T.count; ++t) {
            s_item0[t] = at;
            at += (uint32_t)T.n[t];
        }
    }
    __syncthreads();
    const int64_t total_rows = T.row_end[T.count - 1];
    const bool unit = T.unit != 0;
    double sum = 0.0;
    float top = 0.0f;
    int t = 0;
    for (int64_t g = blockIdx.x; g < total_rows; g += gridDim.x) {
        while (g >= T.row_end[t]) ++t;
        const int64_t r = g - (t ? T.row_end[t - 1] : 0);
        const int64_t idx = (r * NT + tid) * kLaneW;
        const bool ok = idx < T.n[t];
        float v[kLaneW], x[kLaneW], gmax;
        widen(ok ? load_raw<DT>(T.ptr[t], idx) : zero_raw<DT>(), v);
        const float m = block_constant<I, SIGNED>(v, gmax, &s_wide);
        const bool safe = row_is_safe(gmax, ok);
        normalise16<true>(v, m, safe && DT::code == BF16::code, x);
        if (!ok) continue;
        top = fmaxf(top, gmax);
        const float am = unit ? 1.0f : fabsf(m);
        double part[2] = {0.0, 0.0};
#pragma unroll
        for (int k = 0; k < kLaneW; ++k) {  // (m x)^2: with the x of the other sums the error is free of cancellation
            const double e = (double)x[k] * (double)am;
            part[k & 1] = fma(e, e, part[k & 1]);
        }
        sum += part[0] + part[1];
        // 32-byte aligned: the tensors of a launch are whole blocks, of 32 weights at least, and so is what lies before them
        float2* dst = items + s_item0[t] + idx;
        const uint32_t payload = __float_as_uint(am);
#pragma unroll
        for (int k = 0; k < kLaneW; k += 4)
            st_256(dst + k, Raw8{{__float_as_uint(x[k]), payload, __float_as_uint(x[k + 1]), payload, __float_as_uint(x[k + 2]), payload,
                                  __float_as_uint(x[k + 3]), payload}});
    }
    uint32_t bits = __float_as_uint(top);
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        sum += __shfl_xor_sync(kFull, sum, off);
        bits = max(bits, __shfl_xor_sync(kFull, bits, off));
    }
    if (lane == 0) {
        s_sum[warp] = sum;
        s_max[warp] = bits;
    }
    __syncthreads();
    if (tid == 0) {
        double a = 0.0;
        for (int k = 0; k < NT / 32; ++k) {
            a += s_sum[k];
            bits = max(bits, s_max[k]);
        }
        w2[blockIdx.x] = T.accumulate ? w2[blockIdx.x] + a : a;
        tops[blockIdx.x] = T.accumulate ? max(tops[blockIdx.x], bits) : bits;  // non-negative floats order like their bits
        if (!T.accumulate && blockIdx.x == 0) {
            head[0] = n;
            head[4] = 0u;
            w2[kSortParts - 1] = 0.0;  // the short last blocks'
            tops[kSortParts - 1] = 0u;
        }
    }
}

// The short last blocks, after all whole blocks in the sample array: one CTA.  `alone`: there are no whole blocks.
template <class DT, bool SIGNED>
__global__ void __launch_bounds__(kEmTailThreads)
sort_tail_kernel(const EmTails Q, uint32_t at, const uint32_t n, const bool alone, float2* __restrict__ items,
                 uint32_t* __restrict__ head, double* __restrict__ w2, uint32_t* __restrict__ tops)
{
    if (!after_previous()) return;
    __shared__ float s_w[4096];
    __shared__ unsigned long long s_red[kEmTailThreads / 32];
    __shared__ double s_sum[kEmTailThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double sum = 0.0;
    uint32_t top = 0u;
    for (int q = 0; q < Q.count; ++q) {
        const int len = Q.len[q];
        const float m = load_short_block<DT, SIGNED>(Q.ptr[q], len, s_w, s_red);
        top = max(top, __float_as_uint(fabsf(m)));
        for (int i = tid; i < len; i += kEmTailThreads) {
            const float x = normalise(s_w[i], m), am = Q.unit ? 1.0f : fabsf(m);
            const double e = (double)x * (double)am;
            sum = fma(e, e, sum);
            items[at + i] = make_float2(x, am);
        }
        at += (uint32_t)len;
        __syncthreads();  // before the next block overwrites s_w
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(kFull, sum, off);
    if (lane == 0) s_sum[warp] = sum;
    __syncthreads();
    if (tid == 0) {
        double a = 0.0;
        for (int k = 0; k < kEmTailThreads / 32; ++k) a += s_sum[k];
        w2[kSortParts - 1] = Q.accumulate ? w2[kSortParts - 1] + a : a;
        tops[kSortParts - 1] = Q.accumulate ? max(tops[kSortParts - 1], top) : top;
        if (alone && !Q.accumulate) {
            head[0] = n;
            head[4] = 0u;
        }
    }
    if (alone && !Q.accumulate) {
        for (int k = tid; k < kSortParts - 1; k += kEmTailThreads) {
            w2[k] = 0.0;
            tops[k] = 0u;
        }
    }
}

// ---------------------------------------------------------------- ordering passes

// Samples [lo, hi) of CTA c.
__device__ __forceinline__ void sort_part(uint32_t n, uint32_t c, uint32_t& lo, uint32_t& hi)
{
    const uint32_t len = (n + kSortGrid - 1) / kSortGrid;
    lo = min(n, c * len);
    hi = min(n, lo + len);
}

// tops (the second pass): the largest constants of the samples' CTAs, of which one CTA makes one.
template <int SHIFT>
__global__ void __launch_bounds__(kSortThreads)
sort_count_kernel(const float2* __restrict__ in, uint32_t* __restrict__ head, uint32_t* __restrict__ counts, const uint32_t* __restrict__ tops)
{
    if (!after_previous()) return;
    if (SHIFT && blockIdx.x == 0 && threadIdx.x < 32) {
        uint32_t top = 0u;
#pragma unroll
        for (int k = 0; k < kSortParts; k += 32) top = max(top, k + threadIdx.x < kSortParts ? tops[k + threadIdx.x] : 0u);
        top = __reduce_max_sync(kFull, top);
        if (threadIdx.x == 0) head[1] = top;
    }
    __shared__ uint32_t s_hist[4][256];  // a copy per eight warps: fewer collisions on crowded digits
    const int tid = threadIdx.x;
    (&s_hist[0][0])[tid] = 0u;
    __syncthreads();
    uint32_t lo, hi;
    sort_part(*head, blockIdx.x, lo, hi);
    for (uint32_t i = lo + tid; i < hi; i += kSortThreads)
        atomicAdd(&s_hist[tid >> 8][(sort_bin(in[i].x) >> SHIFT) & 255], 1u);
    __syncthreads();
    if (tid < 256) counts[blockIdx.x * 256 + tid] = s_hist[0][tid] + s_hist[1][tid] + s_hist[2][tid] + s_hist[3][tid];
}

// Ranks of a warp's PER x 32 items by a digit of eight bits: item k of a lane goes behind rank[k] others of its digit
// (those of smaller k, and of lower lanes at the same k).  cnt[256], zero before, ends as the warp's histogram.
template <int PER, class Digit, class Valid>
__device__ __forceinline__ void rank_in_warp(uint32_t* cnt, int lane, Digit digit, Valid valid, uint32_t (&rank)[PER])
{
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const bool ok = valid(k);
        const uint32_t d = digit(k);
        unsigned peers = __ballot_sync(kFull, ok);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const unsigned with = __ballot_sync(kFull, (d >> b) & 1u);
            peers &= ((d >> b) & 1u) ? with : ~with;
        }
        const uint32_t old = cnt[d];
        __syncwarp();
        if (ok && lane == __ffs(peers) - 1) cnt[d] = old + __popc(peers);
        __syncwarp();
        rank[k] = old + __popc(peers & ((1u << lane) - 1u));
    }
}

// Stable scatter by one digit.  A sample goes to: samples with a smaller digit + samples of the same
// digit in earlier CTAs + in earlier tiles of this CTA + in earlier warps of the tile + earlier in the
// warp (each warp owns 256 consecutive samples of a tile, 32 at a time).  STAGED: a tile is put in order in shared memory first,
// so that neighbouring lanes store neighbouring samples, not 32 cache lines a store.  (A digit's counts per warp go back to shared memory
// as they are added up: kept in registers over the barriers they spilled 90 bytes.)
constexpr int kScatterSmem = kSortTile * 8;
// Fits over so many samples, one per weight, stage them.  Fewer fill a tile in part, and the barriers cost what the stores save.  Staged and
// not, 50 iterations: 2^18 weights 127.8 and 126.9 us, 2^19 129.4 and 130.7, 3 * 2^18 135.0 and 138.4, 2^20 139.9 and 145.6, 2^23 384 and
// 459, 2^24 702 and 890.
constexpr int64_t kStagedMin = 1 << 19;
template <int SHIFT, bool STAGED>
__global__ void __launch_bounds__(kSortThreads)
sort_scatter_kernel(const float2* __restrict__ in, const uint32_t* __restrict__ head, const uint32_t* __restrict__ counts,
                    float2* __restrict__ out)
{
    if (!after_previous()) return;
    extern __shared__ __align__(16) unsigned char s_window[];
    float2* const s_item = reinterpret_cast<float2*>(s_window);  // [kSortTile] STAGED
    __shared__ uint32_t s_cnt[32][256];
    __shared__ uint32_t s_base[256], s_warp[8];
    // of a digit: the place of its first sample in the tile, and where that goes less this place
    __shared__ uint32_t s_first[256], s_place[256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t lo, hi;
    sort_part(*head, blockIdx.x, lo, hi);
    {
        const int seg = tid >> 8, d = tid & 255;
        uint32_t before = 0u, all = 0u;
#pragma unroll
        for (int k = 0; k < (kSortGrid + 3) / 4; ++k) {  // all loads at once: one round trip to L2
            const int c = seg + 4 * k;
            const uint32_t v = c < kSortGrid ? __ldcg(counts + c * 256 + d) : 0u;
            all += v;
            before += (c < (int)blockIdx.x) ? v : 0u;
        }
        s_cnt[seg][d] = before;
        s_cnt[4 + seg][d] = all;
        __syncthreads();
        uint32_t mine = 0u, incl = 0u;
        if (tid < 256) {
            mine = s_cnt[4][tid] + s_cnt[5][tid] + s_cnt[6][tid] + s_cnt[7][tid];
            incl = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, incl, off);
                if (lane >= off) incl += t;
            }
            if (lane == 31) s_warp[warp] = incl;
        }
        __syncthreads();
        if (tid < 256) {
            for (int k = 0; k < warp; ++k) incl += s_warp[k];
            s_base[tid] = incl - mine + s_cnt[0][tid] + s_cnt[1][tid] + s_cnt[2][tid] + s_cnt[3][tid];
        }
        __syncthreads();
    }
    for (uint32_t t0 = lo; t0 < hi; t0 += kSortTile) {
        float2 item[kSortPerThread];
        uint32_t rank[kSortPerThread];
        const uint32_t i0 = t0 + warp * (32 * kSortPerThread) + lane;
#pragma unroll
        for (int k = 0; k < kSortPerThread; ++k) {
            const uint32_t i = i0 + 32 * k;
            item[k] = (i < hi) ? in[i] : make_float2(0.0f, 0.0f);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) s_cnt[warp][lane + 32 * k] = 0u;
        __syncwarp();
        rank_in_warp<kSortPerThread>(s_cnt[warp], lane, [&](int k) { return ((uint32_t)sort_bin(item[k].x) >> SHIFT) & 255u; },
                                     [&](int k) { return i0 + 32 * k < hi; }, rank);
        if constexpr (STAGED) {
            __syncthreads();
            uint32_t mine = 0u, incl = 0u;
            if (tid < 256) {
#pragma unroll 8
                for (int w = 0; w < 32; ++w) {
                    const uint32_t c = s_cnt[w][tid];
                    s_cnt[w][tid] = mine;
                    mine += c;
                }
                incl = mine;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const uint32_t t = __shfl_up_sync(kFull, incl, off);
                    if (lane >= off) incl += t;
                }
                if (lane == 31) s_warp[warp] = incl;
            }
            __syncthreads();
            if (tid < 256) {
                for (int k = 0; k < warp; ++k) incl += s_warp[k];
                const uint32_t first = incl - mine;
                s_first[tid] = first;
                s_place[tid] = s_base[tid] - first;
                s_base[tid] += mine;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kSortPerThread; ++k) {
                const uint32_t d = ((uint32_t)sort_bin(item[k].x) >> SHIFT) & 255u;
                if (i0 + 32 * k < hi) s_item[s_first[d] + s_cnt[warp][d] + rank[k]] = item[k];
            }
            __syncthreads();
            const uint32_t len = min((uint32_t)kSortTile, hi - t0);
#pragma unroll
            for (int k = 0; k < kSortPerThread; ++k) {
                const uint32_t j = tid + k * kSortThreads;
                if (j < len) {
                    const float2 it = s_item[j];
                    out[s_place[((uint32_t)sort_bin(it.x) >> SHIFT) & 255u] + j] = it;
                }
            }
        } else {
            __syncthreads();
            if (tid < 256) {
                uint32_t c[32], run = s_base[tid];
#pragma unroll
                for (int w = 0; w < 32; ++w) c[w] = s_cnt[w][tid];
#pragma unroll
                for (int w = 0; w < 32; ++w) {
                    s_cnt[w][tid] = run;
                    run += c[w];
                }
                s_base[tid] = run;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kSortPerThread; ++k) {
                const uint32_t d = ((uint32_t)sort_bin(item[k].x) >> SHIFT) & 255u;
                if (i0 + 32 * k < hi) out[s_cnt[warp][d] + rank[k]] = item[k];
            }
        }
        __syncthreads();  // s_cnt is cleared for the next tile
    }
}

// ---------------------------------------------------------------- sums of the bins

// What a sample contributes; its payload is |m|.
template <bool MAE>
struct SampleWeight {
    uint32_t max_bits;
    bool unit;
    __device__ __forceinline__ void operator()(float2 it, double& s, unsigned long long& a) const
    {
        a = 0ull;
        const double m = (double)it.y;
        s = MAE ? m : m * m;
        if (MAE) a = unit ? 1ull : (unsigned long long)sort_fixed_weight(it.y, max_bits);
    }
};

template <bool MAE>
__device__ __forceinline__ void sums_reduce(SortSums& t)
{
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        t.s += __shfl_xor_sync(kFull, t.s, off);
        t.sx += __shfl_xor_sync(kFull, t.sx, off);
        if (MAE) t.a += __shfl_xor_sync(kFull, t.a, off);
    }
}
__device__ __forceinline__ void sums_add(SortSums& t, const SortSums& v)
{
    t.s += v.s;
    t.sx += v.sx;
    t.a += v.a;
}

// ---------------------------------------------------------------- crowded bins
//
// The bins are fine where normalised weights of model layers lie, but data can put any number of samples into one:
// few distinct values (weights that have been quantised before) or a narrow range of x.  Looked through by a warp, such bins
// made a fit of 2^24 weights of sixteen levels 4.4 ms long (MSE) and one of medians 100 ms, whatever streaming it takes (0.4
// and 5.2 ms for 8 iterations).  So the windows that hold part of a crowded bin are put in full order, with running sums
// beside them; what a threshold takes of the bin, and where its weight reaches a half, is then found by bisection in every
// window, a lane each: 1.1 and 1.3 ms, of which 0.8 are the ordering that other data takes as well.  An iteration now costs
// at most a few bisections (14 steps of an access to L2 each) per 2^20 samples of a crowded bin, and median step.
// Other data pays for a launch that finds nothing to do (two for medians) and for the test of the flag: 12 iterations over 2^20
// weights 92.9 -> 97.0 us (50 of them 140.5 -> 137.6, for no known reason), 12 of medians 119.5 -> 124.9.

// One CTA per window of kSortWindow samples: four stable passes of eight bits by the key of x in shared memory, then the
// running sums (exclusive within the window, every fourth sample).
struct WindowScratch {
    float2 item[kSortWindow];
    uint32_t cnt[kSortThreads / 32][256];
    uint32_t warp[8];
    SortSums sum[kSortThreads / 32];
};
template <bool MAE>
__global__ void __launch_bounds__(kSortThreads)
sort_windows_kernel(const SortWs W, SampleWeight<MAE> weight)
{
    if (!after_previous()) return;
    if (W.n_items[4] == 0u) return;
    constexpr int NT = kSortThreads, PER = kSortWindow / NT, NW = NT / 32;
    extern __shared__ __align__(16) unsigned char s_window[];
    WindowScratch& S = *reinterpret_cast<WindowScratch*>(s_window);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n = W.n_items[0];
    weight.max_bits = W.n_items[1];
    for (uint32_t lo = blockIdx.x * kSortWindow; lo < n; lo += gridDim.x * kSortWindow) {
        const uint32_t len = min(kSortWindow, n - lo);
        bool crowded = false;
        for (uint32_t i = tid; i < len; i += NT) {
            const float2 it = W.b[lo + i];
            const int b = sort_bin(it.x);
            crowded = crowded || (!one_value_bin(b) && W.start[b + 1] - W.start[b] > kSortCrowd);
            S.item[i] = it;
        }
        if (!__syncthreads_or(crowded)) continue;
        const uint32_t i0 = warp * (32 * PER) + lane;
        for (int shift = 0; shift < 32; shift += 8) {
            float2 item[PER];
            uint32_t rank[PER];
#pragma unroll
            for (int k = 0; k < PER; ++k) item[k] = (i0 + 32 * k < len) ? S.item[i0 + 32 * k] : make_float2(0.0f, 0.0f);
#pragma unroll
            for (int k = 0; k < 8; ++k) S.cnt[warp][lane + 32 * k] = 0u;
            __syncwarp();
            rank_in_warp<PER>(S.cnt[warp], lane, [&](int k) { return (sort_key(item[k].x) >> shift) & 255u; },
                              [&](int k) { return i0 + 32 * k < len; }, rank);
            __syncthreads();
            uint32_t mine = 0u, incl = 0u;  // samples of smaller digits, then those of the same digit in earlier warps
            if (tid < 256) {
                for (int w = 0; w < NW; ++w) mine += S.cnt[w][tid];
                incl = mine;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const uint32_t t = __shfl_up_sync(kFull, incl, off);
                    if (lane >= off) incl += t;
                }
                if (lane == 31) S.warp[warp] = incl;
            }
            __syncthreads();
            if (tid < 256) {
                for (int k = 0; k < warp; ++k) incl += S.warp[k];
                uint32_t run = incl - mine;
                for (int w = 0; w < NW; ++w) {
                    const uint32_t c = S.cnt[w][tid];
                    S.cnt[w][tid] = run;
                    run += c;
                }
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < PER; ++k)
                if (i0 + 32 * k < len) S.item[S.cnt[warp][(sort_key(item[k].x) >> shift) & 255u] + rank[k]] = item[k];
            __syncthreads();
        }
        for (uint32_t i = tid; i < len; i += NT) W.b[lo + i] = S.item[i];
        // a thread adds up PER samples in a row
        auto add = [&](SortSums& t, uint32_t i) {
            if (i >= len) return;
            const float2 it = S.item[i];
            SortSums v;
            weight(it, v.s, v.a);
            v.sx = v.s * (double)it.x;
            sums_add(t, v);
        };
        SortSums incl{0.0, 0.0, 0ull};
        for (int k = 0; k < PER; ++k) add(incl, tid * PER + k);
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const SortSums u{__shfl_up_sync(kFull, incl.s, off), __shfl_up_sync(kFull, incl.sx, off),
                             MAE ? __shfl_up_sync(kFull, incl.a, off) : 0ull};
            if (lane >= off) sums_add(incl, u);
        }
        if (lane == 31) S.sum[warp] = incl;
        SortSums run{__shfl_up_sync(kFull, incl.s, 1), __shfl_up_sync(kFull, incl.sx, 1), MAE ? __shfl_up_sync(kFull, incl.a, 1) : 0ull};
        if (lane == 0) run = SortSums{0.0, 0.0, 0ull};
        __syncthreads();
        for (int k = 0; k < warp; ++k) sums_add(run, S.sum[k]);
        for (int k = 0; k < PER; ++k) {
            const uint32_t i = tid * PER + k;
            if (k % 4 == 0 && i < len) W.before[(lo + i) / 4] = run;
            add(run, i);
        }
        __syncthreads();  // the next window overwrites the samples
    }
}

// Windows that a warp looks into at once, per lane: as many independent bisections in flight.
constexpr int kWindowsPerLane = 4;

// Sums of the samples of a window in front of position i (`first`: the window's first sample).
template <bool MAE>
__device__ __forceinline__ SortSums sums_before(const SortWs& W, const SampleWeight<MAE>& weight, uint32_t first, uint32_t i)
{
    SortSums t{0.0, 0.0, 0ull};
    if (i <= first) return t;
    const uint32_t q = (i - 1) / 4;
    t = W.before[q];
    for (uint32_t j = 4 * q; j < i; ++j) {
        const float2 it = W.b[j];
        double s;
        unsigned long long a;
        weight(it, s, a);
        t.s += s;
        t.sx += s * (double)it.x;
        t.a += a;
    }
    return t;
}

// This lane's share of the samples of a crowded bin, from ... to - 1, with p <= x < q; the warp's lanes together have all.  (Nothing is looked
// for where p is minus infinity, as it is for what lies below a threshold: 2^20 weights in two bins, squared error, 16.2 -> 11.1 us an iteration.)
template <bool MAE>
__device__ __noinline__ void crowded_sums(const SortWs& W, const SampleWeight<MAE>& weight, uint32_t from, uint32_t to, float p,
                                          float q, SortSums& t)
{
    constexpr int U = kWindowsPerLane;
    const uint32_t last = (to - 1) / kSortWindow;
    const bool cut = p > -__int_as_float(0x7f800000);
    for (uint32_t w0 = from / kSortWindow + (threadIdx.x & 31); w0 <= last; w0 += 32 * U) {
        uint32_t lo[U], hi[U], at_p[U], at_q[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t w = w0 + 32 * u;
            lo[u] = max(from, w * kSortWindow);
            hi[u] = min(to, (w + 1) * kSortWindow);
            if (w > last) lo[u] = hi[u] = to;
            at_p[u] = at_q[u] = lo[u];
        }
        for (uint32_t step = kSortWindow; step; step >>= 1) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (cut && at_p[u] + step <= hi[u] && W.b[at_p[u] + step - 1].x < p) at_p[u] += step;
                if (at_q[u] + step <= hi[u] && W.b[at_q[u] + step - 1].x < q) at_q[u] += step;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (at_q[u] <= at_p[u]) continue;
            const uint32_t first = (lo[u] / kSortWindow) * kSortWindow;
            const SortSums a = sums_before<MAE>(W, weight, first, at_p[u]), b = sums_before<MAE>(W, weight, first, at_q[u]);
            t.s += b.s - a.s;
            t.sx += b.sx - a.sx;
            t.a += b.a - a.a;
        }
    }
}

// First samples of all bins: a thread each, by bisection, in CTAs of their own beside those that form the sums.  (Written by the sums' warps as they
// come to the ends of runs, the gaps between few samples are long chains of stores: 1000 weights, 12 iterations, 89 us and 70 this way,
// 2^14 81.7 and 75.4, 2^20 93.9 and 93.4, medians of 2^24 710 and 701; with a launch before, 80, 81, 99.6 and 969 for the fit as it was then.
// By halves, quarters and eighths 2^18 82.5, 80.9 and 81.3, 2^24 699, 701 and 705.)
//
// Sums: one warp per kSortChunk ordered samples, 32 at a time: a segmented scan over the runs of equal bins.
// A run that lies inside the chunk is a bin's sum; parts of runs that cross the chunk's edges go to
// lead / trail and are put together by sort_group_kernel.  The work is even whatever the distribution (the bins
// of x = +-1 hold 1 / I of the data; a bin of small data is mostly empty).
constexpr int kStartCtas = kSortBins / 256;
template <bool MAE>
__global__ void __launch_bounds__(256)
sort_sums_kernel(const SortWs W, SampleWeight<MAE> weight)
{
    if (!after_previous()) return;
    constexpr int STEPS = kSortChunk / 32, kNone = 1 << 20;
    const uint32_t n = W.n_items[0];
    if (blockIdx.x < kStartCtas) {
        const int bin = (int)(blockIdx.x * 256 + threadIdx.x);
        uint32_t from = 0u, to = n;
        while (from < to) {  // quarters: half the dependent loads that halves take
            const uint32_t part = (to - from + 3u) / 4u;
            uint32_t in_front = 0u;
#pragma unroll
            for (int u = 1; u < 4; ++u) {
                const uint32_t last = from + u * part - 1u;
                const int at = sort_bin(W.b[min(last, to - 1u)].x);
                in_front += (last < to && at < bin) ? 1u : 0u;
            }
            from += in_front * part;
            if (in_front < 3u) to = min(to, from + part - 1u);
        }
        W.start[bin] = from;
        if (bin == 0) W.start[kSortBins] = n;
        return;
    }
    weight.max_bits = W.n_items[1];
    const int lane = threadIdx.x & 31;
    const uint32_t warps = (gridDim.x - kStartCtas) * 8u;
    for (uint32_t c = (blockIdx.x - kStartCtas) * 8u + (threadIdx.x >> 5); (uint64_t)c * kSortChunk < n; c += warps) {
        const uint32_t lo = c * kSortChunk, hi = min(n, lo + kSortChunk);
        float2 it[STEPS];
        SortSums v[STEPS];
        int key[STEPS];
#pragma unroll
        for (int k = 0; k < STEPS; ++k) {
            const uint32_t i = lo + 32 * k + lane;
            it[k] = (i < hi) ? W.b[i] : make_float2(0.0f, 0.0f);
        }
        const int before = lo ? sort_bin(W.b[lo - 1].x) : -1, behind = (hi < n) ? sort_bin(W.b[hi].x) : kNone;
#pragma unroll
        for (int k = 0; k < STEPS; ++k) {
            const uint32_t i = lo + 32 * k + lane;
            v[k] = SortSums{0.0, 0.0, 0ull};
            key[k] = kNone;
            if (i < hi) {
                key[k] = sort_bin(it[k].x);
                weight(it[k], v[k].s, v[k].a);
                v[k].sx = v[k].s * (double)it[k].x;
            }
        }
        SortSums open{0.0, 0.0, 0ull};  // the run that reaches the end of the steps so far (the same in all lanes)
        int open_key = before;
        bool early = true;              // it began before this chunk
#pragma unroll
        for (int k = 0; k < STEPS; ++k) {
            int left = __shfl_up_sync(kFull, key[k], 1);
            if (lane == 0) left = open_key;
            const unsigned heads = __ballot_sync(kFull, key[k] != left);
            if ((heads & 1u) && k > 0 && lane == 0 && open_key != kNone) (early ? W.lead[c] : W.bin[open_key]) = open;
            const unsigned upto = heads & ((2u << lane) - 1u);
            const int from = upto ? 31 - __clz(upto) : 0;
            SortSums t = v[k];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const double s = __shfl_up_sync(kFull, t.s, off), sx = __shfl_up_sync(kFull, t.sx, off);
                const unsigned long long a = MAE ? __shfl_up_sync(kFull, t.a, off) : 0ull;
                if (lane >= from + off) {
                    t.s += s;
                    t.sx += sx;
                    t.a += a;
                }
            }
            if (!upto) sums_add(t, open);
            if (lane < 31 && ((heads >> (lane + 1)) & 1u) && key[k] != kNone) ((early && !upto) ? W.lead[c] : W.bin[key[k]]) = t;
            open.s = __shfl_sync(kFull, t.s, 31);
            open.sx = __shfl_sync(kFull, t.sx, 31);
            if (MAE) open.a = __shfl_sync(kFull, t.a, 31);
            open_key = __shfl_sync(kFull, key[k], 31);
            early = early && heads == 0u;
        }
        if (lane == 0 && open_key != kNone) (early ? W.lead[c] : open_key == behind ? W.trail[c] : W.bin[open_key]) = open;
    }
}

// One warp per group of 32 bins: empty bins are cleared, bins that cross chunks put together (in the
// order of the chunks), and the sums of the group, of the bins in front of each formed.
// Bound by the latency of its loads: with all crossing bins put together one after the other by the whole warp
// it took 14.6 us for 2^20 samples, 3.7 with those of up to kSortFew chunks a lane each.
// Between 4 and 64 chunks as the line the fits of 2^18 to 2^24 weights differ by less than 2 us; at 64 those of 2^18 are 1.5 slower.
constexpr uint32_t kSortFew = 16;
// A bin of very many chunks (crowded, or one of a single value: the zeros of sparse data) is put together by the whole CTA:
// 2^24 samples within a tenth of a binade took 1910 us by a warp; 2^20 took 132, 32 this way.
constexpr uint32_t kSortMany = 128;
template <bool MAE>
__global__ void __launch_bounds__(256)
sort_group_kernel(const SortWs W)
{
    if (!after_previous()) return;
    const int lane = threadIdx.x & 31, g = blockIdx.x * 8 + (threadIdx.x >> 5), b = g * kSortGroup + lane;
    const uint32_t s = W.start[b], e = W.start[b + 1];
    SortSums t{0.0, 0.0, 0ull};
    const uint32_t c0 = s / kSortChunk, c1 = (e > s) ? (e - 1) / kSortChunk : c0;
    if (e > s && c0 == c1) t = W.bin[b];
    if (e > s && e - s > kSortCrowd && !one_value_bin(b)) W.n_items[4] = 1u;
    // a bin of a few chunks by its lane, the lanes side by side; a longer one by the warp
    const bool few = e > s && c0 != c1 && c1 - c0 <= kSortFew;
    if (few) {
        t = W.trail[c0];
#pragma unroll 4
        for (uint32_t c = c0 + 1; c <= c1; ++c) sums_add(t, W.lead[c]);
    }
    const bool many = e > s && c1 - c0 > kSortMany;
    unsigned spans = __ballot_sync(kFull, e > s && c0 != c1 && !few && !many);
    while (spans) {
        const int who = __ffs(spans) - 1;
        spans &= spans - 1u;
        const uint32_t f = __shfl_sync(kFull, c0, who), l = __shfl_sync(kFull, c1, who);
        SortSums u{0.0, 0.0, 0ull};
#pragma unroll 4
        for (uint32_t c = f + lane; c <= l; c += 32) sums_add(u, (c == f) ? W.trail[c] : W.lead[c]);
        __syncwarp();
        sums_reduce<MAE>(u);
        if (lane == who) t = u;
    }
    __shared__ uint32_t s_first[256], s_last[256], s_many[8];
    __shared__ SortSums s_part[8];
    if (__syncthreads_or(many)) {
        const unsigned wide = __ballot_sync(kFull, many);
        s_first[threadIdx.x] = c0;
        s_last[threadIdx.x] = c1;
        if (lane == 0) s_many[threadIdx.x >> 5] = wide;
        __syncthreads();
        for (int w = 0; w < 8; ++w) {
            for (unsigned left = s_many[w]; left; left &= left - 1u) {
                const int who = w * 32 + __ffs(left) - 1;
                const uint32_t f = s_first[who], l = s_last[who];
                SortSums u{0.0, 0.0, 0ull};
#pragma unroll 4
                for (uint32_t c = f + threadIdx.x; c <= l; c += 256) sums_add(u, (c == f) ? W.trail[c] : W.lead[c]);
                __syncwarp();
                sums_reduce<MAE>(u);
                if (lane == 0) s_part[threadIdx.x >> 5] = u;
                __syncthreads();
                if ((int)threadIdx.x == who)
                    for (int k = 0; k < 8; ++k) sums_add(t, s_part[k]);
                __syncthreads();
            }
        }
    }
    W.bin[b] = t;
    SortSums up = t;  // this bin and those in front of it
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const SortSums u{__shfl_up_sync(kFull, up.s, o), __shfl_up_sync(kFull, up.sx, o), MAE ? __shfl_up_sync(kFull, up.a, o) : 0ull};
        if (lane >= o) sums_add(up, u);
    }
    if (lane == 0) W.pre[b] = SortSums{0.0, 0.0, 0ull};
    if (lane < 31) W.pre[b + 1] = up;
    else W.group[g] = up;
    const uint32_t first = __shfl_sync(kFull, s, 0);
    W.off[b] = (uint16_t)min(s - first, kFarBin);
    if (lane == 0) W.first[g] = first;
    if (b == kSortBins - 1) W.first[kSortGroups] = e;
}

// ---------------------------------------------------------------- all iterations, squared error
//
// What lies below a threshold (em_fit.cuh): the groups in front of its bin's, in shared memory, the bins of the group in front of it
// (one load), and the samples of its bin.  The first samples of all bins are in shared memory (16 bits beside the group's first),
// which leaves one access to L2 in the chain: 1.14 us an iteration over 2^20 fp32 weights (1.60 with cuts found by one warp, whole
// groups added up between them and three barriers), 3.5 over 2^24 (3.9).  Of its 2200 cycles the bin takes 130, its first sample 220,
// the samples 430 or 820, by where in L2 they are, their reduction 230, the barrier and what it waits for 200, the differences 300
// and the quotients with the test of the sums 330.  (The next iteration's samples requested ahead, by the last steps of the
// threshold: 1 to 13 % slower.)
constexpr int kMseLow = (kSortGroups + 1) * 16;      // shared memory: sums of the groups in front, high and low halves,
constexpr int kMseOff = 2 * kMseLow;                 // first samples of the bins,
constexpr int kMseFirst = kMseOff + kSortBins * 2 + 16;  // (and the end) of the groups
constexpr int kMseSmem = kMseFirst + (kSortGroups + 1) * 4;

// The first samples of all bins, into shared memory: 16 bits beside the first of the bin's group (or kFarBin).  Asynchronous.
__device__ __forceinline__ void copy_starts(const SortWs& W, uint16_t* s_off, uint32_t* s_first)
{
    auto copy = [](void* to, const void* from, auto bytes) {
        constexpr int B = decltype(bytes)::value;
        const uint32_t a = (uint32_t)__cvta_generic_to_shared(to);
        if constexpr (B == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(from) : "memory");
        else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(a), "l"(from) : "memory");
    };
    for (int k = threadIdx.x; k < kSortBins / 8; k += blockDim.x) copy(s_off + 8 * k, W.off + 8 * k, std::integral_constant<int, 16>{});
    for (int k = threadIdx.x; k <= kSortGroups; k += blockDim.x) copy(s_first + k, W.first + k, std::integral_constant<int, 4>{});
}

// Sums of the samples with p <= x < q, by a warp; the result is the same in all lanes.
template <bool CROWDED>
__device__ __noinline__ double2 region_sums(const SortWs& W, float p, float q)
{
    const int lane = threadIdx.x & 31;
    const float inf = __int_as_float(0x7f800000);
    const int bp = (p == -inf) ? -1 : sort_bin(p), bq = (q == inf) ? kSortBins : sort_bin(q);
    const int b0 = bp + 1, b1 = max(bq, b0);  // bins strictly inside, as whole groups with up to 31 single bins on either side
    const int g0 = (b0 + kSortGroup - 1) / kSortGroup, g1 = b1 / kSortGroup;
    SortSums t{0.0, 0.0, 0ull};
    auto whole = [&](const SortSums* v) { t.s += __ldg(&v->s), t.sx += __ldg(&v->sx); };
    if (b0 + lane < min(b1, g0 * kSortGroup)) whole(W.bin + b0 + lane);
    for (int g = g0 + lane; g < g1; g += 32) whole(W.group + g);
    if (g1 >= g0 && g1 * kSortGroup + lane < b1) whole(W.bin + g1 * kSortGroup + lane);
    auto cut = [&](int b) {
        if (one_value_bin(b)) {  // in or out as a whole
            if (lane == 0 && value_of_bin(b) >= p && value_of_bin(b) < q) whole(W.bin + b);
            return;
        }
        const uint32_t from = __ldg(W.start + b), to = __ldg(W.start + b + 1);
        if (CROWDED && to - from > kSortCrowd) {
            crowded_sums<false>(W, SampleWeight<false>{}, from, to, p, q, t);
            return;
        }
        for (uint32_t i = from + lane; i < to; i += 32) {
            const float2 it = __ldg(W.b + i);
            if (!(it.x >= p && it.x < q)) continue;
            const double m = (double)it.y, s = m * m;
            t.s += s;
            t.sx += s * (double)it.x;
        }
        __syncwarp();
    };
    if (bp >= 0) cut(bp);
    if (bq < kSortBins && bq != bp) cut(bq);
    __syncwarp();
    sums_reduce<false>(t);
    return make_double2(t.s, t.sx);
}

// CROWDED: a copy of the loop that also knows crowded bins.  Apart, because the calls in it cost the other one registers.
template <bool CROWDED>
__device__ __forceinline__ void fit_mse(const SortWs& W, const SortFit& F)
{
    extern __shared__ __align__(16) unsigned char s_fit[];
    double2* const s_high = reinterpret_cast<double2*>(s_fit);           // {s, sx} of the groups in front of a group
    double2* const s_low = reinterpret_cast<double2*>(s_fit + kMseLow);
    uint16_t* const s_off = reinterpret_cast<uint16_t*>(s_fit + kMseOff);
    uint32_t* const s_first = reinterpret_cast<uint32_t*>(s_fit + kMseFirst);
    // What lies below threshold k - 1: whole groups (high, low), the rest.  Entry 0: nothing, entry 16: everything.  Two sets, used
    // in turn.
    __shared__ double2 s_below[2][3][kLevels + 1];
    __shared__ float2 s_cut[2][kLevels + 1];  // the threshold, and how many samples lie below it
    __shared__ float s_level[2][kLevels];
    __shared__ int s_stop;  // the iteration behind whose barrier all leave
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float inf = __int_as_float(0x7f800000);
    if (tid == 0) s_stop = 0x7fffffff, s_off[kSortBins] = 0u;
    copy_starts(W, s_off, s_first);
    // running sums of the groups, four to a thread
    {
        constexpr int PER = kSortGroups / kFitThreads;
        TwoSum s[PER], x[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const SortSums* g = W.group + tid * PER + k;
            s[k] = TwoSum{g->s, 0.0}, x[k] = TwoSum{g->sx, 0.0};
        }
        static_assert(PER == 4, "a tree of two levels");
        TwoSum ts = two_add(two_add(s[0], s[1]), two_add(s[2], s[3])), tx = two_add(two_add(x[0], x[1]), two_add(x[2], x[3]));
        auto scan = [&](TwoSum& as, TwoSum& ax) {  // inclusive, over the warp
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const TwoSum us = two_shfl_up(as, off), ux = two_shfl_up(ax, off);
                if (lane >= off) as = two_add(us, as), ax = two_add(ux, ax);
            }
        };
        scan(ts, tx);
        // (the room of the loop's sums serves for the warps' totals)
        if (lane == 31) s_below[0][0][warp] = make_double2(ts.h, tx.h), s_below[0][1][warp] = make_double2(ts.l, tx.l);
        __syncthreads();
        TwoSum ws{0.0, 0.0}, wx = ws;
        if (lane < warp) {
            const double2 h = s_below[0][0][lane], l = s_below[0][1][lane];
            ws = TwoSum{h.x, l.x}, wx = TwoSum{h.y, l.y};
        }
        scan(ws, wx);  // lane 31: all warps in front of this one
        TwoSum rs = two_shfl_up(ts, 1), rx = two_shfl_up(tx, 1);
        if (lane == 0) rs = rx = TwoSum{0.0, 0.0};
        rs = two_add(TwoSum{__shfl_sync(kFull, ws.h, 31), __shfl_sync(kFull, ws.l, 31)}, rs);
        rx = two_add(TwoSum{__shfl_sync(kFull, wx.h, 31), __shfl_sync(kFull, wx.l, 31)}, rx);
#pragma unroll
        for (int k = 0; k <= PER; ++k) {
            if (k == PER && tid < kFitThreads - 1) break;  // behind the last group: everything
            s_high[tid * PER + k] = make_double2(rs.h, rx.h);
            s_low[tid * PER + k] = make_double2(rs.l, rx.l);
            if (k < PER) rs = two_add(rs, s[k]), rx = two_add(rx, x[k]);
        }
    }
    // warps 0 to 14: lane k has level warp + k % 2, those on either side of the warp's threshold; the last warp: lane l has level l
    const bool last = warp == kLevels - 1;
    const int mine = last ? lane & (kLevels - 1) : warp + (lane & 1);
    const bool fixed = (F.fixed_mask >> mine) & 1u;
    float lv = F.codebook[mine];
    double w2 = 0.0;
    if (last) {
        for (int k = lane; k < kSortParts; k += 32) w2 += W.w2[k];
#pragma unroll
        for (int off = 16; off; off >>= 1) w2 += __shfl_xor_sync(kFull, w2, off);
    }
    copies_done();
    __syncthreads();
    if (tid < 2) {
        const double2 none = make_double2(0.0, 0.0);
        for (int k = 0; k < 3; ++k) s_below[tid][k][0] = none;
        s_below[tid][0][kLevels] = s_high[kSortGroups];
        s_below[tid][1][kLevels] = s_low[kSortGroups];
        s_below[tid][2][kLevels] = none;
        s_cut[tid][0] = make_float2(-inf, __uint_as_float(0u));
        s_cut[tid][kLevels] = make_float2(inf, __uint_as_float(s_first[kSortGroups]));
    }
    if (last) {
        squared_errors(F, w2, s_level, s_below, s_stop);
        return;
    }
    for (int iter = 0; iter < F.iters; ++iter) {
        const int set = iter & 1;
        const float p = __fmul_rn(__fadd_rn(lv, __shfl_xor_sync(kFull, lv, 1)), 0.5f);
        const int b = sort_bin(p);
        const bool one = one_value_bin(b);                        // in or out as a whole
        const int at = (one && value_of_bin(b) < p) ? b + 1 : b;  // whole bins in front of this one
        // All loads are requested before anything is used, and without branches around them: a lane that has nothing to load loads
        // something else.
        const uint32_t o0 = s_off[at], o1 = s_off[b + 1], f0 = s_first[at / kSortGroup], f1 = s_first[(b + 1) / kSortGroup];
        const double2 whole = ((lane & 1) ? s_low : s_high)[at / kSortGroup];
        uint32_t from = f0 + o0, to = f1 + o1;
        if (max(o0, o1) == kFarBin) {
            if (o0 == kFarBin) from = __ldg(W.start + at);
            if (o1 == kFarBin) to = __ldg(W.start + b + 1);
        }
        if (one) to = from;
        const double rest = __ldg(reinterpret_cast<const double*>(W.pre + min(at, kSortBins - 1)) + (lane >> 4));
        double ls = 0.0, lx = 0.0;
        uint32_t below = 0u;
        if (CROWDED && to - from > kSortCrowd) {
            SortSums in{0.0, 0.0, 0ull};
            crowded_sums<false>(W, SampleWeight<false>{}, from, to, -inf, p, in);
            ls = in.s, lx = in.sx;
            below = lane == 0 ? ~from - (uint32_t)warp : 0u;  // not counted: no two thresholds alike
        } else {
            // 64 samples at once, which is all of most bins, then 128
            auto add = [&](auto count, uint32_t i) {
                constexpr int U = decltype(count)::value;
                float2 it[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t j = i + 32 * u < to ? i + 32 * u : 0u;
                    it[u] = __ldg(W.b + j);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const bool in = i + 32 * u < to && it[u].x < p;
                    const double x = (double)it[u].x, m = (double)it[u].y, sv = m * m, xv = sv * x;
                    ls += in ? sv : 0.0;
                    lx += in ? xv : 0.0;
                    below += in ? 1u : 0u;
                }
            };
            add(std::integral_constant<int, 2>{}, from + lane);
            for (uint32_t i = from + 64; i < to; i += 128) add(std::integral_constant<int, 4>{}, i + lane);
        }
        __syncwarp();
        below = __reduce_add_sync(kFull, below);
        // both sums at once: half the warp goes on with each
        const bool a = lane & 16;
        double v = (a ? lx : ls) + __shfl_xor_sync(kFull, a ? ls : lx, 16);
        v += ((lane & 15) || at == kSortBins) ? 0.0 : rest;
#pragma unroll
        for (int off = 8; off; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
        if ((lane & 15) == 0) (a ? s_below[set][2][warp + 1].y : s_below[set][2][warp + 1].x) = v;
        if ((lane | 1) == 3) s_below[set][lane & 1][warp + 1] = whole;
        if (lane == 4) s_cut[set][warp + 1] = make_float2(p, __uint_as_float(from + below));
        if (lane == 8 || (lane == 9 && warp == kLevels - 2)) s_level[set][mine] = lv;
        __syncthreads();
        // the sums of the two regions, and their levels
        const int stop = s_stop;
        const double2 r0 = s_below[set][2][mine], r1 = s_below[set][2][mine + 1], h0 = s_below[set][0][mine], h1 = s_below[set][0][mine + 1];
        const double2 l0 = s_below[set][1][mine], l1 = s_below[set][1][mine + 1];
        const float2 c0 = s_cut[set][mine], c1 = s_cut[set][mine + 1];
        double s0 = ((h1.x - h0.x) + (l1.x - l0.x)) + (r1.x - r0.x);
        const double s1 = ((h1.y - h0.y) + (l1.y - l0.y)) + (r1.y - r0.y);
        float moved = (float)(s1 / s0);
        const bool empty = __float_as_uint(c0.y) == __float_as_uint(c1.y);
        const unsigned by_itself = __ballot_sync(kFull, !fixed & !empty & too_rough(s0, s1, r0, r1, h0.x, h1.x));
        if (stop <= iter) break;
        if (by_itself & 3u) {
            for (int k = 0; k < 2; ++k) {
                if (!((by_itself >> k) & 1u)) continue;
                const double2 t = region_sums<CROWDED>(W, __shfl_sync(kFull, c0.x, k), __shfl_sync(kFull, c1.x, k));
                if ((lane & 1) == k) s0 = t.x, moved = (float)(t.y / t.x);
            }
        }
        if (!fixed && !empty && s0 > 0.0) lv = moved;
    }
    // (a stop: the levels have not moved since the iteration before)
    if (lane == 0 || (lane == 1 && warp == kLevels - 2))
        if (!fixed) F.codebook[mine] = lv;
}

__global__ void __launch_bounds__(kFitThreads, 1)
sort_fit_mse_kernel(const SortWs W, const SortFit F)
{
    if (!after_previous()) return;
    if (W.n_items[4] != 0u) fit_mse<true>(W, F);
    else fit_mse<false>(W, F);
}

// ---------------------------------------------------------------- all iterations, absolute error

// Sum of a 64-bit integer over the warp (modulo 2^64), 27 bits at a time.
__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v)
{
    const uint32_t lo = __reduce_add_sync(kFull, (uint32_t)v & 0x7ffffffu);
    const uint32_t mi = __reduce_add_sync(kFull, (uint32_t)(v >> 27) & 0x7ffffffu);
    const uint32_t hi = __reduce_add_sync(kFull, (uint32_t)(v >> 54));
    return (unsigned long long)lo + ((unsigned long long)mi << 27) + ((unsigned long long)hi << 54);
}


// The sample of a crowded bin, from ... to - 1, with which the weight of its samples reaches the goal.  It is one of those with p <= x < q; c0 of the
// weight lies below p, c1 below q; it is near `guess`.  Called by a whole warp.  (Medians of 2^20 weights in two bins, 18 iterations, 1140 us looked
// for among all samples of a bin, 985 between the thresholds, 957 with the level as the first place to look; about zero 3240, 2830 and 1845.)
__device__ __noinline__ float crowded_median(const SortWs& W, const SampleWeight<true>& weight, uint32_t from, uint32_t to, float p, float guess,
                                             float q, unsigned long long goal, unsigned long long c0, unsigned long long c1)
{
    constexpr int U = kWindowsPerLane;
    const uint32_t w0 = from / kSortWindow + (threadIdx.x & 31), last = (to - 1) / kSortWindow;
    // weight of the bin's samples with keys up to k, the largest of these keys, and the smallest key beyond
    auto upto = [&](uint32_t k, uint32_t& end, uint32_t& begin) -> unsigned long long {
        unsigned long long sum = 0ull;
        uint32_t top = 0u, next = 0xffffffffu;
        for (uint32_t w = w0; w <= last; w += 32 * U) {
            uint32_t lo[U], hi[U], at[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t v = w + 32 * u;
                lo[u] = max(from, v * kSortWindow);
                hi[u] = min(to, (v + 1) * kSortWindow);
                if (v > last) lo[u] = hi[u] = to;
                at[u] = lo[u];
            }
            for (uint32_t step = kSortWindow; step; step >>= 1) {
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (at[u] + step <= hi[u] && sort_key(W.b[at[u] + step - 1].x) <= k) at[u] += step;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (lo[u] == hi[u]) continue;
                if (at[u] < hi[u]) next = min(next, sort_key(W.b[at[u]].x));
                if (at[u] == lo[u]) continue;
                top = max(top, sort_key(W.b[at[u] - 1].x));
                const uint32_t first = (lo[u] / kSortWindow) * kSortWindow;
                sum += sums_before<true>(W, weight, first, at[u]).a - sums_before<true>(W, weight, first, lo[u]).a;
            }
        }
        __syncwarp();
        end = __reduce_max_sync(kFull, top);
        begin = __reduce_min_sync(kFull, next);
        return warp_sum64(sum);
    };
    // every window is in order: the bin's first and last keys are those of the windows' parts of it
    uint32_t k0 = 0xffffffffu, k1 = 0u;
    for (uint32_t w = w0; w <= last; w += 32) {
        k0 = min(k0, sort_key(W.b[max(from, w * kSortWindow)].x));
        k1 = max(k1, sort_key(W.b[min(to, (w + 1) * kSortWindow) - 1].x));
    }
    __syncwarp();
    k0 = max(__reduce_min_sync(kFull, k0), sort_key(p));
    k1 = min(__reduce_max_sync(kFull, k1), sort_key(q) - 1u);
    for (int step = 0; k0 < k1; ++step) {  // behind the first step as in the search over few samples
        const uint32_t d = k1 - k0;
        const float at = step % 3 == 0 ? 0.5f : (float)(goal - c0) / (float)(c1 - c0);
        const uint32_t km = step ? k0 + min((uint32_t)((float)d * at), d - 1u) : min(max(sort_key(guess), k0), k1 - 1u);
        uint32_t end, begin;
        const unsigned long long c = upto(km, end, begin);
        if (c >= goal) k1 = end, c1 = c;
        else k0 = begin, c0 = c;
    }
    return sort_key_value(k0);
}

constexpr int kFitMaeThreads = 2 * kFitThreads;  // a warp per threshold and level, as many for the error

// Behind a barrier warp l looks for the median of region l: the first sample, in the order of x, with which the weight reaches half
// of the region's.  The weights are integers, so a region is exactly the difference of two sums.  A second barrier, and the levels
// are there.  Sixteen more warps add up beside this what the error of the iteration needs, and warp 15, which has no threshold, writes
// the error of the iteration before.
//
// The source, by a warp, results the same in all lanes:  weight(v): of what lies below v;  sums(v): {s, sx} of it, all(): of everything, in
//              lanes 0 to 3 the doubles of a Below;
//              median(goal, at, a0, a1): the first sample with which the weight of all samples from the first on reaches the goal; it is known to
//              be in the region that `at` tells, below whose ends the weights a0 and a1 lie
struct FitMaeShared {
    unsigned long long below[2][kLevels + 1];  // weight below threshold k - 1; entry 0: nothing, entry 16: everything
    float level[2][kLevels];
    Below at[2][2 * kLevels];                  // what lies below the levels, and below the thresholds above them
    int stop;
};
template <class Source>
__device__ __forceinline__ void fit_mae_loop(Source& source, FitMaeShared& S, unsigned long long weight, const SortFit& F)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < 2) S.below[tid][0] = 0ull, S.below[tid][kLevels] = weight;
    if (tid == 0) S.stop = 0;
    if (tid < kLevels) S.level[0][tid] = F.codebook[tid];
    __syncthreads();
    // the error of iteration `at`, by warp 15
    auto error_of = [&](int at) {
        const int l = lane & (kLevels - 1);
        const float* const lvs = S.level[at & 1];
        const FitPoints p = points_of(l, lvs[max(l - 1, 0)], lvs[l], lvs[min(l + 1, kLevels - 1)]);
        double err = half_error(lane, p, lvs[l], S.at[at & 1][lower_end_of(lane)], S.at[at & 1][lane]);
#pragma unroll
        for (int off = 16; off; off >>= 1) err += __shfl_xor_sync(kFull, err, off);
        err = fmax(err, 0.0) / (double)F.n_total;
        if (lane == 0 && F.err_log) F.err_log[at] = err;
        return err;
    };
    int iter = 0;
    if (warp >= kLevels) {
        // ---- what the error needs of a threshold and of a level, beside the others' search for the next levels
        const int l = warp - kLevels;
        float known = 0.0f;
        double part = source.all();
        auto put = [&](int set, int at, double v) {
            if (lane < 4) reinterpret_cast<double*>(&S.at[set][at])[lane] = v;
        };
        if (l == kLevels - 1) put(0, 2 * kLevels - 1, part), put(1, 2 * kLevels - 1, part);
        for (; iter < F.iters; ++iter) {
            const int set = iter & 1;
            const FitPoints at = points_of(l, S.level[set][max(l - 1, 0)], S.level[set][l], S.level[set][min(l + 1, kLevels - 1)]);
            if (l < kLevels - 1) put(set, kLevels + l, source.sums(at.hi));
            __syncthreads();
            if (S.stop) return;
            if (iter == 0 || __float_as_uint(at.mid) != __float_as_uint(known)) {
                part = source.sums(at.mid);
                known = at.mid;
            }
            put(set, l, part);
            __syncthreads();
        }
        return;
    }
    // ---- warp w: threshold w and level w
    const bool fixed = (F.fixed_mask >> warp) & 1u, cuts = warp < kLevels - 1;
    float lv = S.level[0][warp];
    for (; iter < F.iters; ++iter) {
        const int set = iter & 1;
        float above = 0.0f;  // the next level
        if (cuts) {
            above = S.level[set][warp + 1];
            const unsigned long long a = source.weight(__fmul_rn(__fadd_rn(lv, above), 0.5f));
            if (lane == 0) S.below[set][warp + 1] = a;
        } else {
            if (iter) {
                const double err = error_of(iter - 1);
                const int l = lane & (kLevels - 1);
                // no level has moved: the remaining iterations would repeat this one bit for bit
                if (__all_sync(kFull, __float_as_uint(S.level[set][l]) == __float_as_uint(S.level[set ^ 1][l]))) {
                    if (lane == 0) S.stop = 1;
                    if (F.err_log)
                        for (int k = iter + lane; k < F.iters; k += 32) F.err_log[k] = err;
                }
            }
        }
        __syncthreads();
        if (S.stop) break;
        const unsigned long long a0 = S.below[set][warp], a1 = S.below[set][warp + 1];
        const FitPoints at = points_of(warp, warp ? S.level[set][warp - 1] : 0.0f, lv, above);
        // (levels that do not ascend have regions without samples)
        if (a1 != a0 && !(at.lo > at.hi) && !fixed) lv = source.median(a0 + (a1 - a0) - (a1 - a0) / 2ull, at, a0, a1);
        if (lane == 0) S.level[set ^ 1][warp] = lv;
        __syncthreads();
    }
    if (warp == kLevels - 1 && iter == F.iters && iter) error_of(iter - 1);
    if (lane == 0 && !fixed) F.codebook[warp] = lv;
}

// What lies below a threshold: as for the squared error.  The place of a median: in the running sums of the groups (shared memory,
// 64 entries a step), then of the group's bins (one load), then among the samples of one bin.
// An iteration over 2^20 fp32 weights 6.5 -> 3.1 us, over 2^24 33 -> 14.5 (before: two warps to a region, whole groups added up and
// searched one after the other, cut bins first).  Bound by its chain: three loads from L2 of 430 or 820 cycles each, the
// reductions, two barriers; over 2^24 weights by the passes over the 500 samples of a bin (of up to 64 samples every lane adds
// up what is not behind its own, in one pass: 2^20 weights 3.75 -> 3.1).
constexpr int kMaeOff = ((kSortGroups + 1) * 8 + 15) / 16 * 16;  // shared memory: weights in front of the groups, first samples of the bins,
constexpr int kMaeFirst = kMaeOff + kSortBins * 2 + 16;         // (and the end) of the groups
constexpr int kMaeSmem = kMaeFirst + (kSortGroups + 1) * 4;

template <bool CROWDED>
struct MaeSamples {
    const SortWs& W;
    const SampleWeight<true>& weights;
    const double* group_sums;                 // what lies in front of a group, the four doubles of a Below
    SharedTable<unsigned long long> group_a;
    SharedTable<uint16_t> off;
    SharedTable<uint32_t> group_first;
    __device__ __forceinline__ uint32_t start_of(int b) const  // first sample of bin b <= kSortBins
    {
        const uint32_t o = off[b], f = group_first[b / kSortGroup];
        return o == kFarBin ? __ldg(W.start + b) : f + o;
    }
    // This lane's share of what lies below v, less the whole groups in front of the one that is returned; what lies in front of that one, a double
    // to a lane (asked for before the samples).
    template <bool SUMS>
    __device__ __forceinline__ int below(float v, SortSums& t, double& front) const
    {
        const int lane = threadIdx.x & 31;
        const int b = sort_bin(v);
        const bool one = one_value_bin(b);                        // in or out as a whole
        const int at = (one && value_of_bin(b) < v) ? b + 1 : b;  // whole bins in front of this one
        const uint32_t from = start_of(at), to = one ? from : start_of(b + 1);
        t = SortSums{0.0, 0.0, 0ull};
        const unsigned long long pre =
            __ldg(reinterpret_cast<const unsigned long long*>(W.pre + min(at, kSortBins - 1)) + (SUMS ? (lane & 1) : 2));
        if (SUMS) front = group_sums[4 * (at / kSortGroup) + (lane & 3)];
        if (CROWDED && to - from > kSortCrowd) {
            crowded_sums<true>(W, weights, from, to, -__int_as_float(0x7f800000), v, t);
        } else {
            auto add = [&](auto count, uint32_t i) {  // 64 samples at once, which is all of most bins, then 128
                constexpr int U = decltype(count)::value;
                float2 it[U];
#pragma unroll
                for (int u = 0; u < U; ++u) it[u] = __ldg(W.b + (i + 32 * u < to ? i + 32 * u : 0u));
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    double s;
                    unsigned long long a;
                    weights(it[u], s, a);
                    const bool in = i + 32 * u < to && it[u].x < v;
                    const double sx = s * (double)it[u].x;
                    if (SUMS) {
                        t.s += in ? s : 0.0;
                        t.sx += in ? sx : 0.0;
                    } else {
                        t.a += in ? a : 0ull;
                    }
                }
            };
            add(std::integral_constant<int, 2>{}, from + lane);
            for (uint32_t i = from + 64; i < to; i += 128) add(std::integral_constant<int, 4>{}, i + lane);
        }
        __syncwarp();
        if (at < kSortBins) {
            if (SUMS && lane == 0) t.s += __longlong_as_double((long long)pre);
            if (SUMS && lane == 1) t.sx += __longlong_as_double((long long)pre);
            if (!SUMS && lane == 0) t.a += pre;
        }
        return at / kSortGroup;
    }
    __device__ __forceinline__ unsigned long long weight(float v) const
    {
        SortSums t;
        double none;
        const int g = below<false>(v, t, none);
        return warp_sum64(t.a) + group_a[g];
    }
    __device__ __forceinline__ double sums(float v) const
    {
        SortSums t;
        double front;
        below<true>(v, t, front);
        const int lane = threadIdx.x & 31;
        const bool h = lane & 16;
        double u = (h ? t.sx : t.s) + __shfl_xor_sync(kFull, h ? t.s : t.sx, 16);
#pragma unroll
        for (int o = 8; o; o >>= 1) u += __shfl_xor_sync(kFull, u, o);
        const double rest = __shfl_sync(kFull, u, lane & 1 ? 16 : 0);
        return (lane & 2) ? front + rest : front;
    }
    __device__ __forceinline__ double all() const { return group_sums[4 * kSortGroups + (threadIdx.x & 3)]; }
    __device__ __forceinline__ float median(unsigned long long goal, const FitPoints& at, unsigned long long a0, unsigned long long a1) const
    {
        // the last group in front of which there is less than the goal: 32 groups of 64, then one of 64
        const int lane = threadIdx.x & 31, c = __popc(__ballot_sync(kFull, group_a[64 * (lane + 1)] < goal));
        const unsigned long long u = group_a[64 * c + 1 + lane], v = group_a[64 * c + 33 + lane];
        const int g = 64 * c + __popc(__ballot_sync(kFull, u < goal)) + __popc(__ballot_sync(kFull, v < goal));
        const unsigned long long before = group_a[g], pre = __ldg(&W.pre[g * kSortGroup + lane].a);
        const int in = __popc(__ballot_sync(kFull, before + pre < goal)) - 1, b = g * kSortGroup + in;
        const unsigned long long front = before + __shfl_sync(kFull, pre, in), need = goal - front;  // of the bin's weight
        if (one_value_bin(b)) return value_of_bin(b);
        const uint32_t s0 = start_of(b), e = start_of(b + 1);
        if (CROWDED && e - s0 > kSortCrowd)
            return crowded_median(W, weights, s0, e, at.lo, at.mid, at.hi, need, max(a0, front) - front, min(a1 - front, __ldg(&W.bin[b].a)));
        auto get = [&](uint32_t i, uint32_t& k, uint32_t& a) {
            const float2 it = __ldg(W.b + (i < e ? i : s0));
            double s;
            unsigned long long w;
            weights(it, s, w);
            k = i < e ? sort_key(it.x) : 0xffffffffu;
            a = i < e ? (uint32_t)w : 0u;  // (31 bits)
        };
        if (e - s0 <= 64u) {
            // Few samples: one or two to a lane, which adds up for each all those that are not behind it.
            auto among = [&](auto count) -> float {
                constexpr int N = decltype(count)::value;
                uint32_t key[N], mine[N], first = 0xffffffffu;
                unsigned long long sum[N];
#pragma unroll
                for (int r = 0; r < N; ++r) {
                    get(s0 + 32 * r + lane, key[r], mine[r]);
                    sum[r] = 0ull;
                }
#pragma unroll
                for (int r = 0; r < N; ++r) {
                    const int here = min((int)(e - s0) - 32 * r, 32);
#pragma unroll 4
                    for (int j = 0; j < here; ++j) {
                        const uint32_t k = __shfl_sync(kFull, key[r], j), w = __shfl_sync(kFull, mine[r], j);
#pragma unroll
                        for (int q = 0; q < N; ++q) sum[q] += k <= key[q] ? w : 0u;
                    }
                }
#pragma unroll
                for (int q = 0; q < N; ++q)
                    if (sum[q] >= need) first = min(first, key[q]);  // (no sample: the last key of all)
                return sort_key_value(__reduce_min_sync(kFull, first));
            };
            return e - s0 <= 32u ? among(std::integral_constant<int, 1>{}) : among(std::integral_constant<int, 2>{});
        }
        // The goal is reached at one of the keys k0 ... k1 of the bin's samples; c0 of the bin's weight lies below k0, c1 up to
        // k1.  The next key to split at is where even weights would put it (every third time the middle), and the ends move to
        // samples: a handful of steps, where halving the keys takes one per bit in which they differ.
        constexpr int R = 4;
        uint32_t key[R], wt[R], kmin = 0xffffffffu, kmax = 0u;
        unsigned long long c0 = 0ull, c1 = __ldg(&W.bin[b].a);
#pragma unroll
        for (int r = 0; r < R; ++r) get(s0 + 32 * r + lane, key[r], wt[r]);
        auto each = [&](auto fn) {
#pragma unroll
            for (int r = 0; r < R; ++r) fn(key[r], wt[r]);
            for (uint32_t i = s0 + 32 * R + lane; i < e; i += 32 * 2 * R) {
                uint32_t k[2 * R], a[2 * R];
#pragma unroll
                for (int r = 0; r < 2 * R; ++r) get(i + 32 * r, k[r], a[r]);
#pragma unroll
                for (int r = 0; r < 2 * R; ++r) fn(k[r], a[r]);
            }
            __syncwarp();
        };
        each([&](uint32_t k, uint32_t) {
            if (k != 0xffffffffu) {
                kmin = min(kmin, k);
                kmax = max(kmax, k);
            }
        });
        uint32_t k0 = __reduce_min_sync(kFull, kmin), k1 = __reduce_max_sync(kFull, kmax);
        for (int step = 1; k0 < k1; ++step) {
            const uint32_t d = k1 - k0;
            const float part = step % 3 == 0 ? 0.5f : (float)(need - c0) / (float)(c1 - c0);
            const uint32_t km = k0 + min((uint32_t)((float)d * part), d - 1u);
            uint32_t end = 0u, begin = 0xffffffffu;
            unsigned long long sum = 0ull;
            each([&](uint32_t k, uint32_t a) {
                if (k <= km) {
                    sum += a;
                    end = max(end, k);
                } else {
                    begin = min(begin, k);
                }
            });
            sum = warp_sum64(sum);
            if (sum >= need) k1 = __reduce_max_sync(kFull, end), c1 = sum;
            else k0 = __reduce_min_sync(kFull, begin), c0 = sum;
        }
        return sort_key_value(k0);
    }
};

// CROWDED: the kernel for data with crowded bins.  Both are launched, the flag of such bins tells which one runs: with both
// loops in one kernel 2^22 fp32 weights, 12 iterations, take 252.9 us against 246.2, 2^20 125.2 against 124.9.
template <bool CROWDED>
__global__ void __launch_bounds__(kFitMaeThreads, 1)
sort_fit_mae_kernel(const __grid_constant__ SortWs W, const __grid_constant__ SortFit F)
{
    if (!after_previous()) return;
    if ((W.n_items[4] != 0u) != CROWDED) return;
    extern __shared__ __align__(16) unsigned char s_fit[];
    unsigned long long* const s_a = reinterpret_cast<unsigned long long*>(s_fit);
    uint16_t* const s_off = reinterpret_cast<uint16_t*>(s_fit + kMaeOff);
    uint32_t* const s_first = reinterpret_cast<uint32_t*>(s_fit + kMaeFirst);
    __shared__ FitMaeShared S;
    SampleWeight<true> weights;
    weights.max_bits = W.n_items[1];
    weights.unit = F.metric >= 2;
    if (threadIdx.x == 0) s_off[kSortBins] = 0u;
    copy_starts(W, s_off, s_first);
    // What lies in front of the groups goes where the digits' counts were, which have served: in shared memory beside the first samples it would leave
    // 28 KB of L1, and bisections in crowded bins live on L1 (2^20 weights in two bins 58 us an iteration, 68 without it).
    static_assert((kSortGroups + 1) * sizeof(Below) <= (size_t)kSortGrid * 256 * 4, "room for the running sums");
    Below* const sums = reinterpret_cast<Below*>(W.counts);
    if (threadIdx.x < kFitThreads)
        running_sums<kSortGroups / kFitThreads, TwoPair>(true, kSortGroups, [&](int g) { return TwoPair{{W.group[g].s, 0.0}, {W.group[g].sx, 0.0}}; },
                                                         [&](int g, const TwoPair& v) {
                                                             sums[g] = Below{make_double2(v.s.h, v.x.h), make_double2(v.s.l, v.x.l)};
                                                         });
    else
        running_sums<kSortGroups / kFitThreads, unsigned long long>(true, kSortGroups, [&](int g) { return W.group[g].a; },
                                                                    [&](int g, unsigned long long v) { s_a[g] = v; });
    copies_done();
    __syncthreads();
    MaeSamples<CROWDED> source{W, weights, reinterpret_cast<const double*>(sums), SharedTable(s_a), SharedTable(s_off), SharedTable(s_first)};
    fit_mae_loop(source, S, s_a[kSortGroups], F);
}

// ---------------------------------------------------------------- host side

namespace {

template <bool MAE>
int sums_and_iterations(const SortWs& W, const SortFit& F, cudaStream_t st)
{
    SampleWeight<MAE> weight{};
    weight.unit = F.metric >= 2;
    const int64_t ctas = (F.n_max + 8 * kSortChunk - 1) / (8 * kSortChunk);
    launch_after(sort_sums_kernel<MAE>, kStartCtas + (int)(ctas < 8 * kSMs ? ctas : 8 * kSMs), 256, 0, st, W, weight);
    launch_after(sort_group_kernel<MAE>, kSortGroups / 8, 256, 0, st, W);
    auto order_windows = [&]() -> int {
        constexpr auto kern = sort_windows_kernel<MAE>;
        constexpr int smem = (int)sizeof(WindowScratch);
        if (const int rc = ensure_dynamic_smem<kern>(smem)) return rc;
        const int64_t windows = (F.n_max + kSortWindow - 1) / kSortWindow;
        launch_after(kern, (int)(windows < kSMs ? windows : kSMs), kSortThreads, smem, st, W, weight);
        return BOF4_OK;
    };
    const bool may_crowd = F.n_max > kSortCrowd;  // no more samples than make a crowded bin do not
    if constexpr (MAE) {
        constexpr auto plain = sort_fit_mae_kernel<false>;
        if (const int rc = ensure_dynamic_smem<plain>(kMaeSmem)) return rc;
        launch_after(plain, 1, kFitMaeThreads, kMaeSmem, st, W, F);
        if (may_crowd) {
            if (const int rc = order_windows()) return rc;
            constexpr auto crowded = sort_fit_mae_kernel<true>;
            if (const int rc = ensure_dynamic_smem<crowded>(kMaeSmem)) return rc;
            launch_after(crowded, 1, kFitMaeThreads, kMaeSmem, st, W, F);
        }
    } else {
        if (may_crowd)
            if (const int rc = order_windows()) return rc;
        if (const int rc = ensure_dynamic_smem<sort_fit_mse_kernel>(kMseSmem)) return rc;
        launch_after(sort_fit_mse_kernel, 1, kFitThreads, kMseSmem, st, W, F);
    }
    BOF4_CUDA_TRY(cudaGetLastError());
    return BOF4_OK;
}

template <class DT, bool SG>
int samples(const EmTensors& T, int block_size, uint32_t first, uint32_t n, const SortWs& W, cudaStream_t st)
{
#define BOF4_SORT_I(I_) \
    case I_: launch_after(sort_samples_kernel<DT, I_, SG>, 2 * kSMs, 512, 0, st, T, first, n, W.a, W.n_items, W.w2, W.first); break;
    switch (block_size) {
        BOF4_SORT_I(32) BOF4_SORT_I(64) BOF4_SORT_I(128) BOF4_SORT_I(256) BOF4_SORT_I(512) BOF4_SORT_I(1024)
        BOF4_SORT_I(2048) BOF4_SORT_I(4096)
    }
#undef BOF4_SORT_I
    BOF4_CUDA_TRY(cudaGetLastError());
    return BOF4_OK;
}

}  // namespace

// Samples are in W.a, their number in *W.n_items: orders them, sums the bins, runs the iterations.
static int sorted_run(const SortWs& W, const SortFit& F, cudaStream_t st)
{
    const bool staged = F.n_max >= kStagedMin;
    auto pass = [&](auto shift, const float2* in, float2* out) -> int {
        constexpr int S = decltype(shift)::value;
        launch_after(sort_count_kernel<S>, kSortGrid, kSortThreads, 0, st, in, W.n_items, W.counts, W.first);
        if (staged) {
            constexpr auto kern = sort_scatter_kernel<S, true>;
            if (const int rc = ensure_dynamic_smem<kern>(kScatterSmem)) return rc;
            launch_after(kern, kSortGrid, kSortThreads, kScatterSmem, st, in, W.n_items, W.counts, out);
        } else {
            launch_after(sort_scatter_kernel<S, false>, kSortGrid, kSortThreads, 0, st, in, W.n_items, W.counts, out);
        }
        return BOF4_OK;
    };
    int rc;
    if ((rc = pass(std::integral_constant<int, 0>{}, W.a, W.b)) || (rc = pass(std::integral_constant<int, 8>{}, W.b, W.a))) return rc;
    SortWs V = W;  // the ordered samples are in the first array
    V.a = W.b;
    V.b = W.a;
    V.before = reinterpret_cast<SortSums*>(W.b);
    BOF4_CUDA_TRY(cudaGetLastError());
    const bool mae = F.metric == BOF4_METRIC_MAE || F.metric == BOF4_METRIC_MAE_NORMALIZED;
    return mae ? sums_and_iterations<true>(V, F, st) : sums_and_iterations<false>(V, F, st);
}

int sorted_fit(const EmArgs& a, float* d_codebook, uint32_t fixed_mask, int iters, double* d_err_log, void* d_ws,
               size_t ws_bytes, cudaStream_t st, bool* done)
{
    *done = false;
    if (a.n_total > kSortMaxDirect || !ordering_pays(a.w_dtype, a.n_total, a.metric, iters, false)) return BOF4_OK;
    SortWs W;
    if (sorted_layout(d_ws, a.n_total, &W) > ws_bytes) return BOF4_OK;
    *done = true;
    const uint32_t n = (uint32_t)a.n_total;
    const bool alone = !has_whole_blocks(a);
    const bool sg = a.norm == BOF4_NORM_SIGNED;
    uint32_t at = 0;
    int calls = 0;
    int rc = for_each_tensor_chunk(a, 512 * kLaneW, [&](const EmTensors& T) -> int {
        const uint32_t first = at;
        for (int t = 0; t < T.count; ++t) at += (uint32_t)T.n[t];
        if (a.w_dtype == BOF4_F32)
            return sg ? samples<F32, true>(T, a.block_size, first, n, W, st) : samples<F32, false>(T, a.block_size, first, n, W, st);
        return sg ? samples<BF16, true>(T, a.block_size, first, n, W, st) : samples<BF16, false>(T, a.block_size, first, n, W, st);
    }, &calls);
    if (rc) return rc;
    rc = for_each_tail_chunk(a, [&](const EmTails& Q) -> int {
        if (a.w_dtype == BOF4_F32) {
            if (sg) launch_after(sort_tail_kernel<F32, true>, 1, kEmTailThreads, 0, st, Q, at, n, alone, W.a, W.n_items, W.w2, W.first);
            else launch_after(sort_tail_kernel<F32, false>, 1, kEmTailThreads, 0, st, Q, at, n, alone, W.a, W.n_items, W.w2, W.first);
        } else {
            if (sg) launch_after(sort_tail_kernel<BF16, true>, 1, kEmTailThreads, 0, st, Q, at, n, alone, W.a, W.n_items, W.w2, W.first);
            else launch_after(sort_tail_kernel<BF16, false>, 1, kEmTailThreads, 0, st, Q, at, n, alone, W.a, W.n_items, W.w2, W.first);
        }
        for (int q = 0; q < Q.count; ++q) at += (uint32_t)Q.len[q];
        BOF4_CUDA_TRY(cudaGetLastError());
        return BOF4_OK;
    });
    if (rc) return rc;
    SortFit F{};
    F.metric = a.metric;
    F.n_total = a.n_total;
    F.n_max = a.n_total;
    F.codebook = d_codebook;
    F.fixed_mask = fixed_mask;
    F.iters = iters;
    F.err_log = d_err_log;
    return sorted_run(W, F, st);
}

}  // namespace bof4
