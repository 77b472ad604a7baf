// Iterations of a codebook fit over the cells of em_cells.cu.
//
//   sums   a thread per place in the order of x: the cell's sums, and what lies in front of it in its block of 512 places
//   fit    all iterations in one CTA (em_fit.cuh).  What lies below a threshold is what lies in front of its place, and the place is
//          worked out from the threshold's bits: so many fractions lie below it.
//
// A value's place: x = RN(a / b 2^-k) lies below a threshold with the 24-bit significand Q in the same binade exactly if the fraction lies below
// (2 Q - 1) / 2^24, halfway to the number before (no fraction with b < 256 is halfway between two floats), which is a
// comparison of integers; for a negative threshold the magnitudes up to it are counted, with 2 Q + 1.
#include <type_traits>

#include "em_cells.cuh"

namespace bof4 {

// The cell at a place and its normalised weight; false: there is none.
template <class Table>
__device__ __forceinline__ bool cell_at(int place, const Table& value_of, uint32_t& cell, float& x)
{
    const int i = abs(place - kCellOne);
    const bool neg = place < kCellOne;
    x = 0.0f;
    cell = kZeroCell;
    if (place >= kCellPlaces) return false;
    if (i == 0) return true;
    if (i == kCellOne) {
        cell = neg ? kCellDepth : 0;
        x = 1.0f;
    } else if (i < kPlaceBinades) {
        const uint32_t e = (uint32_t)i - 1u;
        cell = (uint32_t)kDeepCells + e + (neg ? kDeepExps : 0);
        x = __uint_as_float(e ? e << 23 : 0x400000u);
    } else {
        const int t = i - kPlaceBinades, e = 40 - t / kCellFractions;
        const int f = value_of[t % kCellFractions], a = f >> 7, b = f & 127;
        const int d = 128 * (a >= b ? e : e - 1) + b - a;
        if (d >= kCellDepth) return false;  // 2^-40 is a deep cell
        cell = (uint32_t)(b * kCellRow + (neg ? kCellDepth : 0) + d);
        x = __fdiv_rn(__uint_as_float((uint32_t)(0x3f80 + b - d) << 16), __uint_as_float((uint32_t)(0x3f80 + b) << 16));
    }
    if (neg) x = -x;
    return true;
}

// The first place whose x is not below p (kCellPlaces: none); GROUP lanes have the same p, and the warp is whole.  The fractions in front of the
// part of the binade that p lies in are counted beforehand; of the next ones, four to a part on average, a lane looks at
// each, or where every lane has a p of its own, the place among the part's is found by halving.
template <int GROUP, class Table>
__device__ __forceinline__ int place_of(float p, const Table& value_of)
{
    const uint32_t bits = __float_as_uint(p) & 0x7fffffffu, q = (bits & 0x7fffffu) | 0x800000u;
    const bool neg = p < 0.0f;
    const uint32_t half = 2u * q + (neg ? 1u : 0xffffffffu);
    const int part = (int)(q / (0x800000u / kCellParts)) - kCellParts;
    auto in_front = [&](int i) {
        const int f = value_of[i], a = (f >> 7) + 128, b = (f & 127) + 128;
        return ((unsigned long long)(uint32_t)(a < b ? 2 * a : a) << 24) < (unsigned long long)(uint32_t)b * half;
    };
    int n = value_of[kCellFractions + part];
    if constexpr (GROUP == 1) {
        int end = value_of[kCellFractions + min(part + 1, kCellParts - 1)];
        if (part == kCellParts - 1) end = kCellFractions;
        while (n < end) {
            const int mid = (n + end) >> 1;
            const bool in = in_front(mid);
            n = in ? mid + 1 : n;
            end = in ? end : mid;
        }
        __syncwarp();
    } else {
        const int lane = threadIdx.x & 31, i = lane & (GROUP - 1);
        constexpr uint32_t kMask = 0xffffffffu >> (32 - GROUP);
        int more;
        do {
            const bool in = n + i < kCellFractions && in_front(min(n + i, kCellFractions - 1));
            more = __popc(__ballot_sync(kFull, in) >> (lane & ~(GROUP - 1)) & kMask);
            n += more;
        } while (__any_sync(kFull, more == GROUP));
    }
    // magnitudes below that of p (neg: up to it), zero among them
    const int e = (int)(bits >> 23);
    int below;
    if (bits >= 0x3f800000u) {
        below = (neg || bits > 0x3f800000u) ? kCellOne + 1 : kCellOne;
        if (bits > 0x7f800000u) below = kCellOne;  // not a number: all but one
    } else if (e >= 87) {
        below = kPlaceBinades + (e - 87) * kCellFractions + n;
        if (!neg && bits == 87u << 23) below = kPlaceBinades - 1;  // 2^-40 itself is a deep cell
    } else if (e > 0) {
        below = 1 + e + ((neg || (bits & 0x7fffffu)) ? 1 : 0);
    } else {
        below = bits == 0u ? 0 : 1 + ((bits > 0x400000u || (neg && bits == 0x400000u)) ? 1 : 0);
    }
    return neg ? kCellOne + 1 - below : kCellOne + below;
}

// ---------------------------------------------------------------- sums

template <bool MAE>
__device__ __forceinline__ void cell_sums(const CellsWs& W, uint32_t cell, double scale, double& s, unsigned long long& a)
{
    const ulonglong2 v = W.acc[cell];
    s = ((double)v.y * 18446744073709551616.0 + (double)v.x) * scale;
    a = MAE ? W.acc_a[cell] : 0ull;
}

// Bound by its gathers from L2 (neighbours in the order of x have different significands of the constant) and the shuffles of its sums,
// so blocks without a weight, about two thirds of near-Gaussian data's, end early, and one warp puts the warps' sums together for all: 13.7 us
// over 2^22 or 2^26 weights, 24.5 with every thread adding up the warps in front of its own and no block left out.
template <bool MAE>
__global__ void __launch_bounds__(kCellBlock)
cells_sums_kernel(const CellsWs W)
{
    if (!after_previous()) return;
    constexpr int NW = kCellBlock / 32, PART = kCellPart / 32;
    __shared__ CellBlock s_warp[NW];
    __shared__ double2 s_front[NW];
    __shared__ unsigned long long s_a[NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, place = (int)blockIdx.x * kCellBlock + tid;
    const double scale = *cells_scale(W);
    uint32_t cell;
    float x;
    double s = 0.0;
    unsigned long long a = 0ull;
    if (cell_at(place, W.value_of, cell, x)) cell_sums<MAE>(W, cell, scale, s, a);
    if (!__syncthreads_or(s != 0.0)) {  // (a weight of the medians comes with one of the sums)
        W.front[place] = make_double2(0.0, 0.0);
        if (tid == 0) W.block[blockIdx.x] = CellBlock{0.0, 0.0, 0.0};
        if (MAE) {
            W.front_a[place] = 0ull;
            if (tid % kCellPart == 0) W.part_a[place / kCellPart] = 0ull;
        }
        return;
    }
    const double sx = s * (double)x;
    double is = s, ix = sx, q = sx * (double)x;
    unsigned long long ia = a;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double us = __shfl_up_sync(kFull, is, off), ux = __shfl_up_sync(kFull, ix, off);
        const unsigned long long ua = MAE ? __shfl_up_sync(kFull, ia, off) : 0ull;
        if (lane >= off) is += us, ix += ux, ia += ua;
        if (!MAE) q += __shfl_xor_sync(kFull, q, off);
    }
    if (lane == 31) {
        s_warp[warp] = CellBlock{is, ix, q};
        s_a[warp] = ia;
    }
    double fs = __shfl_up_sync(kFull, is, 1), fx = __shfl_up_sync(kFull, ix, 1);
    if (lane == 0) fs = fx = 0.0;
    __syncthreads();
    if (warp == 0) {
        CellBlock v{0.0, 0.0, 0.0};
        if (lane < NW) v = s_warp[lane];
        double ts = v.s, tx = v.sx;
#pragma unroll
        for (int off = 1; off < NW; off <<= 1) {
            const double us = __shfl_up_sync(kFull, ts, off), ux = __shfl_up_sync(kFull, tx, off);
            if (lane >= off) ts += us, tx += ux;
            v.sxx += __shfl_xor_sync(kFull, v.sxx, off);
        }
        if (lane < NW - 1) s_front[lane + 1] = make_double2(ts, tx);
        if (lane == NW - 1) s_front[0] = make_double2(0.0, 0.0), W.block[blockIdx.x] = CellBlock{ts, tx, v.sxx};
    }
    if (MAE) {
        unsigned long long fa = ia - a;
        for (int w = warp / PART * PART; w < warp; ++w) fa += s_a[w];
        W.front_a[place] = fa;
        if (tid % kCellPart == kCellPart - 1) W.part_a[place / kCellPart] = fa + a;
    }
    __syncthreads();
    const double2 f = s_front[warp];
    W.front[place] = make_double2(f.x + fs, f.y + fx);
}

// ---------------------------------------------------------------- iterations

constexpr int kCellPer = (kCellBlocks + kFitThreads - 1) / kFitThreads;  // blocks per thread

// {s, sx} of p <= x < q, by a warp; the same in all lanes.
__device__ __noinline__ double2 cell_region(const CellsWs& W, float p, float q)
{
    const int lane = threadIdx.x & 31;
    const int from = place_of<32>(p, W.value_of), to = place_of<32>(q, W.value_of);
    const int b0 = (from + kCellBlock - 1) / kCellBlock, b1 = to / kCellBlock;
    const double scale = *cells_scale(W);
    double s = 0.0, x = 0.0;
    auto single = [&](int i0, int i1) {
        for (int i = i0 + lane; i < i1; i += 32) {
            uint32_t cell;
            float v;
            double w;
            unsigned long long a;
            if (!cell_at(i, W.value_of, cell, v)) continue;
            cell_sums<false>(W, cell, scale, w, a);
            s += w, x += w * (double)v;
        }
    };
    single(from, min(to, b0 * kCellBlock));
    for (int b = b0 + lane; b < b1; b += 32) s += W.block[b].s, x += W.block[b].sx;
    if (b1 >= b0) single(b1 * kCellBlock, to);
    __syncwarp();
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        s += __shfl_xor_sync(kFull, s, off);
        x += __shfl_xor_sync(kFull, x, off);
    }
    return make_double2(s, x);
}

constexpr int kCellValues = (kCellFractions + kCellParts) * 2;  // bytes of value_of

// ---- squared error

// Part of an array in shared memory, of one warp: the neighbourhood of a threshold, which moves little from one iteration to the next.
// A load from L2 takes 430 or 820 cycles, by where in L2 it goes, and fifteen warps wait for the longest.
template <int N>
struct Window {
    uint32_t base;   // shared memory
    int first;       // of the array; far below zero: nothing yet
    int last;        // the entry that was asked for before
    bool on_its_way;
    __device__ __forceinline__ Window(double2* p) : base((uint32_t)__cvta_generic_to_shared(p)), first(-2 * N), last(-2 * N), on_its_way(false) {}
    // Entry i of the array; where it is not at hand it is loaded, and its neighbourhood asked for if the step to it was small (with
    // the first iterations' steps the copies would only stand in the way of the others' loads).
    __device__ __forceinline__ double2 entry(const double2* array, int i, int size)
    {
        if (on_its_way) {
            copies_done();
            __syncwarp();
            on_its_way = false;
        }
        const bool near = abs(i - last) < N / 4;
        last = i;
        if ((uint32_t)(i - first) < (uint32_t)N) {
            double2 v;
            asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(base + (uint32_t)(i - first) * 16u) : "memory");
            return v;
        }
        const double2 v = __ldg(array + i);
        if (near) {
            __syncwarp();  // what it holds has been read
            first = min(max(i - N / 2, 0), size - N);
#pragma unroll
            for (int k = threadIdx.x & 31; k < N; k += 32)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + (uint32_t)k * 16u), "l"(array + first + k) : "memory");
            on_its_way = true;
        }
        return v;
    }
};

// An iteration over 2^26 bf16 weights took 1.61 us with cells put in the order of 65,536 bins by sorting, 1.10 with running sums over
// these bins, 1.11 with places and all sums loaded, 0.9 this way; 1.45 with all thresholds in one warp, a lane each, and no barrier (the chain
// of a single warp is longer than a barrier and the waiting for others).
constexpr int kWindow = 256;
constexpr int kCellsMseLow = (kCellBlocks + 1) * 16;
constexpr int kCellsMseValues = 2 * kCellsMseLow;
constexpr int kCellsMseWindows = kCellsMseValues + kCellValues;
constexpr int kCellsMseSmem = kCellsMseWindows + (kLevels - 1) * kWindow * 16;
__global__ void __launch_bounds__(kFitThreads, 1)
cells_fit_mse_kernel(const __grid_constant__ CellsWs W, const __grid_constant__ SortFit F)
{
    if (!after_previous()) return;
    extern __shared__ __align__(16) unsigned char s_fit[];
    double2* const s_high = reinterpret_cast<double2*>(s_fit);  // {s, sx} of the blocks in front of a block
    double2* const s_low = reinterpret_cast<double2*>(s_fit + kCellsMseLow);
    uint16_t* const s_value = reinterpret_cast<uint16_t*>(s_fit + kCellsMseValues);
    // What lies below threshold k - 1: whole blocks (high, low), the rest.  Entry 0: nothing, entry 16: everything.  Two sets, used
    // in turn.
    __shared__ double2 s_below[2][3][kLevels + 1];
    __shared__ float2 s_cut[2][kLevels + 1];  // the threshold, and its place
    __shared__ float s_level[2][kLevels];
    __shared__ int s_stop;  // the iteration behind whose barrier all leave
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float inf = __int_as_float(0x7f800000);
    if (tid == 0) s_stop = 0x7fffffff;
    copy_in(s_value, W.value_of, kCellValues);
    double w2 = 0.0;
    if (warp == kLevels - 1) {
#pragma unroll 8
        for (int k = lane; k < kCellBlocks; k += 32) w2 += W.block[k].sxx;
#pragma unroll
        for (int off = 16; off; off >>= 1) w2 += __shfl_xor_sync(kFull, w2, off);
    }
    // running sums of the blocks, six to a thread
    {
        constexpr int PER = (kCellBlocks + kFitThreads - 1) / kFitThreads;
        static_assert(kCellBlocks < PER * kFitThreads, "what lies in front of the end has a thread");
        TwoSum s[PER], x[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const bool in = tid * PER + k < kCellBlocks;
            const CellBlock* b = W.block + (in ? tid * PER + k : 0);
            s[k] = TwoSum{in ? b->s : 0.0, 0.0}, x[k] = TwoSum{in ? b->sx : 0.0, 0.0};
        }
        TwoSum ts = s[0], tx = x[0];
#pragma unroll
        for (int k = 1; k < PER; ++k) ts = two_add(ts, s[k]), tx = two_add(tx, x[k]);
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
        for (int k = 0; k < PER; ++k) {
            if (tid * PER + k > kCellBlocks) break;  // [kCellBlocks]: everything
            s_high[tid * PER + k] = make_double2(rs.h, rx.h);
            s_low[tid * PER + k] = make_double2(rs.l, rx.l);
            rs = two_add(rs, s[k]), rx = two_add(rx, x[k]);
        }
    }
    copies_done();
    __syncthreads();
    const SharedTable<double2> high(s_high), low(s_low);
    const SharedTable<uint16_t> value_of(s_value);
    Window<kWindow> window(reinterpret_cast<double2*>(s_fit + kCellsMseWindows) + min(warp, kLevels - 2) * kWindow);
    // warps 0 to 14: lane k has level warp + k % 2, those on either side of the warp's threshold; the last warp: lane l has level l
    const bool last = warp == kLevels - 1;
    const int mine = last ? lane & (kLevels - 1) : warp + (lane & 1);
    const bool fixed = (F.fixed_mask >> mine) & 1u;
    float lv = F.codebook[mine];
    if (tid < 2) {
        const double2 none = make_double2(0.0, 0.0);
        for (int k = 0; k < 3; ++k) s_below[tid][k][0] = none;
        s_below[tid][0][kLevels] = s_high[kCellBlocks];
        s_below[tid][1][kLevels] = s_low[kCellBlocks];
        s_below[tid][2][kLevels] = none;
        s_cut[tid][0] = make_float2(-inf, __uint_as_float(0u));
        s_cut[tid][kLevels] = make_float2(inf, __uint_as_float((uint32_t)kCellPlaces));
    }
    if (last) {
        squared_errors(F, w2, s_level, s_below, s_stop);
        return;
    }
    for (int iter = 0; iter < F.iters; ++iter) {
        const int set = iter & 1;
        const float p = __fmul_rn(__fadd_rn(lv, __shfl_xor_sync(kFull, lv, 1)), 0.5f);
        const int place = place_of<32>(p, value_of);
        const double2 whole = ((lane & 1) ? low : high)[place / kCellBlock];
        if ((lane | 1) == 3) s_below[set][lane & 1][warp + 1] = whole;
        if (lane == 4) s_cut[set][warp + 1] = make_float2(p, __uint_as_float((uint32_t)place));
        const double2 rest = window.entry(W.front, place, kCellBlocks * kCellBlock);
        if (lane == 0) s_below[set][2][warp + 1] = rest;
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
                const double2 t = cell_region(W, __shfl_sync(kFull, c0.x, k), __shfl_sync(kFull, c1.x, k));
                if ((lane & 1) == k) s0 = t.x, moved = (float)(t.y / t.x);
            }
        }
        if (!fixed && !empty && s0 > 0.0) lv = moved;
    }
    // (a stop: the levels have not moved since the iteration before)
    if (lane == 0 || (lane == 1 && warp == kLevels - 2))
        if (!fixed) F.codebook[mine] = lv;
    copies_done();  // nothing of this CTA is in flight when it ends
}

// ---- absolute error
//
// Warp l forms what lies below the two thresholds beside level l and looks for the median between them: the first cell, in the order of
// x, with which the weight reaches half of the region's.  Its part is found by three steps of 32 entries in shared memory, its place
// among the 128 of the part by one round of loads.  One more warp, with half a region per lane, adds up the error
// and stops the others when no level has moved.
// An iteration over eight layers of a 7B-shaped model 5.6 us with sorted cells, 2.5 with running sums over 65,536 bins, 1.9 with places and
// sixteen warps for the error, a barrier before the medians, 1.41 with one warp for it and no such barrier, 1.30 with what an iteration's
// error needs loaded behind the one before and 32 errors divided at once (2^22 and 2^26 weights).
constexpr int kCellsMaeThreads = kFitThreads + 32;
constexpr int kCellsMaeHigh = ((kCellPartsAll + 1) * 8 + 15) / 16 * 16;       // shared memory: weights in front of the parts, {s, sx} in
constexpr int kCellsMaeLow = kCellsMaeHigh + (kCellBlocks + 1) * 16;          // front of the blocks, high and low halves,
constexpr int kCellsMaeValues = kCellsMaeLow + (kCellBlocks + 1) * 16;        // value_of
constexpr int kCellsMaeSmem = kCellsMaeValues + kCellValues;
__global__ void __launch_bounds__(kCellsMaeThreads, 1)
cells_fit_mae_kernel(const __grid_constant__ CellsWs W, const __grid_constant__ SortFit F)
{
    if (!after_previous()) return;
    extern __shared__ __align__(16) unsigned char s_fit[];
    unsigned long long* const s_a = reinterpret_cast<unsigned long long*>(s_fit);
    double2* const s_high = reinterpret_cast<double2*>(s_fit + kCellsMaeHigh);
    double2* const s_low = reinterpret_cast<double2*>(s_fit + kCellsMaeLow);
    uint16_t* const s_value = reinterpret_cast<uint16_t*>(s_fit + kCellsMaeValues);
    __shared__ float s_level[2][kLevels];
    __shared__ int s_stop;  // the iteration behind whose barrier all leave
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    copy_in(s_value, W.value_of, kCellValues);
    if (tid < kLevels) s_level[0][tid] = F.codebook[tid];
    if (tid == 0) s_stop = 0x7fffffff;
    CellBlock* const s_block = reinterpret_cast<CellBlock*>(s_high);  // the blocks' sums, before the running sums take their place
    static_assert(kCellBlocks * sizeof(CellBlock) + 16 <= 2 * (kCellBlocks + 1) * sizeof(double2), "room for the blocks' sums");
    copy_in(s_block, W.block, kCellBlocks * (int)sizeof(CellBlock));
    copy_in(s_a, W.part_a, kCellPartsAll * 8);
    copies_done();
    __syncthreads();
    running_sums<kCellPer, TwoPair>(warp < kLevels, kCellBlocks, [&](int b) { return TwoPair{{s_block[b].s, 0.0}, {s_block[b].sx, 0.0}}; },
                                    [&](int b, const TwoPair& v) {
                                        s_high[b] = make_double2(v.s.h, v.x.h);
                                        s_low[b] = make_double2(v.s.l, v.x.l);
                                    });
    running_sums<kCellPartsAll / kFitThreads + 1, unsigned long long>(warp < kLevels, kCellPartsAll, [&](int p) { return s_a[p]; },
                                                                     [&](int p, unsigned long long v) { s_a[p] = v; });
    __syncthreads();
    const SharedTable<uint16_t> value_of(s_value);
    const SharedTable<unsigned long long> parts_a(s_a);
    if (warp == kLevels) {
        // ---- the error, a half region to a lane
        const SharedTable<double2> high(s_high), low(s_low);
        const int l = lane & (kLevels - 1), from = lower_end_of(lane);
        float before = __int_as_float(0x7fc00001);
        double err = 0.0, kept = 0.0;
        // Of iteration k, formed behind the loads of the next one; 32 are kept, a lane each, and written together.
        Below end;
        double2 rest;
        FitPoints at;
        auto add_up = [&](int k) {
            end.low.x += rest.x, end.low.y += rest.y;
            const Below begin{make_double2(__shfl_sync(kFull, end.high.x, from), __shfl_sync(kFull, end.high.y, from)),
                              make_double2(__shfl_sync(kFull, end.low.x, from), __shfl_sync(kFull, end.low.y, from))};
            err = half_error(lane, at, before, begin, end);
#pragma unroll
            for (int off = 16; off; off >>= 1) err += __shfl_xor_sync(kFull, err, off);
            if (lane == (k & 31)) kept = err;
            if ((k & 31) == 31 && F.err_log) F.err_log[k - 31 + lane] = fmax(kept, 0.0) / (double)F.n_total;
        };
        int iter = 0;
        for (; iter < F.iters; ++iter) {
            const float* const lvs = s_level[iter & 1];
            const float lv = lvs[l];
            const FitPoints now = points_of(l, lvs[max(l - 1, 0)], lv, lvs[min(l + 1, kLevels - 1)]);
            const int place = place_of<1>(lane < kLevels ? now.mid : now.hi, value_of);
            const double2 next = __ldg(W.front + place);
            if (iter) add_up(iter - 1);
            // the levels have stopped to move: the iterations from this one on repeat the one before bit for bit
            const bool same = __all_sync(kFull, __float_as_uint(lv) == __float_as_uint(before));
            if (same && lane == 0) s_stop = iter;
            __syncthreads();
            if (same) break;
            before = lv, at = now, rest = next;
            end = Below{high[place / kCellBlock], low[place / kCellBlock]};
        }
        if (iter == F.iters) add_up(iter - 1);
        if (F.err_log) {
            if (lane < (iter & 31)) F.err_log[(iter & ~31) + lane] = fmax(kept, 0.0) / (double)F.n_total;
            for (int k = iter + lane; k < F.iters; k += 32) F.err_log[k] = fmax(err, 0.0) / (double)F.n_total;
        }
        return;
    }
    // ---- warp l: level l
    const bool fixed = (F.fixed_mask >> warp) & 1u;
    float lv = s_level[0][warp];
    for (int iter = 0; iter < F.iters; ++iter) {
        const int set = iter & 1;
        if (!fixed) {
            // half the warp has the threshold below, half that above
            const bool up = lane & 16, end = up ? warp == kLevels - 1 : warp == 0;
            const float other = s_level[set][min(max(warp + (up ? 1 : -1), 0), kLevels - 1)], inf = __int_as_float(0x7f800000);
            const int place = place_of<16>(end ? (up ? inf : -inf) : __fmul_rn(__fadd_rn(lv, other), 0.5f), value_of);
            const unsigned long long a = __ldg(W.front_a + place) + parts_a[place / kCellPart];
            const unsigned long long a0 = __shfl_sync(kFull, a, 0), a1 = __shfl_sync(kFull, a, 16);
            // (levels that do not ascend have regions without samples)
            if (a1 != a0 && __shfl_sync(kFull, place, 0) < __shfl_sync(kFull, place, 16)) {
                const unsigned long long goal = a0 + (a1 - a0) - (a1 - a0) / 2ull;
                // the last part in front of which there is less than the goal
                constexpr int S1 = (kCellPartsAll + 31) / 32, S2 = (S1 + 31) / 32;
                static_assert(S2 <= 32, "three steps");
                auto less = [&](int i) { return parts_a[min(i, kCellPartsAll)] < goal; };
                int b = S1 * __popc(__ballot_sync(kFull, less(S1 * (lane + 1))));
                b += S2 * __popc(__ballot_sync(kFull, S2 * (lane + 1) < S1 && less(b + S2 * (lane + 1))));
                b += __popc(__ballot_sync(kFull, lane < S2 && less(b + 1 + lane)));
                b = min(b, kCellPartsAll - 1);
                // the last of its places with less in front
                constexpr int U = kCellPart / 32;
                unsigned long long f[U];
#pragma unroll
                for (int k = 0; k < U; ++k) f[k] = __ldg(W.front_a + b * kCellPart + 32 * k + lane);
                const unsigned long long need = goal - parts_a[b];
                int n = b * kCellPart - 1;
#pragma unroll
                for (int k = 0; k < U; ++k) n += __popc(__ballot_sync(kFull, f[k] < need));
                uint32_t cell;
                cell_at(n, value_of, cell, lv);
            }
            if (lane == 0) s_level[set ^ 1][warp] = lv;
        } else if (lane == 0) {
            s_level[set ^ 1][warp] = lv;
        }
        __syncthreads();
        if (s_stop <= iter) break;
    }
    if (lane == 0 && !fixed) F.codebook[warp] = lv;
}

int cells_run(const CellsWs& W, const SortFit& F, cudaStream_t st)
{
    if (F.metric == BOF4_METRIC_MAE || F.metric == BOF4_METRIC_MAE_NORMALIZED) {
        if (const int rc = ensure_dynamic_smem<cells_fit_mae_kernel>(kCellsMaeSmem)) return rc;
        launch_after(cells_sums_kernel<true>, kCellBlocks, kCellBlock, 0, st, W);
        launch_after(cells_fit_mae_kernel, 1, kCellsMaeThreads, kCellsMaeSmem, st, W, F);
    } else {
        if (const int rc = ensure_dynamic_smem<cells_fit_mse_kernel>(kCellsMseSmem)) return rc;
        launch_after(cells_sums_kernel<false>, kCellBlocks, kCellBlock, 0, st, W);
        launch_after(cells_fit_mse_kernel, 1, kFitThreads, kCellsMseSmem, st, W, F);
    }
    BOF4_CUDA_TRY(cudaGetLastError());
    return BOF4_OK;
}

}  // namespace bof4
