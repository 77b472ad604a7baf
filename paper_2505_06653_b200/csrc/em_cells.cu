// Codebook fit of bf16 data over its distinct normalised weights (see em_sorted.cuh).
//
// A bf16 number has an 8-bit significand, so w / m is (a / b) 2^e with a and b in 128 ... 255: whatever
// the size of the data, the normalised weights of magnitude 2^-40 and more take at most 128 * 128 * 2 * 40
// values, and the fit only needs the sum of the sample weights (m^2 or |m|) of each.  The data is read
// twice, once for the block constants and once for the counts; then a fit of any number of iterations
// works on 1.3 million cells (of which near-Gaussian data occupies about 0.4 million).
//
//   blocks      block constants (bf16, stored) and the number of blocks per magnitude; HBM bound
//   plan        first position of every magnitude, units of work; the order of the fractions a / b
//   order       block addresses grouped by magnitude
//   accumulate  a unit is some blocks of ONE magnitude |m|: with m fixed, the cell of a weight is the
//               difference of the two bit patterns, so the counts of a unit are 10240 words of shared
//               memory and a weight costs a subtraction, a comparison and one shared-memory reduction,
//               whose rate bounds it (4.6 cycles per 32 weights; a counter per lane for four binades, so that no two
//               lanes meet at a bank, takes two reductions of 4.4 each: 811 -> 1570 us; two
//               weights at a time without a predicate where all are counted: 2^26 weights 56 -> 51 us, 1.6 * 10^9 827 -> 811);
//               when the unit is done its counts times the weight of |m| are added to the cells
//   then        sums of the cells in the order of x, and all iterations (em_cells_fit.cu)
//
// A cell is (significand of m, sign, distance of the bit patterns).  Cell sums are integers (128 bits, a
// fixed-point scale relative to the largest |m|; exact while |m| is within 2^-38 of it), so they do not
// depend on the order of the additions.  Normalised weights of 2^-40 and less in magnitude are told apart by sign and
// exponent only (deep cells): they count as the power of two at or below them.  Whether a lane's sixteen weights have
// any is seen from the largest distance among them, a three-way maximum per four weights: eight layers of a 7B-shaped model, medians,
// 1850 -> 1857 us (1897 with a two-way maximum, 1994 with the smallest magnitude that is not zero).
#include "em_cells.cuh"
#include "lane32.cuh"

namespace bof4 {

constexpr int kCellCounts = 2 * kCellDepth + 2 * kDeepExps;  // counters of a unit: one magnitude, zeros left out
constexpr int kMags = 32768;                      // magnitudes of a bf16 number
constexpr int kCellBaseMax = 8192;                // bound on where a unit's counters begin in shared memory: behind the system's
                                                  // kilobyte and the kernel's own variables
constexpr int kCellThreads = 512;
constexpr int kCellCtas = 3;                      // per SM
constexpr int kOrderGroup = 8;                   // blocks that a thread of the ordering takes at a time
// Below, a fit has one sample per weight.  That is no longer the faster way (20 iterations, MSE and MAE, one sample per weight against
// this way: 2^17 weights 77 and 106 us against 73 and 85, 2^19 83 and 120 against 73 and 85, 2^20 93 and 142 against 74 and 87, 2^21 126 and
// 187 against 75 and 89; the two crossed here while the cells were sorted), but small fits have not got the limits that the cells have (weights
// below 2^-40 and constants below 2^-38, see the header), and take 16 bytes a weight where the cells take 64 MB.
constexpr int64_t kCellsMinN = (int64_t)3 << 19;
constexpr int kMagTiny = 48 * 128;                // |m| below 2^-79: subnormal weights within 40 binades

bool cells_apply(int w_dtype, int64_t n) { return w_dtype == BOF4_BF16 && n >= kCellsMinN; }

constexpr int kMaxExtraUnits = 16 * kSMs;  // units beyond one per magnitude: blocks / unit size

static int unit_blocks(int64_t blocks, int block_size)
{
    const int64_t least = 131072 / block_size, even = (blocks + kMaxExtraUnits - 1) / kMaxExtraUnits;
    return (int)(even > least ? even : least);
}

static size_t cells_layout(void* base, int64_t n, int block_size, CellsWs* W)
{
    char* p = static_cast<char*>(base);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* q = p ? p + off : nullptr;
        off += align_up(bytes, 256);
        return q;
    };
    const size_t blocks = (size_t)(n / block_size) + 1;
    CellsWs L;
    L.hist = reinterpret_cast<uint32_t*>(take((size_t)kMags * 4));
    L.scal = reinterpret_cast<uint32_t*>(take(256));
    L.acc = reinterpret_cast<ulonglong2*>(take((size_t)kCells * 16));
    L.acc_a = reinterpret_cast<unsigned long long*>(take((size_t)kCells * 8));  // the four arrays above are cleared together
    L.cursor = reinterpret_cast<uint32_t*>(take((size_t)kMags * 4));
    L.units = reinterpret_cast<CellUnit*>(take((size_t)(kMags + kMaxExtraUnits) * sizeof(CellUnit)));
    L.order = reinterpret_cast<unsigned long long*>(take(blocks * 8));
    L.consts = reinterpret_cast<uint16_t*>(take(align_up(blocks, kOrderGroup) * 2));
    L.value_of = reinterpret_cast<uint16_t*>(take((size_t)(kCellFractions + kCellParts) * 2));
    L.front = reinterpret_cast<double2*>(take((size_t)kCellBlocks * kCellBlock * 16));
    L.front_a = reinterpret_cast<unsigned long long*>(take((size_t)kCellBlocks * kCellBlock * 8));
    L.block = reinterpret_cast<CellBlock*>(take((size_t)kCellBlocks * sizeof(CellBlock)));
    L.part_a = reinterpret_cast<unsigned long long*>(take((size_t)kCellPartsAll * 8));
    if (W) *W = L;
    return off;
}

size_t cells_workspace_bytes(int64_t n, int block_size)
{
    return cells_layout(nullptr, n, block_size, nullptr);
}

// ---------------------------------------------------------------- weights and cells of one magnitude

// Bit pattern of a bf16 value scaled by 2^64 (exact; makes subnormal values normal).
__device__ __forceinline__ uint32_t scaled16(uint32_t bits)
{
    return __float_as_uint(__uint_as_float(bits << 16) * 0x1p64f) >> 16;
}

// The sample weight of |m| (per weight) as an integer times 2^shift.
struct MagWeight {
    uint32_t b;       // significand, 128 ... 255
    uint32_t base;    // b^2, b or 1
    int shift;
    uint32_t fixed;   // MAE: weight of the median
};
constexpr int kMseScale = 76, kMaeScale = 84;  // 2^33 weights of the largest |m| stay below 2^128

__device__ __forceinline__ int true_exponent(uint32_t mag)  // biased exponent, extended below the normal range
{
    return mag < (uint32_t)kMagTiny ? (int)(scaled16(mag) >> 7) - 64 : (int)(mag >> 7);
}
__device__ __forceinline__ MagWeight mag_weight(uint32_t mag, uint32_t max_mag, int metric)
{
    MagWeight r;
    const uint32_t s = mag < (uint32_t)kMagTiny ? scaled16(mag) : mag;
    r.b = 128u + (s & 127u);
    const int k = true_exponent(max_mag) - true_exponent(mag);
    if (metric >= 2) {
        r.base = 1u;
        r.shift = kMaeScale;
        r.fixed = 1u;
    } else if (metric == BOF4_METRIC_MSE) {
        r.base = r.b * r.b;
        r.shift = kMseScale - 2 * k;
        r.fixed = 0u;
    } else {
        r.base = r.b;
        r.shift = kMaeScale - k;
        r.fixed = sort_fixed_weight(__uint_as_float(mag << 16), max_mag << 16);
    }
    return r;
}
__device__ __forceinline__ double cell_scale(uint32_t max_mag, int metric)
{
    if (metric >= 2) return ldexp(1.0, -kMaeScale);
    const int e = true_exponent(max_mag) - 134;  // |m| = b 2^(exponent - 134)
    return metric == BOF4_METRIC_MSE ? ldexp(1.0, 2 * e - kMseScale) : ldexp(1.0, e - kMaeScale);
}

__device__ __forceinline__ void cell_add(const CellsWs& W, uint32_t cell, unsigned long long count, const MagWeight& m, bool mae)
{
    const unsigned long long v = count * m.base;
    unsigned long long lo, hi = 0ull;
    if (m.shift >= 64) {
        lo = 0ull;
        hi = v << (m.shift - 64);
    } else if (m.shift > 0) {
        lo = v << m.shift;
        hi = v >> (64 - m.shift);
    } else {
        lo = m.shift > -64 ? v >> (-m.shift) : 0ull;
    }
    unsigned long long* p = reinterpret_cast<unsigned long long*>(W.acc + cell);
    if (lo) {
        const unsigned long long old = atomicAdd(p, lo);
        if (old + lo < old) ++hi;
    }
    if (hi) atomicAdd(p + 1, hi);
    if (mae && m.fixed) atomicAdd(W.acc_a + cell, count * m.fixed);
}

// ---------------------------------------------------------------- block constants

template <int I, bool SIGNED>
__global__ void __launch_bounds__(1024, 1)
cells_blocks_kernel(const EmTensors T, const int64_t first_block, uint32_t* __restrict__ hist, uint16_t* __restrict__ consts)
{
    if (!after_previous()) return;
    extern __shared__ uint32_t s_hist[];  // [kMags]
    __shared__ WideScratch s_wide;
    __shared__ const void* s_ptr[kEmMaxTensors];
    __shared__ int64_t s_n[kEmMaxTensors], s_row_end[kEmMaxTensors], s_block0[kEmMaxTensors];
    const int tid = threadIdx.x;
    for (int k = tid; k < kMags; k += 1024) s_hist[k] = 0u;
    if (tid < T.count) {
        s_ptr[tid] = T.ptr[tid];
        s_n[tid] = T.n[tid];
        s_row_end[tid] = T.row_end[tid];
    }
    if (tid == 0) {
        int64_t b = first_block;
        for (int t = 0; t < T.count; ++t) {
            s_block0[t] = b;
            b += T.n[t] / I;
        }
    }
    __syncthreads();
    const int64_t total_rows = T.row_end[T.count - 1];
    int t_cur = 0;
    auto fetch = [&](int64_t g, int64_t& block) -> Raw32 {  // block: this lane's block, or -1 past the end
        block = -1;
        if (g < total_rows) {
            while (g >= s_row_end[t_cur]) ++t_cur;
            const int64_t r = g - (t_cur ? s_row_end[t_cur - 1] : 0);
            const int64_t idx = (r * 1024 + tid) * kLW;
            if (idx < s_n[t_cur]) {
                block = s_block0[t_cur] + idx / I;
                if (idx & (I - 1)) block |= (int64_t)1 << 62;  // not the block's first lane
                return load_raw32(s_ptr[t_cur], idx);
            }
        }
        return zero_raw32();
    };
    auto row = [&](const Raw32& raw, int64_t block) {
        uint32_t u[16];
        words_of(raw, u);
        float mx, mn, g;
        lane_minmax32(u, mx, mn);
        const float m = block_constant32<I, SIGNED>(u, mx, mn, g, &s_wide);
        if (block >= 0 && !(block >> 62)) {
            const uint32_t b = __float_as_uint(m) >> 16;
            consts[block] = (uint16_t)b;
            atomicAdd(&s_hist[b & 0x7fffu], 1u);
        }
    };
    int64_t g = blockIdx.x, ba, bb;
    const int64_t GS = gridDim.x;
    Raw32 a = fetch(g, ba), b;
    while (g < total_rows) {  // two row buffers used in turn
        b = fetch(g + GS, bb);
        row(a, ba);
        g += GS;
        if (g >= total_rows) break;
        a = fetch(g + GS, ba);
        row(b, bb);
        g += GS;
    }
    __syncthreads();
    for (int k = tid; k < kMags; k += 1024)
        if (s_hist[k]) atomicAdd(&hist[k], s_hist[k]);
}

// ---------------------------------------------------------------- plan

// One CTA, 32 magnitudes per thread, 1024 apart: positions of the magnitudes in the ordered list, the units of work,
// the largest magnitude and the scale of the cell sums.  The magnitudes that most blocks have are neighbours (a binade
// has 128), so they lie with different threads; with 32 neighbours to a thread one of them wrote most of the
// units (2^26 weights 20 us against 7, 2^30 26 against 11).  The order of the magnitudes in the list is of no account.
// The other CTAs put the fractions in order meanwhile.
__global__ void __launch_bounds__(1024)
cells_plan_kernel(const CellsWs W, uint32_t per_unit, int metric)
{
    if (!after_previous()) return;
    if (blockIdx.x) {
        const uint32_t f = (blockIdx.x - 1) * kFractionThreads + threadIdx.x;
        if (threadIdx.x >= kFractionThreads) return;
        if (f < kCellFractions) W.value_of[fraction_rank(f >> 7, f & 127u)] = (uint16_t)f;
        else W.value_of[f] = (uint16_t)fractions_below(f - kCellFractions);
        return;
    }
    __shared__ uint32_t s_blocks[32], s_units[32], s_top;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_top = W.scal[2];
    uint32_t c[32], blocks = 0u, units = 0u, top = 0u;
#pragma unroll
    for (int k = 0; k < 32; ++k) c[k] = W.hist[k * 1024 + tid];
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        blocks += c[k];
        if (c[k]) {
            units += (c[k] + per_unit - 1) / per_unit;
            top = (uint32_t)(k * 1024 + tid);
        }
    }
    uint32_t ib = blocks, iu = units;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t x = __shfl_up_sync(kFull, ib, off), y = __shfl_up_sync(kFull, iu, off);
        if (lane >= off) {
            ib += x;
            iu += y;
        }
    }
    __syncthreads();
    if (lane == 31) {
        s_blocks[warp] = ib;
        s_units[warp] = iu;
    }
    top = __reduce_max_sync(kFull, top);
    if (lane == 0) atomicMax(&s_top, top);
    __syncthreads();
    for (int k = 0; k < warp; ++k) {
        ib += s_blocks[k];
        iu += s_units[k];
    }
    uint32_t at = ib - blocks, u = iu - units;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const uint32_t mag = (uint32_t)(k * 1024 + tid);
        W.cursor[mag] = at;
        for (uint32_t done = 0; done < c[k]; done += per_unit)
            W.units[u++] = CellUnit{mag, at + done, min(per_unit, c[k] - done)};
        at += c[k];
    }
    if (tid == 1023) {
        W.scal[0] = iu;
        W.scal[1] = 0u;
    }
    if (tid == 0) {
        W.scal[3] = s_top;
        *cells_scale(W) = cell_scale(s_top, metric);
    }
}

// ---------------------------------------------------------------- order

// Few blocks: every CTA takes a contiguous part of them, counts its magnitudes, reserves room for them in the
// list, then writes the addresses.  The order inside a magnitude does not matter (sums of integers).
__global__ void __launch_bounds__(1024, 1)
cells_order_few_kernel(const EmTensors T, const int64_t first_block, const int64_t n_blocks, int block_size, const CellsWs W)
{
    if (!after_previous()) return;
    extern __shared__ uint32_t s_pos[];  // [kMags]
    __shared__ const char* s_ptr[kEmMaxTensors];
    __shared__ int64_t s_end[kEmMaxTensors];  // first block behind the tensor
    const int tid = threadIdx.x;
    for (int k = tid; k < kMags; k += 1024) s_pos[k] = 0u;
    if (tid == 0) {
        int64_t b = first_block;
        for (int t = 0; t < T.count; ++t) {
            // address that block 0 would have
            s_ptr[t] = static_cast<const char*>(T.ptr[t]) - b * block_size * 2;
            b += T.n[t] / block_size;
            s_end[t] = b;
        }
    }
    __syncthreads();
    const int64_t part = (n_blocks + gridDim.x - 1) / gridDim.x;
    const int64_t lo = first_block + (int64_t)blockIdx.x * part;
    const int64_t hi = min(first_block + n_blocks, lo + part);
#pragma unroll 4
    for (int64_t i = lo + tid; i < hi; i += 1024) atomicAdd(&s_pos[W.consts[i] & 0x7fffu], 1u);
    __syncthreads();
    for (int k = tid; k < kMags; k += 1024)
        if (s_pos[k]) s_pos[k] = atomicAdd(&W.cursor[k], s_pos[k]);
    __syncthreads();
    int t = 0;
#pragma unroll 4
    for (int64_t i = lo + tid; i < hi; i += 1024) {
        while (i >= s_end[t]) ++t;
        const uint32_t c = W.consts[i];
        const unsigned long long p = reinterpret_cast<unsigned long long>(s_ptr[t] + i * block_size * 2);
        W.order[atomicAdd(&s_pos[c & 0x7fffu], 1u)] = p | ((unsigned long long)(c >> 15) << 63);
    }
}

// Every CTA takes a contiguous part of the blocks, 8192 at a time: ranks them within their magnitudes, reserves room for
// every magnitude in the list, puts the tile in order in shared memory and writes its addresses, so that neighbouring lanes
// write neighbouring places.  The order inside a magnitude does not matter (sums of integers).  Writing each address from
// the lane that has the block, 32 cache lines a store, took 207 us for the 25 million blocks of eight layers of a 7B-shaped
// model, 113 this way (fits of 2^28 and 2^30 weights 10 and 60 us faster).  Bound by the counters, whose lanes collide on common
// magnitudes, and the chain of a tile: the reservation in global memory, five barriers.  (A lane counting for all of its
// magnitude in the warp, by __match_any_sync: 248 us.)
// Fewer blocks in a launch are written directly.  Fits of 8 iterations, directly and in tiles: 2^16 blocks (2^22 weights) 132.7 us and
// 136.6, 3 * 2^17 156 and 163, 2^19 173.3 and 173.7, 2^20 207 and 205.5, 2^22 417 and 404.  (Constants spread over six binades in every
// tensor: 2^19 the same, 2^20 210 and 216, 2^21 295 and 299, 2^22 445 and 445.)
constexpr int64_t kOrderFew = 1 << 19;
constexpr int kOrderTile = 1024 * kOrderGroup;
static_assert(kOrderTile == 1 << 13, "13 bits for a place in a tile");
constexpr int kOrderSmem = kMags * 4 + kOrderTile * (4 + 4 + 2);
__global__ void __launch_bounds__(1024, 1)
cells_order_kernel(const EmTensors T, const int64_t first_block, const int64_t n_blocks, int block_size, const CellsWs W)
{
    if (!after_previous()) return;
    extern __shared__ __align__(16) uint32_t s_pos[];  // [kMags] blocks of a magnitude in the tile, then its slot and first place
    uint32_t* const s_item = s_pos + kMags;            // [kOrderTile] slot, sign, block in the tile
    uint32_t* const s_delta = s_item + kOrderTile;     // [kOrderTile] per slot: place in the list less place in the tile
    uint16_t* const s_mag = reinterpret_cast<uint16_t*>(s_delta + kOrderTile);  // [kOrderTile] per slot
    __shared__ const char* s_ptr[kEmMaxTensors];
    __shared__ int64_t s_end[kEmMaxTensors];  // first block behind the tensor
    __shared__ uint32_t s_slots, s_warp[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = tid; k < kMags / 4; k += 1024) reinterpret_cast<uint4*>(s_pos)[k] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
        int64_t b = first_block;
        for (int t = 0; t < T.count; ++t) {
            // address that block 0 would have
            s_ptr[t] = static_cast<const char*>(T.ptr[t]) - b * block_size * 2;
            b += T.n[t] / block_size;
            s_end[t] = b;
        }
        s_slots = 0u;
    }
    __syncthreads();
    // groups of eight blocks, of which the first and the last of the launch may belong to others in part
    const int64_t end = first_block + n_blocks, g0 = first_block / kOrderGroup, groups = (end + kOrderGroup - 1) / kOrderGroup - g0;
    const int64_t part = (groups + gridDim.x - 1) / gridDim.x;
    const int64_t lo = g0 + (int64_t)blockIdx.x * part, hi = min(g0 + groups, lo + part);
    const uint4* consts = reinterpret_cast<const uint4*>(W.consts);  // (room for whole groups: cells_layout)
    uint4 next = lo + tid < hi ? consts[lo + tid] : make_uint4(0u, 0u, 0u, 0u);
    int t = 0;
    for (int64_t tile = lo; tile < hi; tile += 1024) {
        const int64_t g = tile + tid, i0 = g * kOrderGroup;
        const uint32_t w[4] = {next.x, next.y, next.z, next.w};
        if (g + 1024 < hi) next = consts[g + 1024];
        const int from = g < hi ? (int)max(first_block - i0, (int64_t)0) : kOrderGroup;
        const int to = (int)min(end - i0, (int64_t)kOrderGroup);
        uint32_t rank[kOrderGroup];
#pragma unroll
        for (int k = 0; k < kOrderGroup; ++k) {
            const uint32_t mag = (w[k >> 1] >> (16 * (k & 1))) & 0x7fffu;
            rank[k] = k >= from && k < to ? atomicAdd(&s_pos[mag], 1u) : 1u;
        }
#pragma unroll
        for (int k = 0; k < kOrderGroup; ++k)
            if (rank[k] == 0u) s_mag[atomicAdd(&s_slots, 1u)] = (uint16_t)((w[k >> 1] >> (16 * (k & 1))) & 0x7fffu);
        __syncthreads();
        const uint32_t slots = s_slots;
        uint32_t placed = 0u;  // blocks of the slots before
        for (uint32_t j0 = 0; j0 < slots; j0 += 1024) {
            const uint32_t j = j0 + tid;
            uint32_t mag = 0u, count = 0u, at = 0u;
            if (j < slots) {
                mag = s_mag[j];
                count = s_pos[mag];
                at = atomicAdd(&W.cursor[mag], count);
            }
            uint32_t incl = count;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t x = __shfl_up_sync(kFull, incl, off);
                if (lane >= off) incl += x;
            }
            if (j0) __syncthreads();  // s_warp of the round before has been read
            if (lane == 31) s_warp[warp] = incl;
            __syncthreads();
            const uint32_t mine = s_warp[lane];
            const uint32_t before = __reduce_add_sync(kFull, lane < warp ? mine : 0u), all = __reduce_add_sync(kFull, mine);
            const uint32_t place = placed + before + incl - count;
            if (j < slots) {
                s_pos[mag] = j << 13 | place;
                s_delta[j] = at - place;
            }
            placed += all;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kOrderGroup; ++k) {
            if (k < from || k >= to) continue;
            const uint32_t c = w[k >> 1] >> (16 * (k & 1)), e = s_pos[c & 0x7fffu];
            s_item[(e & (kOrderTile - 1)) + rank[k]] = (e >> 13) << 14 | ((c >> 15) & 1u) << 13 | (uint32_t)(tid * kOrderGroup + k);
        }
        __syncthreads();
        for (uint32_t j = tid; j < slots; j += 1024) s_pos[s_mag[j]] = 0u;
        if (tid == 0) s_slots = 0u;
        const int64_t b0 = tile * kOrderGroup;
        while (max(b0, first_block) >= s_end[t]) ++t;
        const bool one = min(b0 + kOrderTile, end) <= s_end[t];  // the tile lies in one tensor
        const char* const base = s_ptr[t];
#pragma unroll 4
        for (uint32_t p = tid; p < placed; p += 1024) {
            const uint32_t e = s_item[p];
            const int64_t i = b0 + (e & (kOrderTile - 1));
            const char* from_tensor = base;
            if (!one) {
                int u = t;
                while (i >= s_end[u]) ++u;
                from_tensor = s_ptr[u];
            }
            const unsigned long long a = reinterpret_cast<unsigned long long>(from_tensor + i * block_size * 2);
            W.order[s_delta[e >> 14] + p] = a | ((unsigned long long)((e >> 13) & 1u) << 63);
        }
        __syncthreads();  // the next tile overwrites what has been read here
    }
}

// ---------------------------------------------------------------- accumulate

__device__ __forceinline__ void cell_count(uint32_t base, uint32_t d, uint32_t negative)
{
    // positive weights at distance d, negative ones kCellDepth further on; a zero is not counted (the zeros of a unit are
    // what is missing from its number of weights), nor is a weight of 2^-40 of the constant and less (deep_cell)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.lt.u32 p, %0, %2;\n\t"
        "@p red.shared.add.u32 [%1], 1;\n\t}" ::"r"(d),
        "r"(base + d * 4u + (negative ? (uint32_t)kCellDepth * 4u : 0u)), "n"(kCellDepth)
        : "memory");
}

// Which of the deep cells a weight of 2^-40 of the constant and less counts in, or -1 where its quotient is zero.  w: bit pattern
// relative to the constant's sign, mag: the constant's.
__device__ __forceinline__ int deep_cell(uint32_t w, uint32_t mag)
{
    const float x = __fdiv_rn(__uint_as_float((w & 0x7fffu) << 16), __uint_as_float(mag << 16));
    return x == 0.0f ? -1 : (int)(__float_as_uint(x) >> 23) + ((w & 0x8000u) ? kDeepExps : 0);
}
__device__ __noinline__ void deep_count(uint32_t* cnt, uint32_t u, uint32_t mag, bool tiny)
{
    for (int h = 0; h < 2; ++h, u >>= 16) {
        const uint32_t w = u & 0xffffu, a = w & 0x7fffu;
        if (a == 0u || (tiny ? scaled16(mag) - scaled16(a) : mag - a) < (uint32_t)kCellDepth) continue;
        const int at = deep_cell(w, mag);
        if (at >= 0) atomicAdd(cnt + at, 1u);
    }
}

__global__ void __launch_bounds__(kCellThreads, kCellCtas)
cells_accumulate_kernel(const CellsWs W, int lanes_shift, int metric)
{
    if (!after_previous()) return;
    extern __shared__ uint32_t s_cnt[];  // [kCellCounts]
    __shared__ CellUnit s_unit;
    __shared__ uint32_t s_seen[kCellThreads / 32];
    static_assert(1024 + sizeof(s_unit) + sizeof(s_seen) + 256 <= kCellBaseMax, "base below");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(s_cnt);
    const uint32_t units = W.scal[0], max_mag = W.scal[3];
    const bool mae = metric == BOF4_METRIC_MAE || metric == BOF4_METRIC_MAE_NORMALIZED;
    for (int k = tid; k < kCellCounts; k += kCellThreads) s_cnt[k] = 0u;
    while (true) {
        __syncthreads();
        if (tid == 0) {
            const uint32_t u = atomicAdd(&W.scal[1], 1u);
            s_unit = (u < units) ? W.units[u] : CellUnit{0u, 0u, 0u};
        }
        __syncthreads();
        const CellUnit U = s_unit;
        if (U.count == 0u) break;
        const unsigned long long* list = W.order + U.first;
        const uint32_t pieces = U.count << lanes_shift, mask = (1u << lanes_shift) - 1u;  // pieces of 16 weights
        auto load = [&](uint32_t q, uint32_t& flip) -> Raw8 {
            const unsigned long long p = __ldg(list + (q >> lanes_shift));
            flip = (p >> 63) ? 0x80008000u : 0u;
            return ld_stream256(reinterpret_cast<const char*>(p & 0x7fffffffffffffffull) + (q & mask) * 32u);
        };
        if (U.mag == 0u) {
            // all-zero blocks: every weight is a zero (below)
        } else if (U.mag >= (uint32_t)kMagTiny) {
            const uint32_t deep = U.mag - (uint32_t)kCellDepth;  // largest magnitude that goes to a deep cell
            const uint32_t both = U.mag * 0x10001u;
            // Two weights at a time: their distances (no weight is beyond the constant: no borrow between the halves), then
            // the addresses of their counters, two to a word: they have to stay below 2^16.
            static_assert(2 * kCellDepth * 4 + kCellBaseMax <= 1 << 16, "an address would carry into the other half");
            const uint32_t base2 = base * 0x10001u;
            auto use = [&](const Raw8& r, uint32_t flip) {
                constexpr uint32_t kCounted = (uint32_t)(kCellDepth - 1) * 0x10001u;
#pragma unroll
                for (int h = 0; h < 8; h += 4) {
                    uint32_t d[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) d[k] = both - (r.u[h + k] & 0x7fff7fffu);
                    // the largest distance, or the largest that is counted
                    if (__vimax3_u16x2(__vimax3_u16x2(d[0], d[1], d[2]), d[3], kCounted) == kCounted) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const uint32_t negative = ((r.u[h + k] ^ flip) >> 15) & 0x10001u;
                            const uint32_t at = negative * (uint32_t)(kCellDepth * 4) + base2 + d[k] * 4u;
                            asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(at & 0xffffu) : "memory");
                            asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(at >> 16) : "memory");
                        }
                    } else {  // a zero, or a weight for a deep cell
                        uint32_t least = 0xffffffffu;  // the smallest magnitude less one: zeros wrap to the top
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const uint32_t u = r.u[h + k] ^ flip;
                            cell_count(base, d[k] & 0xffffu, u & 0x8000u);
                            cell_count(base, d[k] >> 16, u & 0x80000000u);
                            least = __viaddmin_u16x2(u & 0x7fff7fffu, 0xffffffffu, least);
                        }
                        if ((least & 0xffffu) < deep || (least >> 16) < deep)
                            for (int k = 0; k < 4; ++k) deep_count(s_cnt + 2 * kCellDepth, r.u[h + k] ^ flip, U.mag, false);
                    }
                }
            };
            uint32_t fa, fb, q = tid;
            Raw8 a, b;
            if (q < pieces) a = load(q, fa);
            while (q < pieces) {  // two buffers used in turn
                if (q + kCellThreads < pieces) b = load(q + kCellThreads, fb);
                use(a, fa);
                q += kCellThreads;
                if (q >= pieces) break;
                if (q + kCellThreads < pieces) a = load(q + kCellThreads, fa);
                use(b, fb);
                q += kCellThreads;
            }
        } else {  // subnormal weights may occur: compare scaled bit patterns
            const uint32_t mag = scaled16(U.mag);
            for (uint32_t q = tid; q < pieces; q += kCellThreads) {
                uint32_t flip;
                const Raw8 r = load(q, flip);
                for (int k = 0; k < 8; ++k) {
                    const uint32_t u = r.u[k] ^ flip;
                    cell_count(base, mag - (scaled16(u & 0xffffu) & 0x7fffu), u & 0x8000u);
                    cell_count(base, mag - (scaled16(u >> 16) & 0x7fffu), u & 0x80000000u);
                    deep_count(s_cnt + 2 * kCellDepth, u, U.mag, true);
                }
            }
        }
        __syncthreads();
        const MagWeight m = mag_weight(U.mag, max_mag, metric);
        const uint32_t row = (m.b - 128u) * (uint32_t)kCellRow;
        uint32_t seen = 0u;
        for (int k = tid; k < kCellCounts; k += kCellThreads) {
            const uint32_t v = s_cnt[k];
            if (v) {
                s_cnt[k] = 0u;
                seen += v;
                // (all of +-1 share a cell, whatever the significand)
                const uint32_t first = k >= 2 * kCellDepth ? (uint32_t)(kDeepCells - 2 * kCellDepth) : k % kCellDepth ? row : 0u;
                cell_add(W, first + (uint32_t)k, v, m, mae);
            }
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) seen += __shfl_xor_sync(kFull, seen, off);
        if (lane == 0) s_seen[warp] = seen;
        __syncthreads();
        if (tid == 0) {
            for (int k = 1; k < kCellThreads / 32; ++k) seen += s_seen[k];
            const uint32_t zeros = pieces * 16u - seen;
            // an all-zero block has weight zero, except where every sample weighs one
            if (zeros && (U.mag != 0u || metric >= 2)) cell_add(W, kZeroCell, zeros, m, mae);
        }
    }
}

// The short last blocks: `add` = 0 takes the largest magnitude (before the plan), 1 adds their weights.
template <bool SIGNED>
__global__ void __launch_bounds__(kEmTailThreads)
cells_tail_kernel(const EmTails Q, const CellsWs W, int metric, int add)
{
    if (!after_previous()) return;
    __shared__ float s_w[4096];
    __shared__ unsigned long long s_red[kEmTailThreads / 32];
    const bool mae = metric == BOF4_METRIC_MAE || metric == BOF4_METRIC_MAE_NORMALIZED;
    for (int q = 0; q < Q.count; ++q) {
        const int len = Q.len[q];
        const float m = load_short_block<BF16, SIGNED>(Q.ptr[q], len, s_w, s_red);
        const uint32_t mag = (__float_as_uint(m) >> 16) & 0x7fffu;
        if (!add) {
            if (threadIdx.x == 0) atomicMax(&W.scal[2], mag);
        } else if (mag != 0u || metric >= 2) {
            const MagWeight mw = mag_weight(mag, W.scal[3], metric);
            const bool tiny = mag < (uint32_t)kMagTiny;
            const uint32_t ms = tiny ? scaled16(mag) : mag;
            for (int i = threadIdx.x; i < len; i += kEmTailThreads) {
                const uint32_t w0 = (__float_as_uint(s_w[i]) >> 16) ^ ((__float_as_uint(m) >> 16) & 0x8000u);
                const uint32_t w = tiny ? scaled16(w0) : w0, d = ms - (w & 0x7fffu);
                const bool deep = mag != 0u && d >= (uint32_t)kCellDepth && (w0 & 0x7fffu) != 0u;
                const int at = deep ? deep_cell(w0, mag) : -1;
                uint32_t cell = kZeroCell;
                if (at >= 0) cell = (uint32_t)(kDeepCells + at);
                else if (mag != 0u && d < (uint32_t)kCellDepth)
                    cell = (d ? (mw.b - 128u) * (uint32_t)kCellRow : 0u) + d + ((w & 0x8000u) ? kCellDepth : 0u);
                cell_add(W, cell, 1ull, mw, mae);
            }
        }
        __syncthreads();  // before the next block overwrites s_w
    }
}

// ---------------------------------------------------------------- host side

namespace {

template <bool SG>
int blocks_pass(const EmTensors& T, int block_size, int64_t first, const CellsWs& W, cudaStream_t st)
{
    constexpr int smem = kMags * 4;
#define BOF4_CELLS_I(I_)                                                                  \
    case I_: {                                                                            \
        constexpr auto kern = cells_blocks_kernel<I_, SG>;                                \
        if (const int rc = ensure_dynamic_smem<kern>(smem)) return rc;                    \
        launch_after(kern, kSMs, 1024, smem, st, T, first, W.hist, W.consts);                       \
        break;                                                                            \
    }
    switch (block_size) {
        BOF4_CELLS_I(32) BOF4_CELLS_I(64) BOF4_CELLS_I(128) BOF4_CELLS_I(256) BOF4_CELLS_I(512) BOF4_CELLS_I(1024)
        BOF4_CELLS_I(2048) BOF4_CELLS_I(4096)
    }
#undef BOF4_CELLS_I
    BOF4_CUDA_TRY(cudaGetLastError());
    return BOF4_OK;
}

}  // namespace

int cells_fit(const EmArgs& a, float* d_codebook, uint32_t fixed_mask, int iters, double* d_err_log, void* d_ws,
              size_t ws_bytes, cudaStream_t st, bool* done)
{
    *done = false;
    if (!cells_apply(a.w_dtype, a.n_total) || !ordering_pays(a.w_dtype, a.n_total, a.metric, iters, true)) return BOF4_OK;
    CellsWs W;
    if (cells_layout(d_ws, a.n_total, a.block_size, &W) > ws_bytes) return BOF4_OK;
    *done = true;
    int64_t blocks = 0;
    for (int t = 0; t < a.n_tensors; ++t) blocks += a.h_n[t] / a.block_size;
    const bool sg = a.norm == BOF4_NORM_SIGNED;
    BOF4_CUDA_TRY(cudaMemsetAsync(W.hist, 0, reinterpret_cast<char*>(W.cursor) - reinterpret_cast<char*>(W.hist), st));
    auto tails = [&](int add) {
        return for_each_tail_chunk(a, [&](const EmTails& Q) -> int {
            if (sg) launch_after(cells_tail_kernel<true>, 1, kEmTailThreads, 0, st, Q, W, a.metric, add);
            else launch_after(cells_tail_kernel<false>, 1, kEmTailThreads, 0, st, Q, W, a.metric, add);
            BOF4_CUDA_TRY(cudaGetLastError());
            return BOF4_OK;
        });
    };
    auto of = [&](const EmTensors& T) {
        int64_t b = 0;
        for (int t = 0; t < T.count; ++t) b += T.n[t] / a.block_size;
        return b;
    };
    int rc = tails(0), calls = 0;
    if (rc) return rc;
    int64_t first = 0;
    rc = for_each_tensor_chunk(a, 1024 * kLW, [&](const EmTensors& T) -> int {
        const int64_t f = first;
        first += of(T);
        return sg ? blocks_pass<true>(T, a.block_size, f, W, st) : blocks_pass<false>(T, a.block_size, f, W, st);
    }, &calls);
    if (rc) return rc;
    launch_after(cells_plan_kernel, 1 + (kCellFractions + kCellParts) / kFractionThreads, 1024, 0, st, W, (uint32_t)unit_blocks(blocks, a.block_size), a.metric);
    BOF4_CUDA_TRY(cudaGetLastError());
    first = 0;
    rc = for_each_tensor_chunk(a, 1024 * kLW, [&](const EmTensors& T) -> int {
        const int64_t f = first, nb = of(T);
        first += nb;
        if (nb < kOrderFew) {
            if (const int e = ensure_dynamic_smem<cells_order_few_kernel>(kMags * 4)) return e;
            launch_after(cells_order_few_kernel, kSMs, 1024, kMags * 4, st, T, f, nb, a.block_size, W);
        } else {
            if (const int e = ensure_dynamic_smem<cells_order_kernel>(kOrderSmem)) return e;
            launch_after(cells_order_kernel, kSMs, 1024, kOrderSmem, st, T, f, nb, a.block_size, W);
        }
        BOF4_CUDA_TRY(cudaGetLastError());
        return BOF4_OK;
    }, &calls);
    if (rc) return rc;
    int shift = 0;
    while ((16 << shift) < a.block_size) ++shift;
    constexpr int smem = kCellCounts * 4;
    if ((rc = ensure_dynamic_smem<cells_accumulate_kernel>(smem))) return rc;
    launch_after(cells_accumulate_kernel, kCellCtas * kSMs, kCellThreads, smem, st, W, shift, a.metric);
    BOF4_CUDA_TRY(cudaGetLastError());
    if ((rc = tails(1))) return rc;
    SortFit F{};
    F.metric = a.metric;
    F.n_total = a.n_total;
    F.codebook = d_codebook;
    F.fixed_mask = fixed_mask;
    F.iters = iters;
    F.err_log = d_err_log;
    return cells_run(W, F, st);
}

}  // namespace bof4
