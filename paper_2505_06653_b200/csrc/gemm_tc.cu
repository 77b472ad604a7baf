// Decode fused into a batched consumer on the tensor cores: Y = W_q X^T for 16 ... 64 right-hand
// sides (App. E.2 times token generation; with several tokens or sequences in flight the
// matrix-vector product of gemv.cu becomes this small-N matrix product, and the decode of Eq. 3
// amortises over the batch).
//
// Reading (the paper gives no arithmetic for a fused consumer): the A operand is the dequantised
// weight rounded to bf16, bit for bit what bof4_dequantize writes (Eq. 3, then round to nearest
// even), X is bf16, products are exact and the sums are accumulated in fp32 by the tensor cores.
//
// One CTA per SM.  The work is cut into lines (128 bytes of codes of each of 128 rows: four k-blocks of 64
// weights), tile after tile, and every CTA has an equal, contiguous part of them; a tile that is shared by
// several CTAs is summed, in their order, by the one that completes it last (a ticket: nobody waits).  Warps
// with one job each, coupled by mbarriers, run through the whole part without a CTA-wide barrier:
//
//   1 codes       code lines by TMA into a ring
//   16 producers  four groups of four with a k-block of the line each, a thread per row: decode to bf16 through a
//                 table of level pairs (one 8-byte read, one packed multiplication and one conversion per code
//                 byte; [byte][lane], so the bank only depends on the lane) and store the row into TENSOR
//                 MEMORY (tcgen05.st, two weights per 32-bit column), from where tcgen05.mma takes its A operand
//   1 X           the 64 columns of X by TMA, in the K-major 128-byte-swizzled layout of the B operand
//   2 issuers     for the even and the odd k-blocks, an accumulator each: four tcgen05.mma (M = 128, N = batch,
//                 K = 16), tcgen05.commit hands the stage back
//   4 results     read the accumulators of a part of a tile (there are two sets) while the next part runs
//
// What bounds it: the data path of shared memory.  The accesses of a k-block need 300 wavefronts (its 8192 weights at 32 per
// 128-byte wavefront, 256; codes, constants and X the rest); its codes take HBM 182 cycles (4096 bytes at 22.5 bytes a clock and
// SM).  Counted are 473 wavefronts and 551 cycles a k-block while an SM is active (28672 x 8192 x 32, 194 k-blocks per SM; with
// an outlier list 490 and 746, 65 % of the issue slots); what the other 170 wavefronts are is not known.  The rest of a
// launch, about 9 us at any size, is set-up, first loads, cut tiles and drain.  A decoded tile in shared memory
// would add as much again for its write and the tensor cores' read; decoding in registers by byte permutes
// takes 460 cycles of the half-rate integer pipe.  Warps with global loads of their own in flight paid their
// latency at every publication of a k-block, hence the TMA ring; one issuing warp takes 500 cycles per k-block
// beside the producers, hence two; one CTA per tile and part spent 8 us on set-up, first loads and epilogue.
//
// OPQ (Sec. 3.3, decoding side): a position in the outlier list holds its stored bf16 value instead of
// the decoded weight; the producers replace it in their registers.  The warps of the results sort the list's
// entries of a batch of lines into short lists per line, warp and half k-block beforehand (two searches and one
// pass over the tile's entries, beside the main loop).
//
// Measured: 28672 x 8192 x 32 69 us (90 with a list of 0.06 %), 4096 x 4096 x 32 13 us (17); the form with one CTA
// per tile and K split that stored its tile in shared memory took 170 (210) and 13 (17) us.
//
// Every wait is bounded: a time-out sets the status word, everybody leaves, and the kernel frees its tensor
// memory and returns.
#include <atomic>
#include <chrono>
#include <type_traits>

#include <cuda.h>

#include "common.cuh"

namespace bof4 {

constexpr int kTcGroups = 4;      // producer groups of four warps, a k-block each; k-blocks of a code line
constexpr int kTcM = 128;         // rows per CTA = tensor-memory lanes
constexpr int kTcK = 64;          // weights per k-block: one 128-byte swizzle row of bf16
constexpr int kTcLines = 4;       // ring of code lines
constexpr int kTcBatch = 32, kTcEntries = 1536;  // OPQ: lines of a batch, and outliers
constexpr int kTcAhead = 8;       // lines that L2 is asked for before the ring is
constexpr int kTcMaxN = 64;       // columns of an accumulator
constexpr int kTcIssuers = 2;     // warps that issue, an accumulator each
constexpr int kTcACols = kTcK / 2;               // tensor-memory columns of a stage of A
constexpr int kTcTmemCols = 512;                 // power of two >= accumulator and stages of A
// Stages of A and X, and columns of an accumulator, for up to 32 and up to 64 right-hand sides: what tensor
// memory holds beside the four accumulators.  With eight stages (two per producer group) the round trip store -
// multiply - release is not covered.
template <bool WIDE>
struct TcGeo {
    static constexpr int stages = WIDE ? 8 : 12, acc = WIDE ? 64 : 32, x_bytes = acc * kTcK * 2;
    static_assert(2 * kTcIssuers * acc + stages * kTcACols <= kTcTmemCols, "tensor memory");
    static_assert(stages % kTcIssuers == 0, "a stage belongs to one issuing warp");
};
constexpr int kTcLineBytes = kTcM * 128;         // 16 KiB
constexpr int kTcPairBytes = 256 * 32 * 8;       // level pairs per code byte, a column per lane
constexpr int kTcXBytes = 64 * 1024;                  // all stages of X
constexpr int kTcSmem = kTcXBytes + kTcLines * kTcLineBytes + kTcPairBytes + 1024;  // + slack to align to 1024 bytes
constexpr uint32_t kTcSpinLimit = 1u << 16;      // try_wait calls before a wait gives up (a k-block takes microseconds)
// warps: 0 ... 15 produce, then issuers, X, constants and codes, results
constexpr int kTcIssue = kTcGroups * 4, kTcX = kTcIssue + kTcIssuers, kTcCodes = kTcX + 1, kTcEpilogue = kTcCodes + 1;
constexpr int kTcThreads = 32 * (kTcEpilogue + 4);  // 24 warps: 80 registers each

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of a K-major tile in the 128-byte swizzled layout: start
// address and offsets in units of 16 bytes, leading offset 1 (unused for swizzled K-major), stride
// between 8-row groups 1024 bytes, descriptor version 1, layout type 2 (128-byte swizzle).
__device__ __forceinline__ uint64_t tc_smem_desc(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3fffu);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor: fp32 accumulator, bf16 x bf16, both K-major, M = 128, N = n.
__host__ __device__ inline uint32_t tc_instr_desc(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTcM >> 4) << 24);
}

__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity)
{
    for (uint32_t it = 0; it < kTcSpinLimit; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(1000u)  // suspended for up to a microsecond instead of polling
            : "memory");
        if (ok) return true;
    }
    return false;
}

// A block constant as it is in memory; widened where it is used, so that nothing waits for the load before.
template <class ST>
struct TcConst;
template <>
struct TcConst<F32> {
    float v;
    __device__ __forceinline__ void load(const void* scales, int64_t b)
    {
        asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(static_cast<const float*>(scales) + b));
    }
    __device__ __forceinline__ float value() const { return v; }
};
template <>
struct TcConst<BF16> {
    uint16_t v;
    __device__ __forceinline__ void load(const void* scales, int64_t b)
    {
        asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(static_cast<const uint16_t*>(scales) + b));
    }
    __device__ __forceinline__ float value() const { return __uint_as_float((uint32_t)v << 16); }
};

// Eight codes (even element in the high nibble of its byte) to eight bf16 values (Eq. 3, round to nearest even).
__device__ __forceinline__ void tc_lookup8(uint32_t w, float2 mm, uint32_t pairs, uint32_t lane8, uint32_t* o)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        // byte * 256 + lane * 8 in one permute
        const uint32_t off = __byte_perm(w, lane8, 0x5504u | ((uint32_t)k << 4));
        float2 l;
        asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(l.x), "=f"(l.y) : "r"(pairs + off));
        const float2 v = __fmul2_rn(mm, l);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o[k]) : "f"(v.y), "f"(v.x));
    }
}

// Brackets the first entry of the ascending list with idx >= key to 32 places, by one warp: a guess from the
// key's place in the matrix does it in one step for lists of evenly spread outliers, any other list takes
// steps of a factor of 32.
__device__ __forceinline__ int2 tc_bracket(const int32_t* __restrict__ idx, int k_end, int64_t key, int64_t n, int lane)
{
    int lo = 0, hi = k_end;  // the entry lies in [lo, hi]
    const int g = max((int)((double)k_end * ((double)key / (double)n)) - 512, 0);
    for (int step = 0; hi - lo > 32; ++step) {
        // 32 probes; the entries before the last probe that is below the key are below it as well
        const int first = step == 0 ? g : lo, stride = step == 0 ? 32 : (hi - lo + 31) / 32;
        const int at = min(first + lane * stride, k_end);
        const int cnt = __popc(__ballot_sync(kFull, at < hi && (int64_t)__ldg(idx + at) < key));
        const int above = first + cnt * stride;  // the first probe that is not below the key
        if (cnt > 0) lo = max(lo, above - stride + 1);
        if (cnt < 32) hi = min(hi, max(above, lo));
    }
    return make_int2(lo, hi);
}

__device__ __forceinline__ void tc_arrive(unsigned long long* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tc_load_box(uint32_t dst, const CUtensorMap* map, unsigned long long* bar, uint32_t bytes, int x, int y)
{
    const uint32_t b = smem_u32(bar);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 :
                 : "r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(b), "r"(x), "r"(y)
                 : "memory");
}
// Sixteen 32-bit columns of the warp's 32 rows in tensor memory.
__device__ __forceinline__ void tc_store16(uint32_t addr, const uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        :
        : "r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
          "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}

// Eight 32-bit columns of the warp's 32 rows from tensor memory.
__device__ __forceinline__ void tc_load8(uint32_t addr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// The tensor-core instructions that the lane with lead = 1 has issued arrive on `bar` when they have completed.
__device__ __forceinline__ void tc_commit(unsigned long long* bar, uint32_t lead)
{
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar)), "r"(lead)
        : "memory");
}

// ---------------------------------------------------------------- division of the work
//
// The lines (128 bytes of codes of 128 rows, four k-blocks) of all tiles, tile after tile, are dealt in
// contiguous, equal parts to the CTAs, in units of one line (or, without a workspace, of one tile): CTA i has
// the units from start(i) up to start(i + 1), the first `extra` CTAs one more than the others.
struct TcWork {
    int tiles, per_tile, ctas;  // row tiles, lines per tile, CTAs
    int unit;                   // lines per unit: 1 or per_tile
    int each, extra;            // units per CTA, and the remainder
    unsigned long long epoch;   // names this launch in the tickets, low byte zero
    __device__ int start(int i) const { return (i * each + min(i, extra)) * unit; }  // first line
    // the CTA that has line l (unit = 1)
    __device__ int owner(int l) const
    {
        const uint32_t longer = (uint32_t)extra * (uint32_t)(each + 1);
        return (uint32_t)l < longer ? (int)((uint32_t)l / (uint32_t)(each + 1)) : extra + (int)(((uint32_t)l - longer) / (uint32_t)each);
    }
};
__host__ __device__ inline size_t tc_ticket_bytes(int64_t tiles) { return ((size_t)tiles * 8 + 255) / 256 * 256; }
__host__ __device__ inline size_t tc_ws_bytes(int64_t tiles, int64_t ctas, int n_rhs)
{
    return tc_ticket_bytes(tiles) + (size_t)ctas * 2 * kTcM * n_rhs * 4;  // a CTA has at most two parts of tiles
}

// A tile's ticket.  The cell needs no preparation: every CTA that has a part of the tile first makes sure that
// it carries the launch's 56-bit epoch (with no arrivals yet), long before it arrives; the last arrival clears it.
__device__ __forceinline__ void tc_ticket_open(unsigned long long* cell, unsigned long long epoch)
{
    unsigned long long old = *reinterpret_cast<volatile unsigned long long*>(cell);
    while ((old & ~255ull) != epoch) {
        const unsigned long long seen = atomicCAS(cell, old, epoch);
        if (seen == old) break;
        old = seen;  // somebody else opened it or arrived: at most `ctas` rounds
    }
}

template <class ST, bool HALF, bool OPQ, bool WIDE>  // HALF: blocks of 32 weights, two constants per row and k-block
__global__ void __launch_bounds__(kTcThreads, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap code_map, const void* __restrict__ scales, int64_t cols, int block_shift,
               const float* __restrict__ levels, const __grid_constant__ CUtensorMap x_map, int n_rhs,
               float* __restrict__ y, int* __restrict__ status, const int32_t* __restrict__ out_idx,
               const uint16_t* __restrict__ out_val, const int64_t* __restrict__ n_out, int64_t capacity,
               const TcWork work, unsigned char* __restrict__ ws)
{
    constexpr int kStages = TcGeo<WIDE>::stages, kAcc = TcGeo<WIDE>::acc, kXBytes = TcGeo<WIDE>::x_bytes;
    extern __shared__ unsigned char s_dyn[];
    // full[s]: stage s holds a k-block (one arrival per producer warp; one and the TMA bytes for X); empty[s]: the
    // tensor cores have read it (tcgen05.commit); line_full / line_empty: the same for the ring of code lines
    // and constants; acc_full / acc_empty: the accumulators of a part of a tile are complete / have been read;
    // batch_full / batch_empty: the same for the outliers of a batch of lines
    __shared__ __align__(8) unsigned long long s_full[kStages], s_empty[kStages], s_line_full[kTcLines], s_line_empty[kTcLines],
        s_acc_full[2], s_acc_empty[2], s_batch_full[2], s_batch_empty[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail, s_sums;
    __shared__ int s_sum[2];                        // tiles that this CTA sums
    // OPQ: the weights to replace in a batch of lines of one tile, {lane, column of the k-block, value}, as a list per
    // line, producer warp and half of its k-block
    constexpr int kEntries = OPQ ? kTcEntries : 1;
    __shared__ uint32_t s_entry[2][kEntries];
    __shared__ uint16_t s_next[2][kEntries];
    __shared__ __align__(8) uint32_t s_head[2][OPQ ? kTcBatch : 1][2 * kTcIssue];
    __shared__ int s_batch_lines[2], s_count;       // lines of a batch, negative: more entries than there is room for
    __shared__ int2 s_bound[4];                     // brackets of the first list entry of the tiles tile0 + k, at k & 3
    if (!after_previous()) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t tiles = (smem_u32(s_dyn) + 1023u) & ~1023u;  // 1024-byte aligned: the swizzle atoms start here
    unsigned char* tiles_ptr = s_dyn + (tiles - smem_u32(s_dyn));
    const uint32_t code_ring = tiles + kTcXBytes;
    unsigned char* const s_pairs = tiles_ptr + kTcXBytes + kTcLines * kTcLineBytes;
    const int per_tile = work.per_tile;
    const int begin = work.start((int)blockIdx.x), finish = work.start((int)blockIdx.x + 1), lines = finish - begin;  // this CTA's lines
    const int tile0 = (int)((uint32_t)begin / (uint32_t)per_tile), in0 = begin - tile0 * per_tile;
    // wait of a whole warp; false (and the failure noted): it ran out
    auto warp_wait = [&](unsigned long long* bar, uint32_t parity) -> bool {
        if (__all_sync(kFull, tc_wait(smem_u32(bar), parity))) return true;
        if (lane == 0) s_fail = 1;
        return false;
    };
    // the n-th use (from 0) of ring entry k of a ring: full has completed n times before it is waited for with
    // parity n & 1, empty is first waited for at the second use
    auto parity = [](int n) { return (uint32_t)(n & 1); };

    // ---- set-up.  The threads that request codes and X set their barriers up themselves and request what the
    // empty rings hold at once; everybody else learns of the barriers below.
    auto init = [&](unsigned long long* bar, int count) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    };
    auto load_codes = [&](int n, int tile, int in) {  // this CTA's n-th line: line `in` of a tile
        const int ls = n % kTcLines;
        tc_load_box(code_ring + (uint32_t)ls * kTcLineBytes, &code_map, &s_line_full[ls], kTcLineBytes, in * 128, tile * kTcM);
    };
    auto load_x = [&](int q, int kb) {  // its q-th k-block: k-block kb of the columns
        const int s = q % kStages;
        tc_load_box(tiles + (uint32_t)s * kXBytes, &x_map, &s_full[s], (uint32_t)n_rhs * 128u, kb * kTcK, 0);
    };
    if (tid == kTcCodes * 32) {
        for (int s = 0; s < kTcLines; ++s) {
            init(&s_line_full[s], 1);
            init(&s_line_empty[s], 4 * kTcGroups);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int n = 0, tile = tile0, in = in0; n < min(lines, kTcLines); ++n) {
            load_codes(n, tile, in);
            if (++in == per_tile) in = 0, ++tile;
        }
    } else if (tid == kTcX * 32) {
        for (int s = 0; s < kStages; ++s) {
            init(&s_full[s], 4 + 1);
            init(&s_empty[s], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int q = 0, in = in0; q < min(lines * kTcGroups, kStages); ++q) {
            load_x(q, in * kTcGroups + q % kTcGroups);
            if (q % kTcGroups == kTcGroups - 1 && ++in == per_tile) in = 0;
        }
    } else if (tid == 0) {
        if (blockIdx.x == 0) *status = 0;  // long before any wait can have run out
        s_fail = s_sums = 0;
        for (int b = 0; b < 2; ++b) {
            init(&s_acc_full[b], kTcIssuers);
            init(&s_acc_empty[b], 4);
            init(&s_batch_full[b], 4);
            init(&s_batch_empty[b], 4 * kTcGroups);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // OPQ: the four warps of the results look the outlier lists of the first two parts up meanwhile
    const int f = tid - kTcEpilogue * 32, r_own = (warp & 3) * 32 + lane, w4 = warp - kTcEpilogue;
    const int segs = lines ? (in0 + lines - 1) / per_tile + 1 : 0;
    int k_end = 0, first_batch = 0;
    auto sync = [] { asm volatile("bar.sync 1, 128;" ::: "memory"); };
    // The four warps leave together or not at all after a wait (they meet at barriers).
    auto all4 = [](bool ok) -> bool {
        uint32_t r;
        asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, 1, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(r) : "r"(ok ? 1u : 0u) : "memory");
        return r != 0u;
    };
    auto bound = [&](int k) {  // by one warp
        const int2 p = tc_bracket(out_idx, k_end, (int64_t)min(tile0 + k, work.tiles) * kTcM * cols, (int64_t)work.tiles * kTcM * cols, lane);
        if (lane == 0) s_bound[k & 3] = p;
    };
    // Batch b: the outliers of up to kTcBatch lines of part `seg` from line `in` of its tile on; returns the lines.
    // All entries of the tile are read (coalesced, most batches are a whole part) and those of the batch kept.
    auto batch = [&](int b, int seg, int in, int most) -> int {
        const int buf = b & 1, lo = s_bound[seg & 3].x, hi = s_bound[(seg + 1) & 3].y;
        // so many lines that three quarters of the room are expected to be taken
        int n = min(min(most, kTcBatch), (int)max((int64_t)(kTcEntries * 3 / 4) * per_tile / max(hi - lo, 1), (int64_t)1));
        for (int k = f; k < n * 2 * kTcIssue; k += 128) s_head[buf][k / (2 * kTcIssue)][k % (2 * kTcIssue)] = 0xffffu;
        if (f == 0) s_count = 0;
        sync();
        const uint32_t first = (uint32_t)((int64_t)(tile0 + seg) * kTcM * cols), nc = (uint32_t)cols, c_lo = (uint32_t)in * (kTcGroups * kTcK);
        for (int k0 = lo + f; k0 < hi; k0 += 4 * 128) {
            uint32_t i[4];
            uint16_t v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + u * 128;
                i[u] = k < hi ? (uint32_t)__ldg(out_idx + k) - first : 0xffffffffu;
                v[u] = k < hi ? __ldg(out_val + k) : (uint16_t)0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t r = i[u] / nc, c = i[u] - r * nc - c_lo, line = c / (kTcGroups * kTcK);
                if (r >= (uint32_t)kTcM || c >= nc || line >= (uint32_t)n) continue;  // (c >= nc: before the batch)
                const int slot = atomicAdd(&s_count, 1);
                if (slot >= kEntries) continue;
                s_entry[buf][slot] = (r & 31u) << 27 | (c % kTcK) << 16 | v[u];
                const uint32_t w = (c / kTcK) % kTcGroups * 4 + (r >> 5);
                s_next[buf][slot] = (uint16_t)atomicExch(&s_head[buf][line][2 * w + (c / (kTcK / 2)) % 2], (uint32_t)slot);
            }
        }
        sync();
        if (f == 0) s_batch_lines[buf] = s_count > kEntries ? -n : n;
        return n;
    };
    if (warp < kTcIssue) {
        const float mine = __ldg(levels + (lane & 15));  // level l sits in the lanes with (lane & 15) == l
#pragma unroll 4
        for (int e = tid; e < 256 * 32; e += kTcIssue * 32) {
            const int byte = e >> 5;
            reinterpret_cast<float2*>(s_pairs)[e] = make_float2(__shfl_sync(kFull, mine, byte >> 4), __shfl_sync(kFull, mine, byte & 15));
        }
    }
    if (warp == kTcIssue) {  // tensor memory: the 128 x N fp32 accumulators, then the stages of A
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTcTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    // the others start without waiting for the four warps of the results
    if (warp < kTcEpilogue) {
        asm volatile("bar.sync 2, %0;" ::"n"(kTcEpilogue * 32) : "memory");
        asm volatile("bar.arrive 3, %0;" ::"n"(kTcThreads) : "memory");
    } else {
        if (OPQ && segs) {
            // the brackets of a list that fills its arrays, while the count is on its way
            int64_t count;
            asm volatile("ld.global.nc.s64 %0, [%1];" : "=l"(count) : "l"(n_out));
            k_end = (int)capacity;
            bound(w4);
            if (count < capacity) {
                k_end = (int)count;
                bound(w4);
            }
            sync();
            first_batch = batch(0, 0, in0, min(lines, per_tile - in0));
        }
        asm volatile("bar.sync 3, %0;" ::"n"(kTcThreads) : "memory");
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;

    if (warp < kTcIssue) {
        // ---- producers: group g decodes k-block g of every line; the thread's row of a k-block is 64 weights.
        // A warp reaches the 32 rows of tensor memory that its number modulo 4 names.
        const int group = warp >> 2, a_row = (warp & 3) * 32 + lane;
        const uint32_t a_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(2 * kTcIssuers * kAcc);
        const uint32_t lane8 = (uint32_t)lane * 8u, pairs = smem_u32(s_pairs);
        // block constants of this thread's k-block, three lines ahead (past the end: the last ones again); a row's
        // constants of a few lines share a sector, which the first of them brings in
        TcConst<ST> c0, c1, c2, d0, d1, d2;
        int ct = tile0, ci = in0;
        auto constants = [&](TcConst<ST>& c, TcConst<ST>& d) {
            const int64_t first = ((int64_t)ct * kTcM + a_row) * cols + min((int64_t)(ci * kTcGroups + group) * kTcK, cols - kTcK);
            c.load(scales, first >> block_shift);
            if (HALF) d.load(scales, (first >> block_shift) + 1);
            if (ct * per_tile + ci + 1 < finish && ++ci == per_tile) ci = 0, ++ct;
        };
        constants(c0, d0);
        constants(c1, d1);
        constants(c2, d2);
        int tile = tile0, in = in0, bat = 0, left = 0, at = 0;  // OPQ
        bool crowded = false;
        // Replaces the outliers of half h (32 columns, 16 registers) of the thread's row of a k-block.
        // (head, entry: the first of its list, read well before.)
        auto outliers = [&](uint32_t (&v)[16], int h, int tile, int in, uint32_t head, uint32_t entry) {
            auto replace = [&](bool mine, int c, uint32_t value) {  // c: column of the half
                const uint32_t sel = (c & 1) ? 0x5410u : 0x3254u;
#define BOF4_TC_PUT(j_) v[j_] = mine ? __byte_perm(v[j_], value, sel) : v[j_];
                switch (c >> 1) {  // the same for all lanes: one indirect branch
                    case 0: BOF4_TC_PUT(0) break;
                    case 1: BOF4_TC_PUT(1) break;
                    case 2: BOF4_TC_PUT(2) break;
                    case 3: BOF4_TC_PUT(3) break;
                    case 4: BOF4_TC_PUT(4) break;
                    case 5: BOF4_TC_PUT(5) break;
                    case 6: BOF4_TC_PUT(6) break;
                    case 7: BOF4_TC_PUT(7) break;
                    case 8: BOF4_TC_PUT(8) break;
                    case 9: BOF4_TC_PUT(9) break;
                    case 10: BOF4_TC_PUT(10) break;
                    case 11: BOF4_TC_PUT(11) break;
                    case 12: BOF4_TC_PUT(12) break;
                    case 13: BOF4_TC_PUT(13) break;
                    case 14: BOF4_TC_PUT(14) break;
                    case 15: BOF4_TC_PUT(15) break;
                }
#undef BOF4_TC_PUT
            };
            if (!crowded) {
                while (head != 0xffffu) {
                    replace((int)(entry >> 27) == lane, (int)((entry >> 16) & 31u), entry & 0xffffu);
                    head = s_next[bat & 1][head];
                    if (head != 0xffffu) entry = s_entry[bat & 1][head];
                }
            } else {  // more outliers than there is room for: every lane looks its own part of the list up
                const int64_t first = ((int64_t)tile * kTcM + a_row) * cols + (int64_t)(in * kTcGroups + group) * kTcK + h * (kTcK / 2);
                const int64_t list_end = min(*n_out, capacity), behind = min(first + kTcK / 2, ((int64_t)tile * kTcM + a_row + 1) * cols);
                int64_t lo = 0, hi = list_end;
                while (lo < hi) {
                    const int64_t mid = (lo + hi) >> 1;
                    if ((int64_t)__ldg(out_idx + mid) < first) lo = mid + 1;
                    else hi = mid;
                }
                for (; lo < list_end; ++lo) {
                    const int64_t i = (int64_t)__ldg(out_idx + lo);
                    if (i >= behind) break;
                    if (i >= first) replace(true, (int)(i - first), (uint32_t)__ldg(out_val + lo));
                }
                __syncwarp();
            }
        };
        for (int n = 0; n < lines; ++n) {
            const int ls = n % kTcLines, q = n * kTcGroups + group, s = q % kStages;
            if (!warp_wait(&s_line_full[ls], parity(n / kTcLines))) break;
            uint32_t head0 = 0xffffu, head1 = 0xffffu, entry0 = 0u, entry1 = 0u;
            if (OPQ) {
                if (left == 0) {  // the next batch
                    if (!warp_wait(&s_batch_full[bat & 1], parity(bat >> 1))) break;
                    left = s_batch_lines[bat & 1];
                    crowded = left < 0;
                    left = abs(left);
                    at = 0;
                }
                const uint2 heads = *reinterpret_cast<const uint2*>(&s_head[bat & 1][at][2 * warp]);
                head0 = crowded ? 0xffffu : heads.x, head1 = crowded ? 0xffffu : heads.y;
                if (head0 != 0xffffu) entry0 = s_entry[bat & 1][head0];
                if (head1 != 0xffffu) entry1 = s_entry[bat & 1][head1];
            }
            uint32_t w[8];
            // the thread's 32 bytes: chunks 2 g and 2 g + 1 of its row's line (128-byte swizzle)
            const uint32_t row = code_ring + (uint32_t)ls * kTcLineBytes + (uint32_t)a_row * 128u;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(w[4 * h]), "=r"(w[4 * h + 1]), "=r"(w[4 * h + 2]), "=r"(w[4 * h + 3])
                             : "r"(row + (uint32_t)(((2 * group + h) ^ (a_row & 7)) * 16)));
            const float m = c0.value(), m2 = HALF ? d0.value() : m;
            c0 = c1, c1 = c2;
            if (HALF) d0 = d1, d1 = d2;
            constants(c2, d2);
            uint32_t v[16];
#pragma unroll
            for (int j = 0; j < 4; ++j) tc_lookup8(w[j], make_float2(m, m), pairs, lane8, v + 4 * j);
            if (OPQ) outliers(v, 0, tile, in, head0, entry0);
            // the tensor cores must have read what the stage held
            if (q >= kStages && !warp_wait(&s_empty[s], parity(q / kStages - 1))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t dst = a_lane + (uint32_t)(s * kTcACols);
            tc_store16(dst, v);
            uint32_t u[16];
#pragma unroll
            for (int j = 0; j < 4; ++j) tc_lookup8(w[4 + j], make_float2(m2, m2), pairs, lane8, u + 4 * j);
            if (OPQ) {
                outliers(u, 1, tile, in, head1, entry1);
                ++at;
                if (--left == 0) {
                    __syncwarp();
                    if (lane == 0) tc_arrive(&s_batch_empty[bat & 1]);
                    ++bat;
                }
                if (++in == per_tile) in = 0, ++tile;
            }
            tc_store16(dst + 16u, u);
            if (lane == 0) tc_arrive(&s_line_empty[ls]);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) tc_arrive(&s_full[s]);
        }
    } else if (warp < kTcX) {
        // ---- the issuing warps: wait for a full stage, issue its four instructions, let tcgen05.commit hand
        // the stage back.  The whole warp takes every step and everything but the lane's predicate is the same for
        // all threads (the number of the warp is a constant here), so that the operands stay in uniform registers.
        auto issue = [&](auto which_c) {
            constexpr int which = decltype(which_c)::value;
            const uint32_t lead = lane == 0 ? 1u : 0u, idesc = tc_instr_desc(n_rhs);
            const uint64_t db0 = tc_smem_desc(tiles);
            int in = in0, seg = 0;
            uint32_t acc = 0u;
            for (int n = 0; n < lines; ++n) {
                const int buf = seg & 1;
                const uint32_t d = tmem + (uint32_t)((buf * kTcIssuers + which) * kAcc);
                if (acc == 0u && seg >= 2 && !warp_wait(&s_acc_empty[buf], parity((seg >> 1) - 1))) return;
#pragma unroll
                for (int j = 0; j < kTcGroups / kTcIssuers; ++j) {
                    const int q = n * kTcGroups + kTcIssuers * j + which, s = q % kStages;
                    if (!warp_wait(&s_full[s], parity(q / kStages))) return;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t a = tmem + (uint32_t)(2 * kTcIssuers * kAcc + s * kTcACols);
                    const uint64_t db = db0 + (uint64_t)(s * (kXBytes >> 4));
#pragma unroll
                    for (int kk = 0; kk < kTcK / 16; ++kk) {  // 16 of K: eight columns of A, +2 in the address field of B
                        asm volatile(
                            "{\n\t.reg .pred p, q;\n\t"
                            "setp.ne.b32 p, %4, 0;\n\t"
                            "setp.ne.b32 q, %5, 0;\n\t"
                            "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                            :
                            : "r"(d), "r"(a + (uint32_t)(8 * kk)), "l"(db + (uint64_t)(2 * kk)), "r"(idesc), "r"(acc), "r"(lead)
                            : "memory");
                        acc = 1u;
                    }
                    tc_commit(&s_empty[s], lead);
                }
                if (++in == per_tile || n + 1 == lines) {  // the end of a part of a tile
                    tc_commit(&s_acc_full[buf], lead);
                    in = 0, ++seg, acc = 0u;
                }
            }
        };
        if (warp == kTcIssue) issue(std::integral_constant<int, 0>{});
        else issue(std::integral_constant<int, 1>{});
    } else if (warp == kTcX) {
        // ---- X: the 64 columns of a k-block
        int in = (in0 + kStages / kTcGroups) % per_tile;
        for (int q = kStages; q < lines * kTcGroups; ++q) {
            if (!warp_wait(&s_empty[q % kStages], parity(q / kStages - 1))) break;
            if (lane == 0) load_x(q, in * kTcGroups + q % kTcGroups);
            if (q % kTcGroups == kTcGroups - 1 && ++in == per_tile) in = 0;
        }
    } else if (warp == kTcCodes) {
        // ---- code lines beyond the first ones, brought into L2 kTcAhead lines before
        int tile = tile0, in = in0, pt = tile0, pi = in0;
        auto step = [&](int& t, int& i) {
            if (++i == per_tile) i = 0, ++t;
        };
        for (int n = 0; n < kTcAhead; ++n) step(pt, pi);
        for (int n = 0; n < lines; ++n) {
            if (n + kTcAhead < lines) {
                if (lane == 0)
                    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(reinterpret_cast<uint64_t>(&code_map)),
                                 "r"(pi * 128), "r"(pt * kTcM)
                                 : "memory");
                step(pt, pi);
            }
            if (n >= kTcLines) {
                if (!warp_wait(&s_line_empty[n % kTcLines], parity(n / kTcLines - 1))) break;
                if (lane == 0) load_codes(n, tile, in);
            }
            step(tile, in);
        }
    } else {
        // ---- results of the parts of tiles; OPQ: the list entries of the next part's rows before that
        unsigned long long* const tickets = reinterpret_cast<unsigned long long*>(ws);
        if (f == 0 && segs) {
            if (in0 || lines < per_tile) tc_ticket_open(tickets + tile0, work.epoch);
            if (segs > 1 && (in0 + lines) % per_tile) tc_ticket_open(tickets + tile0 + segs - 1, work.epoch);
        }
        // The result of a part of a tile; false: a wait ran out.
        auto result = [&](int seg) -> bool {
            const int buf = seg & 1;
            if (!all4(warp_wait(&s_acc_full[buf], parity(seg >> 1)))) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int tile = tile0 + seg, t0 = tile * per_tile;
            const bool all = begin <= t0 && finish >= t0 + per_tile;
            float* const parts = reinterpret_cast<float*>(ws + tc_ticket_bytes(work.tiles));
            const int64_t slab = (int64_t)kTcM * n_rhs;
            float* dst = all ? y + tile * slab : parts + (2 * (int64_t)blockIdx.x + (begin <= t0 ? 1 : 0)) * slab;
            dst += (int64_t)r_own * n_rhs;
            const uint32_t src = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(buf * kTcIssuers * kAcc);
            for (int c0 = 0; c0 < n_rhs; c0 += 8) {
                uint32_t a[8], b[8];
                tc_load8(src + (uint32_t)c0, a);
                tc_load8(src + (uint32_t)(kAcc + c0), b);
                float v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = __uint_as_float(a[k]) + __uint_as_float(b[k]);
                *reinterpret_cast<float4*>(dst + c0) = make_float4(v[0], v[1], v[2], v[3]);
                *reinterpret_cast<float4*>(dst + c0 + 4) = make_float4(v[4], v[5], v[6], v[7]);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) tc_arrive(&s_acc_empty[buf]);
            if (all) return true;
            // A part of a tile: whoever completes the tile last sums its parts, below.
            const int others = work.owner(t0 + per_tile - 1) - work.owner(t0);
            __threadfence();
            sync();
            if (f == 0 && (int)(atomicAdd(tickets + tile, 1ull) & 255ull) == others) {
                tickets[tile] = 0ull;
                s_sum[s_sums++] = tile;
            }
            return true;
        };
        if (!OPQ) {
            for (int seg = 0; seg < segs; ++seg)
                if (!result(seg)) break;
        } else {
            // Batch after batch, one ahead of the results: while the result of a part is waited for, the producers
            // have the batch behind it.
            int line = 0, in = in0, seg = 0, done = 0;
            bool ok = true;
            for (int b = 0; line < lines && ok; ++b) {
                int n = first_batch;
                if (b > 0) {
                    if (b >= 2) ok = all4(warp_wait(&s_batch_empty[b & 1], parity((b >> 1) - 1)));
                    if (!ok) break;
                    n = batch(b, seg, in, min(lines - line, per_tile - in));
                }
                __syncwarp();
                sync();
                if (lane == 0) tc_arrive(&s_batch_full[b & 1]);
                const int ended = seg;  // parts before this one are complete in earlier batches
                line += n;
                if ((in += n) == per_tile) {
                    in = 0, ++seg;
                    if (w4 == 3) bound(seg + 2);  // ([seg], [seg + 1] are there)
                    sync();
                }
                for (; ok && done < ended; ++done) ok = result(done);
            }
            for (; ok && done < segs; ++done) ok = result(done);
        }
    }
    // Every loop above is bounded, so every warp gets here.
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (s_fail) {
        // copies and tensor-core instructions issued before the time-out may still be under way: they take
        // microseconds; give them a bounded 100 before shared and tensor memory go away
        if (tid == 0) atomicExch(status, 1);
        for (int i = 0; i < 100; ++i) __nanosleep(1000);
    }
    for (int k = 0; k < s_sums; ++k) {  // the parts in the order of the CTAs; all but the first begin inside the tile
        const int tile = s_sum[k], t0 = tile * per_tile, i0 = work.owner(t0), i1 = work.owner(t0 + per_tile - 1);
        const int64_t slab = (int64_t)(kTcM / 4) * n_rhs;
        __threadfence();
        const float4* parts = reinterpret_cast<const float4*>(ws + tc_ticket_bytes(work.tiles));
        const float4* head = parts + (int64_t)(2 * i0 + (work.start(i0) <= t0 ? 1 : 0)) * slab;
        const float4* next = parts + (int64_t)(2 * i0 + 2) * slab;
        float4* dst = reinterpret_cast<float4*>(y) + tile * slab;
        const int more = i1 - i0;
        for (int e = tid; e < (int)slab; e += kTcThreads) {
            float4 sum = __ldcg(head + e);
            for (int i = 0; i < more; i += 8) {  // eight on their way at a time
                float4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = i + u < more ? __ldcg(next + (int64_t)(2 * (i + u)) * slab + e) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    sum.x += v[u].x;
                    sum.y += v[u].y;
                    sum.z += v[u].z;
                    sum.w += v[u].w;
                }
            }
            dst[e] = sum;
        }
    }
    if (warp == kTcIssue)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols) : "memory");
}

}  // namespace bof4

using namespace bof4;

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Tensor map of a row-major matrix of 2-byte or 1-byte elements with a box of 128 bytes x box_rows and the
// 128-byte swizzle: X lands in the layout that the tcgen05 descriptor of the B operand names, a code
// line in one that sixteen-byte reads of neighbouring rows find without bank conflicts.
int make_map(const void* p, bool bytes, int64_t cols, int64_t rows, int box_rows, CUtensorMap* map)
{
    static std::atomic<EncodeTiledFn> known{nullptr};
    EncodeTiledFn fn = known.load(std::memory_order_relaxed);
    if (!fn) {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        BOF4_CUDA_TRY(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q));
        if (!f || q != cudaDriverEntryPointSuccess) {
            set_error("bof4_gemm_tc: the driver does not provide cuTensorMapEncodeTiled");
            return BOF4_ERR_CUDA;
        }
        fn = reinterpret_cast<EncodeTiledFn>(f);
        known.store(fn, std::memory_order_relaxed);
    }
    const int esize = bytes ? 1 : 2;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * esize};
    const cuuint32_t box[2] = {(cuuint32_t)(128 / esize), (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn(map, bytes ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(p), dims,
                          strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("bof4_gemm_tc: cuTensorMapEncodeTiled failed with code %d", (int)r);
        return BOF4_ERR_CUDA;
    }
    return BOF4_OK;
}

// A name for every launch, no two alike: 56 bits that mix a counter with the time the library was loaded.
unsigned long long next_epoch()
{
    static std::atomic<unsigned long long> counter{(unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count()};
    unsigned long long z = counter.fetch_add(1) * 0x9e3779b97f4a7c15ull;  // odd: distinct values stay distinct
    z ^= z >> 29;
    z &= ~255ull;
    return z ? z : 256ull;
}

}  // namespace

extern "C" int bof4_gemm_tc(const uint8_t* d_codes, const void* d_scales, int scale_dtype, int64_t rows, int64_t cols,
                            int block_size, const float* d_codebook, const void* d_x, int n_rhs,
                            const int32_t* d_out_idx, const void* d_out_val, const int64_t* d_n_out, int64_t capacity,
                            float* d_y, int* d_status, void* d_ws, size_t ws_bytes, void* stream)
{
    const char* fn = "bof4_gemm_tc";
    if (!valid_block_size(block_size)) {
        set_error("%s: block_size %d is not a power of two in 32 ... 4096", fn, block_size);
        return BOF4_ERR_SHAPE;
    }
    if (scale_dtype != BOF4_F32 && scale_dtype != BOF4_BF16) {
        set_error("%s: unknown scale dtype %d", fn, scale_dtype);
        return BOF4_ERR_DTYPE;
    }
    if (rows < 0 || cols < 0 || rows % kTcM || cols % kTcK || cols % block_size || n_rhs < 16 || n_rhs > kTcMaxN ||
        n_rhs % 16) {
        set_error("%s: rows must be a multiple of 128, cols of 64 and of block_size, n_rhs one of 16, 32, 48, 64", fn);
        return BOF4_ERR_SHAPE;
    }
    const bool opq = d_out_idx != nullptr;
    if (opq && (!d_out_val || !d_n_out || capacity < 0)) {
        set_error("%s: outlier list needs d_out_idx, d_out_val and d_n_out together and a capacity >= 0", fn);
        return BOF4_ERR_INVALID_ARG;
    }
    if (opq && rows * cols > 0x7fffffffLL) {
        set_error("%s: outlier indices are 32-bit, rows * cols must not exceed 2^31 - 1", fn);
        return BOF4_ERR_SHAPE;
    }
    if (rows == 0) return BOF4_OK;
    if (!d_codes || !d_scales || !d_codebook || !d_x || !d_y || !d_status) {
        set_error("%s: NULL pointer", fn);
        return BOF4_ERR_INVALID_ARG;
    }
    if (((uintptr_t)d_codes & 15u) || ((uintptr_t)d_x & 15u)) {
        set_error("%s: d_codes and d_x must be 16-byte aligned", fn);
        return BOF4_ERR_INVALID_ARG;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cols == 0) {
        BOF4_CUDA_TRY(cudaMemsetAsync(d_status, 0, sizeof(int), st));
        BOF4_CUDA_TRY(cudaMemsetAsync(d_y, 0, (size_t)rows * n_rhs * sizeof(float), st));
        return BOF4_OK;
    }
    // One CTA per SM, each with an equal part of the lines (stream-K): no wave is ever partly empty.  Without a
    // workspace for the parts of tiles that this gives, whole tiles per CTA.
    const int64_t tiles = rows / kTcM, per_tile = (cols / kTcK + kTcGroups - 1) / kTcGroups, lines = tiles * per_tile;
    if (lines > 0x3fffffff || tiles * kTcM > 0x7fffffff) {
        set_error("%s: matrix too large", fn);
        return BOF4_ERR_SHAPE;
    }
    int64_t ctas = lines < kSMs ? lines : kSMs, fit = 0;
    if (d_ws && !((uintptr_t)d_ws & 15u) && ws_bytes > tc_ws_bytes(tiles, 0, n_rhs))
        fit = (int64_t)((ws_bytes - tc_ws_bytes(tiles, 0, n_rhs)) / ((size_t)2 * kTcM * n_rhs * 4));
    if (fit < ctas) ctas = fit;
    TcWork work{};
    work.tiles = (int)tiles;
    work.per_tile = (int)per_tile;
    work.unit = 1;
    if (ctas < tiles && ctas < kSMs) {  // no workspace, or less than whole tiles need
        ctas = tiles < kSMs ? tiles : kSMs;
        work.unit = (int)per_tile;
    }
    work.ctas = (int)ctas;
    work.each = (int)(lines / work.unit / ctas);
    work.extra = (int)(lines / work.unit % ctas);
    work.epoch = next_epoch();
    int rc, block_shift = 0;
    while ((1 << block_shift) < block_size) ++block_shift;
    CUtensorMap x_map, code_map;
    if ((rc = make_map(d_x, false, cols, n_rhs, n_rhs, &x_map)) || (rc = make_map(d_codes, true, cols / 2, rows, kTcM, &code_map)))
        return rc;
    const bool list = opq && capacity > 0;
    const uint16_t* val = static_cast<const uint16_t*>(d_out_val);
#define BOF4_TC_W(ST_, HALF_, OPQ_, WIDE_)                                                                                       \
    {                                                                                                                      \
        constexpr auto kern = gemm_tc_kernel<ST_, HALF_, OPQ_, WIDE_>;                                                            \
        if ((rc = ensure_dynamic_smem<kern>(kTcSmem))) return rc;                                                          \
        launch_after(kern, work.ctas, kTcThreads, kTcSmem, st, code_map, d_scales, cols, block_shift, d_codebook, x_map, n_rhs, d_y, \
                     d_status, d_out_idx, val, d_n_out, capacity, work, static_cast<unsigned char*>(d_ws));                          \
    }
#define BOF4_TC_GO(ST_, HALF_, OPQ_) { if (n_rhs > 32) BOF4_TC_W(ST_, HALF_, OPQ_, true) else BOF4_TC_W(ST_, HALF_, OPQ_, false) }
#define BOF4_TC_ST(ST_)                                                             \
    if (block_size == 32) {                                                         \
        if (list) BOF4_TC_GO(ST_, true, true) else BOF4_TC_GO(ST_, true, false)     \
    } else {                                                                        \
        if (list) BOF4_TC_GO(ST_, false, true) else BOF4_TC_GO(ST_, false, false)   \
    }
    if (scale_dtype == BOF4_F32) { BOF4_TC_ST(F32) } else { BOF4_TC_ST(BF16) }
#undef BOF4_TC_ST
#undef BOF4_TC_GO
#undef BOF4_TC_W
    BOF4_CUDA_TRY(cudaGetLastError());
    return BOF4_OK;
}
