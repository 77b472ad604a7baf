// Decode fused into a batched consumer on the tensor cores: Y = W_q X^T for 16 ... 64 right-hand
// sides (App. E.2 times token generation; with several tokens or sequences in flight the
// matrix-vector product of gemv.cu becomes this small-N matrix product, and the decode of Eq. 3
// amortises over the batch).
//
// Reading (the paper gives no arithmetic for a fused consumer): the A operand is the dequantised
// weight rounded to bf16, bit for bit what bof4_dequantize writes (Eq. 3, then round to nearest
// even), X is bf16, products are exact and the sums are accumulated in fp32 by the tensor cores.
//
// One CTA owns 128 rows of W and a range of K.  The codes come by TMA, four k-blocks of 64 weights (a
// 128-byte line of every row) at a time into a ring; two warps bring the block constants beside them.
// Sixteen producer warps, four groups of four with a k-block each and a thread per row, decode to bf16 and
// store the row into TENSOR MEMORY (tcgen05.st, two weights per 32-bit column), from where tcgen05.mma takes
// its A operand: the decoded matrix never touches shared memory, whose bandwidth (16 KiB written by the
// producers and read again by the tensor cores per k-block, 256 cycles) bound the earlier form.  The
// producers have no global load in flight either: publishing a k-block waited for it.
//
// Decode: the products of a block constant with the 16 levels are formed once per row and k-block, rounded
// to bf16 and split into a table of low and a table of high bytes (four registers each); eight codes are
// then looked up with byte permutes: two per table half, one that chooses between the halves by the
// code's top bit, one that interleaves low and high bytes.  About 3 instructions per weight, on the half-rate
// integer pipe, which bounds the kernel: 370 cycles per k-block and SM.
//
// OPQ (Sec. 3.3, decoding side): a position in the outlier list holds its stored bf16 value instead of
// the decoded weight; the producer warp replaces it in tensor memory.  Two more warps find the list's part
// for the tile and the entries of every row meanwhile.
//
// The 64 columns of X of a k-block come by TMA in the K-major 128-byte-swizzled layout that the tcgen05
// shared-memory descriptor names; their bytes and one arrival per producer warp complete the stage's
// "full" mbarrier.  One thread waits for the stages in order and issues four tcgen05.mma each (M = 128,
// N = batch, K = 16); its tcgen05.commit arrives on the stage's "empty" mbarrier.  No CTA-wide barrier in
// the loop.  Every wait is bounded: a time-out sets the status word, the issuing thread still commits and
// waits (bounded) for what it has issued, and the kernel frees its tensor memory and returns.
//
// Matrices with few row tiles are split along K over the CTAs of a cluster (up to 8), whose partial products
// are summed in rank order through distributed shared memory: no workspace and no second launch.
#include <cooperative_groups.h>
#include <cuda.h>

#include "common.cuh"

namespace bof4 {

constexpr int kTcGroups = 4;      // producer groups of four warps, a k-block each; k-blocks of a code line
constexpr int kTcM = 128;         // rows per CTA = tensor-memory lanes
constexpr int kTcK = 64;          // weights per k-block: one 128-byte swizzle row of bf16
constexpr int kTcStages = 8;
constexpr int kTcLines = 4;       // ring of code lines
constexpr int kTcMaxN = 64;       // columns of the accumulator
constexpr int kTcACols = kTcK / 2;               // tensor-memory columns of a stage of A
constexpr int kTcTmemCols = 512;                 // power of two >= accumulator and stages of A
static_assert(kTcMaxN + kTcStages * kTcACols <= kTcTmemCols, "tensor memory");
constexpr int kTcBBytes = kTcMaxN * kTcK * 2;    // 8 KiB
constexpr int kTcLineBytes = kTcM * 128;         // 16 KiB
constexpr int kTcScaleFloats = 2 * kTcGroups * kTcM;  // constants of a line (two per k-block for blocks of 32 weights)
constexpr int kTcSmem = kTcStages * kTcBBytes + kTcLines * (kTcLineBytes + kTcScaleFloats * 4) + 1024;  // + slack to align to 1024 bytes
constexpr uint32_t kTcSpinLimit = 1u << 16;      // try_wait calls before a wait gives up (a k-block takes microseconds)
constexpr int kTcMaxSplit = 8;                   // CTAs of a cluster (portable size)
// warps: 0 issues, 1 ... 16 produce, 17 requests code lines, 18 X, 19 and 20 bring constants, 21 and 22 look outlier rows up
constexpr int kTcFinders = 64;
__host__ __device__ constexpr int tc_threads(bool opq) { return 32 * (kTcGroups * 4 + 5) + (opq ? kTcFinders : 0); }

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

template <class ST>
__device__ __forceinline__ float tc_scale(const void* scales, int64_t b);
template <>
__device__ __forceinline__ float tc_scale<F32>(const void* scales, int64_t b)
{
    return __ldg(static_cast<const float*>(scales) + b);
}
template <>
__device__ __forceinline__ float tc_scale<BF16>(const void* scales, int64_t b)
{
    return __uint_as_float((uint32_t)__ldg(static_cast<const uint16_t*>(scales) + b) << 16);
}

__device__ __forceinline__ uint32_t tc_prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// The 16 levels times a block constant, rounded to bf16 (Eq. 3 and the operand's rounding), as a table of
// low bytes and one of high bytes.
struct TcTable {
    uint32_t lo[4], hi[4];
};
__device__ __forceinline__ TcTable tc_table(float m, const float2 (&lv)[8])
{
    TcTable t;
    uint32_t p[8];
    const float2 mm = make_float2(m, m);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float2 v = __fmul2_rn(mm, lv[k]);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p[k]) : "f"(v.y), "f"(v.x));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        t.lo[k] = tc_prmt(p[2 * k], p[2 * k + 1], 0x6420u);
        t.hi[k] = tc_prmt(p[2 * k], p[2 * k + 1], 0x7531u);
    }
    return t;
}
// Eight codes (even element in the high nibble of its byte) to eight bf16 values.
__device__ __forceinline__ void tc_decode8(uint32_t w, const TcTable& t, uint32_t* o)
{
    const uint32_t sel = w & 0x77777777u, half = ((w >> 1) & 0x44444444u) | 0x32103210u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t s = h ? sel >> 16 : sel, c = h ? half >> 16 : half;
        const uint32_t lo = tc_prmt(tc_prmt(t.lo[0], t.lo[1], s), tc_prmt(t.lo[2], t.lo[3], s), c);
        const uint32_t hi = tc_prmt(tc_prmt(t.hi[0], t.hi[1], s), tc_prmt(t.hi[2], t.hi[3], s), c);
        o[2 * h] = tc_prmt(lo, hi, 0x4051u);      // bytes of codes 1 0 3 2: low half of a pair is the even one
        o[2 * h + 1] = tc_prmt(lo, hi, 0x6273u);
    }
}

// First entry of the ascending list with idx >= key, by one warp: a guess from the key's place in the
// matrix narrows the range to 32 entries in one step for lists of evenly spread outliers; any other list
// takes steps of a factor of 32.
__device__ __forceinline__ int64_t tc_lower_bound(const int32_t* __restrict__ idx, int64_t k_end, int64_t key, int64_t n, int lane)
{
    int64_t lo = 0, hi = k_end;  // the answer lies in [lo, hi]
    int64_t g = (int64_t)((double)k_end * ((double)key / (double)n)) - 512;
    g = g < 0 ? 0 : g;
    for (int step = 0; hi > lo; ++step) {
        // 32 probes; the entries before the last probe that is below the key are below it as well
        const int64_t first = step == 0 ? g : lo, stride = step == 0 ? 32 : (hi - lo + 31) / 32;
        const int64_t at = first + lane * stride;
        const int cnt = __popc(__ballot_sync(kFull, at < hi && (int64_t)__ldg(idx + at) < key));
        const int64_t above = first + (int64_t)cnt * stride;  // the first probe that is not below the key
        if (cnt > 0) lo = above - stride + 1;
        if (cnt < 32 && above < hi) hi = above;
        if (step > 0 && stride == 1) break;
    }
    return lo;
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

template <class ST, bool HALF, bool OPQ>  // HALF: blocks of 32 weights, two constants per row and k-block
__global__ void __launch_bounds__(tc_threads(OPQ), 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap code_map, const void* __restrict__ scales, int64_t cols, int block_shift,
               const float* __restrict__ levels, const __grid_constant__ CUtensorMap x_map, int n_rhs,
               float* __restrict__ y, int* __restrict__ status, const int32_t* __restrict__ out_idx,
               const uint16_t* __restrict__ out_val, const int64_t* __restrict__ n_out, int64_t capacity)
{
    constexpr int NT = tc_threads(OPQ);
    extern __shared__ unsigned char s_dyn[];
    // full[s]: stage s holds a k-block (one arrival per producer warp; one and the TMA bytes for X); empty[s]: the
    // tensor cores have read it (tcgen05.commit); line_full / line_empty: the same for the ring of code lines
    // and constants; done: every instruction of the CTA has completed; rows: s_beg and s_end are set
    __shared__ __align__(8) unsigned long long s_full[kTcStages], s_empty[kTcStages], s_line_full[kTcLines], s_line_empty[kTcLines],
        s_done, s_rows;
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    __shared__ int s_beg[kTcM], s_end[kTcM];  // OPQ: the list entries of every row of the tile inside the CTA's columns
    __shared__ long long s_part[2];           // OPQ: the tile's part of the list
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t tiles = (smem_u32(s_dyn) + 1023u) & ~1023u;  // 1024-byte aligned: the swizzle atoms start here
    unsigned char* tiles_ptr = s_dyn + (tiles - smem_u32(s_dyn));
    const uint32_t code_ring = tiles + kTcStages * kTcBBytes;
    float* const scale_ring = reinterpret_cast<float*>(tiles_ptr + kTcStages * kTcBBytes + kTcLines * kTcLineBytes);
    const int64_t row0 = (int64_t)blockIdx.x * kTcM;
    // the CTA's k-blocks: its share of the cluster's, in whole lines
    const int splits = (int)gridDim.y, rank = (int)blockIdx.y, kb_all = (int)(cols / kTcK);
    const int lines_all = (kb_all + kTcGroups - 1) / kTcGroups;
    const int line0 = (int)((int64_t)lines_all * rank / splits), lines = (int)((int64_t)lines_all * (rank + 1) / splits) - line0;
    const int kb0 = line0 * kTcGroups, kblocks = min(kb_all - kb0, lines * kTcGroups);
    // wait of a whole warp; false (and the failure noted): it ran out
    auto warp_wait = [&](unsigned long long* bar, uint32_t parity) -> bool {
        if (__all_sync(kFull, tc_wait(smem_u32(bar), parity))) return true;
        if (lane == 0) s_fail = 1;
        return false;
    };

    if (tid == 0) {
        if (blockIdx.x == 0 && rank == 0) *status = 0;  // long before any wait can have run out
        s_fail = 0;
        auto init = [&](unsigned long long* bar, int count) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
        };
        for (int s = 0; s < kTcStages; ++s) {
            init(&s_full[s], 4 + 1);
            init(&s_empty[s], 1);
        }
        for (int s = 0; s < kTcLines; ++s) {
            init(&s_line_full[s], 2);
            init(&s_line_empty[s], 4 * kTcGroups);
        }
        init(&s_done, 1);
        init(&s_rows, kTcFinders / 32);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {  // tensor memory: the 128 x N fp32 accumulator, then the stages of A
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTcTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;

    if (warp == 0) {
        // ---- the issuing warp: one thread waits for a full stage, issues its four instructions and
        // lets tcgen05.commit hand the stage back
        if (lane == 0) {
            const uint32_t idesc = tc_instr_desc(n_rhs);
            bool ok = true;
            for (int kb = 0; kb < kblocks; ++kb) {
                const int s = kb % kTcStages;
                if (!tc_wait(smem_u32(&s_full[s]), (uint32_t)((kb / kTcStages) & 1))) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a = tmem + (uint32_t)(kTcMaxN + s * kTcACols);
                const uint64_t db = tc_smem_desc(tiles + (uint32_t)s * kTcBBytes);
#pragma unroll
                for (int kk = 0; kk < kTcK / 16; ++kk) {  // 16 of K: eight columns of A, +2 in the address field of B
                    const uint32_t acc = (kb > 0 || kk > 0) ? 1u : 0u;
                    asm volatile(
                        "{\n\t.reg .pred p;\n\t"
                        "setp.ne.b32 p, %4, 0;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, {%5, %5, %5, %5}, p;\n\t}"
                        :
                        : "r"(tmem), "r"(a + (uint32_t)(8 * kk)), "l"(db + (uint64_t)(2 * kk)), "r"(idesc), "r"(acc), "r"(0u)
                        : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 smem_u32(&s_empty[s]))
                             : "memory");
            }
            // whatever has been issued arrives on `done` when it has completed (also after a time-out)
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&s_done))
                         : "memory");
            if (!ok) s_fail = 1;
            if (!tc_wait(smem_u32(&s_done), 0u)) s_fail = 1;
        }
    } else if (warp <= kTcGroups * 4) {
        // ---- producers: group g decodes k-blocks g, g + 4, ...; the thread's row of a k-block is 64 weights.
        // A warp reaches the 32 rows of tensor memory that its number modulo 4 names.
        const int group = (warp - 1) >> 2, a_row = (warp & 3) * 32 + lane;
        const uint32_t a_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)kTcMaxN;
        float2 lv[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) lv[k] = __ldg(reinterpret_cast<const float2*>(levels) + k);
        // OPQ: the row's next list entry, as a column of this CTA, and its value
        int at = 0, end = 0, next = INT32_MAX;
        uint32_t value = 0u;
        const int base = OPQ ? (int)((row0 + a_row) * cols + (int64_t)kb0 * kTcK) : 0;  // indices fit 31 bits
        auto entry = [&]() {
            next = at < end ? __ldg(out_idx + at) - base : INT32_MAX;
            value = at < end ? (uint32_t)__ldg(out_val + at) : 0u;
        };
        for (int kb = group, line = 0; kb < kblocks; kb += kTcGroups, ++line) {
            const int ls = line % kTcLines, s = kb % kTcStages;
            if (!warp_wait(&s_line_full[ls], (uint32_t)((line / kTcLines) & 1))) break;
            uint32_t w[8];
            // the thread's 32 bytes: chunks 2 g and 2 g + 1 of its row's line (128-byte swizzle)
            const uint32_t row = code_ring + (uint32_t)ls * kTcLineBytes + (uint32_t)a_row * 128u;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(w[4 * h]), "=r"(w[4 * h + 1]), "=r"(w[4 * h + 2]), "=r"(w[4 * h + 3])
                             : "r"(row + (uint32_t)(((2 * group + h) ^ (a_row & 7)) * 16)));
            const float* sc = scale_ring + ls * kTcScaleFloats + (HALF ? 2 * group : group) * kTcM + a_row;
            const float m = sc[0], m2 = HALF ? sc[kTcM] : 0.0f;
            TcTable tab = tc_table(m, lv);
            uint32_t v[16];
#pragma unroll
            for (int j = 0; j < 4; ++j) tc_decode8(w[j], tab, v + 4 * j);
            // the tensor cores must have read what the stage held (k-block kb - stages)
            if (kb >= kTcStages && !warp_wait(&s_empty[s], (uint32_t)(((kb / kTcStages) - 1) & 1))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t dst = a_lane + (uint32_t)(s * kTcACols);
            tc_store16(dst, v);
            if (HALF) tab = tc_table(m2, lv);
            uint32_t u[16];
#pragma unroll
            for (int j = 0; j < 4; ++j) tc_decode8(w[4 + j], tab, u + 4 * j);
            tc_store16(dst + 16u, u);
            if (lane == 0) tc_arrive(&s_line_empty[ls]);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            if (OPQ) {
                if (kb == group) {  // the row's part of the list, found meanwhile
                    if (!warp_wait(&s_rows, 0u)) break;
                    at = s_beg[a_row], end = s_end[a_row];
                    entry();
                }
                const int c0 = kb * kTcK;
                while (next < c0) {  // the other groups' entries
                    ++at;
                    entry();
                }
                __syncwarp();
                // one entry of one row at a time: the column it shares with its neighbour comes back from tensor
                // memory, the row's half of it is replaced (about two entries per warp and k-block)
                unsigned hits;
                while ((hits = __ballot_sync(kFull, next < c0 + kTcK)) != 0u) {
                    const int src = __ffs(hits) - 1, c = __shfl_sync(kFull, next, src) - c0;
                    const uint32_t a = dst + (uint32_t)(c >> 1);
                    uint32_t r;
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(a));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (lane == src) {
                        r = (c & 1) ? (r & 0xffffu) | (value << 16) : (r & 0xffff0000u) | value;
                        ++at;
                        entry();
                    }
                    __syncwarp();
                    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(a), "r"(r) : "memory");
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) tc_arrive(&s_full[s]);
        }
    } else if (warp == kTcGroups * 4 + 1) {
        // ---- code lines: 128 bytes of each of the 128 rows
        for (int line = 0; line < lines; ++line) {
            const int ls = line % kTcLines;
            if (line >= kTcLines && !warp_wait(&s_line_empty[ls], (uint32_t)(((line / kTcLines) - 1) & 1))) break;
            if (lane == 0)
                tc_load_box(code_ring + (uint32_t)ls * kTcLineBytes, &code_map, &s_line_full[ls], kTcLineBytes, (line0 + line) * 128, (int)row0);
        }
    } else if (warp == kTcGroups * 4 + 2) {
        // ---- X: the 64 columns of a k-block
        for (int kb = 0; kb < kblocks; ++kb) {
            const int s = kb % kTcStages;
            if (kb >= kTcStages && !warp_wait(&s_empty[s], (uint32_t)(((kb / kTcStages) - 1) & 1))) break;
            if (lane == 0) tc_load_box(tiles + (uint32_t)s * kTcBBytes, &x_map, &s_full[s], (uint32_t)n_rhs * 128u, (kb0 + kb) * kTcK, 0);
        }
    } else if (warp <= kTcGroups * 4 + 4) {
        // ---- block constants of every other line, as fp32 [k-block][row]
        constexpr int PER = HALF ? 2 : 1;
        for (int line = warp - (kTcGroups * 4 + 3); line < lines; line += 2) {
            const int ls = line % kTcLines;
            float v[4 * kTcGroups * PER];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int64_t first = (row0 + lane + 32 * r) * cols + (int64_t)kb0 * kTcK;
#pragma unroll
                for (int q = 0; q < kTcGroups * PER; ++q) {
                    const int kb = min(line * kTcGroups + q / PER, kblocks - 1);
                    v[q * 4 + r] = tc_scale<ST>(scales, (first + kb * kTcK + (q % PER) * 32) >> block_shift);
                }
            }
            if (line >= kTcLines && !warp_wait(&s_line_empty[ls], (uint32_t)(((line / kTcLines) - 1) & 1))) break;
#pragma unroll
            for (int q = 0; q < kTcGroups * PER; ++q)
#pragma unroll
                for (int r = 0; r < 4; ++r) scale_ring[ls * kTcScaleFloats + q * kTcM + lane + 32 * r] = v[q * 4 + r];
            __syncwarp();
            if (lane == 0) tc_arrive(&s_line_full[ls]);
        }
    } else if (OPQ) {
        // ---- OPQ: the entries of every row of the tile inside the CTA's columns
        const int f = tid - (kTcGroups * 4 + 5) * 32;
        int64_t k_end = *n_out;
        if (k_end > capacity) k_end = capacity;
        const int64_t n = (int64_t)gridDim.x * kTcM * cols;
        for (int r = f; r < kTcM; r += kTcFinders) s_beg[r] = s_end[r] = 0;
        // first and last entry of the tile, a warp each
        const int64_t p = tc_lower_bound(out_idx, k_end, (row0 + (f < 32 ? 0 : kTcM)) * cols, n, lane);
        if (lane == 0) s_part[f >> 5] = p;
        asm volatile("bar.sync 1, %0;" ::"n"(kTcFinders) : "memory");
        const int64_t lo = s_part[0], hi = s_part[1];
        const uint32_t tile = (uint32_t)(row0 * cols), c_lo = (uint32_t)kb0 * kTcK, c_hi = c_lo + (uint32_t)kblocks * kTcK, nc = (uint32_t)cols;
        // row of entry k if it lies inside the CTA's columns, else -1 (also for what a list that is not ascending holds)
        auto row_of = [&](int64_t k) -> int {
            if (k < lo || k >= hi) return -1;
            const uint32_t i = (uint32_t)__ldg(out_idx + k) - tile, r = i / nc, c = i - r * nc;
            return (r < (uint32_t)kTcM && c >= c_lo && c < c_hi) ? (int)r : -1;
        };
        for (int64_t k = lo + f; k < hi; k += kTcFinders) {
            const int r = row_of(k);
            if (r < 0) continue;
            if (row_of(k - 1) != r) s_beg[r] = (int)k;
            if (row_of(k + 1) != r) s_end[r] = (int)k + 1;
        }
        __syncwarp();
        if (lane == 0) tc_arrive(&s_rows);
    }
    // Every loop above is bounded, so every warp gets here.  After a time-out the issuing thread has
    // still committed and waited (bounded) for what it issued.
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const bool failed = s_fail != 0;
    if (failed) {
        // a TMA copy requested before the time-out may still be writing this CTA's shared memory: it
        // takes microseconds; give it a bounded 100 before the CTA goes away
        if (tid == 0) atomicExch(status, 1);
        for (int i = 0; i < 100; ++i) __nanosleep(1000);
    }
    // the accumulator, one row per thread (warp w reads lanes 32 (w % 4) ...), through shared memory: the stages
    // are free now.  Rows are padded by 16 bytes so that eight neighbouring rows fall into different banks.
    float* part = reinterpret_cast<float*>(tiles_ptr);
    const int pitch = n_rhs + 4;
    if (!failed && warp < 16) {
        float* prow = part + ((warp & 3) * 32 + lane) * pitch;
        for (int c0 = (warp >> 2) * 8; c0 < n_rhs; c0 += 32) {
            uint32_t v[8];
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                         : "r"(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            *reinterpret_cast<uint4*>(prow + c0) = make_uint4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<uint4*>(prow + c0 + 4) = make_uint4(v[4], v[5], v[6], v[7]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    if (splits > 1) cluster.sync();
    else __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols) : "memory");
    // the tile's 128 x n_rhs results are contiguous in y: each CTA of the cluster sums and writes its share
    // of the rows, the ranks' parts in order
    const int quads = n_rhs >> 2, rows_here = kTcM / splits;
    for (int i = tid; i < rows_here * quads; i += NT) {
        const int r = rank * rows_here + i / quads, c = (i % quads) * 4;
        float4 sum = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        for (int q = 0; q < splits; ++q) {
            const float* src = splits > 1 ? cluster.map_shared_rank(part, q) : part;
            const float4 v = *reinterpret_cast<const float4*>(src + r * pitch + c);
            if (q == 0) {
                sum = v;
            } else {
                sum.x += v.x;
                sum.y += v.y;
                sum.z += v.z;
                sum.w += v.w;
            }
        }
        *reinterpret_cast<float4*>(y + (row0 + r) * n_rhs + c) = sum;
    }
    if (splits > 1) cluster.sync();  // nobody leaves while its part is being read
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
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        BOF4_CUDA_TRY(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q));
        if (!f || q != cudaDriverEntryPointSuccess) {
            set_error("bof4_gemm_tc: the driver does not provide cuTensorMapEncodeTiled");
            return BOF4_ERR_CUDA;
        }
        fn = reinterpret_cast<EncodeTiledFn>(f);
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
    if (rows / kTcM > 0x7fffffff) {
        set_error("%s: too many rows", fn);
        return BOF4_ERR_SHAPE;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cols == 0) {
        BOF4_CUDA_TRY(cudaMemsetAsync(d_status, 0, sizeof(int), st));
        BOF4_CUDA_TRY(cudaMemsetAsync(d_y, 0, (size_t)rows * n_rhs * sizeof(float), st));
        return BOF4_OK;
    }
    const int grid = (int)(rows / kTcM);
    // Split along K over a cluster: the choice with the least waves x (k-blocks per CTA + what a CTA costs
    // beside them, about six k-blocks: set-up, pipeline fill and drain, epilogue).
    const int kblocks = (int)(cols / kTcK);
    int splits = 1;
    int64_t best = INT64_MAX;
    for (int cand = 1; cand <= kTcMaxSplit && cand * kTcGroups <= kblocks + kTcGroups - 1; cand *= 2) {
        const int64_t cost = (((int64_t)grid * cand + kSMs - 1) / kSMs) * ((kblocks + cand - 1) / cand + 6);
        if (cost < best) best = cost, splits = cand;
    }
    int rc, block_shift = 0;
    while ((1 << block_shift) < block_size) ++block_shift;
    CUtensorMap x_map, code_map;
    if ((rc = make_map(d_x, false, cols, n_rhs, n_rhs, &x_map)) || (rc = make_map(d_codes, true, cols / 2, rows, kTcM, &code_map)))
        return rc;
    const bool list = opq && capacity > 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, splits);
    cfg.blockDim = dim3(tc_threads(list));
    cfg.dynamicSmemBytes = kTcSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = (unsigned)splits;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const uint16_t* val = static_cast<const uint16_t*>(d_out_val);
#define BOF4_TC_GO(ST_, HALF_, OPQ_)                                                                                        \
    {                                                                                                                       \
        constexpr auto kern = gemm_tc_kernel<ST_, HALF_, OPQ_>;                                                             \
        if ((rc = ensure_dynamic_smem<kern>(kTcSmem))) return rc;                                                           \
        BOF4_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, code_map, d_scales, cols, block_shift, d_codebook, x_map, n_rhs, d_y,  \
                                         d_status, d_out_idx, val, d_n_out, capacity));                                     \
    }
#define BOF4_TC_ST(ST_)                                                             \
    if (block_size == 32) {                                                         \
        if (list) BOF4_TC_GO(ST_, true, true) else BOF4_TC_GO(ST_, true, false)     \
    } else {                                                                        \
        if (list) BOF4_TC_GO(ST_, false, true) else BOF4_TC_GO(ST_, false, false)   \
    }
    if (scale_dtype == BOF4_F32) { BOF4_TC_ST(F32) } else { BOF4_TC_ST(BF16) }
#undef BOF4_TC_ST
#undef BOF4_TC_GO
    return BOF4_OK;
}
