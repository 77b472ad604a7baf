// Codebook fit over samples that are put in order ONCE: what the two ways share (em_sorted.cu: one sample per weight, put in the order of
// bins of x; em_cells.cu and em_cells_fit.cu: one per distinct normalised weight of bf16 data, whose order is known).
//
// The normalised weights x and the block constants do not change from one Lloyd iteration to the next;
// only the thresholds move.  With the samples in ascending order of a 16-bit bin of x and running sums of
// the bins at hand, an iteration needs no pass over the data: what lies below a threshold is a running sum
// plus a few samples of the bin that the threshold cuts, a region is the difference of two such sums, and the weighted median is
// found the same way.  An iteration costs about as much as a handful of L2 accesses, whatever the size
// of the data.
#pragma once

#include "common.cuh"
#include "em_common.cuh"
#include "layout.h"

namespace bof4 {

constexpr int kSortGrid = 148;               // CTAs of the ordering passes, a contiguous part of the samples each
constexpr int kSortBins = 1 << 16;           // bins of x; bin 0 stays empty
constexpr int kSortGroup = 32;               // bins per group sum
constexpr int kSortGroups = kSortBins / kSortGroup;
constexpr uint32_t kFarBin = 0xffffu;
constexpr int kSortChunk = 128;              // samples per warp of the bin sums
constexpr int kSortMinIters = 4;             // shorter fits stream, see ordering_pays
// A bin of more samples than this, crowded, is not looked through sample by sample (em_sorted.cu).  Near-Gaussian data
// of 2^26 weights, the most there can be, has up to 3500 in a bin; 4096 take a warp 10 us.
constexpr uint32_t kSortCrowd = 4096;
constexpr uint32_t kSortWindow = 8192;       // samples put in full order together
constexpr int64_t kSortMaxDirect = (int64_t)1 << 26;  // one sample per weight: 16 bytes of workspace each
constexpr int kSortParts = 2 * kSMs + 1;     // partial sums of w^2: CTAs of the sample kernels, and the short last blocks

// A sample is {x, the magnitude of its block constant}.
struct SortSums {      // per bin, per group, or per part of a bin
    double s, sx;      // sum of the sample weights, sum of weight * x
    unsigned long long a;  // MAE: sum of the fixed-point weights of the median
};

struct SortWs {
    uint32_t* n_items;    // device: [0] samples, [1] bits of the largest block constant, [4] whether a bin is crowded
    double* w2;           // [kSortParts]
    uint32_t* counts;     // [kSortGrid][256]; behind the ordering passes running sums of the groups, see sort_fit_mae_kernel
    uint32_t* start;      // [kSortBins + 1] first sample of every bin
    uint32_t* first;      // [kSortGroups + 1] first sample of every group; before, the largest constants of the samples' CTAs
    uint16_t* off;        // [kSortBins] first sample of a bin in its group, kFarBin: too far, see start
    SortSums *bin, *group;
    SortSums* pre;        // per bin: the bins of its group in front of it
    SortSums *lead, *trail;  // [chunks] part of a bin that began in an earlier chunk / that goes on in the next
    float2 *a, *b;        // samples, ordered samples
    SortSums* before;     // crowded bins: sums of the window's samples in front of every fourth (in the place of a)
};

// Whether a fit of `iters` iterations over n weights is faster with its samples in order than streamed: the ordering is
// paid once, an iteration is cheaper by what it streams.  Both sides by measurement, in us with k = n / 2^20 (blocks of 64;
// other block sizes differ by a few per cent):
//   ordering, less what a streamed fit takes before its first iteration
//             one sample per weight, fp32: 66 (k = 1), 87 (2), 150 (4), 263 (8), 510 (16), 715 (24), 925 (32), 1360 (48), 1815 (64)
//             distinct bf16 weights 43 to 56 (2), 48 to 60 (4), 65 to 80 (16), 81 to 120 (64), 109 to 255 (256)
//   streamed iteration less an ordered one
//             fp32: MSE 15 (1), 15 (2), 19 (4), 25 (8), 34 (16), 49 (24), 61 (32), 83 (48), 105 (64),
//             medians 47 (1), 50 (2), 56 (4), 71 (8), 90 (16), 120 (24), 142 (32), 188 (48), 231 (64)
//             bf16: MSE 16 (2), 16 (4), 31 (16), 76 (64), 264 (256), medians 54, 58, 82, 180, 679
// The lines below lie on the streamed side of these, which takes 9 MB of workspace where ordering takes 16 bytes a weight (64 MB and 10
// bytes a block for bf16 data): a fit at the line has streamed at most two and a half times what the ordering costs.  From 2^25 weights on
// (more than half a gigabyte) that is on purpose: ordering has to save more than it costs, and squared errors over 2^26 weights get by with the
// small workspace up to 32 iterations.  Where they cross, in iterations, and by the figures: fp32 MSE 6 (5) at 2^20, 10 (9) at 2^22, 13 (11) at
// 2^23, 17 (15) at 2^24, 20 (16) at 2^25, 33 (18) at 2^26, medians 4, 4 (3) at 2^22, 7 (4) at 2^23, 9 (6) at 2^24, 11 (7) at 2^25, 19 (8) at
// 2^26; bf16 MSE 6 (3) from 3 * 2^19 to 2^22, 4 (3) from 2^24 on, medians 4 (2).
// Fewer than four iterations are not ordered, although two or three would pay for bf16 data from 2^26 weights on (2^28, three: 1000
// us streamed, about 410 ordered): such a fit gets by with the small workspace.
inline bool ordering_pays(int w_dtype, int64_t n, int metric, int iters, bool cells)
{
    if (iters < kSortMinIters || n < 1) return false;
    const double k = (double)n / (1 << 20);
    const bool mae = metric == BOF4_METRIC_MAE || metric == BOF4_METRIC_MAE_NORMALIZED;
    double order = 105.0 + 1.1 * k, gain = mae ? 50.0 + 1.9 * k : 16.5 + 0.9 * k;
    if (!cells) {
        order = fmax(fmin(46.0 + 35.0 * k, 50.0 + 33.0 * k), 70.0 * k - 1120.0);
        gain = mae ? fmax(47.5, 31.0 + 2.3 * k) : (w_dtype == BOF4_BF16 ? 18.0 : 13.0) + 1.42 * k;
    }
    return iters * gain >= order;
}

// Whether distinct weights serve as samples (em_cells.cu), and the bytes of workspace they take.
bool cells_apply(int w_dtype, int64_t n);
size_t cells_workspace_bytes(int64_t n, int block_size);

// Carves the workspace for up to n samples; returns the bytes used.
size_t sorted_layout(void* base, int64_t n, SortWs* W);

struct SortFit {
    int metric;
    int64_t n_total;
    int64_t n_max;                   // at most this many samples
    float* codebook;
    uint32_t fixed_mask;
    int iters;
    double* err_log;
};

// The whole fit by one of the two ways; *done tells whether it was taken (workspace, size, type,
// number of iterations).
int sorted_fit(const EmArgs& a, float* d_codebook, uint32_t fixed_mask, int iters, double* d_err_log, void* d_ws,
               size_t ws_bytes, cudaStream_t st, bool* done);
int cells_fit(const EmArgs& a, float* d_codebook, uint32_t fixed_mask, int iters, double* d_err_log, void* d_ws,
              size_t ws_bytes, cudaStream_t st, bool* done);

// Bin of a normalised weight, monotone in x: 32768 +- the bin of |x|, which is 0 for x = 0 alone, eight bins per binade
// below 2^-11 (1 ... 215, all of |x| < 2^-38 in the first), bins of width 1 / 32566 from there on (at least the width of the
// ones below), and 32767 for |x| = 1 alone.  Zeros (sparse data) and ones (a weight per block) are the only
// values that data is likely to hold in any number, and no threshold ever has to look into a bin of one value.
constexpr int kBinMinus = 1, kBinZero = 32768, kBinPlus = 65535;
__device__ __forceinline__ int sort_bin(float x)
{
    const float a = fminf(fabsf(x), 1.0f);
    int m;
    if (a >= 0x1p-11f) {
        m = 201 + (int)(a * 32566.0f);
    } else {
        m = 215 - (927 - (int)(__float_as_uint(a) >> 20));
        m = (a == 0.0f) ? 0 : max(m, 1);
    }
    return x < 0.0f ? kBinZero - m : kBinZero + m;
}
__device__ __forceinline__ bool one_value_bin(int b) { return b == kBinMinus || b == kBinZero || b == kBinPlus; }
__device__ __forceinline__ float value_of_bin(int b) { return b == kBinMinus ? -1.0f : b == kBinPlus ? 1.0f : 0.0f; }

// Order-preserving key of x and back; -0 and +0 share a key.
__device__ __forceinline__ uint32_t sort_key(float x)
{
    const uint32_t u = __float_as_uint(x + 0.0f);
    return u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
}
__device__ __forceinline__ float sort_key_value(uint32_t k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// |m| as a 31-bit fixed-point integer relative to the largest magnitude of the data (see em_mae.cu).
__device__ __forceinline__ uint32_t sort_fixed_weight(float m, uint32_t max_bits)
{
    const uint32_t b = __float_as_uint(fabsf(m));
    const int e = max((int)(b >> 23), 1), emax = max((int)(max_bits >> 23), 1);
    const uint32_t mant = (b & 0x7fffffu) | ((b >> 23) ? 0x800000u : 0u);
    const int sh = e - emax + 7;
    if (sh >= 0) return mant << min(sh, 7);
    return (-sh >= 32) ? 0u : (mant >> (-sh));
}

}  // namespace bof4
