// Cells of distinct normalised weights: what em_cells.cu (their sums) and em_cells_fit.cu (iterations over them) share.
//
// A cell is (significand b of the block constant, sign, distance d of the bit patterns of constant and weight): its normalised weight
// is +-(a / b) 2^-k with d = 128 k + b - a.  The cells are laid out by b, sign and d, so that a unit of work adds to neighbours.
// Their order by x needs no sorting: between two powers of two lie the same 16384 fractions a / b of significands whatever
// the exponent, so the place of a cell in this order is the rank of its fraction and its binade.
#pragma once

#include "em_fit.cuh"

namespace bof4 {

constexpr int kCellDepth = 40 * 128;              // bit-pattern distances told apart: 40 binades
constexpr int kCellRow = 2 * kCellDepth + 1;      // positive, negative, zero
constexpr int kDeepExps = 88;                     // biased exponents of fp32 numbers up to 2^-40
constexpr int kDeepCells = 128 * kCellRow;        // first deep cell: positive ones by exponent, then negative ones
constexpr int kCells = kDeepCells + 2 * kDeepExps;
constexpr uint32_t kZeroCell = 2 * kCellDepth;    // zeros of all significands; +-1 of all are in the first row's cells as well

constexpr int kCellFractions = 128 * 128;         // a / b, between two powers of two
constexpr int kFractionThreads = 256;             // threads of a CTA that put them in order
constexpr int kCellParts = 4096;                  // equal parts of a binade

// Places in the order of x, of one sign: zero, deep cells by exponent, the binades from 2^-40 on, one.  The place of x >= 0 is kCellOne
// behind that of x = -1, which is the first.
constexpr int kPlaceBinades = 1 + kDeepExps;
constexpr int kCellOne = kPlaceBinades + 40 * kCellFractions;  // place of one: as many lie between it and zero
constexpr int kCellPlaces = 2 * kCellOne + 1;
constexpr int kCellBlock = 512;                   // places whose sums are formed together
constexpr int kCellBlocks = kCellPlaces / kCellBlock + 1;  // (behind the last place there is another one, with all in front)
constexpr int kCellPart = 128, kCellPartsAll = kCellBlocks * (kCellBlock / kCellPart);  // parts of blocks, for the weights of the medians

struct CellUnit {
    uint32_t mag, first, count;  // bit pattern of |m|, first block in the ordered list, blocks
};
struct CellBlock {     // sums of a block of places
    double s, sx, sxx;
};
struct CellsWs {
    uint32_t* hist;      // [kMags] blocks per magnitude
    uint32_t* cursor;    // [kMags] next free position of the ordered list
    uint32_t* scal;      // [0] units, [1] next unit, [2] largest magnitude of the short last blocks, [3] of all, [4 ... 5] cells_scale
    ulonglong2* acc;     // [kCells] 128-bit sums of weights
    unsigned long long* acc_a;  // [kCells] fixed-point weights of the medians
    CellUnit* units;
    unsigned long long* order;  // [blocks] address, sign of the constant in bit 63
    uint16_t* consts;           // [blocks]
    uint16_t* value_of;         // [kCellFractions] by rank: (a - 128) * 128 + b - 128; [kCellParts] fractions in front of a part
    double2* front;             // by place: {s, sx} of the places of its block in front of it
    unsigned long long* front_a;  // by place: weight of the places of its part in front of it
    CellBlock* block;             // [kCellBlocks]
    unsigned long long* part_a;   // [kCellPartsAll]
};
__device__ __forceinline__ double* cells_scale(const CellsWs& W) { return reinterpret_cast<double*>(W.scal + 4); }  // undoes the sums' scale

// How many of the fractions y = a / b (a >= b) or 2 a / b (a < b), a and b in 128 ... 255, lie before that of (a0, b0) + 128: in their order,
// equal ones by b.
__device__ __forceinline__ uint32_t fraction_rank(uint32_t a0, uint32_t b0)
{
    const uint32_t a = (a0 + 128u) << (a0 < b0 ? 1 : 0), b = b0 + 128u;
    // y b' = q1 + r1 / b and y b' / 2 = q2 + r2 / 2 b for b' = 128, 129, ...
    uint32_t q1 = 128u * a / b, r1 = 128u * a % b, q2 = q1 >> 1, r2 = r1 + (q1 & 1u) * b;
    const uint32_t dq = a / b, dr = a % b;  // (a / b is 1)
    uint32_t rank = 0u;
#pragma unroll 4
    for (uint32_t c = 128u; c < 256u; ++c) {
        const uint32_t tie = c < b ? 1u : 0u;
        const int n1 = (int)min(r1 || tie ? q1 : q1 - 1u, 255u) - (int)c + 1;            // a' = c ... 255, a' < y c (or equal)
        const int n2 = (int)min(r2 || tie ? q2 : q2 - 1u, c - 1u) - 127;                 // a' = 128 ... c - 1, a' < y c / 2
        rank += (uint32_t)max(n1, 0) + (uint32_t)max(n2, 0);
        q1 += dq, r1 += dr;
        if (r1 >= b) r1 -= b, ++q1;
        q2 = q1 >> 1, r2 = r1 + (q1 & 1u) * b;
    }
    return rank;
}

// How many fractions lie below 1 + part / kCellParts (none of them is nearer to it than 2^-20, so how they are rounded is of no account).
__device__ __forceinline__ uint32_t fractions_below(uint32_t part)
{
    const uint32_t q = kCellParts + part;
    uint32_t n = 0u;
    for (uint32_t b = 128u; b < 256u; ++b) {  // a / b < q / kCellParts, and 2 a / b
        const uint32_t t = b * q - 1u;
        n += (uint32_t)max((int)min(t / kCellParts, 255u) - (int)b + 1, 0) + (uint32_t)max((int)min(t / (2u * kCellParts), b - 1u) - 127, 0);
    }
    return n;
}

// Sums in the order of x and all iterations.
int cells_run(const CellsWs& W, const SortFit& F, cudaStream_t st);

}  // namespace bof4
