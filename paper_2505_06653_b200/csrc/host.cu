// Host-only parts of the C ABI: error strings, the OPQ threshold, the default starting codebook.
#include <limits.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>

#include <atomic>

#include "common.cuh"
#include "em_sorted.cuh"
#include "layout.h"

namespace bof4 {

static thread_local char g_err[512] = "";

void set_error(const char* fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

int cuda_fail(cudaError_t e, const char* what)
{
    set_error("CUDA error %d (%s) in %s", (int)e, cudaGetErrorString(e), what);
    return BOF4_ERR_CUDA;
}

// Where a count is read back: a page of host memory that the device writes, one line per waiting call.  A copy to
// pageable memory and a stream synchronisation take 8 us after the kernels are done, a store seen by a
// polling host 1 us.  The page is allocated once; with all its lines taken a call copies as before.
struct CountSlots {
    static constexpr int kSlots = 64;
    std::atomic<uint64_t> taken{0};
    char* page = nullptr;
    int take()
    {
        uint64_t t = taken.load(std::memory_order_relaxed);
        while (~t) {
            const int k = __builtin_ctzll(~t);
            if (taken.compare_exchange_weak(t, t | (1ull << k), std::memory_order_acquire)) return k;
        }
        return -1;
    }
    void give(int k) { taken.fetch_and(~(1ull << k), std::memory_order_release); }
    volatile int64_t* slot(int k) { return reinterpret_cast<volatile int64_t*>(page + 64 * k); }
};

// The process's page, or NULL if none can be had.
static CountSlots* count_slots()
{
    static CountSlots slots;
    static const bool ok = [] {
        void* p = nullptr;
        if (cudaHostAlloc(&p, 64 * CountSlots::kSlots, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
            (void)cudaGetLastError();
            return false;
        }
        slots.page = static_cast<char*>(p);
        return true;
    }();
    return ok ? &slots : nullptr;
}

__global__ void store_count_kernel(const int64_t* n_out, volatile int64_t* slot)
{
    if (!after_previous()) return;
    *slot = *n_out;
}

}  // namespace bof4

extern "C" {

const char* bof4_last_error(void) { return bof4::g_err; }

size_t bof4_workspace_bytes(int op, int64_t n_max, int block_size, int metric)
{
    if (n_max < 0 || !bof4::valid_block_size(block_size)) return 0;
    if (op == BOF4_OP_EM) {
        if (metric < BOF4_METRIC_MSE || metric > BOF4_METRIC_MAE_NORMALIZED) return 0;
        return bof4::em_workspace_bytes_for(n_max);
    }
    if (op == BOF4_OP_EM_BF16) return bof4_fit_workspace_bytes(n_max, BOF4_BF16, block_size, metric, INT_MAX);
    if (op == BOF4_OP_OPQ) return bof4::opq_layout(n_max).total;
    return 0;
}

size_t bof4_fit_workspace_bytes(int64_t n_total, int w_dtype, int block_size, int metric, int iters)
{
    const size_t need = bof4_workspace_bytes(BOF4_OP_EM, n_total, block_size, metric);
    if (need == 0 || (w_dtype != BOF4_F32 && w_dtype != BOF4_BF16)) return 0;
    const bool cells = bof4::cells_apply(w_dtype, n_total);
    if ((!cells && n_total > bof4::kSortMaxDirect) || !bof4::ordering_pays(w_dtype, n_total, metric, iters, cells)) return need;
    const size_t order = cells ? bof4::cells_workspace_bytes(n_total, block_size) : bof4::sorted_layout(nullptr, n_total, nullptr);
    return need < order ? order : need;
}

// The synchronising half of the two-call pattern: the outlier-producing calls only leave the true
// count on the device; this reads it back and turns an overflow into an error code.
int bof4_outlier_count(const int64_t* d_n_out, int64_t capacity, int64_t* h_n_out, void* stream)
{
    if (!d_n_out || capacity < 0) {
        bof4::set_error("bof4_outlier_count: NULL count pointer or negative capacity");
        return BOF4_ERR_INVALID_ARG;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int64_t count = 0;
    bof4::CountSlots* slots = bof4::count_slots();
    const int k = slots ? slots->take() : -1;
    if (k < 0) {
        BOF4_CUDA_TRY(cudaMemcpyAsync(&count, d_n_out, sizeof(count), cudaMemcpyDeviceToHost, st));
        BOF4_CUDA_TRY(cudaStreamSynchronize(st));
    } else {
        // a slot is given back once its kernel is known to have run; after an error it is not
        volatile int64_t* slot = slots->slot(k);
        *slot = -1;
        bof4::launch_after(bof4::store_count_kernel, 1, 1, 0, st, d_n_out, slot);
        BOF4_CUDA_TRY(cudaGetLastError());
        for (int polls = 0; (count = *slot) < 0; ++polls) {
            if ((polls & 1023) != 1023) continue;
            const cudaError_t e = cudaStreamQuery(st);
            if (e == cudaErrorNotReady) continue;
            BOF4_CUDA_TRY(e);
            count = *slot;  // the stream is done: this is the count, whatever it is
            break;
        }
        std::atomic_thread_fence(std::memory_order_acquire);
        slots->give(k);
    }
    if (h_n_out) *h_n_out = count;
    if (count > capacity) {
        bof4::set_error("outlier list overflow: %lld outliers found, capacity %lld (only the first %lld were "
                        "stored; call again with capacity >= %lld)",
                        (long long)count, (long long)capacity, (long long)capacity, (long long)count);
        return BOF4_ERR_CAPACITY;
    }
    return BOF4_OK;
}

// tau with G(tau) = (1 + q^(1/I)) / 2  <=>  erfc(tau / sqrt 2) = 1 - q^(1/I) = -expm1(ln q / I).
// erfc is strictly decreasing, so bisection on [0, 40] converges to the last bit.
double bof4_opq_threshold(double q, int block_size)
{
    if (!(q > 0.0 && q < 1.0) || block_size < 1) return NAN;
    const double target = -expm1(log(q) / (double)block_size);
    double lo = 0.0, hi = 40.0;
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (erfc(mid * M_SQRT1_2) > target)
            lo = mid;
        else
            hi = mid;
    }
    return 0.5 * (lo + hi);
}

int bof4_default_init(int norm, float h_levels[BOF4_LEVELS], uint32_t* h_fixed_mask)
{
    if (!h_levels || (norm != BOF4_NORM_ABS && norm != BOF4_NORM_SIGNED)) {
        bof4::set_error("bof4_default_init: bad argument");
        return BOF4_ERR_INVALID_ARG;
    }
    for (int k = 0; k < 7; ++k) h_levels[k] = (float)(-1.0 + (double)k / 7.0);
    h_levels[7] = 0.0f;
    for (int k = 1; k <= 8; ++k) h_levels[7 + k] = (float)((double)k / 8.0);
    if (h_fixed_mask)
        *h_fixed_mask = (norm == BOF4_NORM_ABS) ? ((1u << 0) | (1u << 7) | (1u << 15))
                                                : ((1u << 7) | (1u << 15));
    return BOF4_OK;
}

}  // extern "C"
