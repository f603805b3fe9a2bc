// Output blocks handed to the lane groups of the CUDA-core kernels.
#pragma once

#include <atomic>

#include "bsm_internal.cuh"
#include "numeric_debug.cuh"

namespace bsm {
namespace {

constexpr int kGroupThreads = 128;

// Blocks taken from the ticket together, with what a group needs to start one:
// 32 blocks' loads run side by side, one lane each, instead of a chain of
// dependent loads every time a group is done (a warp's other groups wait).
struct Window {
    int32_t item[32], shape[32];
    int32_t p[32], pe[32];          // products [p, pe)
    int64_t xoff[32], yoff[32];     // operands of the first product
    int32_t tn[32];                 // its terms of k
    int32_t ix[32], iy[32];         // operand blocks of the second
};

struct ItemRun {
    Window *w;
    int cur, count;    // entries of the window handed out, and all
    int64_t left;      // blocks not yet taken by any warp, as last seen
};

// true when the window holds a block (a new window is loaded when it is empty)
__device__ __forceinline__ bool items_left(const NumericArgs &a, ItemRun &run, int lane) {
    if (run.cur < run.count) return true;
    // an eighth of a warp's share of what is left, so that the warps end together
    const int chunk = (int)max((int64_t)1, min((int64_t)32, run.left / ((int64_t)gridDim.x * kGroupThreads / 32 * 8)));
    int64_t base = 0;
    if (lane == 0) base = (int64_t)atomicAdd(a.work_counter, (unsigned long long)chunk);
    base = __shfl_sync(0xffffffffu, base, 0);
    run.left = max((int64_t)0, a.n_items - base);
    run.cur = 0;
    run.count = (int)min((int64_t)chunk, run.left);
    if (lane < run.count) {
        const int64_t pos = base + lane;
        const int32_t q = a.item_order ? (int32_t)((uint32_t)a.item_order[pos] & 0x7fffffffu) : (int32_t)pos;
        Window &w = *run.w;
        w.item[lane] = q;
        w.shape[lane] = a.out_blk_rc[q];
        const int32_t p = (int32_t)a.seg_ptr[q], pe = (int32_t)a.seg_ptr[q + 1];
        w.p[lane] = p;
        w.pe[lane] = pe;
        if (p < pe && BSM_DBG_LANE_OK(a, q)) {
            const int32_t ix = a.px[p], iy = a.py[p], rc = a.x_blk_rc[ix];
            if (pe - p > 1) {
                w.ix[lane] = a.px[p + 1];
                w.iy[lane] = a.py[p + 1];
            }
            w.xoff[lane] = a.x_blk_off[ix];
            w.yoff[lane] = a.y_blk_off[iy];
            w.tn[lane] = a.x_trans ? rc_rows(rc) : rc_cols(rc);
        }
    }
    __syncwarp();
    return run.count > 0;
}

// Persistent launch of `kernel`: as many CTAs as fit, or as the blocks need.
template <typename K>
cudaError_t launch_persistent(K kernel, std::atomic<int> &resident, const NumericArgs &a, cudaStream_t s, int *grid) {
    int per_sm = resident.load(std::memory_order_relaxed);  // the same for every device this code runs on
    if (per_sm == 0) {
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kGroupThreads, 0);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        resident.store(per_sm, std::memory_order_relaxed);
    }
    if (a.ctas_per_sm > 0 && a.ctas_per_sm < per_sm) per_sm = a.ctas_per_sm;
    constexpr int warps = kGroupThreads / 32;
    const int64_t need = (a.n_items + warps - 1) / warps, fit = (int64_t)num_sms() * per_sm;
    *grid = (int)(need < fit ? need : fit);
    kernel<<<*grid, kGroupThreads, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace
}  // namespace bsm
