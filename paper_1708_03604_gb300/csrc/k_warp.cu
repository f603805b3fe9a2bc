// Few output blocks on the CUDA cores: a warp per block.
//
// With few blocks for the warps of the GPU there is nothing for lane groups
// (k_group.cu) or register tiles (k_tile.cu) to share: a block's own chain of
// products is what takes the time, so the lanes of a warp split its elements, and
// the loads of as many terms as the registers hold run ahead (wide: 253 registers,
// 8 warps an SM).
#include <cuda_runtime.h>

#include "numeric_items.cuh"
#include "numeric_warp.cuh"

namespace bsm {

namespace {

template <typename T, bool WIDE>
__global__ void __launch_bounds__(kGroupThreads) k_numeric_warp(NumericArgs a) {
    const int lane = threadIdx.x & 31;
    if (a.status && *a.status != 0) return;
    while (true) {
        int64_t t = 0;
        if (lane == 0) t = (int64_t)atomicAdd(a.work_counter, 1ull);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= a.n_items) break;
        const int64_t q = a.item_order ? (int64_t)((uint32_t)a.item_order[t] & 0x7fffffffu) : t;
        BSM_DBG_WARP_SKIP(a, q, lane)
        warp_block<T, WIDE>(a, q, lane);
    }
}

template <typename T, bool WIDE>
cudaError_t launch_build(const NumericArgs &a, cudaStream_t s, int *grid) {
    static std::atomic<int> resident{0};
    return launch_persistent(k_numeric_warp<T, WIDE>, resident, a, s, grid);
}

}  // namespace

cudaError_t launch_numeric_warp(const NumericArgs &a, bool wide, cudaStream_t s, int *grid) {
    if (a.dtype == BSM_FP64) return wide ? launch_build<double, true>(a, s, grid) : launch_build<double, false>(a, s, grid);
    return wide ? launch_build<float, true>(a, s, grid) : launch_build<float, false>(a, s, grid);
}

uint32_t warp_debug_bits(cudaStream_t s) { return read_debug_bits(s); }

}  // namespace bsm
