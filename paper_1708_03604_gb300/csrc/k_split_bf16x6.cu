// The BF16x6 split path's kernels (a translation unit per precision: they compile side by side).
#include "numeric_split.cuh"

namespace bsm {

cudaError_t launch_split_bf16x6(const NumericArgs &a, cudaStream_t s, int threads, int *grid) {
    return launch_tc<BSM_P_BF16x6>(a, s, threads, grid);
}

uint32_t split_bf16x6_debug_bits(cudaStream_t s) { return read_debug_bits(s); }

}  // namespace bsm
