// The image chain on contiguous bundles (as k_image_lean.cu) for launches with a
// camera that takes the packed search for any window (window_search).
#include "k_image_launch.cuh"

namespace rta {

cudaError_t dispatch_image_chain_any(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s) {
    // variant 4 is variant 0's tile in the 64 registers that let three CTAs share an SM; where
    // shared memory holds fewer, variant 0's registers (90) are there to be used: 1,000 images of
    // 4096 pixels x 128 samples, W = 16, 360 us and 370 in 64; 3,000 of 1600 x 100, W = 6, 267 and 276 (rows split)
    if (v == 4 && 3 * smem > SMEM_PER_CTA && (a.arr.max_P > SMALL_PIX || a.max_S >= 64)) v = 0;
    return dispatch_rows<SEARCH_PACKED>(v, a, grid, smem, s);
}

}  // namespace rta
