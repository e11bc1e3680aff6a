// The image chain on contiguous bundles (as k_image_lean.cu) with sliding windows of 4, 5, 7 or 8
// samples: the packed searches of 40, 30 and 25 samples (and the 16-sample camera's window of 5)
// compiled for those widths. The search for any width is slower: 6,000 images of
// 1855 pixels x 40 samples, W = 8, 410 us, here 168 us.
#include "k_image_launch.cuh"

namespace rta {

cudaError_t dispatch_image_chain_win(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s) {
    switch (a.pp.W) {
    case 4: return dispatch_flat_rows<SEARCH_OWN, 4>(v, a, grid, smem, s);
    case 5: return dispatch_flat_rows<SEARCH_OWN, 5>(v, a, grid, smem, s);
    case 7: return dispatch_flat_rows<SEARCH_OWN, 7>(v, a, grid, smem, s);
    case 8: return dispatch_flat_rows<SEARCH_OWN, 8>(v, a, grid, smem, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace rta
