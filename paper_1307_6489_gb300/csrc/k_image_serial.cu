// The image chain on contiguous bundles (as k_image_lean.cu) for launches with a camera whose
// sample count or window has no specialised search and is served best by the serial one
// (window_search).
#include "k_image_launch.cuh"

namespace rta {

cudaError_t dispatch_image_chain_serial(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s) {
    return dispatch_rows<SEARCH_SERIAL>(v, a, grid, smem, s);
}

}  // namespace rta
