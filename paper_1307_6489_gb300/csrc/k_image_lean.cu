// The instantiations of the fused image kernel (k_image_chain.cuh) that run the image chain on
// contiguous bundles whose cameras all have a specialised window search: flat window, neighbour-peak window and digital filter, rows only.
#include "k_image_launch.cuh"

namespace rta {

cudaError_t dispatch_image_chain_lean(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s) {
    if (a.pp.sliding && a.pp.W != 6 && !a.pp.nbpeak && !a.pp.filter)
        return dispatch_image_chain_win(v, a, grid, smem, s);
    return dispatch_rows<SEARCH_OWN>(v, a, grid, smem, s);
}

}  // namespace rta
