// The neighbour-peak instantiations of the fused image kernel (k_image_chain
// with NB = true, k_image_chain.cuh) for byte streams, the integrate-only call and rows with
// masks (rows alone: k_image_lean.cu, k_image_any.cu).
#include "k_image_launch.cuh"

namespace rta {

template <int SEARCH>
static cudaError_t dispatch_nb(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only,
                               int* occ) {
    if (a.smeta) return dispatch_chain<true, true, 0, OUT_ROWS, SEARCH>(v, a, grid, smem, s, occ_only, occ);
    if (a.integrate_only) return dispatch_chain<true, false, 0, OUT_CHARGES, SEARCH>(v, a, grid, smem, s, occ_only, occ);
    return dispatch_chain<true, false, 0, OUT_MASKS, SEARCH>(v, a, grid, smem, s, occ_only, occ);
}

cudaError_t dispatch_image_chain_nb(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only,
                                    int* occ) {
    return a.search == SEARCH_PACKED ? dispatch_nb<SEARCH_PACKED>(v, a, grid, smem, s, occ_only, occ)
                        : dispatch_nb<SEARCH_SERIAL>(v, a, grid, smem, s, occ_only, occ);
}

}  // namespace rta
