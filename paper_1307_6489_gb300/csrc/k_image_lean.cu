// The instantiations of the fused image kernel (k_image_chain.cuh) that run the image chain on
// contiguous bundles whose cameras all have a specialised window search (ANY = false): flat
// window, neighbour-peak window and digital filter, rows only. Compiled apart from the others so
// that the builds run in parallel.
#include "k_image_rows.cuh"

namespace rta {

// The same tile variants as the other window modes (kVariants in k_image.cu).
cudaError_t dispatch_image_chain_lean(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s,
                                      bool occ_only, int* occ) {
    if (a.pp.nbpeak) {
        switch (v) {
        case 0: return launch_rows<8, 1, 2, 6, true>(a, grid, smem, s, occ_only, occ);
        case 1: return launch_rows<4, 2, 2, 6, true>(a, grid, smem, s, occ_only, occ);
        case 2: return launch_rows<8, 2, 2, 6, true>(a, grid, smem, s, occ_only, occ);
        case 3: return launch_rows<4, 1, 2, 6, true>(a, grid, smem, s, occ_only, occ);
        case 4: return launch_rows<8, 1, 3, 6, true>(a, grid, smem, s, occ_only, occ);
        default: return cudaErrorInvalidValue;
        }
    }
    if (a.pp.filter) {
        switch (v) {
        case 0: return launch_rows<8, 1, 2, 6, false, 1>(a, grid, smem, s, occ_only, occ);
        case 1: return launch_rows<4, 2, 2, 6, false, 1>(a, grid, smem, s, occ_only, occ);
        case 2: return launch_rows<8, 2, 2, 6, false, 1>(a, grid, smem, s, occ_only, occ);
        case 3: return launch_rows<4, 1, 2, 6, false, 1>(a, grid, smem, s, occ_only, occ);
        case 4: return launch_rows<8, 1, 3, 6, false, 1>(a, grid, smem, s, occ_only, occ);
        default: return cudaErrorInvalidValue;
        }
    }
    if (a.pp.sliding && a.pp.W != 6 && !occ_only) return dispatch_image_chain_win(v, a, grid, smem, s);
    return dispatch_rows<6>(v, a, grid, smem, s, occ_only, occ);
}

}  // namespace rta
