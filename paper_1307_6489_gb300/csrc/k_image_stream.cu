// The byte-stream instantiations of the fused image kernel (k_image_chain with
// STREAM = true, k_image_chain.cuh): the producer copies each chunk from the
// segments of an ingested stream; with the digital filter (FILTER 1) and without it.
#include "k_image_launch.cuh"

namespace rta {

template <int SEARCH>
static cudaError_t dispatch_stream(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only,
                                   int* occ) {
    return a.pp.filter || occ_only ? dispatch_chain<false, true, 1, OUT_ROWS, SEARCH>(v, a, grid, smem, s, occ_only, occ)
                                   : dispatch_chain<false, true, 0, OUT_ROWS, SEARCH>(v, a, grid, smem, s, occ_only, occ);
}

cudaError_t dispatch_image_chain_stream(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s,
                                        bool occ_only, int* occ) {
    return a.search == SEARCH_PACKED ? dispatch_stream<SEARCH_PACKED>(v, a, grid, smem, s, occ_only, occ)
                        : dispatch_stream<SEARCH_SERIAL>(v, a, grid, smem, s, occ_only, occ);
}

}  // namespace rta
