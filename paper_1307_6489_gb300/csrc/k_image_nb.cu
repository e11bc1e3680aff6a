// The neighbour-peak instantiations of the fused image kernel (k_image_chain
// with NB = true, k_image_chain.cuh), for contiguous bundles and byte streams,
// compiled apart from the other instantiations so that the builds run in
// parallel.
#include "k_image_chain.cuh"

namespace rta {

template <int IW, int PPT, int MB, bool STREAM, int OUT, bool ANY>
static cudaError_t launch_nb(const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occupancy_only,
                             int* occ) {
    auto kern = k_image_chain<IW, PPT, MB, true, STREAM, 0, OUT, ANY>;
    // the dynamic shared-memory opt-in is per device; remember the largest size set
    static size_t attr_bytes[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || attr_bytes[dev] < smem) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_bytes[dev] = smem;
    }
    if (occupancy_only) {
        *occ = 0;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, kern, chain_block(IW, 1), smem);
    }
    kern<<<grid, chain_block(IW, 1), smem, s>>>(a);
    return cudaGetLastError();
}

template <bool STREAM, int OUT, bool ANY>
static cudaError_t dispatch_nb(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only,
                               int* occ) {
    switch (v) {
    case 0: return launch_nb<8, 1, 2, STREAM, OUT, ANY>(a, grid, smem, s, occ_only, occ);
    case 1: return launch_nb<4, 2, 2, STREAM, OUT, ANY>(a, grid, smem, s, occ_only, occ);
    case 2: return launch_nb<8, 2, 2, STREAM, OUT, ANY>(a, grid, smem, s, occ_only, occ);
    case 3: return launch_nb<4, 1, 2, STREAM, OUT, ANY>(a, grid, smem, s, occ_only, occ);
    case 4: return launch_nb<8, 1, 3, STREAM, OUT, ANY>(a, grid, smem, s, occ_only, occ);
    default: return cudaErrorInvalidValue;
    }
}

// The same tile variants as the other window modes (kVariants in k_image.cu): byte-stream
// bundles, the integrate-only call, and rows with masks (rows alone: k_image_lean.cu).
template <bool ANY>
static cudaError_t dispatch_nb_any(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only,
                                   int* occ) {
    if (a.smeta) return dispatch_nb<true, OUT_ROWS, ANY>(v, a, grid, smem, s, occ_only, occ);
    if (a.integrate_only) return dispatch_nb<false, OUT_CHARGES, ANY>(v, a, grid, smem, s, occ_only, occ);
    return dispatch_nb<false, OUT_MASKS, ANY>(v, a, grid, smem, s, occ_only, occ);
}

cudaError_t dispatch_image_chain_nb(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only,
                                    int* occ) {
    return a.any_window ? dispatch_nb_any<true>(v, a, grid, smem, s, occ_only, occ)
                        : dispatch_nb_any<false>(v, a, grid, smem, s, occ_only, occ);
}

}  // namespace rta
