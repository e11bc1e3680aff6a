// The byte-stream instantiations of the fused image kernel (k_image_chain with
// STREAM = true, k_image_chain.cuh): the producer copies each chunk from the
// segments of an ingested stream; with the digital filter (FILTER 1) and without it.
// Compiled apart so the builds run in parallel.
#include "k_image_chain.cuh"

namespace rta {

template <int IW, int PPT, int MB, int FILTER, bool ANY>
static cudaError_t launch_stream(const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occupancy_only,
                                 int* occ) {
    auto kern = k_image_chain<IW, PPT, MB, false, true, FILTER, OUT_ROWS, ANY>;
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

// The same tile variants as the other window modes (kVariants in k_image.cu).
template <bool ANY>
static cudaError_t dispatch_stream(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only,
                                   int* occ) {
    if (!a.pp.filter && !occ_only) {
        switch (v) {
        case 0: return launch_stream<8, 1, 2, 0, ANY>(a, grid, smem, s, occ_only, occ);
        case 1: return launch_stream<4, 2, 2, 0, ANY>(a, grid, smem, s, occ_only, occ);
        case 2: return launch_stream<8, 2, 2, 0, ANY>(a, grid, smem, s, occ_only, occ);
        case 3: return launch_stream<4, 1, 2, 0, ANY>(a, grid, smem, s, occ_only, occ);
        case 4: return launch_stream<8, 1, 3, 0, ANY>(a, grid, smem, s, occ_only, occ);
        default: return cudaErrorInvalidValue;
        }
    }
    switch (v) {
    case 0: return launch_stream<8, 1, 2, 1, ANY>(a, grid, smem, s, occ_only, occ);
    case 1: return launch_stream<4, 2, 2, 1, ANY>(a, grid, smem, s, occ_only, occ);
    case 2: return launch_stream<8, 2, 2, 1, ANY>(a, grid, smem, s, occ_only, occ);
    case 3: return launch_stream<4, 1, 2, 1, ANY>(a, grid, smem, s, occ_only, occ);
    case 4: return launch_stream<8, 1, 3, 1, ANY>(a, grid, smem, s, occ_only, occ);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t dispatch_image_chain_stream(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s,
                                        bool occ_only, int* occ) {
    return a.any_window ? dispatch_stream<true>(v, a, grid, smem, s, occ_only, occ)
                        : dispatch_stream<false>(v, a, grid, smem, s, occ_only, occ);
}

}  // namespace rta
