// Launches of the image chain's kernels (k_image_chain.cuh), compiled in several files so that the
// builds run in parallel.
#pragma once
#include "k_image_chain.cuh"

namespace rta {

// One instantiation: a launch, or with occ_only its CTAs per SM in *occ.
template <int IW, int PPT, int MB, bool NB, bool STREAM, int FILTER, int OUT, int SEARCH, int TAILS = 1, int WIN = 6>
cudaError_t launch_chain(const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only, int* occ) {
    auto kern = k_image_chain<IW, PPT, MB, NB, STREAM, FILTER, OUT, SEARCH, TAILS, WIN>;
    static std::atomic<uint64_t> opted_in{0};
    if (smem > SMEM_PER_CTA) return cudaErrorInvalidValue;
    const cudaError_t e = smem_opt_in(kern, opted_in);
    if (e != cudaSuccess) return e;
    if (occ_only) {
        *occ = 0;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, kern, chain_block(IW, TAILS), smem);
    }
    kern<<<grid, chain_block(IW, TAILS), smem, s>>>(a);
    return cudaGetLastError();
}

// The tile variants (kVariants in k_image.cu).
template <bool NB, bool STREAM, int FILTER, int OUT, int SEARCH, int WIN = 6>
cudaError_t dispatch_chain(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only = false,
                           int* occ = nullptr) {
    switch (v) {
    case 0: return launch_chain<8, 1, 2, NB, STREAM, FILTER, OUT, SEARCH, 1, WIN>(a, grid, smem, s, occ_only, occ);
    case 1: return launch_chain<4, 2, 2, NB, STREAM, FILTER, OUT, SEARCH, 1, WIN>(a, grid, smem, s, occ_only, occ);
    case 2: return launch_chain<8, 2, 2, NB, STREAM, FILTER, OUT, SEARCH, 1, WIN>(a, grid, smem, s, occ_only, occ);
    case 3: return launch_chain<4, 1, 2, NB, STREAM, FILTER, OUT, SEARCH, 1, WIN>(a, grid, smem, s, occ_only, occ);
    case 4:      // registers for three CTAs per SM
        return launch_chain<8, 1, 3, NB, STREAM, FILTER, OUT, SEARCH, 1, WIN>(a, grid, smem, s, occ_only, occ);
    default: return cudaErrorInvalidValue;
    }
}

// Contiguous bundles, rows only, the flat window (of WIN samples in the specialised searches).
template <int SEARCH, int WIN = 6>
cudaError_t dispatch_flat_rows(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s) {
    if (a.small) return launch_chain<8, 1, 2, false, false, 0, OUT_ROWS, SEARCH, SMALL_TAILS, WIN>(a, grid, smem, s, false, nullptr);
    return dispatch_chain<false, false, 0, OUT_ROWS, SEARCH, WIN>(v, a, grid, smem, s);
}

// Contiguous bundles, rows only, any window mode.
template <int SEARCH>
cudaError_t dispatch_rows(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s) {
    if (a.pp.nbpeak) return dispatch_chain<true, false, 0, OUT_ROWS, SEARCH>(v, a, grid, smem, s);
    if (a.pp.filter) return dispatch_chain<false, false, 1, OUT_ROWS, SEARCH>(v, a, grid, smem, s);
    return dispatch_flat_rows<SEARCH>(v, a, grid, smem, s);
}

}  // namespace rta
