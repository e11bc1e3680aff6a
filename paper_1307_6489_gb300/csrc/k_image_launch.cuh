// Launches of the image chain's kernels (k_image_chain.cuh), compiled in several files so that the
// builds run in parallel.
#pragma once
#include <algorithm>

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
    // small cameras: variant 4's tile with a tail warp for each of eight slots, two CTAs an SM (an
    // image of 256 pixels is integrated in a fraction of the time its cleaning and moments take:
    // 2,000 of them 21.4 us, 35.5 with one tail warp for two slots); with rows of 64 samples and more
    // the search sets the pace again (303 of 208 x 100: 30.3 us so, 28.9 with three CTAs an SM)
    if (v == 4 && a.arr.max_P <= SMALL_PIX && a.max_S < 64) {
        const size_t sm8 = chain_smem_bytes(4, a.nstage, a.stage_wave_bytes, a.arr.max_P, 0, 0, SMALL_TAILS);
        const int g8 = int(std::min<int64_t>(a.n_img, 2 * int64_t(a.n_sm)));
        if (sm8 <= SMEM_PER_CTA)
            return launch_chain<8, 1, 2, false, false, 0, OUT_ROWS, SEARCH, SMALL_TAILS, WIN>(a, g8, sm8, s, false, nullptr);
    }
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
