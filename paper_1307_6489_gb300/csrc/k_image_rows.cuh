// Launches of the image chain's kernels for contiguous bundles, rows only, whose cameras all have a
// specialised window search (k_image_lean.cu, k_image_win.cu).
#pragma once
#include <algorithm>

#include "k_image_chain.cuh"

namespace rta {

// WIN: the width of the sliding window; FILTER 1: the digital filter.
template <int IW, int PPT, int MB, int WIN, bool NB = false, int FILTER = 0, int TAILS = 1>
cudaError_t launch_rows(const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occupancy_only, int* occ) {
    auto kern = k_image_chain<IW, PPT, MB, NB, false, FILTER, OUT_ROWS, false, TAILS, WIN>;
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
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, kern, chain_block(IW, TAILS), smem);
    }
    kern<<<grid, chain_block(IW, TAILS), smem, s>>>(a);
    return cudaGetLastError();
}

// The flat window of WIN samples through tile variant v (the order of kVariants in k_image.cu).
template <int WIN>
cudaError_t dispatch_rows(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only, int* occ) {
    // small cameras: variant 4's tile with a tail warp for each of eight slots, two CTAs an SM (an
    // image of 256 pixels is integrated in a fraction of the time its cleaning and moments take:
    // 2,000 of them 21.4 us, 35.5 with one tail warp for two slots); with rows of 64 samples and more
    // the search sets the pace again (303 of 208 x 100: 30.3 us so, 28.9 with three CTAs an SM)
    if (v == 4 && a.arr.max_P <= SMALL_PIX && a.max_S < 64 && !occ_only) {
        const size_t sm8 = chain_smem_bytes(4, a.nstage, a.stage_wave_bytes, a.arr.max_P, 0, 0, SMALL_TAILS);
        const int g8 = int(std::min<int64_t>(a.n_img, 2 * int64_t(a.n_sm)));
        if (sm8 <= size_t(227) * 1024)
            return launch_rows<8, 1, 2, WIN, false, 0, SMALL_TAILS>(a, g8, sm8, s, false, nullptr);
    }
    switch (v) {
    case 0: return launch_rows<8, 1, 2, WIN>(a, grid, smem, s, occ_only, occ);
    case 1: return launch_rows<4, 2, 2, WIN>(a, grid, smem, s, occ_only, occ);
    case 2: return launch_rows<8, 2, 2, WIN>(a, grid, smem, s, occ_only, occ);
    case 3: return launch_rows<4, 1, 2, WIN>(a, grid, smem, s, occ_only, occ);
    case 4: return launch_rows<8, 1, 3, WIN>(a, grid, smem, s, occ_only, occ);   // registers for three CTAs per SM
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace rta
