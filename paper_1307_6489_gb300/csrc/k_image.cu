// The unfused image-stage kernels (k_clean, k_hillas) and the host-side
// launchers of the fused image kernel; the kernels themselves live in
// k_image_chain.cuh, whose neighbour-peak and byte-stream instantiations are
// compiled in k_image_nb.cu and k_image_stream.cu.
#include "k_image_launch.cuh"

namespace rta {

// ------------------------------------------------------------------ unfused stage kernels

// One block per image, a warp per 32-pixel word and a lane per pixel. What an image's pixels need
// from memory -- values straight into ballots, or the charges, times and positions of the pixels
// that count -- is loaded side by side, one latency for all of them (a thread per bitmap word met
// one per set bit). Both kernels are bound by such chains (telescope, camera, pixels, barriers), so
// their time is that of an image times the rounds that the resident blocks make.

// k_clean: a warp takes the same words of an image in every pass and holds its lanes' bits of them, so only what neighbours ask for, the hi and the core bits, is shared: two barriers an
// image, and the next image's hi bits may be written while this one's core bits are still read.
// The neighbours' lists are loaded for the words that have such pixels alone, one after another:
// held for all of a warp's words they took the registers of half the resident blocks. 500, 4,224 and
// 28,160 images of the three presets 9.0, 27.1 and 142 us; 8.4, 35.6 and 220 with the lists
// held, 10.5, 27.5 and 187 with a thread per bitmap word.
constexpr int CLEAN_WARPS = 8;
constexpr int CLEAN_WORDS = RTA_MAX_PIX / 32 / CLEAN_WARPS;      // words a warp has at most
static_assert(CLEAN_WORDS <= 32, "a bit per word");

__global__ void __launch_bounds__(CLEAN_WARPS * 32, 8) k_clean(const CleanArgs a) {
    extern __shared__ __align__(16) uint32_t words[];
    uint32_t *hi = words, *core = words + words_of(a.arr.max_P);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t img = blockIdx.x; img < a.n_img; img += gridDim.x) {
        const int tel = a.img_tel[img];
        const int64_t off = a.pix_off[img];
        if (tel < 0 || tel >= a.arr.n_tel) {
            if (threadIdx.x == 0) atomicOr(a.status, RTA_DEV_BAD_IMAGE);
            continue;
        }
        const DevCam C = a.arr.cams[a.arr.tel_cam[tel]];
        if (off < 0 || off + C.P > a.n_q || C.P > a.arr.max_P) {      // max_P: a captured launch's shared memory
            if (threadIdx.x == 0) atomicOr(a.status, RTA_DEV_BAD_IMAGE);
            continue;
        }
        const int nw = words_of(C.P);
        const float* q = a.q + off + 32 * warp + lane;
        // bit k of this lane: its pixel of the warp's word k (warp + 8 k); of the warp: any pixel of it
        unsigned is_hi = 0, is_lo = 0, any_hi = 0, any_lo = 0;
#pragma unroll
        for (int k0 = 0; k0 < CLEAN_WORDS; k0 += 8) {
            if (warp + CLEAN_WARPS * k0 >= nw) break;
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int at = 32 * CLEAN_WARPS * (k0 + k);
                v[k] = at + 32 * warp + lane < C.P ? __ldg(q + at) : __int_as_float(0x7fc00000);   // NaN: neither
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int w = warp + CLEAN_WARPS * (k0 + k);
                if (w >= nw) break;
                const bool h = v[k] >= a.pp.t_hi, l = v[k] >= a.pp.t_lo;
                const uint32_t bh = __ballot_sync(0xffffffffu, h);
                is_hi |= unsigned(h) << (k0 + k);
                is_lo |= unsigned(l) << (k0 + k);
                any_hi |= unsigned(bh != 0) << (k0 + k);
                any_lo |= unsigned(__any_sync(0xffffffffu, l)) << (k0 + k);
                if (lane == 0) hi[w] = bh;
            }
        }
        __syncthreads();
        // core = hi, with a hi neighbour if asked
        const int mine = warp + CLEAN_WARPS * lane;
        if (lane < CLEAN_WORDS && mine < nw && !((any_hi >> lane) & 1u)) core[mine] = 0u;
        unsigned is_mask = 0;
        for (unsigned m = any_hi; m; m &= m - 1) {
            const int k = __ffs(m) - 1, w = warp + CLEAN_WARPS * k;
            bool on = (is_hi >> k) & 1u;
            if (on && a.pp.core_nb) on = any_neighbour(__ldg(C.nb + (32 * w + lane)), C.K, C.P, hi);
            is_mask |= unsigned(on) << k;
            const uint32_t b = __ballot_sync(0xffffffffu, on);
            if (lane == 0) core[w] = b;
        }
        __syncthreads();
        // mask = core, and lo with a core neighbour
        for (unsigned m = any_lo; m; m &= m - 1) {
            const int k = __ffs(m) - 1, w = warp + CLEAN_WARPS * k;
            if ((is_lo & ~is_mask) >> k & 1u)
                is_mask |= unsigned(any_neighbour(__ldg(C.nb + (32 * w + lane)), C.K, C.P, core)) << k;
        }
        uint8_t* out = a.mask + off + 32 * warp + lane;
        for (int k = 0; warp + CLEAN_WARPS * k < nw; ++k)
            if (32 * (warp + CLEAN_WARPS * k) + lane < C.P) out[32 * CLEAN_WARPS * k] = (is_mask >> k) & 1u;
    }
}

// k_hillas: four warps, so that an SM holds eight images. 500, 4,224 and 28,160 images of the three
// presets 10.5, 32.9 and 200 us, 7,800 of 256 pixels 48 us; 11.3, 40.3, 224 and 90 with eight warps,
// 12.9, 48.5, 400 and 84 with a thread per bitmap word.
constexpr int UNF_WARPS = 4;
constexpr int UNF_WORDS = 8;      // words a warp takes at a time
constexpr int UNF_STEP = UNF_WARPS * UNF_WORDS;

__global__ void __launch_bounds__(UNF_WARPS * 32) k_hillas(const HillasArgs a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ float red[3 * NCW * 8];
    float* sq = reinterpret_cast<float*>(smem_raw);
    float* st = sq + a.arr.max_P;
    float2* sxy = reinterpret_cast<float2*>(st + a.arr.max_P);
    uint32_t* mask = reinterpret_cast<uint32_t*>(sxy + a.arr.max_P);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t img = blockIdx.x; img < a.n_img; img += gridDim.x) {
        const int tel = a.img_tel[img];
        const int64_t off = a.pix_off[img];
        bool bad = tel < 0 || tel >= a.arr.n_tel;
        DevCam C = {};
        if (!bad) {
            C = a.arr.cams[a.arr.tel_cam[tel]];
            bad = off < 0 || off + C.P > a.n_q || C.P > a.arr.max_P;
        }
        if (bad) {
            if (threadIdx.x == 0) {
                atomicOr(a.status, RTA_DEV_BAD_IMAGE);
                write_bad_row(a.out + img);
            }
            continue;
        }
        // charges, times and positions of the cleaned pixels only
        const int nw = words_of(C.P);
        for (int wb = 0; wb < nw; wb += UNF_STEP) {
            bool on[UNF_WORDS];
            float q[UNF_WORDS], t[UNF_WORDS];
            float2 xy[UNF_WORDS];
#pragma unroll
            for (int k = 0; k < UNF_WORDS; ++k) {
                const int p = 32 * (wb + warp + UNF_WARPS * k) + lane;
                on[k] = p < C.P && __ldg(a.mask + off + p) != 0;
            }
#pragma unroll
            for (int k = 0; k < UNF_WORDS; ++k) {
                const int p = 32 * (wb + warp + UNF_WARPS * k) + lane;
                if (on[k]) {
                    q[k] = __ldg(a.q + off + p);
                    if (a.t) t[k] = __ldg(a.t + off + p);
                    xy[k] = __ldg(C.xy + p);
                }
            }
#pragma unroll
            for (int k = 0; k < UNF_WORDS; ++k) {
                const int w = wb + warp + UNF_WARPS * k, p = 32 * w + lane;
                if (w >= nw) break;
                const uint32_t b = __ballot_sync(0xffffffffu, on[k]);
                if (lane == 0) mask[w] = b;
                if (on[k]) {
                    sq[p] = q[k];
                    if (a.t) st[p] = t[k];
                    sxy[p] = xy[k];
                }
            }
        }
        __syncthreads();
        C.xy = sxy;
        hillas_bits<false>(sq, a.t ? st : nullptr, C, mask, red, threadIdx.x, blockDim.x, BlockBar(), a.out + img);
        __syncthreads();
    }
}

// ------------------------------------------------------------------ host-side launchers
// Tile-shape variants of the fused kernel: (integrator warps, pixels per thread).
struct ChainVariant {
    int iw, ppt, min_blocks;   // integrator warps, pixels per thread, CTAs per SM the registers are sized for
};
static const ChainVariant kVariants[RTA_CHAIN_VARIANTS] = {{8, 1, 2}, {4, 2, 2}, {8, 2, 2}, {4, 1, 2}, {8, 1, 3}};

int chain_variant_warps(int v) { return kVariants[v].iw; }
int chain_variant_ppt(int v) { return kVariants[v].ppt; }
int chain_variant_min_blocks(int v) { return kVariants[v].min_blocks; }

int chain_stage_wave_bytes(int v, int max_S) {
    const int chunk = kVariants[v].iw * 32 * kVariants[v].ppt;
    int swb = ((chunk * 2 * max_S + 16) + 127) & ~127;
    const int cap = 48 * 1024;
    return swb < cap ? swb : cap;
}

size_t chain_smem_bytes(int v, int nstage, int stage_wave_bytes, int max_P, int nb_keys, int stream_recs, int tails) {
    const size_t head = ((tails > 1 ? sizeof(ChainSmem<SMALL_TAILS>) : sizeof(ChainSmem<2>)) + 127) & ~size_t(127);
    const size_t words = (max_P + 31) / 32;
    const size_t chunk = size_t(kVariants[v].iw) * 32 * kVariants[v].ppt;
    const size_t keys = nb_keys ? 10 * size_t(max_P) + 16 : 0;   // 64-bit keys, 16-bit candidate ids
    const size_t recs = stream_recs ? 2 * sizeof(StreamImg) + 16 : 0;   // the producer's two stream records
    return head + size_t(nstage) * (stage_wave_bytes + 2 * chunk * 4) + chain_slots(tails) * slot_bytes(max_P) +
           8 * tails * words + 16 +
           keys + recs;
}

int chain_chunk_pixels(int v, int stage_wave_bytes, int S) {
    return chunk_pixels(kVariants[v].iw * 32 * kVariants[v].ppt, stage_wave_bytes, S);
}

// The integrate-only call, and rows with masks; the digital filter as the call says.
template <int SEARCH>
static cudaError_t dispatch_pixels(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s) {
    return a.integrate_only ? dispatch_chain<false, false, 2, OUT_CHARGES, SEARCH>(v, a, grid, smem, s)
                            : dispatch_chain<false, false, 2, OUT_MASKS, SEARCH>(v, a, grid, smem, s);
}

cudaError_t launch_image_chain(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s) {
    // the image chain's rows on a contiguous bundle; then byte streams, and the per-pixel outputs
    // (integrate-only charges and times, cleaning masks)
    if (!a.smeta && !a.integrate_only && !a.mask_out)
        return a.search == SEARCH_PACKED   ? dispatch_image_chain_any(v, a, grid, smem, s)
               : a.search == SEARCH_SERIAL ? dispatch_image_chain_serial(v, a, grid, smem, s)
                                           : dispatch_image_chain_lean(v, a, grid, smem, s);
    if (a.pp.nbpeak) return dispatch_image_chain_nb(v, a, grid, smem, s, false, nullptr);
    if (a.smeta) return dispatch_image_chain_stream(v, a, grid, smem, s, false, nullptr);
    return a.search == SEARCH_PACKED ? dispatch_pixels<SEARCH_PACKED>(v, a, grid, smem, s) : dispatch_pixels<SEARCH_SERIAL>(v, a, grid, smem, s);
}

int chain_occupancy(int v, size_t smem, int kind) {
    int n = 0;
    ChainArgs dummy = {};
    const cudaError_t e = kind == CHAIN_NB       ? dispatch_image_chain_nb(v, dummy, 0, smem, nullptr, true, &n)
                          : kind == CHAIN_STREAM ? dispatch_image_chain_stream(v, dummy, 0, smem, nullptr, true, &n)
                                                 : dispatch_chain<false, false, 2, OUT_MASKS, SEARCH_SERIAL>(v, dummy, 0, smem, nullptr, true, &n);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t launch_clean(const CleanArgs& a, int grid, cudaStream_t s) {
    const size_t smem = size_t(8) * ((a.arr.max_P + 31) / 32);
    k_clean<<<grid, CLEAN_WARPS * 32, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_hillas(const HillasArgs& a, int grid, cudaStream_t s) {
    const size_t smem = size_t(a.arr.max_P) * 16 + size_t(4) * ((a.arr.max_P + 31) / 32) + 16;
    static std::atomic<uint64_t> opted_in{0};
    const cudaError_t e = smem_opt_in(k_hillas, opted_in);
    if (e != cudaSuccess) return e;
    k_hillas<<<grid, UNF_WARPS * 32, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace rta
