// The unfused image-stage kernels (k_clean, k_hillas) and the host-side
// launchers of the fused image kernel; the kernels themselves live in
// k_image_chain.cuh, whose neighbour-peak and byte-stream instantiations are
// compiled in k_image_nb.cu and k_image_stream.cu.
#include "k_image_launch.cuh"

namespace rta {

// ------------------------------------------------------------------ unfused stage kernels

// One block per image, a warp per 32-pixel word and a lane per pixel. What an image's pixels need
// from memory -- values straight into ballots, then the neighbours, or the charges, times and
// positions, of the pixels that count -- is loaded side by side, one latency for all of them (a
// thread per bitmap word met one per set bit). 501 events, 2,320 images: k_hillas 38 -> 26 us,
// k_clean 20.5 -> 22 alone but the two, back to back with the integration, 116 -> 108.
constexpr int UNF_WARPS = 8;
constexpr int UNF_WORDS = 8;      // words a warp takes at a time
constexpr int UNF_STEP = UNF_WARPS * UNF_WORDS;

// w0[w] = {v >= t0}, w1[w] = {v >= t1} of the image's values q (global memory).
__device__ __forceinline__ void threshold_words(const float* q, int P, float t0, float t1, uint32_t* w0, uint32_t* w1) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = words_of(P);
    for (int wb = 0; wb < nw; wb += UNF_STEP) {
        float v[UNF_WORDS];
#pragma unroll
        for (int k = 0; k < UNF_WORDS; ++k) {
            const int p = 32 * (wb + warp + UNF_WARPS * k) + lane;
            v[k] = p < P ? __ldg(q + p) : __int_as_float(0x7fc00000);      // NaN: neither
        }
#pragma unroll
        for (int k = 0; k < UNF_WORDS; ++k) {
            const int w = wb + warp + UNF_WARPS * k;
            if (w >= nw) break;
            const uint32_t b0 = __ballot_sync(0xffffffffu, v[k] >= t0);
            const uint32_t b1 = __ballot_sync(0xffffffffu, v[k] >= t1);
            if (lane == 0) {
                w0[w] = b0;
                w1[w] = b1;
            }
        }
    }
}

__global__ void __launch_bounds__(UNF_WARPS * 32) k_clean(const CleanArgs a) {
    extern __shared__ __align__(16) uint32_t words[];
    const int maxw = words_of(a.arr.max_P);
    uint32_t *hi = words, *lo = hi + maxw, *core = lo + maxw, *mask = core + maxw;
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
        threshold_words(a.q + off, C.P, a.pp.t_hi, a.pp.t_lo, hi, lo);
        __syncthreads();
        // core = hi, with a hi neighbour if asked; mask = core, and lo with a core neighbour. The
        // neighbours of the pixels in lo (hi is part of it) are loaded once for both
        const int nw = words_of(C.P);
        int4 nbr[UNF_WORDS];
        auto fetch = [&](int w0) {
#pragma unroll
            for (int k = 0; k < UNF_WORDS; ++k) {
                const int w = w0 + warp + UNF_WARPS * k;
                if (w < nw && ((lo[w] >> lane) & 1u)) nbr[k] = __ldg(C.nb + (32 * w + lane));
            }
        };
        for (int w0 = 0; w0 < nw; w0 += UNF_STEP) {
            fetch(w0);
#pragma unroll
            for (int k = 0; k < UNF_WORDS; ++k) {
                const int w = w0 + warp + UNF_WARPS * k;
                if (w >= nw) break;
                bool on = (hi[w] >> lane) & 1u;
                if (on && a.pp.core_nb) on = any_neighbour(nbr[k], C.K, C.P, hi);
                const uint32_t b = __ballot_sync(0xffffffffu, on);
                if (lane == 0) core[w] = b;
            }
        }
        __syncthreads();
        for (int w0 = 0; w0 < nw; w0 += UNF_STEP) {
            if (nw > UNF_STEP) fetch(w0);                // else they are still there
#pragma unroll
            for (int k = 0; k < UNF_WORDS; ++k) {
                const int w = w0 + warp + UNF_WARPS * k;
                if (w >= nw) break;
                bool on = (core[w] >> lane) & 1u;
                if (!on && ((lo[w] >> lane) & 1u)) on = any_neighbour(nbr[k], C.K, C.P, core);
                const uint32_t b = __ballot_sync(0xffffffffu, on);
                if (lane == 0) mask[w] = b;
            }
        }
        __syncthreads();
        uint8_t* out = a.mask + off;
        const int quads = C.P >> 2;
        if ((reinterpret_cast<uintptr_t>(out) & 3u) == 0) {
            // four pixels a thread: bits 0..3 spread to the bytes
            for (int g = threadIdx.x; g < quads; g += blockDim.x) {
                const uint32_t b = (mask[g >> 3] >> (4 * (g & 7))) & 15u;
                reinterpret_cast<uint32_t*>(out)[g] = (b * 0x00204081u) & 0x01010101u;
            }
            for (int p = 4 * quads + threadIdx.x; p < C.P; p += blockDim.x) out[p] = bit_of(mask, p) ? 1 : 0;
        } else {
            for (int p = threadIdx.x; p < C.P; p += blockDim.x) out[p] = bit_of(mask, p) ? 1 : 0;
        }
        __syncthreads();
    }
}

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
    const size_t smem = size_t(16) * ((a.arr.max_P + 31) / 32) + 16;
    k_clean<<<grid, UNF_WARPS * 32, smem, s>>>(a);
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
