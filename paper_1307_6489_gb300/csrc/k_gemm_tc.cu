// The dense contractions of the surrogate's training (forward layers, input
// gradients and weight gradients) on the fifth-generation tensor cores:
// D[M x N] = op(A) op(B), BF16 operands, FP32 accumulation in tensor memory,
// the layer's epilogue fused into the read-back.
//
// A CTA of eight warps takes work items (a tile of 128 rows and at most 64 columns
// of D, one K-range of a split reduction) in a grid-stride loop and streams each item's K-chunks of
// A and B through a ring of shared-memory buffers filled by 16-byte
// asynchronous copies. One thread issues the chunk's MMAs (M = 128, N = the tile's
// width, K-steps of 16) into the item's TMEM accumulator and commits them to the
// stage's mbarrier; a stage is refilled once the MMAs that read it are done.
// These layers are small (16 to 73 row tiles) and bound by latency, not by the tensor
// core: tiles of 64 columns put 32 to 146 items on the 152 SMs, and a layer's weight, bias and
// input gradients, which do not depend on one another, share a launch. A training step of 2,048
// events takes 106 us (463 us with full-width tiles, a launch per product and the column sums
// in kernels of 4 and 8 blocks); a chain of twelve launches of 4 to 14 us.
// After an item's last chunk every warp reads its 32 TMEM lanes (rows) and
// applies the epilogue.
//
// Operand staging. An operand stored with K contiguous ("K-major": A as
// [M x K], B as [N x K]) goes to the canonical K-major core-matrix layout of
// rta_tc.cuh. One stored with its rows along K ("MN-major": A as [K x M], B as
// [K x N], the activations and gradients of a weight gradient and the weights
// of a forward layer) goes to the canonical MN-major layout: core matrices of 8
// K-rows x 8 MN-values (16 contiguous bytes per K-row), core matrices adjacent
// in K 128 bytes apart (LBO), groups of 8 MN-values KC x 16 bytes apart (SBO),
// and the instruction descriptor marks the operand as MN-major. Either way a
// 16-byte piece of a stored row lands as one 16-byte piece in shared memory.
#include <algorithm>

#include "rta_mlp_dev.cuh"
#include "rta_tc.cuh"

namespace rta {
namespace {

constexpr int TC_BM = 128;   // rows of a tile = TMEM lanes
// Stages of the ring. The layers have one or two chunks of 128 and a weight gradient's 512-row
// range four, all of which are in flight at once. (Chunks of 64 made the loop's barrier, MMA
// issue and wait eight times a range.)
constexpr int TC_NS = 4;
constexpr int TC_KC = 128;   // K of a chunk (16 for the first layer)
constexpr int TC_SPLIT = 64; // a split's K-range is a multiple of this
constexpr int TC_NT = 256;   // eight warps, two per TMEM lane quarter (each reads half of the columns)
constexpr int TC_BN = 64;    // columns of a tile (16 for the output layer)

// element offset of (row r, k) in an MN-major chunk of KC K-rows
__device__ __forceinline__ int mn_off(int r, int k, int KC) {
    return (r >> 3) * (8 * KC) + (k >> 3) * 64 + (k & 7) * 8 + (r & 7);
}

// 16 bytes global -> shared, zero-filled when !valid (src is not read then)
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}
// Rows [r0, r0 + R) x K-range [k0, k0 + KC) of a stored operand into a stage.
// Rows at or beyond r_end and K at or beyond k_end read as zero. The offsets within the
// chunk are 32-bit and the divisors constants: a CTA's warps have a scheduler each or two,
// so instructions between the copies are time. Eight neighbouring threads take the eight
// 16-byte rows of one core matrix, 128 consecutive bytes of shared memory (threads along a
// stored row instead wrote sixteen pieces to the same banks).
template <bool MN, int KC, int R>
__device__ __forceinline__ void stage_chunk(uint32_t s, const __nv_bfloat16* X, int64_t ld, int64_t r0, int64_t r_end,
                                            int64_t k0, int64_t k_end, int tid) {
    const int rows = int(min(r_end - r0, int64_t(R))), ks = int(min(k_end - k0, int64_t(KC))), l = int(ld);
    if (!MN) {   // stored [rows x K]: 16-byte pieces (row, 8 K-values)
        constexpr int KP = KC / 8;
        X += r0 * ld + k0;
#pragma unroll
        for (int i = 0; i < (R * KP + TC_NT - 1) / TC_NT; ++i) {
            const int p = tid + i * TC_NT, r = (p & 7) + 8 * (p / (8 * KP)), j = (p >> 3) % KP;
            if (R * KP % TC_NT && p >= R * KP) break;
            const bool ok = r < rows && 8 * j < ks;
            cp_async16(s + 2 * uint32_t(canon_off(r, 8 * j, KC)), ok ? X + r * l + 8 * j : X, ok);
        }
    } else {     // stored [K x rows]: 16-byte pieces (K-row, 8 row values)
        constexpr int RP = R / 8;
        X += k0 * ld + r0;
#pragma unroll
        for (int i = 0; i < (KC * RP + TC_NT - 1) / TC_NT; ++i) {
            const int p = tid + i * TC_NT, kk = (p & 7) + 8 * (p / (8 * RP)), j = (p >> 3) % RP;
            if (KC * RP % TC_NT && p >= KC * RP) break;
            const bool ok = kk < ks && 8 * j < rows;
            cp_async16(s + 2 * uint32_t(mn_off(8 * j, kk, KC)), ok ? X + kk * l + 8 * j : X, ok);
        }
    }
}

// Position in a CTA's sequence of (item, chunk). Items: column tiles, then row tiles, then splits.
struct Tiling {
    int64_t m_tiles, n_tiles, n_items, kchunk;
    int bn;                  // columns of a tile
};

struct ChunkIt {
    int64_t item, c, nk, kbeg, m0;
    int z, n0, step;         // step: items to the CTA's next one
    bool valid;
};

__device__ __forceinline__ void it_begin(ChunkIt& t, int64_t item, const Tiling& w, int64_t K, int KC) {
    t.item = item;
    t.valid = item < w.n_items;
    t.c = 0;
    if (!t.valid) return;
    t.n0 = int(item % w.n_tiles) * w.bn;
    const int64_t r = item / w.n_tiles;
    t.m0 = (r % w.m_tiles) * TC_BM;
    t.z = int(r / w.m_tiles);
    t.kbeg = int64_t(t.z) * w.kchunk;
    const int64_t kend = min(K, t.kbeg + w.kchunk);
    t.nk = (kend - t.kbeg + KC - 1) / KC;   // >= 1: the host makes every split non-empty
}

__device__ __forceinline__ void it_next(ChunkIt& t, const Tiling& w, int64_t K, int KC) {
    if (++t.c == t.nk) it_begin(t, t.item + t.step, w, K, KC);
}

__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
    return pack_bf16(__float2bfloat16(lo), __float2bfloat16(hi));
}

// Epilogue of 16 columns [c0, c0 + 16) of row m.
__device__ __forceinline__ void epilogue16(const GemmArgs& g, int64_t m, int64_t M, int c0, int z,
                                           const uint32_t (&r)[16]) {
    float v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
    if (g.epi == EPI_F32_SPLIT) {    // partial sums of split z: [splits][M x N]
        float4* o = reinterpret_cast<float4*>(g.Cf + (int64_t(z) * M + m) * g.N + c0);
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        return;
    }
    if (g.epi == EPI_F32_BIAS) {    // the first n_store columns, plus bias
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (c0 + i < g.n_store) g.Cf[m * g.ldc + c0 + i] = v[i] + g.bias[c0 + i];
        return;
    }
    if (g.epi == EPI_BIAS_RELU_BF16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = fmaxf(v[i] + g.bias[c0 + i], 0.f);
    } else if (g.epi == EPI_MASK_BF16) {
        const uint4* mk = reinterpret_cast<const uint4*>(g.mask + m * g.ldmask + c0);
        const uint4 q0 = mk[0], q1 = mk[1];
        const uint32_t w[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const uint16_t h = uint16_t(w[i / 2] >> (16 * (i & 1)));
            if (!(__bfloat162float(__ushort_as_bfloat16(h)) > 0.f)) v[i] = 0.f;
        }
    }
    uint4* o = reinterpret_cast<uint4*>(g.Cb + m * g.ldc + c0);
    o[0] = make_uint4(bf16x2(v[0], v[1]), bf16x2(v[2], v[3]), bf16x2(v[4], v[5]), bf16x2(v[6], v[7]));
    o[1] = make_uint4(bf16x2(v[8], v[9]), bf16x2(v[10], v[11]), bf16x2(v[12], v[13]), bf16x2(v[14], v[15]));
}

// The items cta, cta + n_cta, ... of one product.
template <bool A_MN, bool B_MN, int KC, int N>
__device__ __forceinline__ void gemm_items(const GemmArgs& g, const Tiling& w, uint32_t tmem_cols, int cta, int n_cta,
                                           uint8_t* sm) {
    constexpr uint32_t a_bytes = TC_BM * KC * 2, b_bytes = N * KC * 2, stage_bytes = a_bytes + b_bytes;
    uint64_t* bar = reinterpret_cast<uint64_t*>(sm + TC_NS * stage_bytes);
    uint32_t* tmem_s = reinterpret_cast<uint32_t*>(bar + TC_NS);
    volatile int* abort_s = reinterpret_cast<volatile int*>(tmem_s + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t M = g.M, K = g.K;

    if (warp == 0) {
        tc_alloc(tmem_s, tmem_cols);
        tc_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < TC_NS; ++i) mbar_init(&bar[i], 1);
        fence_mbar_init();
        *abort_s = 0;
    }
    grid_dependency_wait();                // the operands are the preceding kernels'
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_s;
    const uint32_t s0 = smem_addr(sm);
    const uint32_t idesc = tc_idesc_bf16(TC_BM, N) | (uint32_t(A_MN) << 15) | (uint32_t(B_MN) << 16);
    // LBO: core matrices adjacent in K; SBO: groups of 8 rows (K-major) or 8 MN-values (MN-major)
    const uint32_t sbo = uint32_t(16 * KC);

    ChunkIt prod, cons;
    it_begin(prod, cta, w, K, KC);
    prod.step = n_cta;
    cons = prod;
    auto issue = [&](int stage) {
        const uint32_t sa = s0 + uint32_t(stage) * stage_bytes, sb = sa + a_bytes;
        const int64_t k0 = prod.kbeg + prod.c * KC;
        const int64_t k_end = min(K, prod.kbeg + w.kchunk);
        stage_chunk<A_MN, KC, TC_BM>(sa, g.A, g.lda, prod.m0, M, k0, k_end, tid);
        stage_chunk<B_MN, KC, N>(sb, g.B, g.ldb, prod.n0, g.N, k0, k_end, tid);
        it_next(prod, w, K, KC);
    };
#pragma unroll 1
    for (int s = 0; s < TC_NS - 1; ++s) {
        if (prod.valid) issue(s);
        cp_async_commit();
    }
    int64_t q = 0;
#pragma unroll 1
    while (cons.valid) {
        const int st = int(q % TC_NS);
        cp_async_wait<TC_NS - 2>();        // this thread's pieces of chunk q have landed
        fence_proxy_async_smem();
        if (__syncthreads_or(*abort_s)) break;   // ... and everyone's; one decision for the CTA
        if (tid == 0) {
            tc_fence_after();
            const uint32_t sa = s0 + uint32_t(st) * stage_bytes, sb = sa + a_bytes;
#pragma unroll 1
            for (int kk = 0; kk < KC; kk += 16) {
                const uint64_t da = tc_desc(sa + uint32_t(kk) * 16, 128, sbo);
                const uint64_t db = tc_desc(sb + uint32_t(kk) * 16, 128, sbo);
                tc_mma(tmem, da, db, idesc, cons.c > 0 || kk > 0);
            }
            tc_commit(&bar[st]);
        }
        // refill the stage chunk q - 1 used, once its MMAs are done
        if (q >= 1 && !mbar_wait(&bar[(q - 1) % TC_NS], uint32_t(((q - 1) / TC_NS) & 1), abort_s)) {
            atomicOr(g.status, RTA_DEV_TIMEOUT);
            *abort_s = 1;
        }
        if (prod.valid) issue(int((q + TC_NS - 1) % TC_NS));
        cp_async_commit();
        if (cons.c + 1 == cons.nk) {        // the item's last chunk: epilogue
            if (!mbar_wait(&bar[st], uint32_t((q / TC_NS) & 1), abort_s)) {
                atomicOr(g.status, RTA_DEV_TIMEOUT);
                *abort_s = 1;
            }
            tc_fence_after();
            const int64_t m = cons.m0 + 32 * (warp & 3) + lane;
            const uint32_t t_row = tmem + (uint32_t(32 * (warp & 3)) << 16);
            constexpr int HALF = N >= 32 ? N / 2 : N;
#pragma unroll 1
            for (int c0 = (warp >> 2) * HALF; c0 < N && c0 < ((warp >> 2) + 1) * HALF; c0 += 16) {
                uint32_t r[16];
                tc_ld16(t_row + uint32_t(c0), r);
                if (m < M) epilogue16(g, m, M, cons.n0 + c0, cons.z, r);
            }
            tc_fence_before();             // the next item's MMAs follow the next barrier
        }
        it_next(cons, w, K, KC);
        ++q;
    }
    // teardown: no copy and no MMA of this CTA may still be in flight
    cp_async_wait<0>();
    if (q >= 1 && !mbar_wait(&bar[(q - 1) % TC_NS], uint32_t(((q - 1) / TC_NS) & 1), abort_s))
        atomicOr(g.status, RTA_DEV_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tc_dealloc(tmem, tmem_cols);
}

// A forward layer.
template <int KC, int N>
__global__ void __launch_bounds__(TC_NT) k_gemm_tc(const GemmArgs g, const Tiling w) {
    extern __shared__ __align__(128) uint8_t sm[];
    grid_dependents_launch();
    gemm_items<false, true, KC, N>(g, w, N < 32 ? 32 : N, blockIdx.x, gridDim.x, sm);
}

// A layer's backward pass: the first n_w CTAs take the weight gradient's items, the next n_b eight
// columns each of the bias gradient, the others the input gradient's items.
template <int KC>
__global__ void __launch_bounds__(TC_NT) k_gemm_backward(const GemmArgs gw, const Tiling tw, int n_w, float* bias,
                                                         int n_b, const GemmArgs gx, const Tiling tx) {
    extern __shared__ __align__(128) uint8_t sm[];
    grid_dependents_launch();
    int cta = blockIdx.x;
    if (cta < n_w) {
        gemm_items<true, true, KC, TC_BN>(gw, tw, TC_BN, cta, n_w, sm);
        return;
    }
    cta -= n_w;
    if (cta < n_b) {
        static_assert(TC_NT == COL_NT, "column_sum's block");
        grid_dependency_wait();
        const float s = column_sum(gw.B, gw.K, int(gw.N), 8 * cta, sm);
        if (threadIdx.x < 8) bias[8 * cta + threadIdx.x] = s;
        return;
    }
    if (gx.M > 0) gemm_items<false, false, TC_KC, TC_BN>(gx, tx, TC_BN, cta - n_b, gridDim.x - n_w - n_b, sm);
}

Tiling tile(const GemmArgs& g, int N, int KC, int splits) {
    Tiling w;
    w.bn = N;
    w.m_tiles = (g.M + TC_BM - 1) / TC_BM;
    w.n_tiles = g.N / N;
    const int unit = KC < TC_SPLIT ? KC : TC_SPLIT;
    const int64_t units = (g.K + unit - 1) / unit;
    const int64_t per = (units + splits - 1) / splits;
    w.kchunk = per * unit;
    w.n_items = w.m_tiles * w.n_tiles * ((units + per - 1) / per);
    return w;
}

constexpr size_t tc_smem(int KC, int N) { return size_t(TC_NS) * (TC_BM + N) * KC * 2 + TC_NS * 8 + 16; }

template <int KC, int N>
cudaError_t launch_n(const GemmArgs& g, int n_sm, cudaStream_t s) {
    constexpr size_t smem = tc_smem(KC, N);
    const Tiling w = tile(g, N, KC, 1);
    auto kern = k_gemm_tc<KC, N>;
    static std::atomic<uint64_t> opted_in{0};
    const cudaError_t e = smem_opt_in(kern, opted_in);
    if (e != cudaSuccess) return e;
    // resident CTAs per SM: shared memory and the 512 TMEM columns
    constexpr size_t per_sm = std::max<size_t>(1, std::min<size_t>(size_t(200) * 1024 / smem, 512 / (N < 32 ? 32 : N)));
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(w.n_items, int64_t(n_sm) * int64_t(per_sm)));
    return launch_dependent(kern, unsigned(grid), TC_NT, smem, s, g, w);
}

template <int KC>
cudaError_t launch_backward(const GemmArgs& gw, int splits, float* bias, const GemmArgs* gx, int n_sm, cudaStream_t s) {
    const Tiling tw = tile(gw, TC_BN, KC, splits), tx = gx ? tile(*gx, TC_BN, TC_KC, 1) : Tiling{};
    const size_t smem = std::max(std::max(tc_smem(KC, TC_BN), gx ? tc_smem(TC_KC, TC_BN) : 0), size_t(COL_SMEM));
    static std::atomic<uint64_t> opted_in{0};
    const cudaError_t e = smem_opt_in(k_gemm_backward<KC>, opted_in);
    if (e != cudaSuccess) return e;
    // one CTA per SM: the weight gradient's long items take half of the SMs at most, the bias
    // gradient the SMs its columns need, the input gradient's short items the rest of one wave
    const int n_b = int(gw.N / 8);
    const int n_w = int(std::min<int64_t>(tw.n_items, std::max(1, gx ? n_sm / 2 : n_sm)));
    const int n_x = gx ? int(std::min<int64_t>(tx.n_items, std::max(1, n_sm - n_w - n_b))) : 0;
    return launch_dependent(k_gemm_backward<KC>, unsigned(n_w + n_b + n_x), TC_NT, smem, s, gw, tw, n_w, bias, n_b,
                            gx ? *gx : GemmArgs{}, tx);
}

bool gemm_ok(const GemmArgs& g, bool a_mn, bool b_mn, int splits) {
    if (!(g.N == 16 || (g.N > 0 && g.N <= 256 && g.N % TC_BN == 0)) || g.K < 1 || splits < 1 || g.lda > 65536 ||
        g.ldb > 65536)
        return false;
    // whole 16-byte pieces: MN-major row counts and K-major reductions in multiples of 8
    if ((a_mn ? g.M : g.K) % 8 || (b_mn ? g.N : g.K) % 8) return false;
    const bool f32 = g.epi == EPI_F32_SPLIT || g.epi == EPI_F32_BIAS;
    return !((uintptr_t(g.A) | uintptr_t(g.B) | uintptr_t(f32 ? (const void*)g.Cf : (const void*)g.Cb)) % 16 ||
             (g.lda | g.ldb) % 8 || (!f32 && g.ldc % 8) || (g.epi == EPI_F32_SPLIT && g.ldc != g.N) ||
             (g.epi == EPI_MASK_BF16 && (uintptr_t(g.mask) % 16 || g.ldmask % 8)));
}

}  // namespace

int gemm_tc_splits(int64_t K, int splits) {
    const int unit = K <= 16 ? 16 : TC_SPLIT;
    const int64_t units = (K + unit - 1) / unit;
    const int64_t per = (units + splits - 1) / splits;
    return int((units + per - 1) / per);
}

cudaError_t launch_gemm(const GemmArgs& g, int n_sm, cudaStream_t s) {
    if (g.M <= 0) return cudaSuccess;
    if (!gemm_ok(g, false, true, 1)) return cudaErrorInvalidValue;
    if (g.K <= 16) return g.N == 16 ? launch_n<16, 16>(g, n_sm, s) : launch_n<16, TC_BN>(g, n_sm, s);
    return g.N == 16 ? launch_n<TC_KC, 16>(g, n_sm, s) : launch_n<TC_KC, TC_BN>(g, n_sm, s);
}

cudaError_t launch_gemm_backward(const GemmArgs& gw, int splits, float* bias, const GemmArgs* gx, int n_sm,
                                 cudaStream_t s) {
    if (!gemm_ok(gw, true, true, splits) || gw.N % TC_BN || gw.M <= 0 || !bias ||
        (gx && (!gemm_ok(*gx, false, false, 1) || gx->N % TC_BN || gx->M <= 0)))
        return cudaErrorInvalidValue;
    return gw.K <= 16 ? launch_backward<16>(gw, splits, bias, gx, n_sm, s)
                      : launch_backward<TC_KC>(gw, splits, bias, gx, n_sm, s);
}

}  // namespace rta
