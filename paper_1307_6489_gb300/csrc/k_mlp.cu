// Kernels of the learned deep-sets surrogate (energy, direction offset and
// gamma/hadron score; the paper's Sec. 4.1 asks RT-RECO for energy and
// gamma/hadron separation next to the direction).
//
//   k_features   per event: used images, baseline (two brightest axes), 12 features per image
//   k_pool / k_pool_bwd  sum and mean over an event's images, and back
//   k_loss       loss terms, dL/dy and dL/dG
//   k_update     bias and output-layer gradients, the sums of the split weight gradients, Adam,
//                and the weights' BF16 and tensor-core copies
// (the dense layers, forward and backward, are tensor-core GEMMs: k_gemm_tc.cu)
//
// Row-major matrices throughout. Activations are stored in BF16 (the operand
// type of the next GEMM); biases, the output layer's backward pass and every
// gradient reduction are FP32.
#include "rta_mlp_dev.cuh"
#include "rta_tc.cuh"

namespace rta {

// ------------------------------------------------------------------ features
// SUR_EVT_LANES lanes per event; the inference kernel forms baselines and features the same way.
__global__ void __launch_bounds__(256) k_features(const FeatArgs a) {
    grid_dependents_launch();
    const int gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    const int sub = lane % SUR_EVT_LANES;
    constexpr int GROUPS = 32 / SUR_EVT_LANES;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    const int64_t n_evt = a.n_evt_dev ? min(*a.n_evt_dev, a.n_evt) : a.n_evt;
    const int64_t n_img = a.n_img_dev ? min(*a.n_img_dev, a.n_img) : a.n_img;
    if (a.zero) {
        uint4* z = reinterpret_cast<uint4*>(a.zero);
        const int64_t n16 = a.n_img * (SUR_H * 2 / 16);
        for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n16; i += int64_t(gridDim.x) * blockDim.x)
            z[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    // the whole warp iterates together (the group reductions shuffle across it)
    for (int64_t e0 = int64_t(gwarp) * GROUPS; e0 < n_evt; e0 += nwarps * GROUPS) {
        const int64_t e = e0 + lane / SUR_EVT_LANES;
        int i0 = 0, n = 0;
        bool ok = false;
        if (e < n_evt) {
            i0 = a.evt_off[e];
            const int i1 = a.evt_off[e + 1];
            ok = !(i0 < 0 || i1 < i0 || i1 > n_img);
            n = ok ? i1 - i0 : 0;
        }
        float bx, by;
        int cnt;
        sur_event_baseline(a.h, i0, n, sub, a.used, bx, by, cnt);
        if (e < n_evt && sub == 0) {
            a.base[e] = make_float2(bx, by);
            a.n_used[e] = ok ? cnt : -1;      // -1: malformed event
        }
        for (int k = sub; k < n; k += SUR_EVT_LANES) {
            const rta_hillas_t h = a.h[i0 + k];
            __nv_bfloat162 x[SUR_XPAD / 2];
            sur_image_features(h, a.img_tel[i0 + k], a.tel_cam, a.tel_xy, a.cam_code, a.n_tel, bx, by, x);
            uint4* xr = reinterpret_cast<uint4*>(a.X + int64_t(i0 + k) * SUR_XPAD);
            xr[0] = make_uint4(bf2_bits(x[0]), bf2_bits(x[1]), bf2_bits(x[2]), bf2_bits(x[3]));
            xr[1] = make_uint4(bf2_bits(x[4]), bf2_bits(x[5]), bf2_bits(x[6]), bf2_bits(x[7]));
        }
    }
}

// ------------------------------------------------------------------ pooling
// A warp per event, four channels a lane: an event's rows are read eight at a time (their sums
// stay in image order), and the used images come from one ballot of their flags per 32.
// Bound: the latency of a chain of dependent loads (offsets, flags, rows); 2,048 events of 9,400
// images 9.7 -> 7.0 us (pool) and 23.4 -> 8.0 us (backward, half a warp per row) against a block
// of 128 threads per event that read its flags and rows one after another.
constexpr int POOL_NT = 256;
static_assert(SUR_H == 128, "four channels a lane");

__device__ __forceinline__ float4 bf4(uint2 w) {
    const __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162*>(&w.x), b = *reinterpret_cast<__nv_bfloat162*>(&w.y);
    return make_float4(__low2float(a), __high2float(a), __low2float(b), __high2float(b));
}
__device__ __forceinline__ uint2 pack4(float4 v) {
    return make_uint2(bf2_bits(__floats2bfloat162_rn(v.x, v.y)), bf2_bits(__floats2bfloat162_rn(v.z, v.w)));
}

// P[e] = [sum_used h2 / 40, sum_used h2 / max(1, n_used)] (BF16). The mean multiplies by the
// event's reciprocal count (RN(1 / n)), as the inference kernel does.
__global__ void __launch_bounds__(POOL_NT) k_pool(const PoolArgs a) {
    grid_dependents_launch();
    grid_dependency_wait();
    const int64_t n_evt = a.n_evt_dev ? min(*a.n_evt_dev, a.n_evt) : a.n_evt;
    const int lane = threadIdx.x & 31;
    const uint2* H2 = reinterpret_cast<const uint2*>(a.H2);
    for (int64_t e = (blockIdx.x * int64_t(POOL_NT) + threadIdx.x) >> 5; e < n_evt; e += int64_t(gridDim.x) * (POOL_NT / 32)) {
        const int i0 = a.evt_off[e], i1 = a.evt_off[e + 1];
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        const int n_used = a.n_used[e];
        for (int b = i0; n_used >= 0 && b < i1; b += 32) {
            unsigned used = __ballot_sync(0xffffffffu, b + lane < i1 && a.used[b + lane]);
            while (used) {
                uint2 w[8];
                int n = 0;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (used) {
                        w[k] = H2[int64_t(b + __ffs(used) - 1) * (SUR_H / 4) + lane];
                        used &= used - 1;
                        n = k + 1;
                    }
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (k < n) {
                        const float4 h = bf4(w[k]);
                        s.x += h.x; s.y += h.y; s.z += h.z; s.w += h.w;
                    }
            }
        }
        const float d = 1.f / SUR_POOL_DIV, r = 1.f / fmaxf(1.f, float(n_used));
        uint2* P = reinterpret_cast<uint2*>(a.P + e * 2 * SUR_H);
        P[lane] = pack4(make_float4(s.x * d, s.y * d, s.z * d, s.w * d));
        P[SUR_H / 4 + lane] = pack4(make_float4(s.x * r, s.y * r, s.z * r, s.w * r));
    }
}

// dZ2[i] = used_i * (dP[e][:H] / 40 + dP[e][H:] / max(1, n)) * (H2[i] > 0), BF16.
__global__ void __launch_bounds__(POOL_NT) k_pool_bwd(const PoolArgs a) {
    grid_dependents_launch();
    grid_dependency_wait();
    const int64_t n_evt = a.n_evt_dev ? min(*a.n_evt_dev, a.n_evt) : a.n_evt;
    const int lane = threadIdx.x & 31;
    const uint4* H2 = reinterpret_cast<const uint4*>(a.H2);
    uint4* dZ2 = reinterpret_cast<uint4*>(a.dZ2);
    for (int64_t e = (blockIdx.x * int64_t(POOL_NT) + threadIdx.x) >> 5; e < n_evt; e += int64_t(gridDim.x) * (POOL_NT / 32)) {
        const int n_used = a.n_used[e];
        if (n_used < 0) continue;
        const int i0 = a.evt_off[e], i1 = a.evt_off[e + 1];
        // half a warp per row, eight channels a lane
        const int sub = lane & 15, odd = lane >> 4;
        const uint4* dP = reinterpret_cast<const uint4*>(a.dP + e * 2 * SUR_H);
        const uint4 u = dP[sub], v = dP[SUR_H / 8 + sub];
        const float d = 1.f / SUR_POOL_DIV, r = 1.f / fmaxf(1.f, float(n_used));
        auto comb = [&](float4 x, float4 y) {
            return make_float4(x.x * d + y.x * r, x.y * d + y.y * r, x.z * d + y.z * r, x.w * d + y.w * r);
        };
        const float4 g0 = comb(bf4(make_uint2(u.x, u.y)), bf4(make_uint2(v.x, v.y)));
        const float4 g1 = comb(bf4(make_uint2(u.z, u.w)), bf4(make_uint2(v.z, v.w)));
        for (int b = i0; b < i1; b += 32) {
            const unsigned used = __ballot_sync(0xffffffffu, b + lane < i1 && a.used[b + lane]);
            const int n = min(32, i1 - b);
#pragma unroll 8
            for (int k = odd; k < n; k += 2) {
                const int64_t at = int64_t(b + k) * (SUR_H / 8) + sub;
                const uint4 hw = H2[at];
                const float4 h0 = bf4(make_uint2(hw.x, hw.y)), h1 = bf4(make_uint2(hw.z, hw.w));
                const bool on = (used >> k) & 1u;
                const uint2 lo = pack4(make_float4(on && h0.x > 0.f ? g0.x : 0.f, on && h0.y > 0.f ? g0.y : 0.f,
                                                   on && h0.z > 0.f ? g0.z : 0.f, on && h0.w > 0.f ? g0.w : 0.f));
                const uint2 hi = pack4(make_float4(on && h1.x > 0.f ? g1.x : 0.f, on && h1.y > 0.f ? g1.y : 0.f,
                                                   on && h1.z > 0.f ? g1.z : 0.f, on && h1.w > 0.f ? g1.w : 0.f));
                dZ2[at] = make_uint4(lo.x, lo.y, hi.x, hi.y);
            }
        }
    }
}

// ------------------------------------------------------------------ loss
// A warp per event: its loss term, dL/dy (mean over n_evt events) and dG = (dY V2^T) * (G > 0),
// eight channels a lane (BF16).
__global__ void __launch_bounds__(256) k_loss(const LossArgs a) {
    grid_dependents_launch();
    grid_dependency_wait();
    const int lane = threadIdx.x & 31;
    const float inv_n = 1.f / float(a.n_evt > 1 ? a.n_evt : 1);
    const float ids2 = 1.f / (SUR_DIR_SIGMA * SUR_DIR_SIGMA);
    float4 v2[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v2[k] = bf4(reinterpret_cast<const uint2*>(a.V2b)[lane * 8 + k]);
    for (int64_t e = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; e < a.n_evt;
         e += (int64_t(gridDim.x) * blockDim.x) >> 5) {
        const uint4 gw = reinterpret_cast<const uint4*>(a.G + e * SUR_G)[lane];
        const float4 y = reinterpret_cast<const float4*>(a.Y)[e];
        const float gam = a.is_gamma[e] ? 1.f : 0.f;
        const float2 b = a.base[e];
        const float2 src = a.src[e];
        const float r0 = y.x - a.logE[e];
        const float r1 = y.y - (src.x - b.x), r2 = y.z - (src.y - b.y);
        const float sig = 1.f / (1.f + expf(-y.w));
        const float dy[4] = {2.f * gam * r0 * inv_n, 2.f * gam * r1 * ids2 * inv_n, 2.f * gam * r2 * ids2 * inv_n,
                             (sig - gam) * inv_n};
        if (lane == 0) {
            const float bce = fmaxf(y.w, 0.f) + log1pf(expf(-fabsf(y.w))) - gam * y.w;
            a.lterm[e] = gam * (r0 * r0 + (r1 * r1 + r2 * r2) * ids2) + bce;
            reinterpret_cast<float4*>(a.dY)[e] = make_float4(dy[0], dy[1], dy[2], dy[3]);
        }
        const float4 g0 = bf4(make_uint2(gw.x, gw.y)), g1 = bf4(make_uint2(gw.z, gw.w));
        const float g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
        float d[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            float t = __fmul_rn(dy[0], v2[k].x);
            t = fmaf(dy[1], v2[k].y, t);
            t = fmaf(dy[2], v2[k].z, t);
            t = fmaf(dy[3], v2[k].w, t);
            d[k] = g[k] > 0.f ? t : 0.f;
        }
        const uint2 lo = pack4(make_float4(d[0], d[1], d[2], d[3])), hi = pack4(make_float4(d[4], d[5], d[6], d[7]));
        reinterpret_cast<uint4*>(a.dG + e * SUR_G)[lane] = make_uint4(lo.x, lo.y, hi.x, hi.y);
    }
}

// ------------------------------------------------------------------ gradients and Adam
// One launch ends the step; its blocks, the longest first:
//   UPD_V2     eight rows of V2 each, and c2: sums over events of G dY
//   1          the loss, and the Adam step of the other biases (their gradients are ready: the
//              launches before add up the columns beside their products)
//   UPD_W      a thread per weight of W1, W2, V1: the sum of its partial sums
// and every gradient is followed by its parameter's Adam step in the thread that formed it.
constexpr int UPD_NT = 256;
constexpr int UPD_V2 = SUR_G / 8 + 1;
constexpr int UPD_SPECIAL = UPD_V2 + 1;
constexpr int UPD_WEIGHTS = SUR_XPAD * SUR_H + SUR_H * SUR_H + SUR_G * SUR_G;
constexpr int UPD_W = UPD_WEIGHTS / UPD_NT;
static_assert(UPD_WEIGHTS % UPD_NT == 0 && UPD_NT == 2 * SUR_H && UPD_NT == SUR_G, "whole blocks");

// FP32 master weight; its BF16 copy and, at >= 0, its place in the tensor-core layout follow.
__device__ __forceinline__ void adam_step(const UpdateArgs& a, int64_t i, float g, int64_t at) {
    a.g[i] = g;
    if (!a.apply) return;
    const float m = a.b1 * a.m[i] + (1.f - a.b1) * g;
    const float v = fmaf((1.f - a.b2) * g, g, a.b2 * a.v[i]);
    a.m[i] = m;
    a.v[i] = v;
    const float mh = m / a.bc1, vh = v / a.bc2;
    const float p = a.p[i] - a.lr * mh / (sqrtf(vh) + a.eps);
    a.p[i] = p;
    const __nv_bfloat16 b = __float2bfloat16(p);
    a.pb[i] = b;
    if (at >= 0) a.pk[at] = b;
}

__device__ __forceinline__ float sum_parts(const float* p, int n, int64_t stride) {
    float s = 0.f;
#pragma unroll 8
    for (int z = 0; z < n; ++z) s += p[z * stride];
    return s;
}

__global__ void __launch_bounds__(UPD_NT) k_update(const UpdateArgs a) {
    grid_dependents_launch();
    grid_dependency_wait();
    __shared__ float part[32 * UPD_NT];
    const int tid = threadIdx.x, b = blockIdx.x;
    if (b < UPD_V2) {
        // threads take events t, t + 256, ...; then a tree over the threads, [8 rows x 4][256]
        const bool bias = b == SUR_G / 8;          // a row of ones: c2
        float s[8][4] = {};
        for (int64_t e = tid; e < a.n_evt; e += UPD_NT) {
            const float4 dy = reinterpret_cast<const float4*>(a.dY)[e];
            uint4 gw = make_uint4(0x3F80u, 0u, 0u, 0u);
            if (!bias) gw = *reinterpret_cast<const uint4*>(a.G + e * SUR_G + 8 * b);
            const float4 g0 = bf4(make_uint2(gw.x, gw.y)), g1 = bf4(make_uint2(gw.z, gw.w));
            const float g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                s[k][0] = fmaf(g[k], dy.x, s[k][0]);
                s[k][1] = fmaf(g[k], dy.y, s[k][1]);
                s[k][2] = fmaf(g[k], dy.z, s[k][2]);
                s[k][3] = fmaf(g[k], dy.w, s[k][3]);
            }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
#pragma unroll
            for (int o = 0; o < 4; ++o) part[(k * 4 + o) * UPD_NT + tid] = s[k][o];
        __syncthreads();
        for (int w = UPD_NT / 2; w > 0; w >>= 1) {
            for (int i = tid; i < 32 * w; i += UPD_NT) {
                float* q = part + (i / w) * UPD_NT + i % w;
                *q += q[w];
            }
            __syncthreads();
        }
        if (tid < (bias ? 4 : 32)) {
            const int64_t j = int64_t(b) * 32 + tid;                 // V2, then c2
            adam_step(a, OFF_V2 + j, part[tid * UPD_NT], bias ? -1 : PK_V2P + (j >> 2) * 16 + (j & 3));
        }
        return;
    }
    if (b == UPD_V2) {
        if (tid < SUR_H) adam_step(a, OFF_B1 + tid, a.g[OFF_B1 + tid], -1);
        else adam_step(a, OFF_B2 + tid - SUR_H, a.g[OFF_B2 + tid - SUR_H], -1);
        adam_step(a, OFF_C1 + tid, a.g[OFF_C1 + tid], -1);
        if (!a.d_loss) return;
        float s = 0.f;
        for (int64_t i = tid; i < a.n_evt; i += UPD_NT) s += a.lterm[i];
        part[tid] = s;
        __syncthreads();
        for (int w = UPD_NT / 2; w > 0; w >>= 1) {
            if (tid < w) part[tid] += part[tid + w];
            __syncthreads();
        }
        if (tid == 0) *a.d_loss = part[0] / float(a.n_evt > 1 ? a.n_evt : 1);
        return;
    }
    const int j = (b - UPD_V2 - 1) * UPD_NT + tid;
    if (j < SUR_XPAD * SUR_H) {
        adam_step(a, OFF_W1 + j, sum_parts(a.w1 + j, a.n_w1, SUR_XPAD * SUR_H),
                  PK_W1T + canon_off(j % SUR_H, j / SUR_H, SUR_XPAD));
    } else if (j < SUR_XPAD * SUR_H + SUR_H * SUR_H) {
        const int k = j - SUR_XPAD * SUR_H;
        adam_step(a, OFF_W2 + k, sum_parts(a.w2 + k, a.n_w2, SUR_H * SUR_H),
                  PK_W2T + canon_off(k % SUR_H, k / SUR_H, SUR_H));
    } else {
        const int k = j - SUR_XPAD * SUR_H - SUR_H * SUR_H;
        adam_step(a, OFF_V1 + k, sum_parts(a.v1 + k, a.n_v1, SUR_G * SUR_G),
                  PK_V1T + canon_off(k % SUR_G, k / SUR_G, SUR_G));
    }
}

// ------------------------------------------------------------------ launchers
cudaError_t launch_features(const FeatArgs& a, int grid, cudaStream_t s) {
    k_features<<<grid, 256, 0, s>>>(a);      // (follows a memset: an ordinary launch)
    return cudaGetLastError();
}
cudaError_t launch_pool(const PoolArgs& a, int grid, bool bwd, cudaStream_t s) {
    return launch_dependent(bwd ? k_pool_bwd : k_pool, grid, POOL_NT, 0, s, a);
}
cudaError_t launch_loss(const LossArgs& a, int grid, cudaStream_t s) {
    return launch_dependent(k_loss, grid, 256, 0, s, a);
}
cudaError_t launch_update(const UpdateArgs& a, cudaStream_t s) {
    return launch_dependent(k_update, UPD_SPECIAL + UPD_W, UPD_NT, 0, s, a);
}

}  // namespace rta
