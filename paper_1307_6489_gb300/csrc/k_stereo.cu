// Stereo Hillas intersection (direction and core reconstruction, Sec. 4.1).
//
// Eight lanes per event for events of up to eight images (four such events
// share a warp), a warp for up to 24, the CTA for larger ones. The event's
// images (at most 64) are staged in shared memory; its lanes walk the upper
// triangle of image pairs (i < j) and accumulate the weighted intersections; a
// shuffle tree over those lanes sums the five partial sums. The pair arithmetic
// and its precision are described with the shared pieces in rta_stereo_dev.cuh.
#include <algorithm>

#include "rta_stereo_dev.cuh"

namespace rta {

constexpr int ST_WARPS = 8;
constexpr int ST_NT = ST_WARPS * 32;
constexpr int ST_GL = 8;           // lanes per event for small events
constexpr int ST_EPW = 32 / ST_GL; // small events per warp
constexpr int ST_CTAS = 3;         // resident CTAs per SM (registers)
constexpr int ST_MAX_E = 32;       // events a CTA takes per round
static_assert(ST_GL == STEREO_SMALL_M, "small events take one lane per image slot of their group");

// One image of the bundle staged for the pair loop.
__device__ __forceinline__ int stage_image(const StereoArgs& a, int64_t img, StereoImg* dst) {
    return stereo_stage(a.h[img], a.img_tel[img], a.arr.n_tel, a.arr.tel_xy, a.status, dst);
}

// The CTA takes a.per_cta consecutive events per round and sorts them by image count into three
// lists. The warps take tasks in turn: an event of up to STEREO_WARP_M images each, then up to
// four events of up to STEREO_SMALL_M images side by side, ST_GL lanes each; the larger events
// are then done one after another by the whole CTA. Which of the three an event takes depends on
// its own image count only, so its row does not depend on the events around it (a sub-list of
// events gives the same rows).
// Bound: the longest chain of a CTA (load, pairs, lane combination, about 4 us an event of any
// kind), not arithmetic or memory. So events are spread over one wave of CTAs as far as they go
// and the warps of a CTA share its middle events: 10,000 events 20.9 us (24.4 with 32 events a
// CTA, four to a warp, whose middle events it did one after another), 8 events 6.6 us (9.4).
__global__ void __launch_bounds__(ST_NT, ST_CTAS) k_stereo(const StereoArgs a) {
    __shared__ StereoImg sh[ST_WARPS][RTA_STEREO_MAX_M];
    __shared__ int list[3][ST_MAX_E];                      // event numbers within the round: small, middle, large
    __shared__ int ev_i0[ST_MAX_E], ev_m[ST_MAX_E];
    __shared__ int n_list[3];
    __shared__ DW red[ST_WARPS * 5];
    __shared__ int redi[ST_WARPS * 2];
    static_assert(ST_EPW * STEREO_SMALL_M <= RTA_STEREO_MAX_M && ST_EPW * ST_GL == 32, "small events share the warp");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane / ST_GL, sub = lane % ST_GL;
    StereoImg* im = sh[warp];
    // Launched as a programmatic dependent of the image kernel. When the caller declared the
    // event offsets and counts settled (written before the image kernel started), they are
    // read before the dependency wait: the counts and the first round's offsets.
    if (!a.settled) grid_dependency_wait();
    grid_dependents_launch();
    // a graph captured at capacity reads the bundle's counts at run time
    const int64_t n_evt = a.n_evt_dev ? min(*a.n_evt_dev, a.n_evt) : a.n_evt;
    const int64_t n_img = a.n_img_dev ? min(*a.n_img_dev, a.n_img) : a.n_img;
    bool waited = !a.settled;
    for (int64_t r0 = int64_t(blockIdx.x) * a.per_cta; r0 < n_evt; r0 += int64_t(gridDim.x) * a.per_cta) {
        const int ne = int(min((long long)a.per_cta, (long long)(n_evt - r0)));
        if (warp == 0) {
            int kind = -1;
            if (lane < ne) {
                const int b0 = a.evt_off[r0 + lane], b1 = a.evt_off[r0 + lane + 1];
                if (b0 < 0 || b1 < b0 || b1 > n_img) {         // malformed CSR: flag, never index
                    kind = 3;
                } else {
                    const int m = min(b1 - b0, RTA_STEREO_MAX_M);
                    ev_i0[lane] = b0;
                    ev_m[lane] = m;
                    kind = m <= STEREO_SMALL_M ? 0 : m <= STEREO_WARP_M ? 1 : 2;
                }
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const unsigned who = __ballot_sync(0xffffffffu, kind == k);
                if (kind == k) list[k][__popc(who & ((1u << lane) - 1u))] = lane;
                if (lane == 0) n_list[k] = __popc(who);
            }
            if (!waited) grid_dependency_wait();
            if (kind == 3) {
                atomicOr(a.status, RTA_DEV_BAD_IMAGE);
                rta_stereo_t r = {};
                r.flags = RTA_SF_INVALID;
                a.out[r0 + lane] = r;
            }
        } else if (!waited) {
            grid_dependency_wait();
        }
        waited = true;
        __syncthreads();
        const int n_small = n_list[0], n_mid = n_list[1], n_big = n_list[2];
        for (int t = warp; t < n_mid + (n_small + ST_EPW - 1) / ST_EPW; t += ST_WARPS) {
            if (t < n_mid) {
                const int e = list[1][t], i0 = ev_i0[e], m = ev_m[e];
                int nvalid = 0;
                for (int k = lane; k < m; k += 32) nvalid += stage_image(a, int64_t(i0) + k, im + k);
                __syncwarp();
                CSum acc[5];
                const int npair = pair_sums<32>(im, m, lane, acc);
                const rta_stereo_t r = group_result<32>(acc, npair, nvalid);
                if (lane == 0) a.out[r0 + e] = r;
            } else {
                const int q = (t - n_mid) * ST_EPW + g;        // this group's small event
                const bool on = q < n_small;
                const int e = on ? list[0][q] : 0, i0 = ev_i0[e], m = on ? ev_m[e] : 0;
                StereoImg* gi = im + STEREO_SMALL_M * g;
                int nvalid = 0;
                for (int k = sub; k < m; k += ST_GL) nvalid += stage_image(a, int64_t(i0) + k, gi + k);
                __syncwarp();
                CSum acc[5];
                const int npair = pair_sums<ST_GL>(gi, m, sub, acc);
                const rta_stereo_t r = group_result<ST_GL>(acc, npair, nvalid);
                if (on && sub == 0) a.out[r0 + e] = r;
            }
            __syncwarp();
        }
        // the large events, one at a time, the whole CTA (warp 0's image slots)
        if (n_big > 0) __syncthreads();
        for (int b = 0; b < n_big; ++b) {
            const int e = list[2][b], m = ev_m[e];
            int nvalid = 0;
            if (threadIdx.x < m) nvalid = stage_image(a, int64_t(ev_i0[e]) + threadIdx.x, sh[0] + threadIdx.x);
            stereo_bar<ST_NT>();
            CSum acc[5];
            const int npair = pair_sums<ST_NT>(sh[0], m, threadIdx.x, acc);
            const rta_stereo_t r = cta_result<ST_NT>(acc, npair, nvalid, red, redi);
            if (threadIdx.x == 0) a.out[r0 + e] = r;
        }
        __syncthreads();                                   // the lists are read
    }
    if (!waited) grid_dependency_wait();
}

// Failure-detection self-test: one thread waits on an mbarrier that nothing
// will ever complete, through the same bounded wait the image kernel uses. The
// wait gives up after timeout_ns, the status word gets RTA_DEV_TIMEOUT and the
// kernel returns normally, leaving the context usable.
__global__ void k_wait_selftest(unsigned int* status, uint64_t timeout_ns, unsigned long long* waited_ns) {
    __shared__ uint64_t bar;
    __shared__ int abort;
    if (threadIdx.x != 0) return;
    abort = 0;
    mbar_init(&bar, 1);
    fence_mbar_init();
    const uint64_t t0 = global_ns();
    const bool ok = mbar_wait_ns(&bar, 0, &abort, timeout_ns);
    if (!ok) atomicOr(status, RTA_DEV_TIMEOUT);
    if (waited_ns) *waited_ns = global_ns() - t0;
    // leave no arrival pending: complete the phase ourselves before exiting
    mbar_arrive(&bar);
}

cudaError_t launch_wait_selftest(unsigned int* status, uint64_t timeout_ns, unsigned long long* waited_ns,
                                 cudaStream_t s) {
    k_wait_selftest<<<1, 32, 0, s>>>(status, timeout_ns, waited_ns);
    return cudaGetLastError();
}

cudaError_t launch_stereo(StereoArgs a, int n_sm, cudaStream_t s) {
    // one wave of CTAs, each with as few events as that allows
    const int64_t wave = int64_t(n_sm) * ST_CTAS;
    a.per_cta = int(std::max<int64_t>(1, std::min<int64_t>(ST_MAX_E, (a.n_evt + wave - 1) / wave)));
    const int64_t grid = std::min<int64_t>((a.n_evt + a.per_cta - 1) / a.per_cta, int64_t(n_sm) * 16);
    return launch_dependent(k_stereo, unsigned(std::max<int64_t>(grid, 1)), ST_NT, 0, s, a);
}

}  // namespace rta
