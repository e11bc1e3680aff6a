// Launch-argument blocks of the librta kernels and their host-side launchers.
#pragma once

#include <atomic>

#include "rta_device.cuh"

namespace rta {

constexpr int SMALL_TAILS = 8;
constexpr int SMALL_PIX = 512;      // pixels of the largest camera that counts as small

struct ChainArgs {
    DevArray arr;
    ProcParams pp;
    const uint16_t* wave;
    int64_t n_wave;          // samples in wave
    const int64_t* wave_off;
    const int32_t* img_tel;
    const int64_t* pix_off;  // integrate-only mode, and the rows of mask_out
    int64_t n_q;             // rows of q_out / t_out / mask_out
    int64_t n_img;           // images (capacity when n_img_dev is set)
    const int64_t* n_img_dev;  // optional device-resident image count (<= n_img), read at run time
    float* q_out;            // integrate-only mode
    float* t_out;
    rta_hillas_t* out;       // full mode
    uint8_t* mask_out;       // full mode, optional: cleaning masks
    unsigned int* counter;   // images taken beyond the first of every block; zeroed before the launch when
                             // there are more images than blocks
    unsigned int* status;
    int stage_wave_bytes;    // multiple of 128
    int nstage;
    int max_S;               // longest rows of the array's cameras
    int integrate_only;
    int small;               // the form for small cameras, of SMALL_TAILS slots and tail warps
    int search;              // SEARCH_*: what some camera without a specialised window search needs
    // a byte-stream bundle (rta_ingest's directory): wave is the stream, wave_off unused;
    // smeta: one prepared record per image (k_stream_meta)
    const rta_segment_t* seg;
    const int32_t* img_seg;
    int64_t n_seg;
    const struct StreamImg* smeta;
};

// The search for windows of W in a camera of S samples: SEARCH_OWN, a kernel that has one compiled
// for them; SEARCH_SERIAL, two 16-bit loads per window start; SEARCH_PACKED (PackedRow), which
// works on 16 samples at a time and can lay chunks out in padded runs. rows: flat windows of a
// contiguous bundle, rows only.
//
// The serial search is bound by its shared loads, and those by the banks that a warp's rows share:
// two rows a bank when S % 8 is 2, 4 or 6, four when it is 0 and S / 8 is odd, else more. With one
// or two it is the faster one as a rule, for every output and whatever the images: 0.2 GB of
// 1000-pixel images, W = 4, 1 % of the pixels above t_lo (in brackets nearly all), the packed
// search's time over the serial one's 1.60 (1.41) at 20 samples, 1.38 (1.27) at 31, 1.34 (1.18) at 50,
// 1.06 (1.13) at 60, 1.03 (1.20) at 100, 0.95 (1.11) at 127. With four, 0.94 (1.05) at 24 samples,
// 0.62 (0.83) at 56 and 0.55 (0.73) at 104; with more, 0.70 (0.85) at 16, 0.34 (0.51) at 48, 0.08
// (0.12) at 128. The neighbour peak forms 64-bit keys beside it and gains less from the packed
// search: 1.05 at 24 samples, 1.04 at 16, with W = 16 1.20 at 40 and 1.09 at 56. Windows of one sample are cheaper packed in long rows
// (0.93 at 65 samples, 0.90 at 100).
//
// A fixed window needs no search, but rows of a multiple of 32 samples put a warp's loads on two
// banks or one, and the packed kernels' padded runs spread them: 8 samples of 1000 pixels x 32
// 0.79 of the time, x 64 0.73, x 128 0.83. For up to three samples the runs' copies cost more than
// they save (1.12, 1.20 and 1.01 for one sample). On four banks plain rows are faster
// (5,000 of 2000 x 48, W = 3: 154 us, 175 in padded runs).
enum { SEARCH_OWN = 0, SEARCH_PACKED = 1, SEARCH_SERIAL = 2 };
inline int window_search(const ProcParams& pp, int S, bool rows) {
    if (!pp.sliding) return rows && !pp.filter && S % 32 == 0 && pp.W > 3 ? SEARCH_PACKED : SEARCH_OWN;
    const bool width = pp.W == 6 || (rows && !pp.nbpeak && !pp.filter && pp.W >= 4 && pp.W <= 8);
    if ((width && (S == 40 || S == 30 || S == 25)) || (pp.W == 5 && S == 16 && !pp.nbpeak)) return SEARCH_OWN;
    if (pp.W == 1 && S >= 64) return SEARCH_PACKED;
    if (pp.nbpeak && (S <= 24 || (S % 16 == 8 && 4 * pp.W >= S))) return SEARCH_SERIAL;
    return S % 8 != 0 ? SEARCH_SERIAL : SEARCH_PACKED;
}

// The search of a launch with cameras of both: the serial search loses far more on the other's rows
// than the packed one on its own.
inline int search_of_both(int a, int b) {
    return a == SEARCH_PACKED || b == SEARCH_PACKED ? SEARCH_PACKED : a > b ? a : b;
}

// One image of a byte stream as the image kernel's producer needs it: checked
// once (its segments tile the camera's pixels with 16-byte-aligned runs inside
// the stream) and read with two 16-byte loads at the image boundary; the first
// STREAM_INLINE_SEGS segments inline, the rest from the directory.
constexpr int STREAM_INLINE_SEGS = 4;
struct StreamImg {
    int ok, cam, nseg, seg0;
    long long row;               // first calibration row of the telescope
    int P, S;
    int first[STREAM_INLINE_SEGS];
    int n[STREAM_INLINE_SEGS];
    long long off[STREAM_INLINE_SEGS];
};
cudaError_t launch_stream_meta(const ChainArgs& a, StreamImg* out, int64_t max_img, int n_sm, cudaStream_t s);

struct CleanArgs {
    DevArray arr;
    ProcParams pp;
    const float* q;
    int64_t n_q;
    const int32_t* img_tel;
    const int64_t* pix_off;
    int64_t n_img;
    uint8_t* mask;
    unsigned int* status;
};

struct HillasArgs {
    DevArray arr;
    const float* q;
    const float* t;
    const uint8_t* mask;
    int64_t n_q;
    const int32_t* img_tel;
    const int64_t* pix_off;
    int64_t n_img;
    rta_hillas_t* out;
    unsigned int* status;
};

struct StereoArgs {
    DevArray arr;
    const rta_hillas_t* h;
    const int32_t* img_tel;
    int64_t n_img;
    const int32_t* evt_off;
    int64_t n_evt;             // events (capacity when n_evt_dev is set)
    const int64_t* n_img_dev;  // optional device-resident counts, read at run time
    const int64_t* n_evt_dev;
    rta_stereo_t* out;
    unsigned int* status;
    int settled;               // event offsets and counts were written before the kernel this one follows
                               // on the stream started: they are read before the dependency wait
    int per_cta;               // events a CTA takes per round (set by the launcher)
};

int chain_variant_warps(int v);
int chain_variant_ppt(int v);
int chain_stage_wave_bytes(int v, int max_S);
size_t chain_smem_bytes(int v, int nstage, int stage_wave_bytes, int max_P, int nb_keys = 0, int stream_recs = 0,
                        int tails = 1);
int chain_chunk_pixels(int v, int stage_wave_bytes, int S);
// which instantiation family of the fused kernel a launch uses (the occupancy of
// a family's general instantiation stands for its lean ones: same launch bounds,
// same shared memory)
enum { CHAIN_PLAIN = 0, CHAIN_NB = 1, CHAIN_STREAM = 2 };
int chain_occupancy(int v, size_t smem, int kind = CHAIN_PLAIN);
// the neighbour-peak instantiations (k_image_nb.cu), the lean ones of the image chain on
// contiguous bundles -- flat window, neighbour-peak window, digital filter -- (k_image_lean.cu)
// and the byte-stream ones (k_image_stream.cu)
cudaError_t dispatch_image_chain_nb(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s, bool occ_only,
                                    int* occ);
cudaError_t dispatch_image_chain_lean(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s);
cudaError_t dispatch_image_chain_win(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s);
cudaError_t dispatch_image_chain_serial(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s);
cudaError_t dispatch_image_chain_any(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s);
cudaError_t dispatch_image_chain_stream(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s,
                                        bool occ_only, int* occ);
int chain_variant_min_blocks(int v);
cudaError_t launch_image_chain(int v, const ChainArgs& a, int grid, size_t smem, cudaStream_t s);
cudaError_t launch_clean(const CleanArgs& a, int grid, cudaStream_t s);
cudaError_t launch_hillas(const HillasArgs& a, int grid, cudaStream_t s);
cudaError_t launch_stereo(StereoArgs a, int n_sm, cudaStream_t s);
cudaError_t launch_wait_selftest(unsigned int* status, uint64_t timeout_ns, unsigned long long* waited_ns,
                                 cudaStream_t s);
// stores a message for rta_last_error() on the calling thread
void set_last_error(const char* msg);
// sky map and geometric event rows (k_skymap.cu)
cudaError_t launch_skymap_fill(const rta_event_t* ev, int64_t n_evt, unsigned int* slab, unsigned int* slab_min,
                               cudaStream_t s);
// One window of the transient search (k_skymap.cu): counts from the ring,
// row prefix sums, disk sums, significance, alerts.
struct TransientArgs {
    const unsigned int* slabs;
    int n_slabs;
    unsigned long long use_on, use_off;
    unsigned int *on, *off, *pre_on, *pre_off;   // [256*256], [256*257] work maps
    const int* hw;                               // [2R + 1] disk half-widths
    int R;
    double alpha, s_min;
    int window;
    rta_alert_t* alerts;                         // nullable
    unsigned int* n_alerts;
    unsigned int cap;
    double* sig;                                 // nullable
    int64_t *d_on, *d_off;                       // nullable
};
cudaError_t launch_transient(const TransientArgs& t, cudaStream_t s);
cudaError_t launch_skymap_sum(const unsigned int* slabs, unsigned long long use, unsigned int* out, cudaStream_t s);
cudaError_t launch_stereo_to_events(const rta_stereo_t* st, int64_t n_evt, rta_event_t* ev, cudaStream_t s);
// DL0 byte-stream ingest (k_ingest.cu).
// Packet positions a piece keeps from its walk; past them the packet list walks on. (128 save 2 us
// of 146 on a 5.1 GB stream and made the first call on a context 200 us longer: its workspace then
// passed the allocator's 2 MiB.)
constexpr int ING_SLOTS = 64;
struct IngChunk {            // one piece of the stream
    long long first;         // its first packet (-1: none found)
    long long last;          // its last packet
    long long end;           // where its walk stopped (>= the piece's end, or a fault)
    long long base;          // packets in the pieces before it
    int count;               // packets that start in it
    int err;
};
struct IngHdr {
    long long n_pk;          // packets on the chain (before a framing fault)
    long long first_bad_pk;  // earliest packet with a fault
    long long walk_err_pos;
    unsigned long long crc_ticket;   // next unit of the CRC check
    unsigned int scan_done, sum_done, final_done;   // blocks that have finished a kernel (its last one goes on alone)
    int walk_err;
    int error;
};
struct IngestArgs {
    DevArray arr;
    const uint8_t* stream;
    int64_t n_bytes;
    int64_t n_chunks, chunk_bytes;
    IngChunk* chunks;
    long long* chunk_pos;        // ING_SLOTS per piece
    IngHdr* hdr;
    int64_t* pk_off;             // seg_cap + 1
    int* pk_err;
    int* pk_len;                 // bytes of each packet
    unsigned int* pk_crc;        // CRC register after the whole packet (0: correct, or not checked)
    unsigned long long* pk_scan;
    unsigned long long* blk_sum;
    rta_segment_t* seg;
    int64_t seg_cap;
    int32_t* img_seg;
    int32_t* img_tel;
    int64_t img_cap;
    int32_t* evt_off;
    uint64_t* evt_number;
    int64_t* evt_time;
    int64_t evt_cap;
    int64_t* counts;
    unsigned int* status;
};
int64_t ingest_chunk_bytes(int64_t n_bytes, int64_t seg_cap, int n_sm);
int64_t ingest_max_chunks(int64_t n_bytes, int n_sm);
cudaError_t launch_ingest(const IngestArgs& a, int verify_crc, int n_sm, cudaStream_t s);

// Lookup-table reconstruction and its training sums (k_lut.cu).
struct LutArgs {
    DevArray arr;
    const rta_hillas_t* h;
    const int32_t* img_tel;
    int64_t n_img;
    const int32_t* evt_off;
    int64_t n_evt;
    const rta_stereo_t* stereo;     // reconstruction: the cores
    const float* log_e;             // training: true log10 E per event
    const float* core_xy;           // training: true impact point per event
    const uint8_t* use;             // training: events to take (nullable)
    const float* size_edges;
    int n_size;
    const float* dist_edges;
    int n_dist;
    const unsigned char* lookup;    // reconstruction: the table in lookup form (RTA_LUT_LOOKUP_BYTES a cell)
    double* acc;                    // training sums, 8 per cell
    float cut[4];                   // mscw_lo, mscw_hi, mscl_lo, mscl_hi
    rta_lut_event_t* out;
    unsigned int* status;
    int events_per_block, threads_per_event;
};
int lut_events_per_block(int64_t n_evt, int n_sm);
int lut_threads_per_event(int64_t n_evt, int64_t n_img, int n_sm);
cudaError_t launch_lut_reconstruct(const LutArgs& a, int grid, cudaStream_t s);
cudaError_t launch_lut_accumulate(const LutArgs& a, int grid, cudaStream_t s);
cudaError_t launch_lut_finalize(const double* acc, int64_t n_cells, int min_count, rta_lut_cell_t* cells, int grid,
                                cudaStream_t s);
cudaError_t launch_lut_prepare(const rta_lut_cell_t* cells, int64_t n_cells, void* lookup, int grid, cudaStream_t s);
// Sky-map bin of a direction coordinate: floor((v + 2.56) * 50) in FP32 with
// round-to-nearest and no contraction, -1 outside [0, RTA_SKY_N) (and for NaN).
__device__ __forceinline__ int sky_bin(float v) {
    const float u = __fmul_rn(__fadd_rn(v, 2.56f), 50.0f);
    if (!(u >= 0.f) || !(u < float(RTA_SKY_N))) return -1;
    return int(floorf(u));
}

// The event row of a geometric reconstruction: its direction, no energy or
// gamma/hadron score (NaN), no direction when the intersection is invalid.
__device__ __forceinline__ rta_event_t stereo_event_row(const rta_stereo_t& s) {
    rta_event_t r = {};
    r.log_energy = __int_as_float(0x7fc00000);
    r.gammaness = __int_as_float(0x7fc00000);
    r.dir_x = s.dir_x;
    r.dir_y = s.dir_y;
    r.n_used = s.n_valid;
    r.flags = (s.flags & RTA_SF_INVALID) ? RTA_EF_NO_DIRECTION : 0u;
    return r;
}

// context access for the surrogate (rta_api.cu)
int surrogate_ctx_tables(rta_ctx* c, const int32_t** tel_cam, const float2** tel_xy, int* n_tel, int* device);
// the context's device status word
unsigned int* surrogate_ctx_status(rta_ctx* c);
// The serving loop's passes over a batch gathered on the device (capacities and device
// counts; the counts and tables were written before the image kernel started):
// rta_server.cu calls them, rta_api.cu and rta_surrogate.cu define them.
int serve_image_chain(rta_ctx* c, const uint16_t* d_wave, int64_t n_wave, const int64_t* d_wave_off,
                      const int32_t* d_img_tel, const int64_t* d_n_img, int64_t max_img, int window_mode, int start,
                      int W, float t_hi, float t_lo, int core_nb, rta_hillas_t* d_out, cudaStream_t s);
int serve_stereo(rta_ctx* c, const rta_hillas_t* d_h, const int32_t* d_img_tel, int64_t max_img,
                 const int32_t* d_evt_off, int64_t max_evt, const int64_t* d_n_img, const int64_t* d_n_evt,
                 rta_stereo_t* d_out, cudaStream_t s);
int serve_infer(rta_model* md, const rta_hillas_t* d_h, const int32_t* d_img_tel, int64_t max_img,
                const int32_t* d_evt_off, int64_t max_evt, const int64_t* d_n_img, const int64_t* d_n_evt,
                float fallback_deg, rta_event_t* d_out, cudaStream_t s);
// Host-side check of a bundle's image table against the registered cameras: every
// offset non-negative, a multiple of 8 samples, the image inside n_wave samples; every
// telescope registered. RTA_OK or RTA_E_INVALID / RTA_E_ALIGN with the message set.
int check_bundle_images(rta_ctx* c, const int64_t* h_wave_off, const int32_t* h_img_tel, int64_t n_img,
                        int64_t n_wave);
// ------------------------------------------------------------------ launches
constexpr size_t SMEM_PER_CTA = size_t(227) * 1024;     // the most a CTA can have, and an SM's CTAs together

// Opts a kernel in to the most dynamic shared memory, once on each device. The limit is the same
// for every launch: one sized for a launch of its own could be lowered by another thread before
// that launch.
template <class K>
cudaError_t smem_opt_in(K* kern, std::atomic<uint64_t>& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = uint64_t(1) << (dev & 63);
    if (dev < 64 && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             int(SMEM_PER_CTA - fa.sharedSizeBytes));
    if (e == cudaSuccess && dev < 64) done.fetch_or(bit, std::memory_order_release);
    return e;
}

// A launch as a programmatic dependent of the kernel before it on the stream: a training step's
// kernels after its first, those of an ingest, the stereo, lookup and inference kernels. Each waits
// (grid_dependency_wait) before it reads what that kernel writes.
template <class... P, class... A>
cudaError_t launch_dependent(void (*k)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, P(args)...);
}

}  // namespace rta
