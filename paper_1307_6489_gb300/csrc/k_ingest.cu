// DL0 byte-stream ingest (Sec. 5: telescope data as a telemetry-formatted byte
// stream; the packet layout is documented in include/rta.h). The decoder builds
// a directory of the stream -- segments, images, events -- and copies nothing:
// the image kernel reads each chunk of pixels from the segment that holds it.
//
// Framing: packets follow one another and only a walk from byte 0 knows where
// they start. The stream is cut into pieces (128 KiB to 4 MiB). Each piece looks
// for its first valid packet (16-byte aligned positions, a header whose fields
// hold and whose successor's header holds too; 1,024 positions per round) and walks
// from there to the end of the piece, keeping the first ING_SLOTS packets' positions.
// The walks must join up: piece b's first packet
// is where piece b-1's walk ended. Where they do not (a fault, or a payload that
// happens to look like a header) a single thread walks on from the last joined
// position, and the piece counts are redone from that walk.
//
// Checks: every packet gets the oracle's checks in the oracle's order (framing,
// fixed header fields, camera, segment order, CRC, capacity); the fault reported
// is the one of the earliest packet. The CRC (optional) is computed by warps,
// each up to 32 KiB of a packet, folded in registers, and the parts combined in
// GF(2)[x] modulo the generator.
#include <algorithm>

#include "rta_launch.cuh"

namespace rta {

namespace {

constexpr int ING_SCAN_THREADS = 256;
constexpr int ING_SCAN_UNROLL = 4;                // positions a thread looks at per round
constexpr int ING_JOIN_SMEM = 4096;               // pieces whose counts the join keeps in shared memory

struct PktFields {
    int apid, seq_flags, length, first, n, P, S;
    uint32_t sec, fine;
    uint64_t event;
};

__device__ __forceinline__ uint32_t byte_of(const uint4& a, const uint4& b, int i) {
    const uint4& v = i < 16 ? a : b;
    const int j = i & 15;
    const uint32_t w = j < 4 ? v.x : j < 8 ? v.y : j < 12 ? v.z : v.w;
    return (w >> (8 * (j & 3))) & 0xFFu;
}

__device__ __forceinline__ uint32_t be16(const uint4& a, const uint4& b, int i) {
    return (byte_of(a, b, i) << 8) | byte_of(a, b, i + 1);
}

__device__ __forceinline__ uint32_t be32(const uint4& a, const uint4& b, int i) {
    return (be16(a, b, i) << 16) | be16(a, b, i + 2);
}

// The oracle's framing, header and camera checks of the packet at pos (16-byte
// aligned), in its order; fills f when the header could be read.
// pkt_check: the packet at pos; header_check: the same from the header's 32 bytes, once at least
// 48 bytes are known to be left.
__device__ int header_check(const uint4& a, const uint4& b, int64_t pos, int64_t n_bytes, const DevArray& arr,
                            PktFields& f) {
    const uint32_t w0 = be16(a, b, 0), w1 = be16(a, b, 2);
    f.apid = int(w0 & 0x7FFu);
    f.seq_flags = int(w1 >> 14);
    f.length = int(be16(a, b, 4)) + 7;
    f.sec = be32(a, b, 10);
    f.fine = be16(a, b, 14);
    f.event = (uint64_t(be32(a, b, 16)) << 32) | be32(a, b, 20);
    f.first = int(be16(a, b, 24));
    f.n = int(be16(a, b, 26));
    f.P = int(be16(a, b, 28));
    f.S = int(be16(a, b, 30));
    if ((w0 >> 13) != 0 || ((w0 >> 12) & 1u) != 0 || ((w0 >> 11) & 1u) != 1 || byte_of(a, b, 6) != 0x10 ||
        byte_of(a, b, 7) != RTA_PKT_SERVICE || byte_of(a, b, 8) != RTA_PKT_SUBSERVICE)
        return RTA_STREAM_HEADER;
    const int L = f.length;
    if ((L & 15) || L < 48 || L > RTA_PKT_MAX_BYTES || pos + L > n_bytes) return RTA_STREAM_FRAMING;
    if (48 + 2 * f.n * f.S != L || f.n == 0 || ((f.n * f.S) & 7) || f.first + f.n > f.P) return RTA_STREAM_HEADER;
    const bool starts = f.first == 0, ends = f.first + f.n == f.P;
    const int want = starts && ends ? 3 : starts ? 1 : ends ? 2 : 0;
    if (f.seq_flags != want) return RTA_STREAM_HEADER;
    if (f.apid >= arr.n_tel) return RTA_STREAM_CAMERA;
    const DevCam& C = arr.cams[arr.tel_cam[f.apid]];
    if (C.P != f.P || C.S != f.S) return RTA_STREAM_CAMERA;
    return RTA_STREAM_OK;
}

__device__ int pkt_check(const uint8_t* s, int64_t pos, int64_t n_bytes, const DevArray& arr, PktFields& f) {
    if (n_bytes - pos < 48) return RTA_STREAM_FRAMING;
    const uint4* h = reinterpret_cast<const uint4*>(s + pos);
    return header_check(__ldg(h), __ldg(h + 1), pos, n_bytes, arr, f);
}

// The fixed fields in a header's first 16 bytes: version, type and secondary-header bits, PUS
// version, service and subservice. What fails here fails pkt_check.
__device__ __forceinline__ bool header_like(const uint4& a) {
    return (a.x & 0xF8u) == 0x08u && (a.y >> 16) == ((uint32_t(RTA_PKT_SERVICE) << 8) | 0x10u) &&
           (a.z & 0xFFu) == RTA_PKT_SUBSERVICE;
}

// A position where a packet can start: its checks hold and so do its successor's.
__device__ __forceinline__ bool plausible_start(const uint8_t* s, int64_t pos, int64_t n_bytes, const DevArray& arr) {
    PktFields f, g;
    if (pkt_check(s, pos, n_bytes, arr, f) != RTA_STREAM_OK) return false;
    const int64_t nx = pos + f.length;
    return nx == n_bytes || pkt_check(s, nx, n_bytes, arr, g) == RTA_STREAM_OK;
}

}  // namespace

// The last block of a kernel to finish goes on with what needs all of them (no block waits).
__device__ __forceinline__ bool last_block(unsigned int* done) {
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    __threadfence();
    return last != 0;
}

// ---------------------------------------------------------------- framing
// The walk of one piece (one thread) from ch.first; returns the fault that ends it, at ch.end.
__device__ int walk_piece(const IngestArgs& a, int64_t b, IngChunk& ch) {
    const int64_t c1 = (b + 1) * a.chunk_bytes < a.n_bytes ? (b + 1) * a.chunk_bytes : a.n_bytes;
    int64_t pos = ch.first;
    int code = RTA_STREAM_OK;
    ch.count = 0;
    ch.last = -1;
    auto fetch = [&](int64_t at, uint4& a0, uint4& a1) {
        if (at < 0 || at >= c1 || a.n_bytes - at < 48) return;
        const uint4* h = reinterpret_cast<const uint4*>(a.stream + at);
        a0 = __ldg(h);
        a1 = __ldg(h + 1);
    };
    uint4 h0 = make_uint4(0u, 0u, 0u, 0u), h1 = h0;
    fetch(pos, h0, h1);
    while (pos < c1) {
        if (a.n_bytes - pos < 48) {
            code = RTA_STREAM_FRAMING;
            break;
        }
        // the next header is on its way (from the length alone) while this one is checked
        const uint4 g0 = h0, g1 = h1;
        const int64_t nx = pos + int(be16(g0, g1, 4)) + 7;
        if ((nx & 15) == 0) fetch(nx, h0, h1);
        PktFields f;
        if ((code = header_check(g0, g1, pos, a.n_bytes, a.arr, f)) != RTA_STREAM_OK) break;
        if (ch.count < ING_SLOTS) a.chunk_pos[b * ING_SLOTS + ch.count] = pos;
        ch.last = pos;
        ++ch.count;
        pos += f.length;                          // = nx
    }
    ch.end = pos;
    return code;
}

__device__ void frame_join(const IngestArgs& a);

// One block per piece: its first plausible packet start, 16 KiB a round, then the walk (one
// thread). Then the last block joins the walks.
__global__ void __launch_bounds__(ING_SCAN_THREADS) k_frame_scan(const IngestArgs a) {
    __shared__ long long found;
    grid_dependents_launch();
    const int64_t b = blockIdx.x;
    const int64_t c0 = b * a.chunk_bytes, c1 = c0 + a.chunk_bytes < a.n_bytes ? c0 + a.chunk_bytes : a.n_bytes;
    if (threadIdx.x == 0) found = b == 0 ? 0 : LLONG_MAX;
    __syncthreads();
    for (int64_t r0 = c0; b > 0 && r0 < c1; r0 += 16 * ING_SCAN_THREADS * ING_SCAN_UNROLL) {
        bool hit = false;
        uint4 h[ING_SCAN_UNROLL];
#pragma unroll
        for (int k = 0; k < ING_SCAN_UNROLL; ++k) {
            const int64_t pos = r0 + 16 * (ING_SCAN_THREADS * k + int64_t(threadIdx.x));
            h[k] = pos < c1 && a.n_bytes - pos >= 48 ? __ldg(reinterpret_cast<const uint4*>(a.stream + pos))
                                                     : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < ING_SCAN_UNROLL; ++k) {
            const int64_t pos = r0 + 16 * (ING_SCAN_THREADS * k + int64_t(threadIdx.x));
            if (header_like(h[k]) && plausible_start(a.stream, pos, a.n_bytes, a.arr)) {
                atomicMin(&found, (long long)pos);
                hit = true;
            }
        }
        // the barrier decides for the whole block: a warp that read `found` itself could already
        // see the next round's and leave alone
        if (__syncthreads_or(hit)) break;
    }
    if (threadIdx.x == 0) {
        IngChunk ch = {};
        ch.first = ch.end = ch.last = -1;
        if (found != LLONG_MAX) {
            ch.first = found;
            ch.err = walk_piece(a, b, ch);
        }
        a.chunks[b] = ch;
    }
    if (last_block(&a.hdr->scan_done)) frame_join(a);
}

// Joins the walks (one block). The walks are on the true chain up to the first
// piece whose first packet is not where the previous walk ended; from there one
// thread walks on and rewrites the pieces' starts and counts, stopping at the
// first framing/header/camera fault. Then an exclusive scan of the counts.
__device__ void frame_join(const IngestArgs& a) {
    __shared__ long long first_bad;
    __shared__ int cnt_s[ING_JOIN_SMEM];
    const int64_t nc = a.n_chunks;
    if (threadIdx.x == 0) first_bad = LLONG_MAX;
    __syncthreads();
#pragma unroll 4
    for (int64_t b = threadIdx.x; b < nc; b += blockDim.x) {
        const IngChunk& ch = a.chunks[b];
        if (b < ING_JOIN_SMEM) cnt_s[b] = ch.count;
        bool bad = ch.first < 0 || ch.err != 0;
        if (b > 0) bad = bad || ch.first != a.chunks[b - 1].end;
        if (bad) atomicMin(&first_bad, (long long)b);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t fb = first_bad;
        a.hdr->first_bad_pk = LLONG_MAX;
        a.hdr->walk_err = 0;
        a.hdr->walk_err_pos = -1;
        if (fb != LLONG_MAX) {
            // the true chain is known up to the start of piece fb
            int64_t pos = fb == 0 ? 0 : a.chunks[fb - 1].end;
            for (int64_t b = fb; b < nc; ++b) {
                IngChunk ch = {};
                ch.first = pos;
                const int code = walk_piece(a, b, ch);
                a.chunks[b] = ch;
                if (b < ING_JOIN_SMEM) cnt_s[b] = ch.count;
                pos = ch.end;
                if (code != RTA_STREAM_OK) {
                    a.hdr->walk_err = code;
                    a.hdr->walk_err_pos = pos;
                    for (int64_t r = b + 1; r < nc; ++r) {
                        a.chunks[r].count = 0;
                        if (r < ING_JOIN_SMEM) cnt_s[r] = 0;
                    }
                    break;
                }
            }
        }
    }
    __syncthreads();
    // exclusive scan of the pieces' packet counts, a run of pieces per thread
    __shared__ long long wsum[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t per = (nc + blockDim.x - 1) / blockDim.x, p0 = min((long long)nc, (long long)(per * threadIdx.x)),
                  p1 = min((long long)nc, (long long)(p0 + per));
    long long mine = 0;
    auto count_of = [&](int64_t b) { return b < ING_JOIN_SMEM ? cnt_s[b] : a.chunks[b].count; };
    for (int64_t b = p0; b < p1; ++b) mine += count_of(b);
    long long incl = mine;
    for (int d = 1; d < 32; d <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += u;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    long long base = incl - mine, total = 0;
    for (int w = 0; w < int(blockDim.x >> 5); ++w) {
        if (w < warp) base += wsum[w];
        total += wsum[w];
    }
    for (int64_t b = p0; b < p1; ++b) {
        a.chunks[b].base = base;
        base += count_of(b);
    }
    if (threadIdx.x == 0) a.hdr->n_pk = total;
}

// ---------------------------------------------------------------- per-packet checks
// One block per piece: its packets' offsets (the first seg_cap + 1 packets of the stream), from
// the positions its walk kept and, past those, by walking on; then segment order, and the scan
// values: image start (high word), event start (low).
__global__ void __launch_bounds__(64) k_pkt_check(const IngestArgs a) {
    grid_dependents_launch();
    grid_dependency_wait();
    const int64_t b = blockIdx.x;
    const IngChunk ch = a.chunks[b];
    const int64_t n = a.hdr->n_pk < a.seg_cap + 1 ? a.hdr->n_pk : a.seg_cap + 1;
    const int count = int(max(0ll, min((long long)ch.count, (long long)n - ch.base)));
    if (count == 0) return;
    const int kept = min(count, ING_SLOTS);
    for (int j = threadIdx.x; j < kept; j += blockDim.x) a.pk_off[ch.base + j] = a.chunk_pos[b * ING_SLOTS + j];
    if (threadIdx.x == 0 && kept < count) {
        PktFields f;
        int64_t pos = a.chunk_pos[b * ING_SLOTS + kept - 1];
        for (int j = kept; j < count; ++j) {
            pkt_check(a.stream, pos, a.n_bytes, a.arr, f);
            pos += f.length;
            a.pk_off[ch.base + j] = pos;
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < count; j += blockDim.x) {
        const int64_t k = ch.base + j;
        PktFields f;
        pkt_check(a.stream, a.pk_off[k], a.n_bytes, a.arr, f);     // passed in the walk
        int err = 0;
        bool new_event = f.first == 0;
        if (k > 0) {
            int64_t before;                      // the packet before this one, maybe an earlier piece's last
            if (j > 0) {
                before = a.pk_off[k - 1];
            } else {
                int64_t e = b - 1;
                while (a.chunks[e].count == 0) --e;
                before = a.chunks[e].last;
            }
            PktFields g;
            pkt_check(a.stream, before, a.n_bytes, a.arr, g);
            if (g.first + g.n < g.P) {
                if (f.apid != g.apid || f.event != g.event || f.first != g.first + g.n) err = RTA_STREAM_SEGMENT;
            } else if (f.first != 0) {
                err = RTA_STREAM_SEGMENT;
            }
            new_event = new_event && f.event != g.event;
        } else if (f.first != 0) {
            err = RTA_STREAM_SEGMENT;
        }
        // the stream may not end inside an image (only when the walk reached the end)
        if (!err && k == a.hdr->n_pk - 1 && !a.hdr->walk_err && f.first + f.n < f.P) err = RTA_STREAM_SEGMENT;
        a.pk_err[k] = err;
        a.pk_len[k] = f.length;
        a.pk_crc[k] = 0u;
        a.pk_scan[k] = (uint64_t(f.first == 0) << 32) | uint64_t(new_event);
    }
}

// ---------------------------------------------------------------- CRC
namespace {

// Product of two polynomials of degree < 16 (degree < 31): a multiply by one bit of x is a shift
// of y or nothing.
__device__ __forceinline__ uint32_t gf_mul(uint32_t x, uint32_t y) {
    uint32_t p = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) p ^= (x & (1u << i)) * y;
    return p;
}

// A polynomial of degree < 31 modulo x^16 + x^12 + x^5 + 1: the part at x^16 and above, taken
// down three times.
__device__ __forceinline__ uint32_t gf_mod(uint32_t p) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t t = p >> 16;
        p = (p & 0xFFFFu) ^ t ^ (t << 5) ^ (t << 12);
    }
    return p;
}

// x^(128 k) modulo the generator, k < 256: a register carried over k 16-byte words of zeros.
struct CrcPowers {
    uint16_t x[256];
    constexpr CrcPowers() : x() {
        uint32_t r = 1;
        for (int k = 0; k < 256; ++k) {
            x[k] = uint16_t(r);
            for (int i = 0; i < 128; ++i) r = (r & 0x8000u) ? ((r << 1) ^ 0x11021u) : (r << 1);
        }
    }
};
__device__ constexpr CrcPowers kCrcPowers{};

constexpr int CRC_THREADS = 256;
constexpr int CRC_BLOCK = 4096;                   // bytes a warp takes per step
constexpr int CRC_UNIT = 8;                       // steps of a work unit at most
static_assert(CRC_UNIT <= 8, "the folded words' top byte");
constexpr int CRC_UNITS = (RTA_PKT_MAX_BYTES / CRC_BLOCK + CRC_UNIT - 1) / CRC_UNIT;   // units of the longest packet

}  // namespace

// For a correct packet, running the CRC register over all L bytes -- the CRC field included,
// most significant byte first -- ends at 0 (the register after the message equals the field,
// and two bytes equal to the register clear it). The register is linear in the message, so the
// packet's 16-byte words can be taken in any grouping, and zeros in front of the message do not
// count: the packet is cut into 4096-byte blocks from its end, the first one padded in front.
// A warp step takes a block, eight words a lane (l, l + 32, ...: coalesced). The same word of the
// next block follows 8 * 4096 bits later, and since x has order 32767 modulo the generator,
// x^32768 is x: a lane's words of successive blocks fold into one polynomial, R <- R x + word, a
// funnel shift and an XOR per 32 bits. At the end of a unit (up to CRC_UNIT blocks) the folded
// words' registers come from byte-parallel arithmetic -- a 32-bit register holds the same byte of
// four of them, and a byte step is nine shifts and three-input logic operations for all four
//   t = hi ^ d; t ^= t >> 4;  hi = lo ^ t << 4 ^ t >> 3;  lo = t ^ t << 5   (per byte, truncated)
// -- each is carried to the end of its block by x^(128 k), the warp's sum over the blocks that
// follow by a power of x below 16, and XORed into the packet's register; the preset 0xFFFF is
// the first two bytes inverted. 0 must be left.
// Bound: memory. A 0.5 GB stream takes 87 us, 5.9 TB/s (225 us with four lookup tables
// per lane in shared memory, a packet to a warp: 9,900 packets on 4,864 warps, three rounds; 107
// with every word's register formed in byte-parallel arithmetic: integer issue).
__global__ void __launch_bounds__(CRC_THREADS, 3) k_pkt_crc(const IngestArgs a) {
    grid_dependents_launch();
    grid_dependency_wait();
    const int lane = threadIdx.x & 31;
    const int64_t n = a.hdr->n_pk < a.seg_cap + 1 ? a.hdr->n_pk : a.seg_cap + 1;
    const int64_t tickets = n * CRC_UNITS;
    unsigned long long ticket = 0;               // lane 0's, asked for a unit ahead
    if (lane == 0) ticket = atomicAdd(&a.hdr->crc_ticket, 1ull);
    for (;;) {
        const int64_t unit = int64_t(__shfl_sync(0xffffffffu, ticket, 0));
        if (unit >= tickets) break;
        if (lane == 0) ticket = atomicAdd(&a.hdr->crc_ticket, 1ull);
        const int64_t k = unit / CRC_UNITS;
        const int part = int(unit % CRC_UNITS);
        const int L = a.pk_len[k], words = L >> 4;               // L is a multiple of 16
        const int blocks = (words + 255) >> 8, pad = blocks * 256 - words;
        const int b0 = part * CRC_UNIT, b1 = min(blocks, b0 + CRC_UNIT);
        if (b0 >= b1) continue;
        const uint4* p = reinterpret_cast<const uint4*>(a.stream + a.pk_off[k]);
        uint32_t R[8][5] = {};                    // most significant word first
#pragma unroll 1
        for (int b = b0; b < b1; ++b) {
            const int w0 = b * 256 + lane - pad;
            uint4 q[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) q[j] = w0 + 32 * j >= 0 ? __ldg(p + w0 + 32 * j) : make_uint4(0u, 0u, 0u, 0u);
            if (b == 0) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (w0 + 32 * j == 0) q[j].x ^= 0xFFFFu;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                R[j][0] = __funnelshift_l(R[j][1], R[j][0], 1);
                R[j][1] = __funnelshift_l(R[j][2], R[j][1], 1) ^ __byte_perm(q[j].x, 0u, 0x0123);
                R[j][2] = __funnelshift_l(R[j][3], R[j][2], 1) ^ __byte_perm(q[j].y, 0u, 0x0123);
                R[j][3] = __funnelshift_l(R[j][4], R[j][3], 1) ^ __byte_perm(q[j].z, 0u, 0x0123);
                R[j][4] = (R[j][4] << 1) ^ __byte_perm(q[j].w, 0u, 0x0123);
            }
        }
        uint32_t v = 0;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            uint32_t hi = 0u, lo = 0u;
            auto byte_step = [&](uint32_t d) {
                uint32_t t = hi ^ d;
                t ^= (t >> 4) & 0x0F0F0F0Fu;
                hi = lo ^ ((t << 4) & 0xF0F0F0F0u) ^ ((t >> 3) & 0x1F1F1F1Fu);
                lo = t ^ ((t << 5) & 0xE0E0E0E0u);
            };
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const uint32_t A = R[4 * g][k], B = R[4 * g + 1][k], C = R[4 * g + 2][k], D = R[4 * g + 3][k];
                const uint32_t ab0 = __byte_perm(A, B, 0x5140), cd0 = __byte_perm(C, D, 0x5140);
                if (k > 0) {                      // the first word holds at most CRC_UNIT - 1 bits
                    const uint32_t ab1 = __byte_perm(A, B, 0x7362), cd1 = __byte_perm(C, D, 0x7362);
                    byte_step(__byte_perm(ab1, cd1, 0x7632));
                    byte_step(__byte_perm(ab1, cd1, 0x5410));
                    byte_step(__byte_perm(ab0, cd0, 0x7632));
                }
                byte_step(__byte_perm(ab0, cd0, 0x5410));
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t r = __byte_perm(lo, hi, 0x0040u | uint32_t(j * 0x11)) & 0xFFFFu;
                v ^= gf_mul(r, kCrcPowers.x[255 - lane - 32 * (4 * g + j)]);
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) v ^= __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) atomicXor(a.pk_crc + k, gf_mod(gf_mul(gf_mod(v), 1u << (blocks - b1))));
    }
}

// ---------------------------------------------------------------- scan of the packets' start flags
// Inclusive scan of 64-bit values (image starts in the high word, event starts
// in the low word) in blocks of 1024; the last block forms the blocks' offsets.
__device__ void scan_blocks(const IngestArgs& a, int64_t n_blk);

__global__ void __launch_bounds__(1024) k_pkt_scan(const IngestArgs a) {
    grid_dependents_launch();
    grid_dependency_wait();
    __shared__ unsigned long long wsum[32];
    const int64_t n = a.hdr->n_pk < a.seg_cap + 1 ? a.hdr->n_pk : a.seg_cap + 1;
    const int64_t k = int64_t(blockIdx.x) * 1024 + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long v = k < n ? a.pk_scan[k] : 0ull;
    unsigned long long incl = v;
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long u = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += u;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        unsigned long long w = wsum[lane];
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long u = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += u;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    incl += warp > 0 ? wsum[warp - 1] : 0ull;
    if (k < n) a.pk_scan[k] = incl;
    if (threadIdx.x == 1023) a.blk_sum[blockIdx.x] = incl;
    if (last_block(&a.hdr->sum_done)) scan_blocks(a, gridDim.x);
}

__device__ void scan_blocks(const IngestArgs& a, int64_t n_blk) {
    // one block: exclusive offsets of the blocks, 1024 at a time
    __shared__ unsigned long long wsum[32];
    __shared__ unsigned long long carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t t0 = 0; t0 < n_blk; t0 += 1024) {
        const int64_t b = t0 + threadIdx.x;
        const unsigned long long v = b < n_blk ? a.blk_sum[b] : 0ull;
        unsigned long long incl = v;
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long u = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += u;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            unsigned long long w = wsum[lane];
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned long long u = __shfl_up_sync(0xffffffffu, w, d);
                if (lane >= d) w += u;
            }
            wsum[lane] = w;
        }
        __syncthreads();
        const unsigned long long before = carry + (warp > 0 ? wsum[warp - 1] : 0ull) + incl - v;
        if (b < n_blk) a.blk_sum[b] = before;
        __syncthreads();
        if (threadIdx.x == 1023) carry = before + v;
        __syncthreads();
    }
}

__device__ void ingest_verdict(const IngestArgs& a);

// Adds the block offsets; then the CRC, capacities, and the earliest faulty packet. The last
// block gives the verdict.
__global__ void __launch_bounds__(1024) k_pkt_final(const IngestArgs a) {
    grid_dependents_launch();
    grid_dependency_wait();
    const int64_t n = a.hdr->n_pk < a.seg_cap + 1 ? a.hdr->n_pk : a.seg_cap + 1;
    const int64_t k = int64_t(blockIdx.x) * 1024 + threadIdx.x;
    if (k < n) {
        const unsigned long long incl = a.pk_scan[k] + a.blk_sum[blockIdx.x];
        a.pk_scan[k] = incl;
        const int64_t img = int64_t(incl >> 32) - 1, evt = int64_t(incl & 0xFFFFFFFFull) - 1;
        int err = a.pk_err[k];
        if (!err && a.pk_crc[k] != 0u) err = RTA_STREAM_CRC;
        if (!err && (k >= a.seg_cap || img >= a.img_cap || evt >= a.evt_cap)) err = RTA_STREAM_CAPACITY;
        a.pk_err[k] = err;
        if (err) atomicMin(reinterpret_cast<unsigned long long*>(&a.hdr->first_bad_pk), (unsigned long long)k);
    }
    if (last_block(&a.hdr->final_done) && threadIdx.x == 0) ingest_verdict(a);
}

// The verdict (one thread): the earliest faulty packet, else the walk's fault.
__device__ void ingest_verdict(const IngestArgs& a) {
    IngHdr& h = *a.hdr;
    const int64_t n = h.n_pk < a.seg_cap + 1 ? h.n_pk : a.seg_cap + 1;
    int64_t* c = a.counts;
    int err = 0;
    int64_t pos = -1;
    if (h.first_bad_pk < n) {
        err = a.pk_err[h.first_bad_pk];
        pos = a.pk_off[h.first_bad_pk];
    } else if (h.walk_err) {
        err = h.walk_err;
        pos = h.walk_err_pos;
    }
    h.error = err;
    c[4] = err;
    c[5] = pos;
    c[3] = 0;
    if (err) {
        c[0] = c[1] = c[2] = 0;
        atomicOr(a.status, RTA_DEV_BAD_STREAM);
        return;
    }
    const unsigned long long last = n > 0 ? a.pk_scan[n - 1] : 0ull;
    c[0] = n;
    c[1] = int64_t(last >> 32);
    c[2] = int64_t(last & 0xFFFFFFFFull);
    if (a.img_seg) a.img_seg[c[1]] = int32_t(n);
    if (a.evt_off) a.evt_off[c[2]] = int32_t(c[1]);
}

// The directory (nothing on a fault).
__global__ void __launch_bounds__(256) k_pkt_emit(const IngestArgs a) {
    grid_dependency_wait();      // (what follows on the stream is not this launch's to start early)
    if (a.hdr->error) return;
    const int64_t n = a.hdr->n_pk;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        PktFields f;
        const int64_t pos = a.pk_off[k];
        pkt_check(a.stream, pos, a.n_bytes, a.arr, f);
        rta_segment_t sg;
        sg.offset = pos + RTA_PKT_HEADER_BYTES;
        sg.first_pixel = f.first;
        sg.n_pixels = f.n;
        a.seg[k] = sg;
        const unsigned long long incl = a.pk_scan[k];
        const unsigned long long prev = k > 0 ? a.pk_scan[k - 1] : 0ull;
        const int64_t img = int64_t(incl >> 32) - 1, evt = int64_t(incl & 0xFFFFFFFFull) - 1;
        if ((incl >> 32) != (prev >> 32)) {
            a.img_seg[img] = int32_t(k);
            a.img_tel[img] = f.apid;
            atomicAdd(reinterpret_cast<unsigned long long*>(a.counts + 3), (unsigned long long)(f.P) * f.S);
        }
        if ((incl & 0xFFFFFFFFull) != (prev & 0xFFFFFFFFull)) {
            a.evt_off[evt] = int32_t(img);
            a.evt_number[evt] = f.event;
            if (a.evt_time) a.evt_time[evt] = int64_t(f.sec) * 1000000000 + (int64_t(f.fine) * 1000000000) / 65536;
        }
    }
}

// ---------------------------------------------------------------- the image kernel's per-image records
// One thread per image of an ingested stream: the directory checked once (a
// known telescope; segments that tile the camera's pixels in order, 16-byte
// aligned, inside the stream) and packed for the producer.
__global__ void __launch_bounds__(256) k_stream_meta(const ChainArgs a, StreamImg* out, int64_t max_img) {
    const int64_t n = a.n_img_dev ? (*a.n_img_dev < max_img ? *a.n_img_dev : max_img) : max_img;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        StreamImg m = {};
        const int tel = a.img_tel[i];
        bool ok = tel >= 0 && tel < a.arr.n_tel;
        if (ok) {
            m.cam = a.arr.tel_cam[tel];
            const DevCam C = a.arr.cams[m.cam];
            m.P = C.P;
            m.S = C.S;
            m.row = a.arr.tel_row[tel];
            ok = m.row >= 0;
        }
        const int seg0 = a.img_seg[i], seg1 = a.img_seg[i + 1];
        ok = ok && seg0 >= 0 && seg1 > seg0 && seg1 <= a.n_seg;
        int next = 0;
        for (int k = seg0; ok && k < seg1; ++k) {
            const rta_segment_t sg = a.seg[k];
            ok = sg.first_pixel == next && sg.n_pixels > 0 && (sg.offset & 15) == 0 &&
                 ((int64_t(sg.n_pixels) * m.S) & 7) == 0 && sg.offset >= 0 &&
                 sg.offset + int64_t(sg.n_pixels) * m.S * 2 <= 2 * a.n_wave;
            if (k - seg0 < STREAM_INLINE_SEGS) {
                m.first[k - seg0] = sg.first_pixel;
                m.n[k - seg0] = sg.n_pixels;
                m.off[k - seg0] = sg.offset;
            }
            next += sg.n_pixels;
        }
        m.ok = ok && next == m.P;
        m.seg0 = seg0;
        m.nseg = ok ? seg1 - seg0 : 0;
        out[i] = m;
    }
}

// ---------------------------------------------------------------- launchers
cudaError_t launch_stream_meta(const ChainArgs& a, StreamImg* out, int64_t max_img, int n_sm, cudaStream_t s) {
    const int g = int(std::min<int64_t>((max_img + 255) / 256, int64_t(n_sm) * 8));
    k_stream_meta<<<g > 0 ? g : 1, 256, 0, s>>>(a, out, max_img);
    return cudaGetLastError();
}

// A piece's walk is serial (about 0.7 us a packet), so short streams are cut into smaller pieces;
// but every piece reads half a packet on average to find its first one, and all blocks should be
// resident at once (eight an SM), so pieces grow with the stream: to 1 MiB, and to 4 MiB as far as
// the segment capacity promises at most twice as many packets in one as the piece keeps. 5.2 GB
// without the CRC in pieces of 1 and of 4 MiB: 200 and 153 us with packets of 51 kB (81 a piece of
// 4 MiB), 524 and 661 us with 12 kB, 2,016 and 2,988 us with 3 kB.
int64_t ingest_chunk_bytes(int64_t n_bytes, int64_t seg_cap, int n_sm) {
    int64_t c = int64_t(128) << 10;
    while (c * n_sm * 8 < n_bytes &&
           (c < (int64_t(1) << 20) || (c < (int64_t(4) << 20) && 2 * c * seg_cap <= 2 * ING_SLOTS * n_bytes)))
        c <<= 1;
    return c;
}

// The most pieces that a stream of up to n_bytes comes to, whatever its packets: the workspace is
// sized by it, so that it never grows for a shorter stream (which may come to more pieces).
int64_t ingest_max_chunks(int64_t n_bytes, int n_sm) {
    const int64_t kib128 = (n_bytes + (int64_t(128) << 10) - 1) >> 17, mib = (n_bytes + (int64_t(1) << 20) - 1) >> 20;
    return std::min<int64_t>(kib128, std::max<int64_t>(mib, int64_t(n_sm) * 8));
}

cudaError_t launch_ingest(const IngestArgs& a, int verify_crc, int n_sm, cudaStream_t s) {
    const int64_t nc = a.n_chunks;
    const int64_t max_pk = a.seg_cap + 1;
    const int64_t n_blk = (max_pk + 1023) / 1024;
    cudaError_t e;
    if ((e = cudaMemsetAsync(a.hdr, 0, sizeof(IngHdr), s)) != cudaSuccess) return e;
    k_frame_scan<<<unsigned(nc), ING_SCAN_THREADS, 0, s>>>(a);
    // from here on programmatic dependents: ingest with CRC and reconstruction of a 0.5 GB stream
    // 254 us, 264 with ordinary launches
    if ((e = launch_dependent(k_pkt_check, unsigned(nc), 64, 0, s, a)) != cudaSuccess) return e;
    if (verify_crc) {
        // three CTAs an SM; warps take units as they finish others
        const int64_t wpb = CRC_THREADS / 32;
        const int64_t g = std::min<int64_t>((max_pk * CRC_UNITS + wpb - 1) / wpb, int64_t(n_sm) * 3);
        if ((e = launch_dependent(k_pkt_crc, unsigned(g), CRC_THREADS, 0, s, a)) != cudaSuccess) return e;
    }
    if ((e = launch_dependent(k_pkt_scan, unsigned(n_blk), 1024, 0, s, a)) != cudaSuccess) return e;
    if ((e = launch_dependent(k_pkt_final, unsigned(n_blk), 1024, 0, s, a)) != cudaSuccess) return e;
    const int g = int(std::min<int64_t>((max_pk + 255) / 256, int64_t(n_sm) * 8));
    return launch_dependent(k_pkt_emit, unsigned(g), 256, 0, s, a);
}

}  // namespace rta
