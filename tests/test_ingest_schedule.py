"""The framing kernel of the byte-stream ingest on the host, one thread of a block after another:
whatever order the threads leave a barrier in, they meet the next one together, and the pieces'
walks join to the oracle's packets. (The kernel's own source, compiled with the host compiler.)"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle  # noqa: F401  (its package holds the decoder)
import synth
from oracle import ingest
from paper_1307_6489_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))

HARNESS = r"""
extern "C" int frame(const uint8_t* stream, int64_t n_bytes, int64_t chunk_bytes, const int32_t* tel_cam, int n_tel,
                     const int32_t* cam_ps, int order, int64_t seg_cap, long long* out) {
    rta::DevCam cams[16] = {};
    for (int c = 0; c < 16; ++c) {
        cams[c].P = cam_ps[2 * c];
        cams[c].S = cam_ps[2 * c + 1];
    }
    rta::IngestArgs a{};
    a.arr.cams = cams;
    a.arr.tel_cam = tel_cam;
    a.arr.n_tel = n_tel;
    a.stream = stream;
    a.n_bytes = n_bytes;
    a.chunk_bytes = chunk_bytes;
    a.n_chunks = (n_bytes + chunk_bytes - 1) / chunk_bytes;
    a.seg_cap = seg_cap;
    std::vector<rta::IngChunk> chunks(a.n_chunks);
    std::vector<long long> pos(a.n_chunks * rta::ING_SLOTS);
    rta::IngHdr hdr = {};
    a.chunks = chunks.data();
    a.chunk_pos = pos.data();
    a.hdr = &hdr;
    emu::mixed = 0;
    for (int64_t b = 0; b < a.n_chunks; ++b)
        emu::run_block(unsigned(b), unsigned(a.n_chunks), rta::ING_SCAN_THREADS, order, [&]() { rta::k_frame_scan(a); });
    out[0] = hdr.n_pk;
    out[1] = hdr.walk_err;
    for (int64_t b = 0; b < a.n_chunks; ++b) {
        out[2 + 3 * b] = chunks[b].first;
        out[3 + 3 * b] = chunks[b].count;
        out[4 + 3 * b] = chunks[b].base;
    }
    return emu::mixed;
}
extern "C" int64_t chunk_bytes(int64_t n, int64_t seg_cap, int n_sm) { return rta::ingest_chunk_bytes(n, seg_cap, n_sm); }
extern "C" int64_t max_chunks(int64_t n, int n_sm) { return rta::ingest_max_chunks(n, n_sm); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    text = open(os.path.join(_build.CSRC, "k_ingest.cu")).read()
    cut = text.index("// ---------------------------------------------------------------- per-packet checks")
    rule = text.index("int64_t ingest_chunk_bytes(")
    rules = text[rule:text.index("cudaError_t launch_ingest(")]
    d = tmp_path_factory.mktemp("emu")
    src = d / "frame.cpp"
    src.write_text('#include "emu.h"\n' + text[:cut] + rules + "}  // namespace rta\n" + HARNESS)
    out = str(d / "frame.so")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", f"-I{os.path.join(HERE, 'cuda_host')}",
                    f"-I{_build.INCLUDE}", f"-I{_build.CSRC}", f"-I{cuda}", str(src), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    P, i64, i32 = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int
    lib.frame.argtypes = [P, i64, i64, P, i32, P, i32, i64, P]
    lib.chunk_bytes.argtypes, lib.chunk_bytes.restype = [i64, i64, i32], i64
    lib.max_chunks.argtypes, lib.max_chunks.restype = [i64, i32], i64
    return lib


@pytest.mark.parametrize("order", [0, 1, 2, 3])
@pytest.mark.parametrize("seg,chunk", [(None, 128 << 10), ({1: 40, 2: 48, 3: 64}, 64 << 10)])
def test_every_order_of_a_blocks_threads_frames_the_stream(lib, seg, chunk, order):
    wl = synth.make_workload(2, 6)
    buf, plan = synth.encode_stream(wl, seg_pixels=seg)
    buf = np.ascontiguousarray(buf)
    cams = {c: (cam.n_pix, cam.n_samples) for c, cam in wl.cams.items()}
    r = ingest.decode_stream(buf, wl.tel_cam, cams, verify_crc=False)
    assert r["error"] == 0
    # the packets' starts, and how many of them each piece holds
    start = r["seg"][:, 0] - 32
    n_chunks = -(-len(buf) // chunk)
    assert n_chunks > 4
    ps = np.zeros(32, np.int32)
    for c, (P, S) in cams.items():
        ps[2 * c:2 * c + 2] = P, S
    tel_cam = np.ascontiguousarray(wl.tel_cam, np.int32)
    data = np.zeros(len(buf) + 64, np.uint8)
    data = data[-data.ctypes.data % 16:][: len(buf)]
    data[:] = buf
    out = np.zeros(2 + 3 * n_chunks, np.int64)
    mixed = lib.frame(data.ctypes.data, len(buf), chunk, tel_cam.ctypes.data, len(tel_cam), ps.ctypes.data, order,
                      len(start), out.ctypes.data)
    assert mixed == 0, f"{mixed} barriers reached from two places"
    assert (out[0], out[1]) == (len(start), 0)
    count = np.bincount(start // chunk, minlength=n_chunks)
    np.testing.assert_array_equal(out[3::3], count)
    np.testing.assert_array_equal(out[4::3], np.cumsum(count) - count)
    first = np.array([start[start >= b * chunk].min() if count[b] else -1 for b in range(n_chunks)])
    np.testing.assert_array_equal(out[2::3][count > 0], first[count > 0])


@pytest.mark.parametrize("packet,largest", [(64, 1), (3000, 1), (11600, 1), (26000, 2), (51468, 4), (65536, 4)])
def test_pieces_of_long_streams_are_bounded_by_the_packets_expected(lib, packet, largest):
    """Pieces grow with the stream to 1 MiB, and beyond only where the capacity expects few enough
    packets in one for the single thread that walks them."""
    for n in np.logspace(5, 10.5, 60).astype(np.int64):
        c = lib.chunk_bytes(int(n), int(n // packet) + 1, 152)
        assert 128 << 10 <= c <= largest << 20
        assert c == 128 << 10 or (c // 2) * 152 * 8 < n             # no larger than the stream asks for
        assert c >= min(1 << 20, n // (152 * 8) // 2)               # and no more pieces than that up to 1 MiB
    assert c == largest << 20


def test_the_workspace_of_a_stream_holds_every_shorter_one(lib):
    """The pieces that the workspace is sized for cover the stream's, and never fall with its length
    (pieces of twice the size come to half as many)."""
    before = 0
    sizes = {int(x) for x in np.logspace(0, 11, 400)} | {(c * 1216 << 17) + d for c in (1, 2, 4, 8, 16, 32)
                                                         for d in (-1, 0, 1, 1 << 17)}
    for n in sorted(sizes):
        most = lib.max_chunks(n, 152)
        assert most >= before
        before = most
        for seg_cap in (0, 1, n // 60000 + 1, n // 12000 + 1, n // 64 + 1):
            c = lib.chunk_bytes(n, seg_cap, 152)
            assert -(-n // c) <= most
