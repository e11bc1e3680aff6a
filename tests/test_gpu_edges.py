"""Edge cases of the CUDA path through the C ABI: empty and malformed inputs,
degenerate images, saturated samples, the generic (non-specialised) integration
paths at the maximum camera size, argument checks, and the full-size bundle on
sampled outputs."""
import time

import numpy as np
import pytest

import oracle
import synth
import paper_1307_6489_gb300 as rta

from gpu_helpers import (DIR_DEG, T_ABS, Dev, compare_hillas, core_ok, hillas_rows, hillas_rows_as_f32, make_ctx,
                         proc_args, stereo_rows, f32_rows_as_oracle)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def arr():
    wl = synth.make_workload(2, 40)
    ctx = make_ctx(wl)
    yield wl, ctx
    ctx.close()


def test_empty_bundle_is_a_no_op(arr):
    wl, ctx = arr
    dev = Dev(wl)
    out = torch.zeros(16, dtype=torch.float32, device="cuda")
    mode, start, W, t_hi, t_lo, core_nb = proc_args(wl)
    rta.rta_image_chain(ctx.handle, dev.wave.data_ptr(), dev.wave.numel(), dev.wave_off.data_ptr(),
                        dev.img_tel.data_ptr(), 0, mode, start, W, t_hi, t_lo, core_nb, out.data_ptr(), 0)
    rta.rta_stereo(ctx.handle, 0, 0, 0, dev.evt_off.data_ptr(), 0, out.data_ptr(), 0)
    assert ctx.check() == 0
    assert float(out.abs().sum()) == 0.0


def test_malformed_images_are_flagged_not_read(arr):
    wl, ctx = arr
    dev = Dev(wl)
    mode, start, W, t_hi, t_lo, core_nb = proc_args(wl)
    good = dev.hillas_buf()
    ctx.image_chain(dev.wave, dev.wave_off, dev.img_tel, mode, start, W, t_hi, t_lo, core_nb, good)
    ctx.check()
    off = dev.wave_off.clone()
    tel = dev.img_tel.clone()
    off[3] += 1                         # not a multiple of 8 samples
    tel[5] = 999                        # no such telescope
    off[7] = dev.wave.numel()           # past the end of the buffer
    off[9] = -8                         # negative
    out = dev.hillas_buf()
    ctx.image_chain(dev.wave, off, tel, mode, start, W, t_hi, t_lo, core_nb, out)
    with pytest.raises(rta.RtaError) as e:
        ctx.check()
    assert e.value.code == rta.RTA_E_DEVICE and e.value.bits & rta.RTA_DEV_BAD_IMAGE
    g = hillas_rows(out, wl.n_img)
    bad = [3, 5, 7, 9]
    for i in bad:
        assert g["flags"][i] & rta.RTA_HF_BAD_INPUT and g["n_pix"][i] == 0
    keep = np.setdiff1d(np.arange(wl.n_img), bad)
    a = out.cpu().numpy().reshape(-1, 16)[keep]
    b = good.cpu().numpy().reshape(-1, 16)[keep]
    np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))
    assert ctx.check() == 0             # the status word was cleared


def test_malformed_event_lists_are_flagged(arr):
    wl, ctx = arr
    dev = Dev(wl)
    h = dev.hillas_buf()
    evt = dev.evt_off.clone()
    evt[2] = wl.n_img + 5               # event 1 ends past n_img, event 2 starts there
    out = dev.stereo_buf()
    ctx.stereo(h, evt, dev.img_tel, out)
    with pytest.raises(rta.RtaError):
        ctx.check()
    s = stereo_rows(out, wl.n_evt)
    assert s["flags"][1] & rta.RTA_SF_INVALID and s["flags"][2] & rta.RTA_SF_INVALID


@pytest.mark.parametrize("level", ["pedestal", "saturated", "zero"])
def test_flat_waveforms(arr, level):
    wl0, ctx = arr
    wl = synth.subset(wl0, np.arange(10))
    wl.wave[:] = {"pedestal": 400, "saturated": 65535, "zero": 0}[level]
    ref = oracle.reconstruct(wl, per_pixel=True)
    dev = Dev(wl)
    mode, start, W, t_hi, t_lo, core_nb = proc_args(wl)
    q = torch.zeros(dev.n_pix, dtype=torch.float32, device="cuda")
    t = torch.zeros(dev.n_pix, dtype=torch.float32, device="cuda")
    ctx.calibrate_integrate(dev.wave, dev.wave_off, dev.img_tel, dev.pix_off, mode, start, W, q, t)
    ctx.check()
    np.testing.assert_array_equal(q.cpu().numpy().view(np.uint32), ref["q"].view(np.uint32))
    assert np.max(np.abs(t.cpu().numpy() - ref["t"])) <= T_ABS
    h, s = dev.hillas_buf(), dev.stereo_buf()
    ctx.reconstruct(dev.wave, dev.wave_off, dev.img_tel, dev.evt_off, mode, start, W, t_hi, t_lo, core_nb, h, s)
    ctx.check()
    compare_hillas(hillas_rows(h, wl.n_img), ref["hillas"], level)
    st = stereo_rows(s, wl.n_evt)
    np.testing.assert_array_equal(st["flags"], ref["stereo"][:, oracle.S["flags"]].astype(np.uint32))


def random_waves(rng, n_img, P, S, xy):
    """Pedestal noise plus a bright Gaussian blob per image (arbitrary camera)."""
    ped = 400 + rng.normal(0, 3, P)
    w = ped[None, :, None] + rng.normal(0, 2, (n_img, P, S))
    for i in range(n_img):
        c = xy[rng.integers(P)]
        r2 = ((xy - c) ** 2).sum(1)
        amp = rng.uniform(50, 3000) * np.exp(-r2 / (2 * rng.uniform(0.01, 0.05)))
        t0 = rng.uniform(3, S - 4)
        k = np.arange(S)
        w[i] += amp[:, None] * np.exp(-((k[None, :] - t0) ** 2) / 4.5)
    return np.clip(np.floor(w + 0.5), 0, 65535).astype(np.uint16), ped


@pytest.mark.parametrize("kind,P,S,W,sliding", [("square", 4096, 128, 16, True), ("hex", 336, 27, 7, True),
                                                ("hex", 1000, 24, 3, False), ("grid", 64, 9, 9, True),
                                                ("square", 2048, 25, 6, True), ("hex", 1764, 30, 6, False)])
def test_generic_paths_and_largest_camera(kind, P, S, W, sliding):
    rng = np.random.default_rng(P + S)
    pitch = 0.1
    xy, nb = synth.lattice(kind, P, pitch)
    n_img = 12
    wave, ped = random_waves(rng, n_img, P, S, xy.astype(np.float64))
    gain = 8 * (1 + rng.normal(0, 0.05, P))
    p16 = np.round(16 * ped).astype(np.int32)
    scale = (1 / (16 * gain * 0.9)).astype(np.float32)
    ctx = rta.Context(0)
    ctx.register_camera(5, xy, nb, S)
    ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), p16, scale)
    start = 0 if sliding else S - W
    flat = wave.reshape(-1)
    d_wave = torch.from_numpy(flat.view(np.int16)).cuda()
    wave_off = torch.arange(n_img, dtype=torch.int64, device="cuda") * (P * S)
    img_tel = torch.zeros(n_img, dtype=torch.int32, device="cuda")
    pix_off = torch.arange(n_img, dtype=torch.int64, device="cuda") * P
    q = torch.zeros(n_img * P, dtype=torch.float32, device="cuda")
    t = torch.zeros(n_img * P, dtype=torch.float32, device="cuda")
    mode = rta.RTA_WINDOW_SLIDING if sliding else rta.RTA_WINDOW_FIXED
    ctx.calibrate_integrate(d_wave, wave_off, img_tel, pix_off, mode, start, W, q, t)
    out = torch.zeros(n_img * 16, dtype=torch.float32, device="cuda")
    ctx.image_chain(d_wave, wave_off, img_tel, mode, start, W, 10.0, 5.0, 1, out)
    ctx.check()
    qg, tg = q.cpu().numpy(), t.cpu().numpy()
    ref_rows = []
    for i in range(n_img):
        qr, tr, _, _ = oracle.integrate(wave[i], p16, scale, sliding, start, W)
        np.testing.assert_array_equal(qg[i * P:(i + 1) * P].view(np.uint32), qr.view(np.uint32))
        assert np.max(np.abs(tg[i * P:(i + 1) * P] - tr)) <= T_ABS
        m = oracle.clean(qr, nb, 10.0, 5.0, 1)
        ref_rows.append(oracle.hillas(xy, qr, tr, m))
    compare_hillas(hillas_rows(out, n_img), np.array(ref_rows), f"{kind}{P}x{S}")
    ctx.close()


@pytest.mark.parametrize("kind,P,S,W", [
    ("hex", 72, 1, 1), ("hex", 72, 2, 2), ("hex", 40, 16, 16), ("hex", 40, 17, 16), ("grid", 64, 31, 3),
    ("hex", 331, 32, 8), ("square", 1030, 48, 5), ("hex", 152, 63, 9), ("square", 257, 64, 16), ("hex", 1855, 40, 7),
    ("hex", 1000, 65, 2), ("square", 516, 96, 15), ("hex", 130, 100, 12), ("square", 1030, 112, 6),
    ("hex", 264, 127, 16), ("square", 2049, 128, 4),
    # widths other than 6 of the 40-, 30- and 25-sample cameras: small and large, odd rows
    ("hex", 1855, 40, 8), ("hex", 1855, 40, 4), ("hex", 331, 40, 5), ("square", 1028, 30, 7), ("hex", 264, 30, 8),
    ("hex", 132, 30, 4), ("hex", 1000, 25, 8), ("square", 2048, 25, 7), ("hex", 264, 25, 5), ("hex", 520, 25, 4)])
def test_any_camera_and_window(kind, P, S, W):
    """The sliding search for cameras and windows without a specialised one: sample counts around
    a word, a block of starts and the split of long rows, odd rows, rows that share banks, pixel
    counts that leave a ragged last chunk, samples from 0 to 12 bits and beyond. Charges bit for
    bit through the integrate-only call; the chain's decisions exact, its rows and the byte-wise
    masks within the usual rules; the same through every tile shape."""
    rng = np.random.default_rng(1000 * S + W)
    xy, nb = synth.lattice(kind, P, 0.1)
    n_img = 5
    wave = rng.integers(380, 421, (n_img, P, S)).astype(np.uint16)
    for i in range(n_img):                          # a bright blob, flat rows, rows of full scale
        d = ((xy - xy[rng.integers(P)]) ** 2).sum(1)
        amp = (np.array([60, 900, 3500, 60000, 200])[i] * np.exp(-d / 0.02)).astype(np.int64)
        k0 = rng.integers(0, S)
        wave[i, :, k0] = np.minimum(wave[i, :, k0] + amp, 65535)
    wave[0, : P // 4] = 400                          # ties: the first window
    wave[1, P // 2] = 4095
    wave[2, P // 3, S // 2:] = 4096
    wave[3, P - 1] = 65535
    wave[4, 0] = 0
    p16 = np.full(P, 16 * 400, np.int32)
    scale = (1 / (16 * 8.0 * rng.uniform(0.9, 1.1, P))).astype(np.float32)
    ctx = rta.Context(0)
    ctx.register_camera(5, xy, nb, S)
    ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), p16, scale)
    d_wave = torch.from_numpy(wave.reshape(-1).view(np.int16)).cuda()
    off = torch.arange(n_img, dtype=torch.int64, device="cuda") * (P * S)
    tel = torch.zeros(n_img, dtype=torch.int32, device="cuda")
    pix = torch.arange(n_img, dtype=torch.int64, device="cuda") * P
    q = torch.zeros(n_img * P, dtype=torch.float32, device="cuda")
    t = torch.zeros_like(q)
    hi, lo = 10.0, 5.0
    mode = rta.RTA_WINDOW_SLIDING
    ref_q, rows, masks = [], [], []
    for i in range(n_img):
        qr, tr, _, _ = oracle.integrate(wave[i], p16, scale, True, 0, W)
        m = oracle.clean(qr, nb, hi, lo, 1)
        ref_q.append((qr, tr))
        masks.append(m)
        rows.append(oracle.hillas(xy, qr, tr, m))
    ctx.calibrate_integrate(d_wave, off, tel, pix, mode, 0, W, q, t)
    qg, tg = q.cpu().numpy().reshape(n_img, P), t.cpu().numpy().reshape(n_img, P)
    for i, (qr, tr) in enumerate(ref_q):
        np.testing.assert_array_equal(qg[i].view(np.uint32), qr.view(np.uint32))
        assert np.max(np.abs(tg[i] - tr)) <= T_ABS
    first = None
    for variant, stages in ((4, 2), (0, 3), (1, 2), (2, 2), (3, 4)):
        try:
            ctx.set_chain_config(variant, stages, 0)
        except rta.RtaError:
            continue                                 # no room for this camera
        out = torch.zeros(n_img * 16, dtype=torch.float32, device="cuda")
        mask = torch.full((n_img * P,), 7, dtype=torch.uint8, device="cuda")
        ctx.image_chain(d_wave, off, tel, mode, 0, W, hi, lo, 1, out)
        with_mask = torch.zeros_like(out)
        ctx.image_chain_masks(d_wave, off, tel, pix, mode, 0, W, hi, lo, 1, mask, with_mask)
        assert ctx.check() == 0
        g = hillas_rows(out, n_img)
        np.testing.assert_array_equal(g["n_pix"], np.array(rows)[:, oracle.H["n_pix"]].astype(np.int32))
        np.testing.assert_array_equal(mask.cpu().numpy().reshape(n_img, P), np.array(masks))
        raw = out.cpu().numpy().view(np.uint32)
        np.testing.assert_array_equal(raw, with_mask.cpu().numpy().view(np.uint32))
        if first is None:
            first = raw
            compare_hillas(g, np.array(rows), f"{kind}{P}x{S} W={W}")
        np.testing.assert_array_equal(raw, first)
    ctx.close()


@pytest.mark.parametrize("S,W", [(9, 9), (17, 16), (20, 3), (25, 12), (30, 3), (31, 8), (50, 2), (63, 9), (65, 6),
                                 (100, 12), (127, 16), (40, 6), (104, 4)])
@pytest.mark.parametrize("mode", [rta.RTA_WINDOW_SLIDING, rta.RTA_WINDOW_FILTER, rta.RTA_WINDOW_NEIGHBOUR])
def test_rows_do_not_depend_on_the_search_that_the_array_takes(mode, S, W):
    """A camera alone in its array, and beside another whose rows share banks (48 samples: the packed
    search for the whole launch): the same rows, masks, charges and times bit for bit, for rows of
    every alignment and several images per block, samples up to full scale among them."""
    P, P2, S2, n_img = 264, 72, 48, 700
    if (P * S) % 8:
        P += 8 - P % 8
    rng = np.random.default_rng(31 * S + W)
    cams = [synth.lattice("hex", P, 0.1), synth.lattice("hex", P2, 0.1)]
    wave = rng.integers(380, 430, (40, P, S)).astype(np.uint16)
    for i in range(40):
        d = ((cams[0][0] - cams[0][0][rng.integers(P)]) ** 2).sum(1)
        k0 = rng.integers(0, S)
        wave[i, :, k0] += (200 * (1 + i % 5) * np.exp(-d / 0.03)).astype(np.uint16)
    wave[3, P // 2] = 65535
    wave[5, 7, S // 2:] = 4096
    wave[6] = 400
    wave2 = rng.integers(380, 430, (40, P2, S2)).astype(np.uint16)
    wave2[:, :9, 20] += 700
    flat = torch.from_numpy(np.concatenate([wave.reshape(-1), wave2.reshape(-1)]).view(np.int16)).cuda()
    kind = np.arange(n_img) % 3 == 2                      # the other camera's images in between
    at = np.where(kind, 40 * P * S + np.arange(n_img) % 40 * (P2 * S2), np.arange(n_img) % 40 * (P * S))
    pixels = np.where(kind, P2, P)
    first = np.cumsum(pixels) - pixels
    got = []
    for both in (False, True):
        ctx = rta.Context(0)
        for c, (xy, nb) in enumerate(cams):
            ctx.register_camera(c, xy, nb, (S, S2)[c])
        n_tel = 2 if both else 1
        ctx.register_array(np.arange(n_tel, dtype=np.int32), np.zeros((n_tel, 2), np.float32),
                           np.full(P + both * P2, 6400, np.int32), np.full(P + both * P2, 1 / 128, np.float32))
        if mode == rta.RTA_WINDOW_FILTER:
            rta.rta_set_filter_weights(ctx.handle, [1 + k % 4 for k in range(W)])
        use = np.arange(n_img) if both else np.flatnonzero(~kind)
        off, pix = (torch.from_numpy(np.ascontiguousarray(a[use]).astype(np.int64)).cuda() for a in (at, first))
        tel = torch.from_numpy(kind[use].astype(np.int32)).cuda()
        q = torch.full((int(pixels.sum()),), float("nan"), device="cuda")
        t, mask = torch.full_like(q, float("nan")), torch.full(q.shape, 7, dtype=torch.uint8, device="cuda")
        h, hm = torch.zeros(len(use) * 16, device="cuda"), torch.zeros(len(use) * 16, device="cuda")
        ctx.calibrate_integrate(flat, off, tel, pix, mode, 0, W, q, t)
        ctx.image_chain(flat, off, tel, mode, 0, W, 4.0, 2.0, 1, h)
        ctx.image_chain_masks(flat, off, tel, pix, mode, 0, W, 4.0, 2.0, 1, mask, hm)
        assert ctx.check() == 0
        ctx.close()
        h, hm = h.cpu().numpy().view(np.uint32).reshape(-1, 16), hm.cpu().numpy().view(np.uint32).reshape(-1, 16)
        np.testing.assert_array_equal(h, hm)
        mine = np.repeat(~kind, pixels)
        got.append((h[~kind[use]], q.cpu().numpy().view(np.uint32)[mine], t.cpu().numpy().view(np.uint32)[mine],
                    mask.cpu().numpy()[mine]))
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
    assert (got[0][0][:, 10] > 0).mean() > 0.3


@pytest.mark.parametrize("kind,P,S,start,W", [
    ("hex", 331, 32, 20, 12), ("square", 1030, 32, 0, 1), ("hex", 1000, 64, 17, 16), ("square", 257, 96, 95, 1),
    ("square", 2049, 128, 112, 16), ("hex", 130, 128, 0, 7), ("square", 1600, 100, 9, 6), ("hex", 1000, 48, 40, 8)])
def test_fixed_window_of_long_rows(kind, P, S, start, W):
    """The fixed window on rows of a multiple of 32 samples (chunks in padded runs, from 64 samples
    two threads a row; four samples and more) and on their neighbours: decisions exact, rows within
    the usual rules, the same through every tile shape, samples up to full scale."""
    rng = np.random.default_rng(100 * S + start)
    xy, nb = synth.lattice(kind, P, 0.1)
    n_img = 7
    wave = rng.integers(380, 421, (n_img, P, S)).astype(np.uint16)
    for i in range(n_img):
        d = ((xy - xy[rng.integers(P)]) ** 2).sum(1)
        amp = (np.array([60, 900, 3500, 60000, 200, 0, 1500])[i] * np.exp(-d / 0.02)).astype(np.int64)
        wave[i, :, start + W // 2] = np.minimum(wave[i, :, start + W // 2] + amp, 65535)
    p16 = np.full(P, 16 * 400, np.int32)
    scale = (1 / (16 * 8.0 * rng.uniform(0.9, 1.1, P))).astype(np.float32)
    ctx = rta.Context(0)
    ctx.register_camera(5, xy, nb, S)
    ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), p16, scale)
    d_wave = torch.from_numpy(wave.reshape(-1).view(np.int16)).cuda()
    off = torch.arange(n_img, dtype=torch.int64, device="cuda") * (P * S)
    tel = torch.zeros(n_img, dtype=torch.int32, device="cuda")
    hi, lo = 10.0, 5.0
    rows = []
    for i in range(n_img):
        qr, tr, _, _ = oracle.integrate(wave[i], p16, scale, False, start, W)
        rows.append(oracle.hillas(xy, qr, tr, oracle.clean(qr, nb, hi, lo, 1)))
    first = None
    for config in (None, (4, 2, 1), (0, 3, 1), (1, 2, 0), (3, 4, 1)):
        try:
            if config:
                ctx.set_chain_config(*config)
        except rta.RtaError:
            continue                                 # no room for this camera
        out = torch.zeros(n_img * 16, dtype=torch.float32, device="cuda")
        ctx.image_chain(d_wave, off, tel, rta.RTA_WINDOW_FIXED, start, W, hi, lo, 1, out)
        assert ctx.check() == 0
        raw = out.cpu().numpy().view(np.uint32)
        if first is None:
            first = raw
            compare_hillas(hillas_rows(out, n_img), np.array(rows), f"{kind}{P}x{S} fixed {start}+{W}")
        np.testing.assert_array_equal(raw, first)
    ctx.close()


@pytest.mark.parametrize("P,S,W,start", [
    (256, 16, 5, -1), (331, 40, 6, -1), (1855, 40, 6, -1), (1600, 100, 6, -1),
    # chunks in padded runs, one thread a row and two: sliding, and the fixed window from `start`
    (331, 32, 6, -1), (264, 48, 16, -1), (1000, 64, 5, -1), (2049, 128, 16, -1), (130, 112, 9, -1),
    (331, 32, 4, 13), (512, 32, 16, 16), (1000, 64, 8, 28), (257, 96, 5, 40), (2049, 128, 16, 56)])
def test_rows_do_not_depend_on_the_launch_size(P, S, W, start):
    """Launches of up to an image per SM (a deeper pipeline), up to the resident CTAs (no counter
    reset) and beyond, images of different brightness in turn (a slot's bitmaps are left zero by
    one for the next, and its stages reused): each image's row is the one it has alone, call after call."""
    rng = np.random.default_rng(P + S)
    kind = "square" if P in (256, 512) else "hex"
    xy, nb = synth.lattice(kind, P, 0.1)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    kinds = 5                                        # distinct images, repeated
    wave = rng.integers(380, 421, (kinds, P, S)).astype(np.uint16)
    for i in range(kinds):
        d = ((xy - xy[rng.integers(P)]) ** 2).sum(1)
        wave[i, :, S // 2 if start < 0 else start + W // 2] += (300 * (i + 1) * np.exp(
            -d / (0.03 + 0.1 * (i % 2)))).astype(np.uint16)
    wave[2] = rng.integers(380, 390, (P, S))         # one with nothing to clean away
    ctx = rta.Context(0)
    ctx.register_camera(5, xy, nb, S)
    ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), np.full(P, 6400, np.int32),
                       np.full(P, 1 / 128, np.float32))
    d_wave = torch.from_numpy(wave.reshape(-1).view(np.int16)).cuda()
    mode = (rta.RTA_WINDOW_SLIDING, 0) if start < 0 else (rta.RTA_WINDOW_FIXED, start)

    def rows(order):
        off = torch.from_numpy(np.asarray(order, np.int64) * (P * S)).cuda()
        tel = torch.zeros(len(off), dtype=torch.int32, device="cuda")
        out = torch.full((len(off) * 16,), -1.0, dtype=torch.float32, device="cuda")
        ctx.image_chain(d_wave, off, tel, *mode, W, 10.0, 5.0, 1, out)
        assert ctx.check() == 0
        return out.cpu().numpy().view(np.uint32).reshape(-1, 16)

    single = np.concatenate([rows([i]) for i in range(kinds)])
    assert (single[:, 10] > 0).sum() >= 3 and single[2, 10] == 0
    for n_img in (kinds, n_sm - 1, n_sm, n_sm + 1, 2 * n_sm, 2 * n_sm + 1, 3 * n_sm, 3 * n_sm + 1, 5 * n_sm, 3, n_sm):
        order = np.arange(n_img) % kinds if n_img % 2 else rng.integers(0, kinds, n_img)
        np.testing.assert_array_equal(rows(order), single[order])
    for config in ((4, 2, 1), (0, 2, 1), (1, 2, 1), (3, 3, 1)):      # one CTA an SM: every slot many times over
        try:
            ctx.set_chain_config(*config)
        except rta.RtaError:
            continue                                 # no room for this camera
        order = rng.integers(0, kinds, 9 * n_sm)
        np.testing.assert_array_equal(rows(order), single[order])
    ctx.close()


def test_argument_checks(arr):
    wl, ctx = arr
    dev = Dev(wl)
    mode, start, W, t_hi, t_lo, core_nb = proc_args(wl)
    out = dev.hillas_buf()
    with pytest.raises(rta.RtaError) as e:
        ctx.image_chain(dev.wave, dev.wave_off, dev.img_tel, mode, start, 26, t_hi, t_lo, core_nb, out)
    assert e.value.code == rta.RTA_E_INVALID            # W = 26 > 25 samples of the small camera
    with pytest.raises(rta.RtaError) as e:
        ctx.image_chain(dev.wave, dev.wave_off, dev.img_tel, mode, start, W, 8.0, 0.0, core_nb, out)
    assert e.value.code == rta.RTA_E_INVALID
    with pytest.raises(rta.RtaError) as e:
        rta.rta_image_chain(ctx.handle, dev.wave.data_ptr() + 2, dev.wave.numel() - 1, dev.wave_off.data_ptr(),
                            dev.img_tel.data_ptr(), wl.n_img, mode, start, W, t_hi, t_lo, core_nb, out.data_ptr(), 0)
    assert e.value.code == rta.RTA_E_ALIGN
    xy, nb = synth.lattice("hex", 7, 0.1)
    with pytest.raises(rta.RtaError) as e:
        ctx.register_camera(9, xy, nb, 5)               # 7 * 5 samples: not a multiple of 8
    assert e.value.code == rta.RTA_E_ALIGN
    with pytest.raises(rta.RtaError) as e:
        rta.rta_register_array(ctx.handle, 1, np.array([11], np.int32), np.zeros(2, np.float32),
                               np.zeros(7, np.int32), np.zeros(7, np.float32))
    assert e.value.code == rta.RTA_E_INVALID            # camera 11 not registered
    assert ctx.check() == 0


def test_stereo_degenerate_events(arr):
    """Single-image events, events whose images are all too small, and one event of 70 images (first 64 used)."""
    wl, ctx = arr
    ref = oracle.reconstruct(wl)
    rows32 = hillas_rows_as_f32(ref["hillas"])
    n = wl.n_img
    # events: [0,1) single image, [1,3) pair, then a big event of up to 70 images, rest as pairs
    big = min(70, n - 3)
    bounds = [0, 1, 3, 3 + big] + list(range(3 + big + 2, n + 1, 2))
    if bounds[-1] != n:
        bounds.append(n)
    evt = np.array(bounds, np.int32)
    rows32[1:3].view(np.int32)[:, 10] = 2                # both images of event 1 below 3 pixels
    h = torch.from_numpy(rows32.reshape(-1)).cuda()
    out = torch.zeros((len(evt) - 1) * 8, dtype=torch.float32, device="cuda")
    ctx.stereo(h, torch.from_numpy(evt).cuda(), torch.from_numpy(wl.img_tel).cuda(), out)
    ctx.check()
    g = stereo_rows(out, len(evt) - 1)
    same = f32_rows_as_oracle(rows32)
    S = oracle.S
    for e in range(len(evt) - 1):
        a, b = evt[e], evt[e + 1]
        b = min(b, a + 64)
        exp = oracle.stereo(same[a:b], wl.tel_xy[wl.img_tel[a:b]].astype(np.float64))
        assert g["flags"][e] == exp[S["flags"]] and g["n_valid"][e] == exp[S["n_valid"]]
        if exp[S["flags"]] == 0:
            assert np.hypot(g["dir_x"][e] - exp[S["dir_x"]], g["dir_y"][e] - exp[S["dir_y"]]) <= DIR_DEG
    assert g["flags"][0] == rta.RTA_SF_INVALID and g["flags"][1] == rta.RTA_SF_INVALID


@pytest.mark.parametrize("n_evt", [1, 2, 9, 457, 913, 15000])
def test_stereo_rows_do_not_depend_on_the_events_around(arr, n_evt):
    """One event to more than a wave of CTAs with several events each, of 0, 1, 2, 8, 9, 24, 25 and
    64 images (the edges of what lanes, warps and CTAs take) in turn: every row equals, bit for
    bit, the row of the same event reconstructed alone; then with two malformed events."""
    wl, ctx = arr
    ref = oracle.reconstruct(wl)
    rows32 = hillas_rows_as_f32(ref["hillas"])
    sizes = np.array([8, 0, 24, 1, 64, 9, 2, 25], np.int64)
    h = torch.from_numpy(np.tile(rows32, (8, 1)).reshape(-1)).cuda()
    tel = torch.from_numpy(np.tile(wl.img_tel, 8)).cuda()
    alone = []
    for k, m in enumerate(sizes):                    # images k .. k + m
        out = torch.zeros(8, dtype=torch.float32, device="cuda")
        ctx.stereo(h[16 * k:], torch.tensor([0, int(m)], dtype=torch.int32, device="cuda"), tel[k:], out)
        alone.append(out.cpu().numpy().view(np.uint32))
    kind = np.arange(n_evt) % 8
    src = torch.from_numpy(np.concatenate([np.arange(k, k + sizes[k]) for k in kind]).astype(np.int64)).cuda()
    off = np.concatenate([[0], np.cumsum(sizes[kind])]).astype(np.int32)
    hh, tt = h.view(-1, 16)[src].reshape(-1), tel[src]
    out = torch.zeros(n_evt * 8, dtype=torch.float32, device="cuda")
    ctx.stereo(hh, torch.from_numpy(off).cuda(), tt, out)
    assert ctx.check() == 0
    got = out.cpu().numpy().view(np.uint32).reshape(-1, 8)
    np.testing.assert_array_equal(got, np.array(alone)[kind])
    if n_evt > 2:
        off[1] = len(src) + 1                        # events 0 and 1 leave the range
        ctx.stereo(hh, torch.from_numpy(off).cuda(), tt, out)
        with pytest.raises(rta.RtaError):
            ctx.check()
        bad = out.cpu().numpy().view(np.uint32).reshape(-1, 8)
        assert bad[0, 5] == rta.RTA_SF_INVALID and bad[1, 5] == rta.RTA_SF_INVALID
        np.testing.assert_array_equal(bad[2:], got[2:])


def test_full_size_bundle_every_event():
    """The benchmark's workload (10,000 events, 46,292 images, ~5 GB) in the
    benchmark's launch configuration, against the oracle on every image and event:
    n_pix and flags exact and every Hillas row within tolerance (the lean kernel
    rta_reconstruct runs), every cleaning mask pixel by pixel (the same kernel
    compiled with the mask output, whose rows are identical bit for bit), every
    stereo row's flags and image count exact, the end-to-end direction within the
    end-to-end bars, and the stereo stage fed the oracle's FP32 rows within 1e-3 deg
    on every event."""
    wl = synth.make_workload(2, 10000)
    ctx = make_ctx(wl)
    dev = Dev(wl)
    mode, start, W, t_hi, t_lo, core_nb = proc_args(wl)
    h, s = dev.hillas_buf(), dev.stereo_buf()
    ctx.reconstruct(dev.wave, dev.wave_off, dev.img_tel, dev.evt_off, mode, start, W, t_hi, t_lo, core_nb, h, s)
    ctx.check()
    mask = torch.full((dev.n_pix,), 7, dtype=torch.uint8, device="cuda")
    hm = torch.full_like(h, float("nan"))
    ctx.image_chain_masks(dev.wave, dev.wave_off, dev.img_tel, dev.pix_off, mode, start, W, t_hi, t_lo, core_nb, mask,
                          hm)
    ctx.check()
    np.testing.assert_array_equal(hm.cpu().numpy().view(np.uint32)[: wl.n_img * 16],
                                  h.cpu().numpy().view(np.uint32)[: wl.n_img * 16])
    ref = oracle.reconstruct(wl, per_pixel=True)
    del dev
    np.testing.assert_array_equal(mask.cpu().numpy(), ref["mask"])
    compare_hillas(hillas_rows(h, wl.n_img), ref["hillas"], "full-size bundle")
    st = stereo_rows(s, wl.n_evt)
    S = oracle.S
    np.testing.assert_array_equal(st["flags"], ref["stereo"][:, S["flags"]].astype(np.uint32))
    np.testing.assert_array_equal(st["n_valid"], ref["stereo"][:, S["n_valid"]].astype(np.int32))
    ok = ref["stereo"][:, S["flags"]] == 0
    assert ok.sum() > 0.4 * wl.n_evt
    d = np.hypot(st["dir_x"][ok] - ref["stereo"][ok, S["dir_x"]], st["dir_y"][ok] - ref["stereo"][ok, S["dir_y"]])
    assert np.percentile(d, 99) <= DIR_DEG and np.median(d) <= 1e-4
    # stage-isolated on every event: both sides get the same FP32 rows
    rows32 = hillas_rows_as_f32(ref["hillas"])
    s2 = torch.zeros(wl.n_evt * 8, dtype=torch.float32, device="cuda")
    ctx.stereo(torch.from_numpy(rows32.reshape(-1)).cuda(), torch.from_numpy(wl.evt_off).cuda(),
               torch.from_numpy(wl.img_tel).cuda(), s2)
    ctx.check()
    g = stereo_rows(s2, wl.n_evt)
    same = f32_rows_as_oracle(rows32)
    exp = np.zeros((wl.n_evt, 6))
    for e in range(wl.n_evt):
        a, b = wl.evt_off[e], wl.evt_off[e + 1]
        exp[e] = oracle.stereo(same[a:b], wl.tel_xy[wl.img_tel[a:b]].astype(np.float64))
    np.testing.assert_array_equal(g["flags"], exp[:, S["flags"]].astype(np.uint32))
    np.testing.assert_array_equal(g["n_valid"], exp[:, S["n_valid"]].astype(np.int32))
    ok = exp[:, S["flags"]] == 0
    assert np.max(np.hypot(g["dir_x"][ok] - exp[ok, S["dir_x"]], g["dir_y"][ok] - exp[ok, S["dir_y"]])) <= DIR_DEG
    assert core_ok(g["core_x"][ok], g["core_y"][ok], exp[ok, S["core_x"]], exp[ok, S["core_y"]]).all()
    ctx.close()


def test_bounded_device_wait_times_out_and_the_context_survives(arr):
    """Failure detection without a GPU fault: a wait that nothing completes gives
    up after its limit, reports RTA_DEV_TIMEOUT, and the next launch works."""
    wl, ctx = arr
    t0 = time.perf_counter()
    waited = rta.rta_selftest_wait_timeout(ctx.handle, 200)
    dt = time.perf_counter() - t0
    assert 0.2e9 <= waited < 2.0e9 and dt < 5.0
    with pytest.raises(rta.RtaError) as e:
        ctx.check()
    assert e.value.code == rta.RTA_E_DEVICE and e.value.bits == rta.RTA_DEV_TIMEOUT
    dev = Dev(wl)
    out = dev.hillas_buf()
    mode, start, W, t_hi, t_lo, core_nb = proc_args(wl)
    ctx.image_chain(dev.wave, dev.wave_off, dev.img_tel, mode, start, W, t_hi, t_lo, core_nb, out)
    assert ctx.check() == 0
    assert (hillas_rows(out, wl.n_img)["n_pix"] > 0).any()


def test_threads_with_cameras_of_different_sizes_do_not_disturb_each_other():
    """Two threads, each with a context, a stream and a camera size of its own, launch the stage kernels
    and the image chain side by side: no launch loses its shared memory to the other's, and every
    row is the one of the thread alone."""
    import threading

    rng = np.random.default_rng(11)
    jobs = []
    for kind, P, S in (("square", 4096, 16), ("hex", 3504, 24)):
        n_img, W = 3, 5
        xy, nb = synth.lattice(kind, P, 0.1)
        ctx = rta.Context(0)
        ctx.register_camera(5, xy, nb, S)
        ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), np.full(P, 6400, np.int32),
                           np.full(P, 1 / 128, np.float32))
        wave = torch.from_numpy(rng.integers(380, 480, n_img * P * S).astype(np.int16)).cuda()
        off = torch.arange(n_img, device="cuda") * (P * S)
        pix = torch.arange(n_img, device="cuda") * P
        tel = torch.zeros(n_img, dtype=torch.int32, device="cuda")
        q, t = torch.zeros(n_img * P, device="cuda"), torch.zeros(n_img * P, device="cuda")
        mask = torch.zeros(n_img * P, dtype=torch.uint8, device="cuda")
        h, hc = torch.zeros(n_img * 16, device="cuda"), torch.zeros(n_img * 16, device="cuda")
        stream = torch.cuda.Stream()

        def work(ctx=ctx, a=(wave, off, tel, pix, q, t, mask, h, hc), s=stream.cuda_stream, W=W, keep=stream):
            wave, off, tel, pix, q, t, mask, h, hc = a
            ctx.calibrate_integrate(wave, off, tel, pix, rta.RTA_WINDOW_SLIDING, 0, W, q, t, stream=s)
            ctx.clean(q, tel, pix, 3.0, 1.5, 1, mask, stream=s)
            ctx.hillas(q, t, mask, tel, pix, h, stream=s)
            ctx.image_chain(wave, off, tel, rta.RTA_WINDOW_SLIDING, 0, W, 3.0, 1.5, 1, hc, stream=s)
            keep.synchronize()
            return h.cpu(), hc.cpu()

        torch.cuda.synchronize()
        jobs.append((ctx, work, work()))
    failed = []

    def loop(work, want):
        try:
            for _ in range(300):
                got = work()
                if not all(torch.equal(g.view(torch.int32), w.view(torch.int32)) for g, w in zip(got, want)):
                    failed.append("rows differ")
                    return
        except rta.RtaError as e:
            failed.append(str(e))

    threads = [threading.Thread(target=loop, args=(work, want)) for _, work, want in jobs]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed
    for ctx, _, want in jobs:
        assert ctx.check() == 0 and int(want[0].view(torch.int32).view(-1, 16)[:, 10].min()) > 0
        ctx.close()


@pytest.mark.parametrize("core_nb", [0, 1])
@pytest.mark.parametrize("P", [8, 31, 33, 256, 257, 1023, 1025, 2049, 4096])
def test_stage_calls_on_more_images_than_fit_at_once(P, core_nb):
    """rta_clean and rta_hillas on charges of every density, NaN and values at the thresholds among
    them, several images per block and rows at odd offsets: masks as the oracle's pixel by pixel,
    rows within the usual rules and the same for every copy of an image."""
    rng = np.random.default_rng(P)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    kinds, n_img, hi, lo = 9, 17 * n_sm + 5, 10.0, 5.0
    xy, nb = synth.lattice("hex", P, 0.1)
    q = rng.normal(0, 2, (kinds, P)).astype(np.float32)
    for i in range(1, kinds):                        # none to nearly all pixels above the thresholds
        pick = rng.random(P) < [0, 0.01, 0.05, 0.2, 0.5, 0.9, 1, 0.1, 0.3][i]
        q[i, pick] = rng.uniform(3, 60, int(pick.sum())).astype(np.float32)
    q[7, ::5], q[7, 1::5], q[7, 2::5] = hi, lo, np.nextafter(np.float32(lo), np.float32(0))
    q[8, ::11] = np.nan
    t = rng.uniform(0, 20, (kinds, P)).astype(np.float32)
    ctx = rta.Context(0)
    ctx.register_camera(5, xy, nb, 8)
    ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), np.full(P, 6400, np.int32),
                       np.full(P, 1 / 128, np.float32))
    step = P + 3
    dq = torch.full((n_img, step), 1e9, dtype=torch.float32, device="cuda")     # (must not be read)
    dt = torch.zeros_like(dq)
    which = torch.arange(n_img, device="cuda") % kinds
    dq[:, :P], dt[:, :P] = torch.from_numpy(q).cuda()[which], torch.from_numpy(t).cuda()[which]
    dq, dt = dq.view(-1), dt.view(-1)
    pix = torch.arange(n_img, dtype=torch.int64, device="cuda") * step
    tel = torch.zeros(n_img, dtype=torch.int32, device="cuda")
    mask = torch.full(dq.shape, 7, dtype=torch.uint8, device="cuda")
    ctx.clean(dq, tel, pix, hi, lo, core_nb, mask)
    out = torch.zeros(n_img * 16, dtype=torch.float32, device="cuda")
    ctx.hillas(dq, dt, mask, tel, pix, out)
    assert ctx.check() == 0
    m = mask.cpu().numpy().reshape(n_img, step)
    assert (m[:, P:] == 7).all()
    ref = [oracle.clean(q[i], nb, hi, lo, core_nb) for i in range(kinds)]
    np.testing.assert_array_equal(m[:, :P], np.array(ref)[np.arange(n_img) % kinds])
    raw = out.cpu().numpy().view(np.uint32).reshape(n_img, 16)
    np.testing.assert_array_equal(raw, raw[:kinds][np.arange(n_img) % kinds])
    rows = np.array([oracle.hillas(xy, q[i], t[i], ref[i]) for i in range(kinds)])
    compare_hillas(hillas_rows(out[: kinds * 16], kinds), rows, f"stages {P}")
    ctx.close()


def test_small_cameras_run_with_the_ctas_that_the_configuration_names():
    """Up to two CTAs per SM, and by default two, variant 4 keeps eight image slots for cameras of at
    most 512 pixels; the configuration reports what is launched, and the rows do not depend on it."""
    P, S, W = 256, 16, 5
    rng = np.random.default_rng(5)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    xy, nb = synth.lattice("square", P, 0.1)
    ctx = rta.Context(0)
    ctx.register_camera(5, xy, nb, S)
    ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), np.full(P, 6400, np.int32),
                       np.full(P, 1 / 128, np.float32))
    n = 4 * n_sm
    wave = torch.from_numpy(rng.integers(380, 480, n * P * S).astype(np.int16)).cuda()
    off = torch.arange(n, dtype=torch.int64, device="cuda") * (P * S)
    tel = torch.zeros(n, dtype=torch.int32, device="cuda")
    seen, rows = {}, {}
    for config in (None, (4, 2, 0), (4, 2, 1), (4, 2, 2), (4, 2, 3), (0, 3, 2)):
        if config:
            ctx.set_chain_config(*config)
        seen[config] = ctx.chain_config()
        for n_img in (7, n_sm, 2 * n_sm + 1, n):
            out = torch.full((n_img * 16,), -1.0, device="cuda")
            ctx.image_chain(wave, off[:n_img], tel[:n_img], rta.RTA_WINDOW_SLIDING, 0, W, 3.0, 1.5, 1, out)
            assert ctx.check() == 0
            want = rows.setdefault(n_img, out)
            assert torch.equal(out.view(torch.int32), want.view(torch.int32)), (config, n_img)
    for config, ctas in ((None, 2), ((4, 2, 0), 2), ((4, 2, 1), 1), ((4, 2, 2), 2), ((4, 2, 3), 3), ((0, 3, 2), 2)):
        assert seen[config]["ctas_per_sm"] == ctas and seen[config]["grid"] == ctas * n_sm, config
    assert seen[(4, 2, 1)]["smem_bytes"] == seen[None]["smem_bytes"] > seen[(4, 2, 3)]["smem_bytes"]
    ctx.close()


@pytest.mark.parametrize("n_img_of_sm", [0.25, 3])
def test_autotuning_a_small_bundle_measures_what_it_records(n_img_of_sm):
    """Tuned on an image per SM at most, the launches that were measured are the ones made afterwards
    (no deeper pipeline in their place); the rows are the untuned ones, there and on more images."""
    P, S, W = 1000, 40, 6
    rng = np.random.default_rng(6)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    xy, nb = synth.lattice("hex", P, 0.1)
    n_img = int(n_img_of_sm * n_sm)
    wave = torch.from_numpy(rng.integers(380, 480, n_img * P * S).astype(np.int16)).cuda()
    off = torch.arange(n_img, dtype=torch.int64, device="cuda") * (P * S)
    tel = torch.zeros(n_img, dtype=torch.int32, device="cuda")
    ctx = rta.Context(0)
    ctx.register_camera(5, xy, nb, S)
    ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), np.full(P, 6400, np.int32),
                       np.full(P, 1 / 128, np.float32))
    args = (rta.RTA_WINDOW_SLIDING, 0, W, 3.0, 1.5, 1)
    ref, out = torch.zeros(n_img * 16, device="cuda"), torch.zeros(n_img * 16, device="cuda")
    ctx.image_chain(wave, off, tel, *args, ref)
    table = ctx.autotune(wave, off, tel, *args, out, reps=1)
    assert torch.equal(out.view(torch.int32), ref.view(torch.int32))
    for e in table:
        assert e["grid"] == min(n_img, e["ctas_per_sm"] * n_sm)
    out.zero_()
    ctx.image_chain(wave, off, tel, *args, out)
    assert ctx.check() == 0
    assert torch.equal(out.view(torch.int32), ref.view(torch.int32))
    ctx.close()
