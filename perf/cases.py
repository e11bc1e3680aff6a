"""The framework's main paths as timed cases: what a real-time reconstruction calls, from the
alert of a handful of events to the 10,000-event bundle, through the public entry points.

Inputs are the seeded synthetic generator's (``synth``): showers planned on the host, waveforms
rendered on the GPU, the pedestals, gains and noise of the telescopes. ``exact`` computes the
same results in 64 bits with plain torch. By definition of the entry points a charge is one FP32
product of an exact integer and the calibration factor, and cleaning and table bins are FP32
comparisons, so those stay FP32 there; everything after them is 64-bit.

Every case has a "kind" (what a program calls) and its sizes:

  reconstruct  Context.reconstruct of an array bundle: waveforms -> Hillas -> direction and core
  camera       Context.image_chain of one camera type: waveforms -> Hillas
  stages       calibrate_integrate, clean and hillas one by one: per-pixel charges, times, masks
  learned      rta_reconstruct_learned: waveforms -> Hillas -> energy, direction, gammaness
  events       rta_stereo and rta_lut_reconstruct on stored Hillas rows
  stream       rta_ingest (every CRC checked) and rta_reconstruct_stream on a DL0 byte stream
  train        a run of training steps of the learned reconstruction, then its saved state
"""
import math

import numpy as np
import torch

import paper_1307_6489_gb300 as rta
import synth

WINDOWS = {"fixed": rta.RTA_WINDOW_FIXED, "sliding": rta.RTA_WINDOW_SLIDING, "filter": rta.RTA_WINDOW_FILTER,
           "neighbour": rta.RTA_WINDOW_NEIGHBOUR}
FILTER_WEIGHTS = (1, 4, 9, 8, 4, 2)     # a pulse-shaped filter over the six-sample window
FALLBACK_DEG = 0.5
LEARN_RATE = 1e-3
ADAM_STEP = 400                         # the training run resumes here
IMAGES_PER_EVENT = 4.63                 # of the 69-telescope array
BYTES_PER_IMAGE = 110_040
SIZE_EDGES = np.float32(10.0) ** np.linspace(1.0, 5.0, 33, dtype=np.float32)
DIST_EDGES = np.linspace(0.0, 1000.0, 21, dtype=np.float32)
LUT_CUTS = (-2.0, 0.9, -2.0, 2.0)       # gamma box: mscw and mscl limits


def listed():
    return [
        # an alert: the few events of a short readout, latency first
        dict(name="alert_8_events", kind="reconstruct", events=8, window="sliding"),
        # the headline bundle: 69 telescopes, 5.1 GB of waveforms
        dict(name="bundle_10000_events", kind="reconstruct", events=10000, window="sliding"),
        # the other signal extractors on an ordinary bundle
        dict(name="filter_2000_events", kind="reconstruct", events=2000, window="filter"),
        dict(name="neighbour_2000_events", kind="reconstruct", events=2000, window="neighbour"),
        # a chunk of the single large camera's stream: 1855 pixels, 40 samples
        dict(name="camera1855_20000_images", kind="camera", camera="large1855", images=20000, pixels=1855, samples=40,
             window="sliding", width=6),
        # the small square camera with a fixed readout window
        dict(name="camera256_2000_images", kind="camera", camera="square256", images=2000, pixels=256, samples=16,
             window="fixed", width=5),
        # a camera the library has no preset for, at the largest size it takes
        dict(name="camera4096_1000_images", kind="camera", camera="square", images=1000, pixels=4096, samples=128,
             window="sliding", width=16),
        # calibration and monitoring: the stages one by one, per-pixel results kept
        dict(name="stages_501_events", kind="stages", events=501, window="sliding"),
        # the learned reconstruction of an ordinary bundle
        dict(name="learned_1000_events", kind="learned", events=1000, window="sliding"),
        # an event list reconstructed again from its stored image parameters
        dict(name="event_list_10000", kind="events", events=10000),
        # the telescopes' byte stream, decoded, checked and reconstructed where it lies
        dict(name="dl0_stream_1000_events", kind="stream", events=1000),
        # training the learned reconstruction: a run of mini-batches and its checkpoint
        dict(name="train_16x2048", kind="train", events=2048, steps=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["reconstruct", "reconstruct", "camera", "camera", "stages", "learned", "events", "stream",
                       "train"])
    if kind == "reconstruct":
        window = rng.choice(["sliding", "sliding", "filter", "neighbour"])
        return dict(kind=kind, events=_log_int(rng, 1, 9000 if window == "sliding" else 3000), window=window)
    if kind == "camera":
        which = rng.choice(["large1855", "square256", "medium1764", "small2048", "square", "hex"])
        if which in ("square", "hex"):
            samples = rng.choice([9, 16, 24, 27, 40, 48, 64, 100, 128])
            pixels = _log_int(rng, 64, 4096)
            pixels = max(64, pixels // 8 * 8) if samples % 8 else pixels
            width = rng.randint(3, min(16, samples))
            window = rng.choice(["sliding", "sliding", "fixed"])
            images = max(1, min(_log_int(rng, 8, 20000), 500_000_000 // (pixels * samples)))
        else:
            pixels, samples = {"large1855": (1855, 40), "square256": (256, 16), "medium1764": (1764, 30),
                               "small2048": (2048, 25)}[which]
            window = rng.choice(["sliding", "fixed"])
            width = rng.choice([5, 6, 8])
            images = _log_int(rng, 8, 18000)
        return dict(kind=kind, camera=which, images=images, pixels=pixels, samples=samples, window=window, width=width)
    if kind == "stages":
        return dict(kind=kind, events=_log_int(rng, 5, 1500), window=rng.choice(["sliding", "neighbour", "filter"]))
    if kind == "learned":
        return dict(kind=kind, events=_log_int(rng, 3, 6000), window="sliding")
    if kind == "events":
        return dict(kind=kind, events=_log_int(rng, 10, 50000))
    if kind == "stream":
        return dict(kind=kind, events=_log_int(rng, 20, 1200))
    return dict(kind=kind, events=_log_int(rng, 256, 4096), steps=rng.randint(4, 16))


# ------------------------------------------------------------------ inputs
def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


_lattices = {}


def _custom_camera(kind, pixels, samples):
    key = (kind, pixels)
    if key not in _lattices:
        _lattices[key] = synth.lattice(kind, pixels, 0.1)
    xy, nb = _lattices[key]
    area = 0.01 * (math.sqrt(3.0) / 2.0 if kind == "hex" else 1.0)
    return synth.Camera(5, pixels, samples, nb.shape[1], 0.1, area, 100.0, xy, nb)


def _custom_workload(case, seed):
    """One telescope with a camera of the case's own lattice, sizes and window."""
    cam = _custom_camera(case["camera"], case["pixels"], case["samples"])
    one = synth.make_workload(1, case["images"], seed=seed, render=False)
    rng = np.random.default_rng(seed)
    ped = 400.0 + rng.normal(0, 5, cam.n_pix)
    gain = 8.0 * (1.0 + rng.normal(0, 0.05, cam.n_pix))
    n = case["images"]
    size = cam.n_pix * cam.n_samples
    one.cams = {5: cam}
    one.tel_cam = np.array([5], np.int32)
    one.tel_pix_off = np.array([0, cam.n_pix], np.int64)
    one.ped, one.gain = ped, gain
    one.p16 = np.round(16 * ped).astype(np.int32)
    one.scale = (1 / (16 * gain * 0.95)).astype(np.float32)
    one.wave_off = np.arange(n, dtype=np.int64) * size
    one.pix_off = np.arange(n + 1, dtype=np.int64) * cam.n_pix
    return one


class State:
    """A bundle on the GPU, its context and output buffers."""


def _array_plan(preset, events, seed):
    """Showers on the array. Which telescopes see an event depends on the number of events alone
    (so that a case has one shape); energy, direction, image sizes, the physical array's
    calibration and the noise are the seed's."""
    wl = synth.make_workload(preset, events, render=False, calib_seed=seed)
    rng = np.random.default_rng(seed + 76)
    light = np.exp(rng.normal(0, 0.3, events))
    shift = rng.normal(0, 0.1, (events, 2))
    wl.seed = seed
    wl.truth[:, 0] *= light
    wl.truth[:, 1:3] += shift
    ell = wl.ell
    ell[:, :, 0] *= light[wl.img_evt, None]
    ell[:, :, 1:3] += shift[wl.img_evt, None, :]
    ell[:, :, 3:5] *= np.exp(rng.normal(0, 0.05, ell[:, :, 3:5].shape))
    return wl


def _plan(case, seed):
    """The case's workload (host plan, no waveforms) and processing arguments."""
    if case["kind"] == "camera" and case["camera"] in ("square", "hex"):
        wl = _custom_workload(case, seed)
        hi, lo, core = 10.0, 5.0, True
    elif case["kind"] == "camera" and case["camera"] in ("square256", "large1855"):
        wl = synth.make_workload(0 if case["camera"] == "square256" else 1, case["images"], seed=seed, render=False)
        hi, lo, core = wl.proc.t_hi, wl.proc.t_lo, wl.proc.core_needs_neighbour
    elif case["kind"] == "camera":          # the array's medium or small telescopes, one type alone
        wl = _single_type(2 if case["camera"] == "medium1764" else 3, case["images"], seed)
        hi, lo, core = 8.0, 4.0, True
    else:
        wl = _array_plan(2, case["events"], seed)
        hi, lo, core = wl.proc.t_hi, wl.proc.t_lo, wl.proc.core_needs_neighbour
    width = case.get("width", wl.proc.W)
    start = min(4, min(c.n_samples for c in wl.cams.values()) - width) if case["window"] == "fixed" else 0
    return wl, (WINDOWS[case["window"]], start, width, hi, lo, core)


def _single_type(cam_id, images, seed):
    wl = synth.make_workload(1, images, seed=seed, render=False)
    cam = synth.camera(cam_id)
    wl.cams = {cam_id: cam}
    wl.tel_cam = np.array([cam_id], np.int32)
    wl.tel_pix_off, wl.ped, wl.gain, wl.p16, wl.scale = synth._calibration(seed, wl.tel_cam, wl.proc, wl.cams)
    size = cam.n_pix * cam.n_samples
    wl.wave_off = np.arange(images, dtype=np.int64) * size
    wl.pix_off = np.arange(images + 1, dtype=np.int64) * cam.n_pix
    return wl


def _calibration(case, wl):
    """The calibration factors: a filter's response replaces the flat window's."""
    if case.get("window") == "filter":
        return (wl.scale * np.float32(len(FILTER_WEIGHTS) / sum(FILTER_WEIGHTS))).astype(np.float32)
    return wl.scale


def _waves(wl):
    """The bundle's waveforms, rendered into device memory."""
    wave = torch.empty(wl.n_samples_total, dtype=torch.int16, device="cuda")
    keep = synth.render_waves_gpu(wl, wave, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    del keep
    return wave


def _context(case, wl):
    ctx = rta.Context(0)
    for c, cam in wl.cams.items():
        ctx.register_camera(c, cam.xy, cam.nb, cam.n_samples)
    ctx.register_array(wl.tel_cam, wl.tel_xy, wl.p16, _calibration(case, wl))
    if case.get("window") == "filter":
        rta.rta_set_filter_weights(ctx.handle, FILTER_WEIGHTS)
    return ctx


def _hillas_views(h):
    """Named views of rta_hillas_t rows: floating fields by unit, and the whole numbers."""
    f, i = h.view(-1, 16), h.view(torch.int32).view(-1, 16)
    return dict(size=f[:, 0], geometry=f[:, 1:5], psi=f[:, 5], polar=f[:, 6:8], time_grad=f[:, 8], time_mean=f[:, 9],
                counts=i[:, 10:12])


def _stereo_views(s):
    f, i = s.view(-1, 8), s.view(torch.int32).view(-1, 8)
    return dict(direction=f[:, 0:2], core=f[:, 2:4], counts=i[:, 4:6])


def _event_views(e):
    f, i = e.view(-1, 8), e.view(torch.int32).view(-1, 8)
    return dict(values=f[:, 0:4], baseline=f[:, 6:8], counts=i[:, 4:6])


def _lut_views(e):
    f, i = e.view(-1, 8), e.view(torch.int32).view(-1, 8)
    return dict(values=f[:, 0:4], counts=i[:, 4:6])


def _zeros(n, dtype=torch.float32):
    return torch.zeros(n, dtype=dtype, device="cuda")


def _params(seed):
    """Weights of a network in mid-training, FP32: He-normal layers, a small output layer."""
    rng = np.random.default_rng(seed + 77)
    p = {}
    for name, shape in rta.SURROGATE_LAYOUT:
        if len(shape) == 2:
            p[name] = rng.normal(0, math.sqrt(2.0 / shape[0]) * (0.2 if name == "V2" else 1.0), shape)
        else:
            p[name] = rng.normal(0, 0.05, shape)
    return {k: v.astype(np.float32) for k, v in p.items()}


def _adam_moments(seed):
    """Adam's moments as a checkpoint holds them: per-parameter gradient scales and their noise."""
    rng = np.random.default_rng(seed + 78)
    n = sum(int(np.prod(s)) for _, s in rta.SURROGATE_LAYOUT)
    scale = 10.0 ** rng.uniform(-2.5, -1.0, n)
    return (0.3 * scale * rng.normal(0, 1, n)).astype(np.float32), (scale * scale).astype(np.float32)


def _hillas_rows(wl, seed):
    """Stored Hillas rows of planned showers: their ellipses with reconstruction noise; some
    images too small to use."""
    rng = np.random.default_rng(seed + 79)
    e = wl.ell[:, 0, :].astype(np.float64)
    n = len(e)
    h = np.zeros((n, 16), np.float32)
    size = np.maximum(e[:, 0], 20.0) * np.exp(rng.normal(0, 0.1, n))
    psi = e[:, 5] + rng.normal(0, 0.05, n)
    psi = psi - np.pi * np.round(psi / np.pi)
    length = np.maximum(e[:, 3], 0.02) * np.exp(rng.normal(0, 0.1, n))
    width = np.minimum(np.maximum(e[:, 4], 0.01) * np.exp(rng.normal(0, 0.1, n)), 0.95 * length)
    x, y = e[:, 1] + rng.normal(0, 0.02, n), e[:, 2] + rng.normal(0, 0.02, n)
    n_pix = np.clip(3 + size / 20.0, 3, 300).astype(np.int32)
    small = rng.uniform(size=n) < 0.08
    n_pix[small] = rng.integers(1, 3, int(small.sum()))
    cols = [size, x, y, length, width, psi, np.hypot(x, y), np.arctan2(y, x), rng.normal(2, 0.6, n),
            rng.normal(8, 1, n)]
    for k, v in enumerate(cols):
        h[:, k] = v
    h.view(np.int32)[:, 10] = n_pix
    return h


def _cam_codes(wl):
    codes = np.zeros(16, np.float32)
    for c, cam in wl.cams.items():
        codes[c] = np.log10(cam.mirror_area) - 2.0
    return codes


def _lut_cells(seed):
    """A filled lookup table, a tenth of its cells unused."""
    rng = np.random.default_rng(seed + 80)
    n = rta.RTA_MAX_CAMS * (len(SIZE_EDGES) - 1) * (len(DIST_EDGES) - 1)
    u = lambda lo, hi: rng.uniform(lo, hi, n).astype(np.float32)
    cells = dict(n=rng.integers(1, 500, n), mean_w=u(0.03, 0.12), sigma_w=u(0.01, 0.05), mean_l=u(0.08, 0.3),
                 sigma_l=u(0.02, 0.1), mean_e=u(-1.5, 2.0), sigma_e=u(0.05, 0.4))
    cells["sigma_w"][rng.uniform(size=n) < 0.1] = 0.0
    return cells


def prepare(case, seed):
    return {"reconstruct": _prepare_bundle, "camera": _prepare_bundle, "stages": _prepare_bundle,
            "learned": _prepare_bundle, "events": _prepare_events, "stream": _prepare_stream,
            "train": _prepare_train}[case["kind"]](case, seed)


def _prepare_bundle(case, seed):
    s = State()
    wl, s.proc = _plan(case, seed)
    s.kind = case["kind"]
    s.ctx = _context(case, wl)
    s.wave = _waves(wl)
    s.wave_off, s.img_tel, s.evt_off = _dev(wl.wave_off), _dev(wl.img_tel), _dev(wl.evt_off)
    s.h = _zeros(wl.n_img * 16)
    s.out = dict(hillas=_hillas_views(s.h))
    if s.kind == "reconstruct":
        s.s = _zeros(wl.n_evt * 8)
        s.out["stereo"] = _stereo_views(s.s)
    elif s.kind == "stages":
        n = int(wl.pix_off[-1])
        s.pix_off = _dev(wl.pix_off[:-1])
        s.q, s.t, s.mask = _zeros(n), _zeros(n), _zeros(n, torch.uint8)
        s.out.update(q=s.q, t=s.t, mask=s.mask)
    elif s.kind == "learned":
        s.model = _model(s.ctx, wl, seed)
        s.e = _zeros(wl.n_evt * 8)
        s.out["events"] = _event_views(s.e)
    return s


class _Model:
    """Owns an rta_model (destroyed before its context)."""

    def __init__(self, ctx, codes):
        self.ctx, self.handle = ctx, rta.rta_surrogate_create(ctx.handle, 1, codes)

    def __del__(self):
        try:
            rta.rta_surrogate_destroy(self.handle)
        except Exception:
            pass


def _model(ctx, wl, seed):
    m = _Model(ctx, _cam_codes(wl))
    rta.rta_surrogate_set_params(m.handle, rta.pack_params(_params(seed)))
    return m


def _prepare_events(case, seed):
    s = State()
    s.kind = "events"
    wl = _array_plan(2, case["events"], seed)
    s.ctx = _context(case, wl)
    s.h = _dev(_hillas_rows(wl, seed).reshape(-1))
    s.img_tel, s.evt_off = _dev(wl.img_tel), _dev(wl.evt_off)
    n = rta.RTA_MAX_CAMS * (len(SIZE_EDGES) - 1) * (len(DIST_EDGES) - 1)
    cells = _dev(rta.lut_cells_from_numpy(**_lut_cells(seed)))
    s.size_edges, s.dist_edges = _dev(SIZE_EDGES), _dev(DIST_EDGES)
    s.lookup = _zeros(n * rta.LUT_LOOKUP_BYTES, torch.uint8)
    rta.rta_lut_prepare(s.ctx.handle, cells.data_ptr(), n, s.lookup.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    s.s, s.e = _zeros(wl.n_evt * 8), _zeros(wl.n_evt * 8)
    s.out = dict(stereo=_stereo_views(s.s), events=_lut_views(s.e))
    return s


def _stream_bytes(wl):
    wl.wave = _waves(wl).cpu().numpy().view(np.uint16)
    return synth.encode_stream(wl)


def _prepare_stream(case, seed):
    s = State()
    s.kind = "stream"
    wl, s.proc = _plan(dict(case, window="sliding"), seed)
    s.ctx = _context(case, wl)
    data, plan = _stream_bytes(wl)
    s.data = torch.from_numpy(data).cuda()
    s.n_seg, s.n_img, s.n_evt = len(plan["img"]), wl.n_img, wl.n_evt
    s.seg = _zeros(s.n_seg * 4, torch.int32)
    s.img_seg, s.img_tel = _zeros(s.n_img + 1, torch.int32), _zeros(s.n_img, torch.int32)
    s.evt_off = _zeros(s.n_evt + 1, torch.int32)
    s.evt_number, s.evt_time = _zeros(s.n_evt, torch.int64), _zeros(s.n_evt, torch.int64)
    s.counts = _zeros(6, torch.int64)
    s.h, s.s = _zeros(s.n_img * 16), _zeros(s.n_evt * 8)
    s.out = dict(segments=s.seg, image_segments=s.img_seg, telescopes=s.img_tel, offsets=s.evt_off,
                 numbers=s.evt_number, times=s.evt_time, counts=s.counts, hillas=_hillas_views(s.h),
                 stereo=_stereo_views(s.s))
    return s


def _train_labels(wl):
    log_e = np.log10(wl.truth[:, 0]).astype(np.float32)
    return log_e, wl.truth[:, 1:3].astype(np.float32), (wl.truth[:, 5] == 0).astype(np.uint8)


def _train_plan(case, seed):
    """The run's events: steps x events of them, and each batch's own image offsets."""
    wl = _array_plan(3, case["events"] * case["steps"], seed)
    b = case["events"]
    offs = np.stack([wl.evt_off[k * b:(k + 1) * b + 1] - wl.evt_off[k * b] for k in range(case["steps"])])
    return wl, _hillas_rows(wl, seed), offs.astype(np.int32)


def _prepare_train(case, seed):
    s = State()
    s.kind = "train"
    wl, rows, offs = _train_plan(case, seed)
    s.ctx = _context(case, wl)
    s.model = _Model(s.ctx, _cam_codes(wl))
    rta.rta_surrogate_set_state(s.model.handle, rta.pack_params(_params(seed)), *_adam_moments(seed), ADAM_STEP)
    s.h, s.img_tel, s.offs = _dev(rows.reshape(-1)), _dev(wl.img_tel), _dev(offs)
    s.log_e, s.src, s.gamma = (_dev(a) for a in _train_labels(wl))
    s.loss = _zeros(case["steps"])
    s.batches = []
    for k in range(case["steps"]):
        e0 = k * case["events"]
        i0, i1 = int(wl.evt_off[e0]), int(wl.evt_off[e0 + case["events"]])
        s.batches.append((s.h.data_ptr() + 64 * i0, s.img_tel.data_ptr() + 4 * i0, i1 - i0, s.offs[k].data_ptr(),
                          case["events"], s.log_e.data_ptr() + 4 * e0, s.src.data_ptr() + 8 * e0,
                          s.gamma.data_ptr() + e0, LEARN_RATE, 1, s.loss[k].data_ptr()))
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    stream = torch.cuda.current_stream().cuda_stream
    if s.kind == "reconstruct":
        s.ctx.reconstruct(s.wave, s.wave_off, s.img_tel, s.evt_off, *s.proc, s.h, s.s)
    elif s.kind == "camera":
        s.ctx.image_chain(s.wave, s.wave_off, s.img_tel, *s.proc, s.h)
    elif s.kind == "stages":
        mode, start, width, hi, lo, core = s.proc
        s.ctx.calibrate_integrate(s.wave, s.wave_off, s.img_tel, s.pix_off, mode, start, width, s.q, s.t)
        s.ctx.clean(s.q, s.img_tel, s.pix_off, hi, lo, core, s.mask)
        s.ctx.hillas(s.q, s.t, s.mask, s.img_tel, s.pix_off, s.h)
    elif s.kind == "learned":
        rta.rta_reconstruct_learned(s.model.handle, s.wave.data_ptr(), s.wave.numel(), s.wave_off.data_ptr(),
                                    s.img_tel.data_ptr(), s.img_tel.numel(), s.evt_off.data_ptr(),
                                    s.evt_off.numel() - 1, *s.proc, FALLBACK_DEG, s.h.data_ptr(), s.e.data_ptr(),
                                    stream)
    elif s.kind == "events":
        s.ctx.stereo(s.h, s.evt_off, s.img_tel, s.s)
        rta.rta_lut_reconstruct(s.ctx.handle, s.h.data_ptr(), s.img_tel.data_ptr(), s.img_tel.numel(),
                                s.evt_off.data_ptr(), s.evt_off.numel() - 1, s.s.data_ptr(), s.lookup.data_ptr(),
                                s.size_edges.data_ptr(), len(SIZE_EDGES) - 1, s.dist_edges.data_ptr(),
                                len(DIST_EDGES) - 1, LUT_CUTS, s.e.data_ptr(), stream)
    elif s.kind == "stream":
        rta.rta_ingest(s.ctx.handle, s.data.data_ptr(), s.data.numel(), 1, s.seg.data_ptr(), s.n_seg,
                       s.img_seg.data_ptr(), s.img_tel.data_ptr(), s.n_img, s.evt_off.data_ptr(),
                       s.evt_number.data_ptr(), s.evt_time.data_ptr(), s.n_evt, s.counts.data_ptr(), stream)
        rta.rta_reconstruct_stream(s.ctx.handle, s.data.data_ptr(), s.data.numel(), s.seg.data_ptr(), s.n_seg,
                                   s.img_seg.data_ptr(), s.img_tel.data_ptr(), s.n_img, s.evt_off.data_ptr(), s.n_evt,
                                   s.counts.data_ptr(), *s.proc, s.h.data_ptr(), s.s.data_ptr(), stream)
    else:
        for batch in s.batches:
            rta.rta_surrogate_train_step(s.model.handle, *batch, stream)
        params, m, v, step = rta.rta_surrogate_get_state(s.model.handle)
        return dict(loss=s.loss, params=params, m=m, v=v, step=step)
    return s.out


def work(case):
    """Bytes every pass must read and write once (waveforms, rows, tables), and its arithmetic."""
    kind = case["kind"]
    if kind == "camera":
        n, size = case["images"], 2.0 * case["pixels"] * case["samples"]
        return dict(bytes=n * (size + 64 + 12) + 28.0 * case["pixels"], flops=n * size)
    if kind == "train":
        img, evt, par = IMAGES_PER_EVENT * case["events"], case["events"], 84_996
        flops = 6.0 * (img * (12 * 128 + 128 * 128) + evt * (256 * 256 + 256 * 4))
        return dict(bytes=case["steps"] * (img * 68.0 + evt * 17.0 + par * 24.0), flops=case["steps"] * flops)
    evt = case["events"]
    img = IMAGES_PER_EVENT * evt
    if kind == "events":
        return dict(bytes=2 * img * 68.0 + evt * (32 + 4 + 32 + 4 + 32.0), flops=img * IMAGES_PER_EVENT * 40)
    tables = 69 * 2000 * 8.0 + 3 * 2000 * 24
    data = img * (BYTES_PER_IMAGE + 64 + 12) + evt * 36 + tables
    flops = img * BYTES_PER_IMAGE
    if kind == "stages":     # charges written once and read twice, times and masks written and read once
        data += img * 2000 * (4 + 4 + 4 + 4 + 4 + 1 + 1.0)
    if kind == "learned":
        flops += 2.0 * (img * (12 * 128 + 128 * 128) + evt * (256 * 256 + 256 * 4))
        data += 84_996 * 2
    if kind == "stream":
        data += img * 2.15 * (48 + 16)
    return dict(bytes=data, flops=flops)


# ------------------------------------------------------------------ the same in 64 bits
def _exact_images(case, wl, proc, wave, pixels=False):
    """Hillas rows (n_img x 12, 64-bit: the ten fields, n_pix, 0) and, when asked, charges and times."""
    mode, start, width, t_hi, t_lo, core_nb = proc
    scale_all = _dev(_calibration(case, wl))
    p16_all = _dev(wl.p16.astype(np.int32))
    rows = torch.zeros(wl.n_img, 10, dtype=torch.float64, device="cuda")
    n_pix = torch.zeros(wl.n_img, dtype=torch.int64, device="cuda")
    q_out = _zeros(int(wl.pix_off[-1])) if pixels else None
    t_out = _zeros(int(wl.pix_off[-1]), torch.float64) if pixels else None
    for c, cam in wl.cams.items():
        P, S = cam.n_pix, cam.n_samples
        images = np.nonzero(wl.tel_cam[wl.img_tel] == c)[0]
        xy = _dev(cam.xy.astype(np.float64))
        nb = _dev(np.where(cam.nb < 0, P, cam.nb).astype(np.int64))
        per = max(1, 40_000_000 // (P * S))
        for k in range(0, len(images), per):
            im = _dev(images[k:k + per])
            tel = _dev(wl.img_tel[images[k:k + per]].astype(np.int64))
            at = _dev(wl.wave_off[images[k:k + per]])[:, None] + torch.arange(P * S, device="cuda")
            x = (wave[at].to(torch.int32) & 0xFFFF).view(-1, P, S)
            cal = _dev(wl.tel_pix_off[:-1])[tel][:, None] + torch.arange(P, device="cuda")
            q, t = _exact_window(x, p16_all[cal], scale_all[cal], mode, start, width, nb)
            if pixels:
                dst = _dev(wl.pix_off[images[k:k + per]])[:, None] + torch.arange(P, device="cuda")
                q_out[dst], t_out[dst] = q, t
            mask = _exact_clean(q, nb, t_hi, t_lo, core_nb)
            rows[im], n_pix[im] = _exact_hillas(q.double(), t, mask, xy)
    return rows, n_pix, q_out, t_out


def _exact_window(x, p16, scale, mode, start, width, nb):
    S = x.shape[2]
    c = torch.nn.functional.pad(torch.cumsum(x, 2, dtype=torch.int32), (1, 0))
    sums = c[:, :, width:] - c[:, :, :-width]
    if mode == rta.RTA_WINDOW_FIXED:
        st = torch.full_like(p16, start)
    else:
        k = torch.arange(S - width + 1, device="cuda", dtype=torch.int32)
        st = 127 - ((sums * 128 + (127 - k)).amax(2) & 127)
    charge = lambda sm: (16 * sm - width * p16).float() * scale
    pick = lambda st: torch.gather(sums, 2, st[:, :, None].long())[:, :, 0]
    if mode == rta.RTA_WINDOW_NEIGHBOUR:
        q0 = charge(pick(st))
        inf = torch.full_like(q0[:, :1], -math.inf)
        far = torch.full_like(st[:, :1], S)
        qn = torch.cat([torch.cat([q0, inf], 1)[:, nb], q0[:, :, None]], 2)
        sn = torch.cat([torch.cat([st, far], 1)[:, nb], st[:, :, None]], 2)
        st = torch.where(qn == qn.amax(2, keepdim=True), sn, S).amin(2)
    total = pick(st)
    num = 16 * total - width * p16
    q = charge(total)
    j = torch.arange(width, device="cuda")
    win = torch.gather(x, 2, st[:, :, None].long() + j).long()
    if mode == rta.RTA_WINDOW_FILTER:
        w = torch.tensor(FILTER_WEIGHTS, device="cuda")
        q = (16 * (win * w).sum(2) - sum(FILTER_WEIGHTS) * p16).float() * scale
    moment = (j * (16 * win - p16[:, :, None])).sum(2).double()
    t = torch.where(num > 0, st + moment / num.double(), st + 0.5 * (width - 1))
    return q, t


def _exact_clean(q, nb, t_hi, t_lo, core_nb):
    near = lambda b: torch.nn.functional.pad(b, (0, 1))[:, nb].any(2)
    hi = q >= t_hi
    core = hi & near(hi) if core_nb else hi
    return core | ((q >= t_lo) & near(core))


def _exact_hillas(q, t, mask, xy):
    q, t = torch.where(mask, q, 0.0), torch.where(mask, t, 0.0)
    size = q.sum(1)
    d = torch.where(size > 0, size, 1.0)
    x, y = xy[:, 0], xy[:, 1]
    cx, cy = (q * x).sum(1) / d, (q * y).sum(1) / d
    dx, dy = x - cx[:, None], y - cy[:, None]
    sxx, syy, sxy = (q * dx * dx).sum(1), (q * dy * dy).sum(1), (q * dx * dy).sum(1)
    psi = 0.5 * torch.atan2(2 * sxy, sxx - syy)
    tm = (q * t).sum(1) / d
    co, si = torch.cos(psi)[:, None], torch.sin(psi)[:, None]
    lon, lat = dx * co + dy * si, dy * co - dx * si
    ll = (q * lon * lon).sum(1)
    lt = (q * lon * (t - tm[:, None])).sum(1)
    n = mask.sum(1)
    grad = torch.where((n >= 2) & (ll > 0), lt / torch.where(ll > 0, ll, 1.0), 0.0)
    rows = torch.stack([size, cx, cy, torch.sqrt(ll / d), torch.sqrt((q * lat * lat).sum(1) / d), psi,
                        torch.hypot(cx, cy), torch.atan2(cy, cx), grad, tm], 1)
    return torch.where((n > 0)[:, None], rows, 0.0), n


def _padded(wl, *columns):
    """Per-image columns as (event, image in event) arrays, and which entries exist."""
    off = wl.evt_off.astype(np.int64)
    m = max(1, int(np.diff(off).max()))
    at = off[:-1, None] + np.arange(m)
    exists = at < off[1:, None]
    at = _dev(np.where(exists, at, 0))
    return [c[at] for c in columns], _dev(exists)


def _exact_stereo(wl, rows, n_pix):
    """Direction and core of every event and which have them."""
    txy = _dev(wl.tel_xy.astype(np.float64))[_dev(wl.img_tel.astype(np.int64))]
    direction = torch.zeros(wl.n_evt, 2, dtype=torch.float64, device="cuda")
    core = torch.zeros_like(direction)
    valid = torch.zeros(wl.n_evt, dtype=torch.bool, device="cuda")
    (h, n, t), exists = _padded(wl, rows, n_pix, txy)
    used = exists & (n >= 3)
    m = h.shape[1]
    a, b = torch.triu_indices(m, m, 1, device="cuda")
    for k in range(0, wl.n_evt, 2000) if m > 1 else ():
        e = slice(k, k + 2000)
        i, j = h[e][:, a], h[e][:, b]
        ti, tj = t[e][:, a], t[e][:, b]
        s = torch.sin(j[:, :, 5] - i[:, :, 5])
        ok = used[e][:, a] & used[e][:, b] & (s.abs() >= 1e-6)
        s = torch.where(ok, s, 1.0)
        flat = lambda v: 1 - v[:, :, 4] / torch.where(v[:, :, 3] > 0, v[:, :, 3], 1.0)
        z = i[:, :, 0] + j[:, :, 0]
        w = s.abs() * i[:, :, 0] * j[:, :, 0] / torch.where(z > 0, z, 1.0) * flat(i) * flat(j)
        w = torch.where(ok, w, 0.0)
        ui = torch.stack([torch.cos(i[:, :, 5]), torch.sin(i[:, :, 5])], 2)
        cj, sj = torch.cos(j[:, :, 5]), torch.sin(j[:, :, 5])
        total = w.sum(1)
        good = total > 0
        for out, pi, pj in ((direction, i[:, :, 1:3], j[:, :, 1:3]), (core, ti, tj)):
            d = pj - pi
            p = pi + ui * ((d[:, :, 0] * sj - d[:, :, 1] * cj) / s)[:, :, None]
            mean = (w[:, :, None] * p).sum(1) / torch.where(good, total, 1.0)[:, None]
            out[e] = torch.where(good[:, None], mean, 0.0)
        valid[e] = good
    return direction, core, valid


def _exact_features(wl, rows, n_pix):
    """Network inputs of every image, which images count, and the events' baselines."""
    (h, n), exists = _padded(wl, rows, n_pix)
    used = exists & (n >= 3)
    count = used.sum(1)
    size = torch.where(used, h[:, :, 0], -1.0)
    order = torch.argsort(size, dim=1, descending=True, stable=True)
    pick = lambda r: torch.gather(h, 1, order[:, r].view(-1, 1, 1).expand(-1, 1, h.shape[2]))[:, 0]
    a, b = pick(0), pick(min(1, h.shape[1] - 1))
    s = torch.sin(b[:, 5] - a[:, 5])
    cross = (count >= 2) & (s.abs() >= 0.1)
    k = ((b[:, 1] - a[:, 1]) * torch.sin(b[:, 5]) - (b[:, 2] - a[:, 2]) * torch.cos(b[:, 5])) / torch.where(cross, s, 1.0)
    hit = torch.stack([a[:, 1] + k * torch.cos(a[:, 5]), a[:, 2] + k * torch.sin(a[:, 5])], 1)
    w = torch.where(used, h[:, :, 0], 0.0)
    mean = (w[:, :, None] * h[:, :, 1:3]).sum(1) / torch.where(w.sum(1) > 0, w.sum(1), 1.0)[:, None]
    base = torch.where(cross[:, None], hit, torch.where((count >= 1)[:, None], mean, 0.0))
    evt = _dev(wl.img_evt.astype(np.int64))
    tel = wl.img_tel.astype(np.int64)
    txy = _dev(wl.tel_xy.astype(np.float64)[tel])
    code = _dev(_cam_codes(wl).astype(np.float64)[wl.tel_cam[tel]])
    d = rows[:, 1:3] - base[evt]
    x = torch.stack([torch.log10(rows[:, 0].clamp(min=1e-3)), d[:, 0], d[:, 1], rows[:, 3], rows[:, 4],
                     torch.cos(2 * rows[:, 5]), torch.sin(2 * rows[:, 5]), rows[:, 8] / 10,
                     torch.hypot(d[:, 0], d[:, 1]), code, txy[:, 0] / 1000, txy[:, 1] / 1000], 1)
    return x, n_pix >= 3, base, count


def _exact_forward(p, x, used, evt, n_evt, count):
    h1 = torch.relu(x @ p["W1"] + p["b1"])
    h2 = torch.relu(h1 @ p["W2"] + p["b2"])
    total = torch.zeros(n_evt, 128, dtype=torch.float64, device="cuda")
    total = total.index_add(0, evt, h2 * used[:, None])
    pool = torch.cat([total / 40.0, total / count.clamp(min=1)[:, None]], 1)
    return torch.relu(pool @ p["V1"] + p["c1"]) @ p["V2"] + p["c2"]


def _exact_hillas_out(rows):
    # an axis has two ends: where it lies along the cut at +-pi/2 (a column of pixels) either is
    # right, and the time gradient along it has either sign
    return dict(size=rows[:, 0], geometry=rows[:, 1:5], psi=None, polar=rows[:, 6:8], time_grad=None,
                time_mean=rows[:, 9], counts=None)


def _exact_train(case, seed):
    wl, hrows, _ = _train_plan(case, seed)
    h = _dev(hrows)
    x, used, base, count = _exact_features(wl, h[:, :10].double(), h.view(torch.int32)[:, 10].long())
    log_e, src, gamma = (_dev(v).double() for v in _train_labels(wl))
    p = {k: _dev(v).double().requires_grad_() for k, v in _params(seed).items()}
    flat_m, flat_v = _adam_moments(seed)
    m = {k: _dev(v).double() for k, v in rta.unpack_params(flat_m).items()}
    v = {k: _dev(u).double() for k, u in rta.unpack_params(flat_v).items()}
    evt = _dev(wl.img_evt.astype(np.int64))
    losses, b = [], case["events"]
    for k in range(case["steps"]):
        e0, e1 = k * b, (k + 1) * b
        i0, i1 = int(wl.evt_off[e0]), int(wl.evt_off[e1])
        y = _exact_forward(p, x[i0:i1], used[i0:i1], evt[i0:i1] - e0, b, count[e0:e1])
        g = gamma[e0:e1]
        r = y[:, 1:3] - (src[e0:e1] - base[e0:e1])
        bce = torch.nn.functional.softplus(y[:, 3]) - g * y[:, 3]
        loss = (g * ((y[:, 0] - log_e[e0:e1]) ** 2 + (r * r).sum(1) / 0.01) + bce).mean()
        losses.append(loss.detach())
        grads = torch.autograd.grad(loss, list(p.values()))
        step = ADAM_STEP + k + 1
        with torch.no_grad():
            for name, g in zip(p, grads):
                m[name] = 0.9 * m[name] + 0.1 * g
                v[name] = 0.999 * v[name] + 0.001 * g * g
                p[name] -= LEARN_RATE * (m[name] / (1 - 0.9 ** step)) / (torch.sqrt(v[name] / (1 - 0.999 ** step)) + 1e-8)
    pack = lambda d: torch.cat([d[k].detach().reshape(-1) for k, _ in rta.SURROGATE_LAYOUT])
    return dict(loss=torch.stack(losses), params=pack(p), m=pack(m), v=pack(v), step=None)


def _exact_lut(wl, rows, n_pix, core, valid, seed):
    """Energy and scaled parameters from the lookup table, the core taken in FP32 as it is stored."""
    cells = {k: _dev(np.asarray(v, np.float64)) for k, v in _lut_cells(seed).items()}
    tel = _dev(wl.img_tel.astype(np.int64))
    evt = _dev(wl.img_evt.astype(np.int64))
    cam = _dev(wl.tel_cam.astype(np.int64))[tel]
    d = core.float()[evt] - _dev(wl.tel_xy)[tel]
    dist = torch.sqrt(d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1])
    iu = torch.bucketize(rows[:, 0].float(), _dev(SIZE_EDGES), right=True) - 1
    ir = torch.bucketize(dist, _dev(DIST_EDGES), right=True) - 1
    n_size, n_dist = len(SIZE_EDGES) - 1, len(DIST_EDGES) - 1
    inside = (iu >= 0) & (iu < n_size) & (ir >= 0) & (ir < n_dist)
    cell = torch.where(inside, (cam * n_size + iu) * n_dist + ir, 0)
    c = {k: v[cell] for k, v in cells.items()}
    ok = inside & valid[evt] & (n_pix >= 3) & (c["sigma_w"] > 0)
    one = lambda s: torch.where(ok, s, 1.0)
    wt = one(c["sigma_e"]) ** -2
    terms = torch.stack([(rows[:, 4] - c["mean_w"]) / one(c["sigma_w"]), (rows[:, 3] - c["mean_l"]) / one(c["sigma_l"]),
                         wt * c["mean_e"], wt, torch.ones_like(wt)], 1) * ok[:, None]
    s = torch.zeros(wl.n_evt, 5, dtype=torch.float64, device="cuda").index_add(0, evt, terms)
    has = s[:, 4] > 0
    n, den = torch.where(has, s[:, 4], 1.0), torch.where(has, s[:, 3], 1.0)
    out = torch.stack([s[:, 2] / den, torch.sqrt(1 / den), s[:, 0] / n, s[:, 1] / n], 1)
    return torch.where(has[:, None], out, 0.0)


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "events":
        wl = _array_plan(2, case["events"], seed)
        h = _dev(_hillas_rows(wl, seed))
        rows, n_pix = h[:, :10].double(), h.view(torch.int32)[:, 10].long()
        direction, core, valid = _exact_stereo(wl, rows, n_pix)
        return dict(stereo=dict(direction=direction, core=core, counts=None),
                    events=dict(values=_exact_lut(wl, rows, n_pix, core, valid, seed), counts=None))
    full = dict(case, window="sliding") if kind == "stream" else case
    wl, proc = _plan(full, seed)
    wave = _waves(wl)
    rows, n_pix, q, t = _exact_images(full, wl, proc, wave, kind == "stages")
    out = dict(hillas=_exact_hillas_out(rows))
    if kind in ("reconstruct", "stream"):
        direction, core, _ = _exact_stereo(wl, rows, n_pix)
        out["stereo"] = dict(direction=direction, core=core, counts=None)
    if kind == "stream":
        out.update({k: None for k in ("segments", "image_segments", "telescopes", "offsets", "numbers", "times",
                                      "counts")})
    if kind == "stages":
        out.update(q=q.double(), t=t, mask=None)
    if kind == "learned":
        direction, _, valid = _exact_stereo(wl, rows, n_pix)
        x, used, base, count = _exact_features(wl, rows, n_pix)
        p = {k: _dev(v).double() for k, v in _params(seed).items()}
        y = _exact_forward(p, x, used, _dev(wl.img_evt.astype(np.int64)), wl.n_evt, count)
        fall = (count >= 2) & (torch.hypot(y[:, 1], y[:, 2]) > FALLBACK_DEG) & valid
        where = torch.where(fall[:, None], direction, base + y[:, 1:3])
        out["events"] = dict(values=torch.cat([y[:, :1], where, torch.sigmoid(y[:, 3:])], 1), baseline=base,
                             counts=None)
    return out
