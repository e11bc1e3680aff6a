"""The step captured as a CUDA graph at capacity, with device-resident counts."""
import numpy as np
import pytest

import synth
import paper_1307_6489_gb300 as rta

from gpu_helpers import Dev, make_ctx, proc_args

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_graph_at_capacity_matches_direct_launches_for_any_count():
    wl = synth.make_workload(2, 200)
    ctx = make_ctx(wl)
    dev = Dev(wl)
    mode, start, W, t_hi, t_lo, core_nb = proc_args(wl)
    h_ref, s_ref = dev.hillas_buf(), dev.stereo_buf()
    ctx.reconstruct(dev.wave, dev.wave_off, dev.img_tel, dev.evt_off, mode, start, W, t_hi, t_lo, core_nb, h_ref, s_ref)
    ctx.check()
    n_img_d = torch.tensor([wl.n_img], dtype=torch.int64, device="cuda")
    n_evt_d = torch.tensor([wl.n_evt], dtype=torch.int64, device="cuda")
    h, s = dev.hillas_buf(), dev.stereo_buf()
    g = rta.rta_graph_create(ctx.handle, dev.wave.data_ptr(), dev.wave.numel(), dev.wave_off.data_ptr(),
                             dev.img_tel.data_ptr(), n_img_d.data_ptr(), wl.n_img, dev.evt_off.data_ptr(),
                             n_evt_d.data_ptr(), wl.n_evt, mode, start, W, t_hi, t_lo, core_nb, h.data_ptr(),
                             s.data_ptr())
    stream = torch.cuda.current_stream().cuda_stream
    try:
        rta.rta_graph_launch(g, stream)
        ctx.check(stream)
        assert torch.equal(h, h_ref) and torch.equal(s, s_ref)
        for n_ev in [57, 1, 200]:
            h.fill_(float("nan"))
            s.fill_(float("nan"))
            n_img = int(wl.evt_off[n_ev])
            n_img_d.fill_(n_img)
            n_evt_d.fill_(n_ev)
            rta.rta_graph_launch(g, stream)
            ctx.check(stream)
            assert torch.equal(h[: n_img * 16], h_ref[: n_img * 16])
            assert torch.equal(s[: n_ev * 8], s_ref[: n_ev * 8])
            assert bool(torch.isnan(h[n_img * 16:]).all()) and bool(torch.isnan(s[n_ev * 8:]).all())
    finally:
        rta.rta_graph_destroy(g)
    ctx.close()


@pytest.mark.parametrize("S0,S1", [(40, 48), (48, 40), (31, 30)])
def test_graph_follows_a_camera_registered_again(S0, S1):
    """A graph captured with a camera of S0 samples launches after the camera was registered again
    with S1, which needs the image kernel for any window where S0 does not (or the reverse): its
    rows are the direct launch's, before and after."""
    P, n_img, W = 264, 9, 6
    rng = np.random.default_rng(S0)
    xy, nb = synth.lattice("hex", P, 0.1)
    n = n_img * P * max(S0, S1)
    wave = torch.from_numpy(rng.integers(380, 480, n).astype(np.int16)).cuda()
    off = torch.zeros(n_img, dtype=torch.int64, device="cuda")
    tel = torch.zeros(n_img, dtype=torch.int32, device="cuda")
    evt = torch.arange(n_img + 1, dtype=torch.int32, device="cuda")
    n_d = torch.tensor([n_img], dtype=torch.int64, device="cuda")
    h, st = torch.zeros(n_img * 16, device="cuda"), torch.zeros(n_img * 8, device="cuda")
    ctx = rta.Context(0)
    ctx.register_camera(5, xy, nb, S0)
    ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), np.full(P, 6400, np.int32),
                       np.full(P, 1 / 128, np.float32))
    args = (rta.RTA_WINDOW_SLIDING, 0, W, 3.0, 1.5, 1)
    g = rta.rta_graph_create(ctx.handle, wave.data_ptr(), n, off.data_ptr(), tel.data_ptr(), n_d.data_ptr(), n_img,
                             evt.data_ptr(), n_d.data_ptr(), n_img, *args, h.data_ptr(), st.data_ptr())
    stream = torch.cuda.current_stream().cuda_stream
    try:
        for S in (S0, S1, S0):
            torch.cuda.synchronize()
            ctx.register_camera(5, xy, nb, S)
            off.copy_(torch.arange(n_img, device="cuda") * (P * S))
            ref, ref_st = torch.zeros_like(h), torch.zeros_like(st)
            ctx.reconstruct(wave, off, tel, evt, *args, ref, ref_st)
            h.fill_(float("nan"))
            rta.rta_graph_launch(g, stream)
            ctx.check(stream)
            assert torch.equal(h.view(torch.int32), ref.view(torch.int32))
            assert torch.equal(st.view(torch.int32), ref_st.view(torch.int32))
            assert int(h.view(torch.int32).view(n_img, 16)[:, 10].min()) > 0
    finally:
        rta.rta_graph_destroy(g)
    ctx.close()


@pytest.mark.parametrize("P", [264, 1000])
@pytest.mark.parametrize("mode,W", [(rta.RTA_WINDOW_SLIDING, 6), (rta.RTA_WINDOW_SLIDING, 8),
                                    (rta.RTA_WINDOW_NEIGHBOUR, 6), (rta.RTA_WINDOW_FILTER, 6)])
def test_a_callers_capture_follows_a_camera_registered_again(mode, W, P):
    """A capture of rta_reconstruct by the caller keeps the image kernel it was captured with, here the
    one that has a compiled search for 40 samples alone. Its rows stay the direct call's when the
    camera comes back with other sample counts (odd, below and above, one that the direct call
    serves with padded runs)."""
    n_img, S0 = 11, 40
    rng = np.random.default_rng(P + W)
    xy, nb = synth.lattice("hex", P, 0.1)
    n = n_img * P * 48
    wave = rng.integers(380, 480, n)
    wave[::97] += 900                                # peaks here and there, and samples beyond 12 bits
    wave[:: 50021] = 5000
    wave = torch.from_numpy(wave.astype(np.int16)).cuda()
    off = torch.arange(n_img, device="cuda") * (P * S0)
    tel = torch.zeros(n_img, dtype=torch.int32, device="cuda")
    evt = torch.tensor([0, 4, 5, 5, n_img], dtype=torch.int32, device="cuda")
    h, st = torch.zeros(n_img * 16, device="cuda"), torch.zeros(4 * 8, device="cuda")
    ctx = rta.Context(0)
    ctx.register_camera(5, xy, nb, S0)
    ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), np.full(P, 6400, np.int32),
                       np.full(P, 1 / 128, np.float32))
    if mode == rta.RTA_WINDOW_FILTER:
        rta.rta_set_filter_weights(ctx.handle, [1, 4, 9, 8, 4, 2])
    args = (mode, 0, W, 3.0, 1.5, 1)
    ctx.reconstruct(wave, off, tel, evt, *args, h, st)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.reconstruct(wave, off, tel, evt, *args, h, st)
    for S in (S0, 31, 48, 24, S0):
        torch.cuda.synchronize()
        ctx.register_camera(5, xy, nb, S)
        off.copy_(torch.arange(n_img, device="cuda") * (P * S))
        ref, ref_st = torch.zeros_like(h), torch.zeros_like(st)
        ctx.reconstruct(wave, off, tel, evt, *args, ref, ref_st)
        h.fill_(float("nan"))
        st.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert ctx.check() == 0
        assert torch.equal(h.view(torch.int32), ref.view(torch.int32)), S
        assert torch.equal(st.view(torch.int32), ref_st.view(torch.int32)), S
        assert int(h.view(torch.int32).view(n_img, 16)[:, 10].min()) > 0
    ctx.close()


def camera_case(rng, n_img, P_max, S_max):
    """Device buffers of n_img images of one telescope, for cameras up to P_max x S_max."""
    n = n_img * P_max * S_max
    wave = torch.from_numpy(rng.integers(380, 480, n).astype(np.int16)).cuda()
    off = torch.zeros(n_img, dtype=torch.int64, device="cuda")
    tel = torch.zeros(n_img, dtype=torch.int32, device="cuda")
    evt = torch.arange(n_img + 1, dtype=torch.int32, device="cuda")
    return wave, off, tel, evt, torch.zeros(n_img * 16, device="cuda"), torch.zeros(n_img * 8, device="cuda")


def register(ctx, P, S, array=True):
    xy, nb = synth.lattice("hex", P, 0.1)
    ctx.register_camera(5, xy, nb, S)
    if array:
        ctx.register_array(np.array([5], np.int32), np.zeros((1, 2), np.float32), np.full(P, 6400, np.int32),
                           np.full(P, 1 / 128, np.float32))


@pytest.mark.parametrize("mode", [rta.RTA_WINDOW_SLIDING, rta.RTA_WINDOW_NEIGHBOUR])
def test_graph_follows_growing_cameras_and_arrays(mode):
    """The graph's launches match the direct call's after the camera came back with more pixels and
    longer rows (of the same kind of search and of the other), the array registered with it; a
    window wider than the rows is refused, and the graph launches again after a longer camera."""
    n_img, W = 9, 6
    wave, off, tel, evt, h, st = camera_case(np.random.default_rng(3), n_img, 2048, 128)
    ctx = rta.Context(0)
    register(ctx, 264, 9)
    n_d = torch.tensor([n_img], dtype=torch.int64, device="cuda")
    args = (mode, 0, W, 3.0, 1.5, 1)
    g = rta.rta_graph_create(ctx.handle, wave.data_ptr(), wave.numel(), off.data_ptr(), tel.data_ptr(), n_d.data_ptr(),
                             n_img, evt.data_ptr(), n_d.data_ptr(), n_img, *args, h.data_ptr(), st.data_ptr())
    stream = torch.cuda.current_stream().cuda_stream
    try:
        for P, S in [(264, 9), (264, 128), (2048, 31), (1000, 5), (1000, 40), (2048, 40), (264, 30), (520, 128)]:
            torch.cuda.synchronize()
            register(ctx, P, S)
            off.copy_(torch.arange(n_img, device="cuda") * (P * S))
            if S < W:
                with pytest.raises(rta.RtaError) as e:
                    rta.rta_graph_launch(g, stream)
                assert e.value.code == rta.RTA_E_INVALID
                continue
            ref, ref_st = torch.zeros_like(h), torch.zeros_like(st)
            ctx.reconstruct(wave, off, tel, evt, *args, ref, ref_st)
            h.fill_(float("nan"))
            rta.rta_graph_launch(g, stream)
            assert ctx.check(stream) == 0
            assert torch.equal(h.view(torch.int32), ref.view(torch.int32)), (P, S)
            assert torch.equal(st.view(torch.int32), ref_st.view(torch.int32)), (P, S)
            assert int(h.view(torch.int32).view(n_img, 16)[:, 10].min()) > 0
    finally:
        rta.rta_graph_destroy(g)
    ctx.close()


@pytest.mark.parametrize("mode,start,W", [(rta.RTA_WINDOW_SLIDING, 0, 6), (rta.RTA_WINDOW_FIXED, 20, 6),
                                          (rta.RTA_WINDOW_NEIGHBOUR, 0, 6)])
def test_a_capture_flags_images_that_it_was_not_set_up_for(mode, start, W):
    """A caller's capture replayed after the camera came back larger than its shared memory, with rows
    too long for its stages or too short for the window: every image is flagged and none read;
    once the camera is the old one again the rows are too. More pixels than the telescope has
    calibration rows for are flagged by direct calls as well."""
    n_img = 9
    wave, off, tel, evt, h, st = camera_case(np.random.default_rng(4), n_img, 520, 128)
    ctx = rta.Context(0)
    S0 = 30 if mode == rta.RTA_WINDOW_FIXED else 9
    register(ctx, 264, S0)
    off.copy_(torch.arange(n_img, device="cuda") * (264 * S0))
    args = (mode, start, W, 3.0, 1.5, 1)
    first, first_st = torch.zeros_like(h), torch.zeros_like(st)
    ctx.reconstruct(wave, off, tel, evt, *args, first, first_st)
    assert ctx.check() == 0
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.reconstruct(wave, off, tel, evt, *args, h, st)

    def flagged(call):
        h.fill_(float("nan"))
        call()
        torch.cuda.synchronize()
        with pytest.raises(rta.RtaError) as e:
            ctx.check()
        assert e.value.code == rta.RTA_E_DEVICE and e.value.bits == rta.RTA_DEV_BAD_IMAGE
        rows = rta.hillas_to_numpy(h.cpu().numpy())
        assert (rows["flags"] & rta.RTA_HF_BAD_INPUT).all() and (rows["n_pix"] == 0).all()

    for P, S in [(520, S0), (264, 24 if mode == rta.RTA_WINDOW_FIXED else 5)] + ([(264, 128)] if S0 == 9 else []):
        torch.cuda.synchronize()
        register(ctx, P, S, array=False)
        flagged(g.replay)
        if P > 264:
            flagged(lambda: ctx.reconstruct(wave, off, tel, evt, *args, h, st))
    register(ctx, 264, S0, array=False)
    g.replay()
    torch.cuda.synchronize()
    assert ctx.check() == 0
    assert torch.equal(h.view(torch.int32), first.view(torch.int32))
    assert torch.equal(st.view(torch.int32), first_st.view(torch.int32))
    ctx.close()
