"""ps_fit_step returns an argument error before it launches anything: no gradient is cleared and the
schedule does not advance."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2412_03451_gb300 import binding as B, scenes as S, splat as SP

# field (None: settings) -> bad values: NULL, misaligned, too small
FUSED = [("rec", 0), ("rec", "+4"), ("rect", 0), ("rect", "+4"), ("key", 0), ("tile_ptr", 0), ("tile_ent", 0), ("tile_key", 0),
         ("capacity", -1), ("capacity", 2 ** 31), ("d_required", 0), ("bin_ws", 0), ("bin_ws", "+16"),
         ("bin_ws_bytes", 64), ("bwd_ws", 0), ("bwd_ws", "+4"), ("bwd_ws_bytes", 64), ("gt_depth", 0),
         ("gt_normal", 0), ("view_sums", 0)]
SEPARATE = [x for x in FUSED if x[0] != "bwd_ws_bytes"] + [
    ("bwd_ws_bytes", 8), ("fwd_ws", 0), ("fwd_ws", "+4"), ("fwd_ws_bytes", 8), ("depth", 0), ("normal", 0), ("dL_dD", 0),
    ("dL_dN", 0)]
SETTINGS = [("flags", B.PS_HARD), ("M", 0), ("M", B.PS_MAX_M + 1), ("tile_w", 12), ("cta_warps", 3), ("z_near", 0.0),
            ("z_far", 0.005), ("w_min", 0.0), ("w_min", 1.0)]
CASES = ([(True, *x) for x in FUSED] + [(False, *x) for x in SEPARATE] +
         [(f, "settings." + k, v) for f in (True, False) for k, v in SETTINGS])


def spoil(buf, settings, field, bad):
    obj, name = (settings, field[9:]) if field.startswith("settings.") else (buf, field)
    setattr(obj, name, getattr(obj, name) + int(bad) if isinstance(bad, str) else bad)


@pytest.mark.parametrize("fused, field, bad", CASES)
def test_refused_on_the_host(fused, field, bad):
    if torch.cuda.is_available():
        pytest.skip("placeholder pointers: for a machine without a GPU, where a launch fails as such")
    _, frame = B.ps_plan_views([96], [128], [0], [0, 4], np.eye(3, 4, dtype=np.float32)[None],
                               np.array([[100, 100, 64, 48]], np.float32), 16, 16)
    frame.views = 256
    buf = B.PsFitBuffers(**{k: 1 << 20 for k, t in B.PsFitBuffers._fields_ if t is ctypes.c_void_p})
    buf.split_acc = buf.split_scale = None
    buf.capacity, buf.bin_ws_bytes, buf.fwd_ws_bytes, buf.bwd_ws_bytes, buf.n_sched = 1000, 1 << 20, 1 << 20, 1 << 20, 3
    s = B.make_settings(20.0, B.filter_margin(20.0))
    call = lambda: B.load().ps_fit_step(4, ctypes.byref(frame), ctypes.byref(s), ctypes.byref(buf), int(fused),
                                        1e-3, 0.9, 0.999, 1e-8, 1e-4, 1, None)
    assert call() == B.PS_ERR_CUDA                      # accepted: it gets as far as a launch
    spoil(buf, s, field, bad)
    assert call() == B.PS_ERR_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("fused", [True, False])
def test_refused_step_changes_nothing(fused):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    room = S.tiny_room(0)
    p = S.perturb_planes(room.gt, 1)
    V, H, W = room.cams.V, room.cams.H, room.cams.W
    r = SP.Renderer([H] * V, [W] * V, [0] * V, [0, p.K])
    r.set_cameras(room.cams.w2c, room.cams.intr)
    flat = SP.planes_to_flat(p.center, p.quat, p.radii, "cuda")
    r.ensure_capacity(flat, 20.0)
    fit = SP.Fitter(r, flat, fused=fused)
    fit.grad.fill_(9.0)
    fit.d_state = torch.full((32,), 7, dtype=torch.uint8, device="cuda")
    fit.d_sched = torch.frombuffer(bytearray(B.step_schedule(4)), dtype=torch.uint8).cuda()
    fit.d_iter = torch.tensor([1], dtype=torch.int32, device="cuda")
    gd, gn = torch.ones(V * H * W, device="cuda"), torch.zeros(V * H * W, 3, device="cuda")
    r.view_sums.fill_(5.0)
    r.rec.fill_(3.0)
    real, todo = B.ps_fit_step, [c for c in CASES if c[0] == fused]
    bad = []

    def spoiled(n, frame, settings, buf, *rest):
        spoil(buf, settings, *todo[len(bad)][1:])
        real(n, frame, settings, buf, *rest)

    B.ps_fit_step = spoiled
    try:
        for _ in todo:
            with pytest.raises(B.PsError):
                fit._library_step(r.make_settings(20.0), gd, gn, r.view_sums, 0, fused,
                                  (fit.d_state, fit.d_sched, 4, fit.d_iter))
            bad.append(0)
    finally:
        B.ps_fit_step = real
    torch.cuda.synchronize()
    assert int(fit.d_iter) == 1 and bool((fit.d_state == 7).all())
    assert bool((fit.grad == 9.0).all()) and bool((r.view_sums == 5.0).all()) and bool((r.rec == 3.0).all())
    assert torch.equal(fit.flat, SP.planes_to_flat(p.center, p.quat, p.radii, "cuda"))
