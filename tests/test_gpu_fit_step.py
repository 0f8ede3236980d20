"""ps_fit_step: one call per optimisation step against the separate calls, and the autograd
forward's growth of its tile lists."""
import numpy as np
import pytest

from paper_2412_03451_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _case(flags=0, seed=1, **kw):
    from paper_2412_03451_gb300 import splat as SP
    room = S.tiny_room(0)
    p = S.perturb_planes(room.gt, seed)
    V, H, W = room.cams.V, room.cams.H, room.cams.W
    r = SP.Renderer([H] * V, [W] * V, [0] * V, [0, p.K], flags=flags, **kw)
    r.set_cameras(room.cams.w2c, room.cams.intr)
    return r, SP.planes_to_flat(p.center, p.quat, p.radii, "cuda"), V * H * W


@pytest.mark.parametrize("fused", [True, False])
@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("flags", [0, 1, 4])                   # rectangle, single radii, Eq. 5
def test_step_equals_separate_calls(fused, split, flags):
    import torch
    from paper_2412_03451_gb300 import binding as B, splat as SP
    out = []
    for marks in (None, []):                                   # marks: stage by stage
        r, flat, n = _case(flags)
        flat[7 * r.P:7 * r.P + 4] = 0.5 * SP.R_MIN              # below the clamp of the radii
        g = torch.Generator(device="cuda").manual_seed(5)
        gd = torch.rand(n, device="cuda", generator=g) + 1
        gn = torch.randn(n, 3, device="cuda", generator=g)
        r.ensure_capacity(flat, 20.0)
        fit = SP.Fitter(r, flat, fused=fused)
        if split:
            fit.enable_split([torch.rand(r.P, device="cuda", generator=g) for _ in range(2)])
        fit.ite = 3
        before = flat.clone()
        sums = fit.step(gd, gn, lam=20.0, marks=marks, batch=1)
        assert fit.ite == 4 and sums is r.view_sums and int(r.status.item()) == 0
        # Adam on the step's own gradient, the two groups apart: the same bits
        p, m, v, k = before, torch.zeros_like(flat), torch.zeros_like(flat), 7 * r.P
        for s, lo in ((slice(0, k), float("nan")), (slice(k, None), SP.R_MIN)):
            B.ps_adam_step(p[s], fit.grad[s], m[s], v[s], fit.lr, fit.b1, fit.b2, fit.eps, 4, clamp_min=lo)
        assert torch.equal(p, flat) and torch.equal(m, fit.m) and torch.equal(v, fit.v)
        assert float(flat[k:].min()) >= np.float32(SP.R_MIN)
        out.append((fit.grad.clone(), sums.clone(), r.depth.clone(), None if not split else fit.split_acc.clone()))
    (g0, s0, d0, a0), (g1, s1, d1, a1) = out
    # the same kernels, whose atomic sums differ in order between any two runs
    assert float((g0 - g1).norm() / g1.norm()) < 1e-5 and float(g1.norm()) > 0
    assert torch.allclose(s0, s1, rtol=1e-6) and torch.equal(d0, d1)
    if split:
        assert float((a0 - a1).norm() / a1.norm()) < 1e-5 and float(a1.norm()) > 0


@pytest.mark.parametrize("capacity", [1, 100, 1 << 16])
def test_autograd_grows_its_lists(capacity):
    import torch
    from paper_2412_03451_gb300 import splat as SP
    ref, flat, n = _case()
    ref.ensure_capacity(flat, 20.0)
    want = [x.clone() for x in ref.forward(flat, 20.0)]
    r, flat, n = _case(capacity=capacity)
    flat.requires_grad_(True)
    D, N = SP.PlaneSplatFunction.apply(flat, r, 20.0)
    assert torch.equal(D, want[0]) and torch.equal(N, want[1])
    assert r.capacity >= int(r.required.item()) and int(r.status.item()) == 0
    g = torch.zeros_like(ref.depth).normal_(generator=torch.Generator(device="cuda").manual_seed(2))
    (got,) = torch.autograd.grad([D], [flat], [g])
    exp = torch.zeros_like(got)
    ref.backward(flat.detach(), exp, g, torch.zeros(n, 3, device="cuda"))
    assert float((got - exp).norm() / exp.norm()) < 1e-5 and float(exp.norm()) > 0


def test_step_with_empty_scenes_and_scenes_without_views():
    # the chain finds a plane's records by its scene's views: more views than lanes per plane, a
    # scene with a view but no planes, planes that no view sees, one view, a trailing empty scene
    import torch
    from paper_2412_03451_gb300 import splat as SP
    room = S.tiny_room(0)
    p = S.perturb_planes(room.gt, 1)
    views = [0, 1, 2, 3, 4, 5, 6, 7, 0, 1, 2]
    K, ptr = 32, [0, 5, 5, 12, 32, 32]
    H, W = room.cams.H, room.cams.W
    n = len(views) * H * W
    g = torch.Generator(device="cuda").manual_seed(5)
    gd, gn = torch.rand(n, device="cuda", generator=g) + 1, torch.randn(n, 3, device="cuda", generator=g)
    out = []
    for marks in (None, []):
        r = SP.Renderer([H] * len(views), [W] * len(views), [0] * 9 + [1] + [3], ptr)
        r.set_cameras(room.cams.w2c[views], room.cams.intr[views])
        flat = SP.planes_to_flat(p.center[:K], p.quat[:K], p.radii[:K], "cuda")
        r.ensure_capacity(flat, 20.0)
        fit = SP.Fitter(r, flat)
        fit.grad.fill_(9.0)
        sums = fit.step(gd, gn, lam=20.0, marks=marks)
        out.append((fit.grad, fit.m, sums))
    (g0, m0, s0), (g1, m1, s1) = out
    gc = SP.flat_views(g0, K)
    assert all(float(x[5:12].abs().max()) == 0.0 for x in gc) and float(gc[0][:5].abs().sum()) > 0
    assert float(gc[0][12:].abs().sum()) > 0
    assert float((g0 - g1).norm() / g1.norm()) < 1e-5 and float((m0 - m1).norm() / m1.norm()) < 1e-5
    assert torch.allclose(s0, s1, rtol=1e-6)
