"""Values below the normal FP32 range (2^-126) count like any others in the splat and the chain:
upstream gradients, quaternions whose squared norm is subnormal, and weights near a w_min there."""
import math

import numpy as np
import pytest

from paper_2412_03451_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _room():
    from paper_2412_03451_gb300 import splat as SP
    room = S.tiny_room(0)
    p = S.perturb_planes(room.gt, 1)
    V, H, W = room.cams.V, room.cams.H, room.cams.W
    r = SP.Renderer([H] * V, [W] * V, [0] * V, [0, p.K])
    r.set_cameras(room.cams.w2c, room.cams.intr)
    flat = SP.planes_to_flat(p.center, p.quat, p.radii, "cuda")
    r.ensure_capacity(flat, 20.0)
    return r, flat, V * H * W


def _grad(r, flat, gD, gN):
    import torch
    r.forward(flat, 20.0)
    g = torch.zeros_like(flat)
    r.backward(flat, g, gD, gN)
    return g.double()


def test_subnormal_upstream_gradient():
    import torch
    r, flat, n = _room()
    gD, gN = torch.ones(n, device="cuda"), torch.zeros(n, 3, device="cuda")
    want = _grad(r, flat, gD, gN)
    s = 2.0 ** -127
    got = _grad(r, flat, gD * s, gN * s) / s
    # global atomics take a warp's sum below 2^-126, here 2, as zero; the sums of up to 32 pixels
    # of one sign with factors t - A of metres and 5 lambda = 100 are mostly far above
    assert float((got - want).norm() / want.norm()) < 0.05


def test_quaternion_with_a_subnormal_squared_norm():
    import torch
    from paper_2412_03451_gb300 import splat as SP
    r, flat, n = _room()
    P = r.P
    c, q, rad = SP.flat_views(flat, P)
    s = 2.0 ** -66
    q /= q.norm(dim=1, keepdim=True)
    tiny = flat.clone()
    SP.flat_views(tiny, P)[1].mul_(s)
    g = torch.Generator(device="cuda").manual_seed(2)
    gD, gN = torch.randn(n, device="cuda", generator=g), torch.randn(n, 3, device="cuda", generator=g)
    want, got = _grad(r, flat, gD, gN), _grad(r, tiny, gD, gN)
    got[3 * P:7 * P] *= s
    # |q|^2 = 2^-132 carries 17 bits, so the axes are 2^-18 off a unit length; steep weights
    # (5 lambda = 100) and flipped pixels make more of that, nowhere near the whole gradient
    for lo, hi in ((0, 3 * P), (3 * P, 7 * P), (7 * P, 11 * P)):
        assert float((got[lo:hi] - want[lo:hi]).norm() / want[lo:hi].norm()) < 0.05


def test_weights_below_a_subnormal_w_min_are_no_candidates():
    import torch
    from paper_2412_03451_gb300 import binding as B, splat as SP
    H, W, f, lam, w_min = 16, 1024, 1000.0, 20.0, 1e-39
    # plane 0 in front ends at P_X = -0.45, plane 1 behind covers everything; with M = 1 a candidate
    # of any weight hides the plane behind it
    z = np.float32([2.0, 3.0])
    r = SP.Renderer([H], [W], [0], [0, 2], M=1)
    make = r.make_settings

    def settings(*a, **kw):
        s = make(*a, **kw)
        s.w_min, s.delta = w_min, B.filter_margin(lam, w_min)
        return s

    r.make_settings = settings
    r.set_cameras(np.eye(3, 4, dtype=np.float32)[None], np.float32([[f, f, W / 2, H / 2]]))
    radii = np.float32([[0.1, 0.1, 2, 2], [9, 9, 9, 9]])
    flat = SP.planes_to_flat(np.float32([[0, 0, z[0]], [0, 0, z[1]]]), np.float32([[1, 0, 0, 0]] * 2), radii, "cuda")
    r.ensure_capacity(flat, lam)
    depth, _ = r.forward(flat, lam)
    D = depth.cpu().numpy().reshape(H, W).astype(np.float64)
    X = z[0] * (np.arange(W) + 0.5 - W / 2) / f
    m = 0.1 - np.abs(X)
    w = np.minimum(1.0, 2 / (1 + np.exp(np.minimum(-5 * lam * m, 700))))
    below, above = w < 0.98 * w_min, w > 1.02 * w_min
    # (a binned tile beside the last candidates holds both planes)
    near = below & (w > 1e-3 * w_min)
    assert near.sum() >= 4 and (above & (w < 1e-38)).sum() >= 1
    assert np.allclose(D[:, below], z[1], rtol=1e-6)
    assert np.allclose(D[:, above], np.broadcast_to(z[0] * w[above], (H, int(above.sum()))), rtol=1e-4, atol=1e-43)
