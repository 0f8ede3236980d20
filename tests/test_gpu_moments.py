"""The eight-float gradient accumulators of the splat kernels (rectangle weight).

The gradient of a record's a_x is taken as that of r^x+ less that of r^x-, which
holds for every pair but one at P = 0 exactly (sgn(0) = 0): the radius moves there
and the plane's centre does not.  m < 0 at P = 0 needs a negative radius, which the
entry points accept.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("single", [False, True])
@pytest.mark.parametrize("axis", [0, 1])
def test_pair_on_the_axis_moves_its_radius_only(axis, single):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_03451_gb300 import binding as B, splat as SP
    H = W = 33
    lam, t, rneg = 20.0, 2.0, -0.01
    radii = np.full(4, 0.6, np.float32)
    radii[2 * axis + (0 if single else 1)] = rneg          # P = 0 takes the - side
    r = SP.Renderer([H], [W], [0], [0, 1], flags=B.PS_SINGLE_RADII if single else 0)
    w2c = np.concatenate([np.eye(3), np.zeros((3, 1))], 1).astype(np.float32)[None]
    r.set_cameras(w2c, np.array([[100.0, 100.0, 16.5, 16.5]], np.float32))
    flat = SP.planes_to_flat(np.array([[0, 0, t]]), np.array([[1, 0, 0, 0]]), radii[None], "cuda")
    r.ensure_capacity(flat, lam)
    # upstream on the pixels of the plane's own axis alone (column or row 16), whose rays have P = 0
    gD = torch.zeros(H, W, device="cuda")
    if axis == 0:
        gD[8:25, 16] = 1.0
    else:
        gD[16, 8:25] = 1.0
    r.forward(flat, lam)
    g = torch.zeros_like(flat)
    r.backward(flat, g, gD.reshape(-1), torch.zeros(H * W, 3, device="cuda"))
    g = g.cpu().numpy().astype(np.float64)
    x = 5 * lam * rneg
    w = 2 / (1 + math.exp(-x))
    want = 17 * t * 5 * lam * w * (1 - w / 2)              # dD/dr = t dw/dm at 17 pixels
    gc, gr = g[:3], g[7:]
    moved = 2 * axis + (0 if single else 1)
    # one exp, one division and a handful of FP32 products per pixel
    assert abs(gr[moved] - want) <= 1e-5 * want
    assert np.all(np.delete(gr, moved) == 0.0)
    assert gc[axis] == 0.0
    # the pixels lie symmetrically about the other axis and D = w t: only the depth moves
    assert abs(gc[2] - 17 * w) <= 1e-5 * 17 * w
