"""A launch that the runtime refuses is reported by the call that made it and by no later one."""
import numpy as np
import pytest

from paper_2412_03451_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def test_refused_launch_is_not_reported_twice():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_03451_gb300 import binding as B, splat as SP
    V = 65536                                          # a grid's y extent ends at 65,535
    r = SP.Renderer([8] * V, [8] * V, [0] * V, [0, 1], tile=(8, 8), capacity=1 << 18)
    r.set_cameras(np.tile(np.eye(3, 4, dtype=np.float32), (V, 1, 1)), np.tile(np.float32([8, 8, 4, 4]), (V, 1)))
    flat = SP.planes_to_flat(np.float32([[0, 0, 2]]), np.float32([[1, 0, 0, 0]]), np.full((1, 4), 0.1, np.float32), "cuda")
    n = V * 64
    with pytest.raises(B.PsError, match="CUDA error"):
        SP.Fitter(r, flat).step(torch.ones(n, device="cuda"), torch.zeros(n, 3, device="cuda"), lam=20.0)
    room = S.tiny_room(0)
    p = S.perturb_planes(room.gt, 1)
    V, H, W = room.cams.V, room.cams.H, room.cams.W
    r = SP.Renderer([H] * V, [W] * V, [0] * V, [0, p.K])
    r.set_cameras(room.cams.w2c, room.cams.intr)
    flat = SP.planes_to_flat(p.center, p.quat, p.radii, "cuda")
    r.ensure_capacity(flat, 20.0)
    depth, _ = r.forward(flat, 20.0)
    torch.cuda.synchronize()
    assert float(depth.max()) > 0
