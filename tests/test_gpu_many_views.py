"""Frames of few and of many views: the tile's view is found at the edges of the warp search's
steps, and the whole step agrees with the separate calls on both sides of its chain's rule."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _renderer(V, K=1, flags=0, side=8):
    """View v of V looks along z from 0.25 (v % 64) behind the origin; sizes differ between views."""
    from paper_2412_03451_gb300 import splat as SP
    H, W = [side + 8 * (v % 3) for v in range(V)], [side + 8 * (v % 2) for v in range(V)]
    r = SP.Renderer(H, W, [0] * V, [0, K], tile=(8, 8), flags=flags)
    w2c = np.tile(np.eye(3, 4, dtype=np.float32), (V, 1, 1))
    w2c[:, 2, 3] = 0.25 * (np.arange(V) % 64)
    r.set_cameras(w2c, np.stack([np.float32([40, 40, w / 2, h / 2]) for h, w in zip(H, W)]))
    return r, H, W


@pytest.mark.parametrize("flags", [0, 2])                     # general walk, hard edge
@pytest.mark.parametrize("V", [1, 31, 32, 33, 64, 1023, 1024, 1025, 2500])
def test_every_tile_finds_its_view(V, flags):
    from paper_2412_03451_gb300 import splat as SP
    r, H, W = _renderer(V, flags=flags)
    flat = SP.planes_to_flat(np.float32([[0, 0, 2]]), np.float32([[1, 0, 0, 0]]), np.full((1, 4), 50, np.float32), "cuda")
    r.ensure_capacity(flat, 300.0)
    depth, _ = r.forward(flat, 300.0)
    want = np.repeat(2 + 0.25 * (np.arange(V) % 64), np.multiply(H, W)).astype(np.float32)
    assert np.array_equal(depth.cpu().numpy(), want)          # exact: n_c . p_c over 1


@pytest.mark.parametrize("flags", [0, 4])
@pytest.mark.parametrize("V", [127, 128, 300])
def test_step_on_both_sides_of_the_chain_rule(V, flags):
    import torch
    from paper_2412_03451_gb300 import splat as SP
    K = 13
    rng = np.random.default_rng(V)
    c = np.stack([rng.uniform(-0.3, 0.3, K), rng.uniform(-0.3, 0.3, K), rng.uniform(1.5, 3.0, K)], 1).astype(np.float32)
    q = (rng.normal(size=(K, 4)) * [1.5, 0.3, 0.3, 0.8]).astype(np.float32)
    out = []
    for marks in (None, []):                                  # marks: stage by stage
        r, H, W = _renderer(V, K, flags, side=16)
        flat = SP.planes_to_flat(c, q, np.full((K, 4), 0.3, np.float32), "cuda")
        r.ensure_capacity(flat, 20.0)
        fit = SP.Fitter(r, flat)
        fit.enable_split([torch.full((K,), 0.5, device="cuda")])
        fit.grad.fill_(9.0)
        g = torch.Generator(device="cuda").manual_seed(1)
        n = int(np.multiply(H, W).sum())
        sums = fit.step(torch.rand(n, device="cuda", generator=g) + 2, torch.randn(n, 3, device="cuda", generator=g),
                        lam=20.0, marks=marks)
        assert int(r.status.item()) == 0
        out.append((fit.grad, fit.m, fit.v, fit.split_acc, sums.float()))
    # the same kernels up to the order in which the views are added
    for a, b in zip(*out):
        assert float((a - b).norm() / b.norm()) < 1e-5 and float(b.norm()) > 0
