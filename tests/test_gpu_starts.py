"""Initial radii of Sec. 3.1 on the device: ps_nn_distance against brute force.

The nearest-other-point distance of every point is checked against an all-pairs
FP64 computation on the host (relative 1e-6: the kernel works in FP32) on point
sets shaped like plane starts (points on the faces of a room, many on one plane,
exact duplicates, a lone far point, a single point), and the two starts that use
it are checked for their seeded content.
"""
import numpy as np
import pytest

from paper_2412_03451_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def brute_nn(p):
    p = p.astype(np.float64)
    d2 = ((p[:, None, :] - p[None, :, :]) ** 2).sum(-1)
    np.fill_diagonal(d2, np.inf)
    return np.sqrt(d2.min(1))


def gpu_nn(p):
    import torch
    from paper_2412_03451_gb300 import binding as B
    t = torch.from_numpy(p.astype(np.float32)).cuda()
    d = torch.empty(len(p), dtype=torch.float32, device="cuda")
    B.ps_nn_distance(t, dist=d)
    torch.cuda.synchronize()
    return d.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("case", ["room", "plane", "duplicates", "outlier", "clusters"])
def test_nn_distance_matches_brute_force(case):
    rng = np.random.default_rng(5)
    if case == "room":
        room = S.large_room(1010, n_rect=600, n_views=4)
        p = S.surface_init(room, 3000, 11).center
    elif case == "plane":
        p = np.concatenate([rng.uniform(-2, 2, (2000, 2)), np.full((2000, 1), 1.5)], 1)
    elif case == "duplicates":
        p = rng.uniform(0, 1, (500, 3))
        p = np.concatenate([p, p[:50]])
    elif case == "outlier":
        p = np.concatenate([rng.uniform(0, 1, (999, 3)), [[40.0, -30.0, 25.0]]])
    else:
        c = rng.uniform(-5, 5, (20, 3))
        p = (c[:, None, :] + 0.01 * rng.normal(size=(20, 100, 3))).reshape(-1, 3)
    p = p.astype(np.float32)
    ref = brute_nn(p)
    got = gpu_nn(p)
    assert np.allclose(got, ref, rtol=1e-6, atol=1e-7), np.max(np.abs(got - ref) / np.maximum(ref, 1e-30))
    if case == "duplicates":
        assert (got[:50] == 0).all()


def test_nn_distance_single_point_and_radii():
    import torch
    from paper_2412_03451_gb300 import starts
    assert np.isinf(gpu_nn(np.zeros((1, 3), np.float32)))[0]
    rng = np.random.default_rng(6)
    p = rng.uniform(0, 3, (777, 3)).astype(np.float32)
    r = starts.nn_radii(torch.from_numpy(p).cuda(), scale=0.5).cpu().numpy()
    ref = np.clip(0.5 * brute_nn(p), starts.R_LO, starts.R_HI)
    assert r.shape == (777, 4) and (r == r[:, :1]).all()
    assert np.allclose(r[:, 0], ref, rtol=1e-6, atol=1e-7)


def test_mono_start_is_seeded_and_matches_host_radii():
    from paper_2412_03451_gb300 import starts
    from oracle import oracle as O
    room = S.large_room(1011, n_rect=600, n_views=4)
    c = room.cams
    D, N, _ = O.raycast(room.gt.center, room.gt.quat, room.gt.radii, c.w2c, c.intr, c.H, c.W)
    a = starts.mono_start(room, D, N, 1500, 3)
    b = starts.mono_start(room, D, N, 1500, 3)
    assert np.array_equal(a.center, b.center) and np.array_equal(a.quat, b.quat)
    assert np.array_equal(a.radii, b.radii)
    host = S.mono_init(room, D, N, 1500, 3)
    assert np.array_equal(a.center, host.center) and np.array_equal(a.quat, host.quat)
    assert np.allclose(a.radii, host.radii, rtol=1e-6, atol=1e-7)
    # centres lie near the ground-truth surfaces seen by the views (degraded depth: a few %)
    assert np.isfinite(a.center).all() and (a.radii > 0).all()


@pytest.mark.parametrize("n", [2, 7, 9, 1024, 1025, 10000, 10001, 20011])
def test_nn_distance_sizes(n):
    # one CTA's queries, one chunk of points and both sides of the all-pairs limit, on a thin slab
    # with a lone far point (many shells); FP32 squares against FP64 distances
    from scipy.spatial import cKDTree
    rng = np.random.default_rng(n)
    p = (rng.uniform(0, 1, (n, 3)) * [4.0, 5.0, 0.01]).astype(np.float32)
    p[n // 2] = [9.0, -7.0, 6.0]
    ref = cKDTree(p.astype(np.float64)).query(p.astype(np.float64), k=2)[0][:, 1]
    assert np.allclose(gpu_nn(p), ref, rtol=1e-6, atol=1e-7)
