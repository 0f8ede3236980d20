"""Edges of the splat and loss kernels: views past one warp's search, pixel quads cut by odd
image sizes and buffer offsets, and depth bounds tightened to a strip."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2412_03451_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("shift", [(0, 0), (1, 0), (0, 3)])
@pytest.mark.parametrize("gt_shift", [0, 2, 4])
def test_loss_quads_and_remainders(shift, gt_shift):
    # views that start at every pixel offset modulo 4, buffers one or three floats past a 16-byte
    # boundary, supervision 0, 2 or 4 pixels further along than the maps
    import torch
    from paper_2412_03451_gb300 import binding as B, splat as SP
    sizes = [(3, 5), (1, 1), (2, 9), (7, 13), (1, 2), (9, 1), (16, 20)]
    H, W = [h for h, _ in sizes], [w for _, w in sizes]
    V, n = len(sizes), sum(h * w for h, w in sizes)
    rng = np.random.default_rng(7)
    D, Dg = rng.uniform(1, 3, n).astype(np.float32), rng.uniform(1, 3, n).astype(np.float32)
    N, Ng = (rng.normal(size=(n, 3)).astype(np.float32) for _ in range(2))
    Dg[rng.random(n) < 0.2] = 0.0
    Dg[3:6] = D[3:6]                                              # sgn(0) = 0
    r = SP.Renderer(H, W, [0] * V, [0, 1])
    eye = np.tile(np.eye(3, 4, dtype=np.float32), (V, 1, 1))
    intr = np.tile(np.array([10, 10, 5, 5], np.float32), (V, 1))
    off = np.concatenate([[0], np.cumsum([h * w for h, w in sizes])])
    r.preplan([eye], [intr], [off[:-1] + gt_shift])
    r.make_settings(20.0)

    def at(a, s, lead=0):
        flat = np.asarray(a, np.float32).reshape(-1)
        buf = torch.full((s + lead + flat.size + 8,), float("nan"), device="cuda")
        buf[s + lead:s + lead + flat.size] = torch.from_numpy(flat).cuda()
        return buf[s:]

    s_map, s_gt = shift
    d, nn = at(D, s_map), at(N, s_map)
    gd, gn = at(Dg, s_gt, gt_shift), at(Ng, s_gt, 3 * gt_shift)
    oD, oN = at(np.full(n, np.nan), s_map), at(np.full(3 * n, np.nan), s_map)
    sums = torch.full((V, 4), 7.0, dtype=torch.float64, device="cuda")
    B.ps_loss(r.frame, r.settings, d, nn, gd, gn, oD, oN, sums)
    oD, oN, sums = oD.cpu().numpy(), oN.cpu().numpy(), sums.cpu().numpy()
    assert np.isnan(oD[n:]).all() and np.isnan(oN[3 * n:]).all()   # nothing past the maps
    for v, (h, w) in enumerate(sizes):
        p = slice(off[v], off[v + 1])
        _, rD, rN, rs = O.loss(D[p].reshape(1, h, w), N[p].reshape(1, h, w, 3),
                               Dg[p].reshape(1, h, w), Ng[p].reshape(1, h, w, 3))
        assert np.array_equal(oD[p], rD.astype(np.float32).reshape(-1)), v
        assert np.abs(oN[3 * off[v]:3 * off[v + 1]].reshape(-1, 3) - rN.reshape(-1, 3)).max() < 1e-5, v
        assert np.allclose(sums[v], rs[0], rtol=1e-5), v


@pytest.mark.parametrize("V", [31, 32, 33, 64, 65])
def test_views_past_one_search_step(V):
    import torch
    from paper_2412_03451_gb300 import splat as SP
    p = S.random_planes_in_view(3, 30, depth_range=(1.0, 3.0), half=(0.2, 0.6))
    cams = S.identity_cameras(V, 24, 40, 30.0, seed=1, jitter=0.1)
    flat = SP.planes_to_flat(p.center, p.quat, p.radii, "cuda")

    def maps(views):
        k = len(views)
        r = SP.Renderer([24] * k, [40] * k, [0] * k, [0, p.K])
        r.set_cameras(cams.w2c[views], cams.intr[views])
        r.ensure_capacity(flat, 20.0)
        D, N = r.forward(flat, 20.0)
        return D.view(k, -1), N.view(k, -1)

    D, N = maps(list(range(V)))
    assert float(D.abs().sum()) > 0
    for v in sorted({0, 1, 30, V // 2, V - 2, V - 1}):
        d1, n1 = maps([v])
        assert torch.equal(D[v], d1[0]) and torch.equal(N[v], n1[0]), v


@pytest.mark.parametrize("lists", [20, 200])
def test_gauss_maps_do_not_depend_on_the_tile(lists):
    # the composited pairs are exact whatever bounds the walk has: planes at every tilt, some seen
    # edge on, lists of one chunk and of several
    import torch
    from paper_2412_03451_gb300 import binding as B, splat as SP
    p = S.random_planes_in_view(lists, lists, depth_range=(0.3, 3.0), half=(0.1, 0.8))
    p.quat[::5] = np.float32([np.sqrt(0.5), np.sqrt(0.5), 0, 0])    # normal along y: edge on at mid height
    cams = S.identity_cameras(2, 45, 83, 40.0, seed=2, jitter=0.1)
    flat = SP.planes_to_flat(p.center, p.quat, p.radii, "cuda")
    out = []
    for tile in ((8, 8), (16, 16), (32, 8)):
        r = SP.Renderer([45] * 2, [83] * 2, [0] * 2, [0, p.K], tile=tile, flags=B.PS_GAUSSIAN)
        r.set_cameras(cams.w2c, cams.intr)
        r.ensure_capacity(flat, 20.0)
        out.append([x.clone() for x in r.forward(flat, 20.0)])
        assert int(r.status.item()) == 0
    assert float(out[0][0].abs().sum()) > 0
    for D, N in out[1:]:
        assert torch.equal(D, out[0][0]) and torch.equal(N, out[0][1])


@pytest.mark.parametrize("tile", [(8, 8), (16, 16), (32, 8)])
@pytest.mark.parametrize("V,warps,K", [(1, 0, 150), (5, 2, 150), (13, 8, 150), (27, 0, 150), (27, 0, 6)])
def test_hard_maps_by_groups_of_strips(tile, V, warps, K):
    # the more views, the more strips of a tile per work item (1, 2, 4 or 8); lists of one chunk and
    # of several, a ragged image, pixels without any plane; each view against its own render
    import torch
    from paper_2412_03451_gb300 import binding as B, splat as SP
    p = S.random_planes_in_view(17, K, depth_range=(0.3, 3.0), half=(0.05, 0.7))
    p.center[1], p.quat[1], p.radii[1] = p.center[0], p.quat[0], p.radii[0]     # a tie: the lower id
    h, w = 470, 629
    cams = S.identity_cameras(V, h, w, 400.0, seed=4, jitter=0.1)
    flat = SP.planes_to_flat(p.center, p.quat, p.radii, "cuda")

    def maps(views, **kw):
        k = len(views)
        r = SP.Renderer([h] * k, [w] * k, [0] * k, [0, p.K], flags=B.PS_HARD, **kw)
        r.set_cameras(cams.w2c[views], cams.intr[views])
        r.ensure_capacity(flat, 20.0)
        D, N = (x.clone() for x in r.forward(flat, 20.0))
        A = r.alpha.clone()
        ids, D2 = r.plane_ids(flat)
        assert torch.equal(D, D2) and torch.equal(A, (D > 0).float()) and torch.equal(ids >= 0, D > 0)
        assert int(r.status.item()) == 0 and not (ids == 1).any()
        return D.view(k, -1), N.view(k, -1), ids.view(k, -1)

    got = maps(list(range(V)), tile=tile, warps=warps)
    covered = float((got[0] > 0).float().mean())
    assert 0 < covered and (covered < 1 or K == 150)
    for v in sorted({0, V // 2, V - 1}):
        one = maps([v])
        for a, b in zip(got, one):
            assert torch.equal(a[v], b[0]), v
    # the nearest candidate by definition, in FP64, at sampled pixels away from edges and ties
    v, rng = V - 1, np.random.default_rng(3)
    D, ids = got[0][v].cpu().numpy(), got[2][v].cpu().numpy()
    K, T = cams.intr[v].astype(np.float64), cams.w2c[v].astype(np.float64)
    q = p.quat.astype(np.float64) / np.linalg.norm(p.quat, axis=1, keepdims=True)
    a, b, c, d = q.T
    vx = np.stack([1 - 2 * (c * c + d * d), 2 * (b * c + a * d), 2 * (b * d - a * c)], 1) @ T[:, :3].T
    vy = np.stack([2 * (b * c - a * d), 1 - 2 * (b * b + d * d), 2 * (c * d + a * b)], 1) @ T[:, :3].T
    n = np.cross(vx, vy)
    pc = p.center.astype(np.float64) @ T[:, :3].T + T[:, 3]
    checked = 0
    for x, y in zip(rng.integers(0, w, 400), rng.integers(0, h, 400)):
        ray = np.array([(x + 0.5 - K[2]) / K[0], (y + 0.5 - K[3]) / K[1], 1.0])
        den = n @ ray
        t = (n * pc).sum(1) / den
        o = t[:, None] * ray - pc
        X, Y = (o * vx).sum(1), (o * vy).sum(1)
        r = p.radii.astype(np.float64)
        m = np.minimum(np.where(X > 0, r[:, 0], r[:, 1]) - abs(X), np.where(Y > 0, r[:, 2], r[:, 3]) - abs(Y))
        near = (abs(den) > 1e-3) & (t > 0.02) & (t < 99)
        if (near & (abs(m) < 1e-3)).any() or (~near & (m > -1e-3)).any():
            continue
        hit = np.where(near & (m >= 0))[0]
        if len(hit) == 0:
            assert ids[y * w + x] == -1
        else:
            order = hit[np.argsort(t[hit], kind="stable")]
            gap = [k for k in order if t[k] > t[order[0]] + 1e-4]
            if len(order) - len(gap) > (2 if order[0] in (0, 1) else 1):
                continue
            assert ids[y * w + x] == order[0] and abs(D[y * w + x] - t[order[0]]) < 1e-4
        checked += 1
    assert checked > 100


@pytest.mark.parametrize("tile,warps", [((8, 8), 0), ((16, 16), 2), ((32, 8), 8)])
@pytest.mark.parametrize("K", [12, 150])
def test_grouped_strips_equal_single_views(tile, warps, K):
    # many strips per warp: the first go in groups of a tile's strips (lists of one chunk, K = 12,
    # stay staged from strip to strip; K = 150: several chunks), the last one by one; a view alone
    # has too few to group.  Forward, plane indices, fused and separate backward.
    import torch
    from paper_2412_03451_gb300 import splat as SP
    p = S.random_planes_in_view(K, K, depth_range=(0.4, 3.0), half=(0.1, 0.6))
    V, h, w = 16, 470, 629
    cams = S.identity_cameras(V, h, w, 400.0, seed=4, jitter=0.1)
    flat = SP.planes_to_flat(p.center, p.quat, p.radii, "cuda")
    n = h * w
    g = torch.Generator(device="cuda").manual_seed(1)
    gd, gn = torch.rand(V * n, device="cuda", generator=g) + 1, torch.randn(V * n, 3, device="cuda", generator=g)

    def run(views):
        k = len(views)
        r = SP.Renderer([h] * k, [w] * k, [0] * k, [0, p.K], tile=tile, warps=warps)
        r.set_cameras(cams.w2c[views], cams.intr[views])
        r.ensure_capacity(flat, 60.0)
        at = slice(views[0] * n, (views[-1] + 1) * n)
        D, N = (x.clone() for x in r.forward(flat, 60.0))
        ids, _ = r.plane_ids(flat, 60.0, hard=False)
        r.project_bin(flat, 60.0)
        fused, sep = torch.zeros_like(flat), torch.zeros_like(flat)
        sums = r.fused(flat, fused, gd[at], gn[at], write_maps=True).clone()
        assert torch.equal(r.depth, D) and torch.equal(r.normal, N)
        r.backward(flat, sep)                          # the fused walk's own dL/dD, dL/dN
        assert int(r.status.item()) == 0
        assert float((fused - sep).norm() / sep.norm()) < 1e-5
        return [D.view(k, -1), N.view(k, -1), ids.view(k, -1), sums], fused.double()

    got, grad = run(list(range(V)))
    total = torch.zeros_like(grad)
    for v in range(V):
        one, g1 = run([v])
        for a, b in zip(got[:3], one[:3]):
            assert torch.equal(a[v], b[0]), v
        assert torch.allclose(got[3][v], one[3][0], rtol=1e-6)
        total += g1
    # FP32 sums of the same pairs in another order
    assert float((grad - total).norm() / total.norm()) < 1e-5
