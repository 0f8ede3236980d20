"""Gradients for world-to-camera blocks that are not orthonormal: scaled, sheared, reflected.

The reference renders Eq. 4-13 with dense float64 tensors (every pair of a pixel and a plane,
sorted by depth) and differentiates it by autograd; it knows nothing of records or moments."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

H, W, F, LAM, K = 24, 32, 30.0, 20.0, 7
TURN = np.array([[np.cos(0.3), 0, np.sin(0.3)], [0, 1, 0], [-np.sin(0.3), 0, np.cos(0.3)]])
BLOCKS = {
    "rotation": TURN,
    "scaled": 1.4 * TURN,
    "sheared": 1.5 * TURN @ np.array([[1, 0.2, 0], [0, 1, 0.1], [0, 0, 1.0]]),
    "stretched": TURN @ np.diag([1.2, 1.6, 1.3]),
    "reflected": TURN @ np.diag([-1.0, 1.0, 1.0]),
}


def setup(block, seed=3):
    """Two views with the given 3x3 block and planes in front of them, float32 arrays."""
    rng = np.random.default_rng(seed)
    w2c = np.stack([np.concatenate([block, [[0.1], [-0.05], [0.2]]], 1),
                    np.concatenate([block @ TURN.T, [[-0.3], [0.1], [0.1]]], 1)]).astype(np.float32)
    pc = np.stack([rng.uniform(-0.8, 0.8, K), rng.uniform(-0.6, 0.6, K), np.linspace(2.0, 3.5, K)], 1)
    c = (pc - w2c[0, :, 3]) @ np.linalg.inv(w2c[0, :, :3].astype(np.float64)).T
    q = rng.normal(size=(K, 4)) * [1.5, 0.3, 0.3, 0.8]
    return c.astype(np.float32), q.astype(np.float32), rng.uniform(0.25, 0.6, (K, 4)).astype(np.float32), w2c


def reference(c, q, r, w2c, gauss, gD, gN):
    import torch
    p = [torch.tensor(x.astype(np.float64), requires_grad=True) for x in (c, q, r)]
    w, x, y, z = (p[1] / p[1].norm(dim=1, keepdim=True)).unbind(1)
    vx = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y)], 1)
    vy = torch.stack([2 * (x * y - w * z), 1 - 2 * (x * x + z * z), 2 * (y * z + w * x)], 1)
    n = torch.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)], 1)
    total = 0.0
    jj, ii = np.meshgrid(np.arange(W) + 0.5, np.arange(H) + 0.5)
    d = torch.tensor(np.stack([(jj - W / 2) / F, (ii - H / 2) / F, np.ones_like(jj)], -1).reshape(-1, 1, 3))
    for v in range(len(w2c)):
        T = torch.tensor(w2c[v].astype(np.float64))
        pc, X, Y, N = p[0] @ T[:, :3].T + T[:, 3], vx @ T[:, :3].T, vy @ T[:, :3].T, n @ T[:, :3].T
        den = (d * N).sum(-1)
        t = (N * pc).sum(-1) / den
        e = t[..., None] * d - pc
        PX, PY = (e * X).sum(-1), (e * Y).sum(-1)
        sX = torch.where(PX > 0, p[2][:, 0], p[2][:, 1])
        sY = torch.where(PY > 0, p[2][:, 2], p[2][:, 3])
        if gauss:
            wt = torch.exp(-0.5 * ((PX / sX) ** 2 + (PY / sY) ** 2))
        else:
            m = torch.minimum(sX - PX.abs(), sY - PY.abs())
            wt = torch.clamp(2 * torch.sigmoid(5 * LAM * m), max=1.0)
        ok = (wt >= 1e-4) & (t > 0.01) & (t < 100.0) & (den.abs() > 1e-6)
        wt = torch.where(ok, wt, torch.zeros_like(wt))
        order = torch.where(ok, t, torch.full_like(t, 1e9)).argsort(1)
        ws, ts = wt.gather(1, order), torch.where(ok, t, torch.zeros_like(t)).gather(1, order)
        front = torch.cumprod(torch.cat([torch.ones_like(ws[:, :1]), 1 - ws[:, :-1]], 1), 1) * ws
        D = (front * ts).sum(1)
        Nm = (front[..., None] * N[order]).sum(1)
        total = total + (D * torch.tensor(gD[v]).double()).sum() + (Nm * torch.tensor(gN[v]).double()).sum()
    return [g.numpy() for g in torch.autograd.grad(total, p)]


@pytest.mark.parametrize("gauss", [False, True])
@pytest.mark.parametrize("block", sorted(BLOCKS))
def test_gradients_for_any_block(block, gauss):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from gpu_cases import grad_errors
    from paper_2412_03451_gb300 import binding as B, splat as SP
    c, q, r, w2c = setup(BLOCKS[block])
    rng = np.random.default_rng(5)
    gD = rng.normal(size=(2, H * W)).astype(np.float32)
    gN = rng.normal(size=(2, H * W, 3)).astype(np.float32)
    want = reference(c, q, r, w2c, gauss, gD, gN)
    R = SP.Renderer([H] * 2, [W] * 2, [0, 0], [0, K], flags=B.PS_GAUSSIAN if gauss else 0)
    R.set_cameras(w2c, np.tile(np.float32([F, F, W / 2, H / 2]), (2, 1)))
    flat = SP.planes_to_flat(c, q, r, "cuda")
    R.ensure_capacity(flat, LAM)
    R.forward(flat, LAM)
    g = torch.zeros_like(flat)
    R.backward(flat, g, torch.from_numpy(gD.reshape(-1)).cuda(), torch.from_numpy(gN.reshape(-1, 3)).cuda())
    # 1e-3 of a plane's gradient, as for orthonormal views against the oracle
    for got, exp in zip(SP.flat_views(g, K), want):
        assert np.abs(exp).max() > 0
        assert grad_errors(got.cpu().numpy(), exp)[0] == 0
    # the whole step's own chain against the separate calls': the same splat sums, in other orders
    gd = torch.rand(2 * H * W, device="cuda") + 2
    gn = torch.randn(2 * H * W, 3, device="cuda")
    steps = []
    for marks in (None, []):
        fit = SP.Fitter(R, flat.clone(), lr=0.0)
        fit.step(gd, gn, lam=LAM, marks=marks)
        steps.append(fit.grad)
    for a, b in zip(SP.flat_views(steps[0], K), SP.flat_views(steps[1], K)):
        assert float((a - b).norm() / b.norm()) < 1e-5
