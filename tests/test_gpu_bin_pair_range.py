"""More (record, tile) pairs than an int numbers: the total and the status say so, and the truncated
lists hold valid record ids, which the splat kernels index with."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIDE, VIEWS = 2048, 33


@pytest.mark.parametrize("planes", [992, 993])            # 65,536 tiles x 33 views x planes around 2^31
def test_pair_totals_past_the_int_range(planes):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_03451_gb300 import binding as B, splat as SP
    K, cap = planes, 100_003
    r = SP.Renderer([SIDE] * VIEWS, [SIDE] * VIEWS, [0] * VIEWS, [0, K], tile=(8, 8), capacity=cap)
    w2c = np.tile(np.concatenate([np.eye(3), np.zeros((3, 1))], 1).astype(np.float32), (VIEWS, 1, 1))
    r.set_cameras(w2c, np.tile(np.float32([1000, 1000, SIDE / 2, SIDE / 2]), (VIEWS, 1)))
    # every plane faces the cameras and covers every pixel
    flat = SP.planes_to_flat(np.float32([[0, 0, 2 + 0.001 * k] for k in range(K)]),
                             np.tile(np.float32([1, 0, 0, 0]), (K, 1)), np.full((K, 4), 9.0, np.float32), "cuda")
    r.tile_ent.fill_(1 << 30)
    r.bin_ws.view(torch.int32).fill_(1 << 30)
    r.project_bin(flat, 300.0)
    total = K * VIEWS * (SIDE // 8) ** 2
    assert (total >= 2 ** 31 - 1) == (planes == 993)
    assert int(r.required.item()) == total
    assert int(r.status.item()) == 1 << B.PS_ERR_CAPACITY
    assert int(r.tile_ptr[-1]) == cap and int(r.tile_ptr[1]) == K
    assert int(r.tile_ent.min()) >= 0 and int(r.tile_ent.max()) < VIEWS * K
    if planes == 992:
        assert torch.equal(r.tile_ent[:K], torch.arange(K, device="cuda", dtype=torch.int32))
    r.splat_forward()
    torch.cuda.synchronize()
