"""The seed network's implicit-GEMM convolutions against im2col + GEMM (the same
library's explicit form): bit-equal outputs, since tap order and K steps agree."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def _case(torch, side, C, Bn, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    Kp = 64 if C == 4 else 9 * C
    x = torch.randn(Bn, side, side, C, device="cuda", generator=g).bfloat16()
    w = (0.1 * torch.randn(64, Kp, device="cuda", generator=g)).bfloat16()
    w[:, 9 * C:] = 0
    return x, w, torch.randn(64, device="cuda", generator=g), Kp


# one tile, fewer tiles than SMs, and more than one tile per SM, for every layer
@pytest.mark.parametrize("side,C", [(64, 4), (32, 64), (16, 64), (8, 64)])
@pytest.mark.parametrize("Bn", [8, 64, 512])
def test_conv_equals_im2col_gemm(torch, side, C, Bn):
    from paper_2412_03451_gb300 import binding as B
    x, w, b, Kp = _case(torch, side, C, Bn, 31 * side + Bn)
    P = Bn * side * side // 4
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    A = torch.empty(P, Kp, dtype=torch.bfloat16, device="cuda")
    ref = torch.empty(P, 64, dtype=torch.bfloat16, device="cuda")
    B.ps_seed_im2col(x, Bn, side, side, C, Kp, A)
    B.ps_gemm_bf16(A, w, b, None, ref, relu=True, err=err)
    y = torch.full_like(ref, 7.0)
    xc = torch.zeros_like(x) if C == 4 else None
    B.ps_seed_conv_fwd(x, Bn, side, C, w, b, y, x_copy=xc, err=err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert torch.equal(y, ref)
    assert xc is None or torch.equal(xc, x)


def test_first_layer_takes_any_alignment(torch):
    from paper_2412_03451_gb300 import binding as B
    x, w, b, _ = _case(torch, 64, 4, 64, 5)
    flat = torch.empty(x.numel() + 1, dtype=torch.bfloat16, device="cuda")
    flat[1:] = x.view(-1)
    xu = flat[1:].view_as(x)                      # 2 bytes past a 16-byte boundary
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    ys = [torch.empty(64 * 1024, 64, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    for src, y in zip((x, xu), ys):
        B.ps_seed_conv_fwd(src, 64, 64, 4, w, b, y, x_copy=torch.empty_like(x), err=err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0 and torch.equal(*ys)
    # without room for the copy, and for a size or batch the kernels do not have, refused
    y = ys[0]
    for bad in (dict(x=xu, side=64, C=4, Bn=64), dict(x=x, side=32, C=4, Bn=64), dict(x=x, side=8, C=64, Bn=7)):
        with pytest.raises(B.PsError):
            B.ps_seed_conv_fwd(bad["x"], bad["Bn"], bad["side"], bad["C"], w, b, y)
