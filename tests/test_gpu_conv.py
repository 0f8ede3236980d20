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


def _explicit_backward(torch, net, x, dout):
    """The backward as separate library calls: im2col, transposed copies, one GEMM per product."""
    from paper_2412_03451_gb300 import binding as B
    from paper_2412_03451_gb300 import seednet as SN
    Bn, bf = net.B, torch.bfloat16

    def empty(*shape, dtype=torch.float32):
        return torch.empty(shape, dtype=dtype, device="cuda")

    def transposed(t, rows, cols):
        out = empty(rows, cols, dtype=bf)
        B.ps_seed_transpose(t, out)
        return out

    gW, gb = [None] * 5, [empty(SN.CH) for _ in range(4)] + [empty(SN.OUT)]
    gW[4] = empty(SN.OUT, SN.CH)
    B.ps_gemm_bf16(transposed(dout, SN.OUT, Bn), transposed(net.h16, SN.CH, Bn), None, gW[4], None, err=net.err)
    B.ps_seed_colsum(dout, gb[4])
    d16, dh, dy = empty(Bn, 128, dtype=bf), empty(Bn, SN.CH), empty(Bn * 16, SN.CH)
    B.ps_cast_bf16(dout, d16)
    B.ps_gemm_bf16(d16, transposed(net.W[4], SN.CH, 128), None, dh, None, err=net.err)
    B.ps_seed_pool_bwd(dh, Bn, 16, SN.CH, dy)
    for i in range(3, -1, -1):
        h, cin, kp = SN.LAYERS[i]
        P = net.Y[i].shape[0]
        dz16, dz32, A, gWp = empty(P, SN.CH, dtype=bf), empty(P, SN.CH), empty(P, kp, dtype=bf), empty(SN.CH, kp)
        B.ps_seed_relu_bwd(dy, net.Y[i], 1.0, dz16, dz32)
        B.ps_seed_im2col(net.Y[i - 1] if i else x, Bn, h, h, cin, kp, A)
        B.ps_gemm_bf16(transposed(dz16, SN.CH, P), transposed(A, kp, P), None, gWp, None, err=net.err)
        gW[i] = gWp[:, :9 * cin]
        B.ps_seed_colsum(dz32, gb[i])
        if i:
            dA, dy = empty(P, kp), empty(net.Y[i - 1].shape[0], SN.CH)
            B.ps_gemm_bf16(dz16, transposed(net._bf16[i], kp, SN.CH), None, dA, None, err=net.err)
            B.ps_seed_col2im(dA, Bn, h, h, cin, kp, dy)
    return gW, gb


@pytest.mark.parametrize("Bn", [64, 192, 320])
def test_backward_equals_explicit_form(torch, Bn):
    from paper_2412_03451_gb300 import seednet as SN
    net = SN.SeedNet(seed=2)
    net.sync_weights()
    g = torch.Generator(device="cuda").manual_seed(Bn)
    x = torch.randn(Bn, 64, 64, 4, device="cuda", generator=g).bfloat16()
    dout = torch.randn(Bn, SN.OUT, device="cuda", generator=g)
    net.forward(x)
    ref_W, ref_b = _explicit_backward(torch, net, x, dout)
    kept = x.clone()
    x.zero_()                                     # the backward has its own copy of the input
    net.grad.fill_(9.0)
    net.backward(dout)
    torch.cuda.synchronize()
    assert int(net.err.item()) == 0
    for i in range(4):                            # the same chain of sums in the same order
        assert torch.equal(net.gW[i], ref_W[i]), i
    # other orders of FP32 sums of n terms: relative to the norm, sqrt(n) roundoffs with room
    eps = 2.0 ** -24

    def rel(a, b):
        return float((a.double() - b.double()).norm() / b.double().norm())

    assert rel(net.gW[4], ref_W[4]) < 8 * eps * Bn ** 0.5
    for i, n in enumerate([Bn * 1024, Bn * 256, Bn * 64, Bn * 16, Bn]):
        assert rel(net.gb[i], ref_b[i]) < 8 * eps * n ** 0.5, i
    assert not torch.equal(kept, x)
