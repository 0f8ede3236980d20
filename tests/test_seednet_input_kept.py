"""The network holds its input until the next forward: a caller may drop a tensor of another stream
as soon as forward returns, while the first layer is still reading it."""
import weakref

import pytest

torch = pytest.importorskip("torch")

from paper_2412_03451_gb300 import seednet as N


def test_input_is_held_until_the_next_forward(monkeypatch):
    for name in ("ps_seed_conv_fwd", "ps_seed_pool", "ps_gemm_bf16"):
        monkeypatch.setattr(N.B, name, lambda *a, **k: None)
    net = N.SeedNet(device="cpu")
    x = torch.zeros(64, 64, 64, 4, dtype=torch.bfloat16)
    ref = weakref.ref(x)
    net.forward(x)
    del x
    assert ref() is not None
    net.forward(torch.zeros(64, 64, 64, 4, dtype=torch.bfloat16))
    assert ref() is None
