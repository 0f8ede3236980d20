"""The seed network's backward takes the upstream gradient of its own batch and nothing else: the
library reads B x 96 floats from it."""
import pytest

torch = pytest.importorskip("torch")

from paper_2412_03451_gb300 import seednet as N


def _net(monkeypatch, rows):
    calls = []
    monkeypatch.setattr(N.B, "ps_seed_backward_ws_bytes", lambda b: 1024)
    monkeypatch.setattr(N.B, "ps_seed_backward", lambda *a, **k: calls.append(a))
    net = N.SeedNet(device="cpu")
    net._alloc(rows)
    return net, calls


@pytest.mark.parametrize("shape", [(64, 96), (128, 95), (128, 8, 12), (128 * 96,), (0, 96), (192, 96)])
def test_other_shapes_are_refused(monkeypatch, shape):
    net, calls = _net(monkeypatch, 128)
    with pytest.raises(ValueError):
        net.backward(torch.zeros(shape))
    assert calls == []


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float64])
def test_other_types_are_refused(monkeypatch, dtype):
    net, calls = _net(monkeypatch, 128)
    with pytest.raises(ValueError):
        net.backward(torch.zeros(128, 96, dtype=dtype))
    assert calls == []


@pytest.mark.parametrize("dout", [torch.zeros(128, 96), torch.zeros(96, 128).T, torch.zeros(128 * 96 + 1)[1:].view(128, 96)])
def test_own_batch_in_any_layout(monkeypatch, dout):
    net, calls = _net(monkeypatch, 128)
    net.backward(dout)
    d = calls[0][5]
    assert d.is_contiguous() and d.data_ptr() % 16 == 0 and torch.equal(d, dout)
