"""The autograd forward enqueues its splat before it knows whether the tile lists fitted; lists that
did not fit are given back only once that splat is done with them."""
import types

import pytest

torch = pytest.importorskip("torch")

from paper_2412_03451_gb300 import scenes as S, splat as SP


@pytest.mark.parametrize("need", [7, 8, 9])
def test_old_lists_are_dropped_after_the_stream_is_idle(monkeypatch, need):
    log = []
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda *a: types.SimpleNamespace(synchronize=lambda: log.append("idle")))
    r = types.SimpleNamespace(_required_host=torch.tensor([need]), capacity=8, status=torch.ones(1, dtype=torch.int32),
                              _alloc_lists=lambda c: log.append(("lists", c)))
    grew = SP.Renderer.grow_if_needed(r)
    if need <= 8:
        assert not grew and log == [] and int(r.status) == 1
    else:
        assert grew and log[0] == "idle" and log[1] == ("lists", int(9 * 1.5) + 1024) and int(r.status) == 0


@pytest.mark.gpu
def test_growth_on_another_stream_than_the_lists(monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    room = S.tiny_room(0)
    p = S.perturb_planes(room.gt, 1)
    V, H, W = room.cams.V, room.cams.H, room.cams.W

    def make(**kw):
        r = SP.Renderer([H] * V, [W] * V, [0] * V, [0, p.K], **kw)
        r.set_cameras(room.cams.w2c, room.cams.intr)
        return r, SP.planes_to_flat(p.center, p.quat, p.radii, "cuda")

    ref, flat = make()
    ref.ensure_capacity(flat, 20.0)
    want = [x.clone() for x in ref.forward(flat, 20.0)]
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(a):
        r, flat = make(capacity=100)
    idle, alloc = [], r._alloc_lists

    def dropped(capacity):
        idle.append(torch.cuda.current_stream().query())
        alloc(capacity)

    monkeypatch.setattr(r, "_alloc_lists", dropped)
    b.wait_stream(a)
    with torch.cuda.stream(b):
        D, N = SP.PlaneSplatFunction.apply(flat, r, 20.0)
        with torch.cuda.stream(a):                     # takes and writes what the old lists left on a
            for n in (25, 100, 1000):
                torch.full((n,), 1 << 30, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert idle == [True] and int(r.status.item()) == 0
    assert torch.equal(D, want[0]) and torch.equal(N, want[1])
