"""The flat parameter buffer [center P*3 | quat P*4 | radii P*4]: its group pointers are those of
the views of its groups, and a buffer of another size or shape is refused."""
import types

import pytest

torch = pytest.importorskip("torch")

from paper_2412_03451_gb300 import splat as SP

P = 5


@pytest.mark.parametrize("shape", [(11 * P - 1,), (11 * P + 1,), (10 * P,), (0,), (P, 11), (1, 11 * P), (11 * (P + 1),)])
def test_other_sizes_and_shapes_are_refused(shape):
    flat = torch.zeros(shape)
    with pytest.raises(RuntimeError):
        SP.flat_views(flat, P)
    with pytest.raises(RuntimeError):
        SP.flat_ptrs(flat, P)
    r = types.SimpleNamespace(P=P)
    with pytest.raises(RuntimeError):
        SP.Renderer.planes_struct(r, flat)
    # the whole step as one call takes pointers alone: it is left to the calls that refuse
    assert not SP.Fitter(r, flat)._one_call()


@pytest.mark.parametrize("flat", [torch.zeros(11 * P), torch.zeros(11 * P + 3)[3:], torch.zeros(22 * P)[::2],
                                  torch.zeros(11 * P, dtype=torch.float64)])
def test_pointers_are_those_of_the_views(flat):
    assert SP.flat_ptrs(flat, P) == tuple(x.data_ptr() for x in SP.flat_views(flat, P))
    plain = flat.is_contiguous() and flat.dtype is torch.float32
    assert SP.Fitter(types.SimpleNamespace(P=P), flat)._one_call() == plain
