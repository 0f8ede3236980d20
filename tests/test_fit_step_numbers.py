"""The whole step takes the same numbers as the separate Adam calls: anything int() and float() take."""
import types

import numpy as np
import pytest

from paper_2412_03451_gb300 import binding as B


@pytest.mark.parametrize("step, lr", [(3, 1e-3), (3.0, 1), (np.float64(3), np.float32(0.5)), (np.int64(3), np.float64(0.5))])
def test_numbers_are_converted(monkeypatch, step, lr):
    calls = []

    def call(*a):
        for x, t in zip(a, B_ARGS):
            t.from_param(x)                        # what ctypes does with the arguments
        calls.append(a)
        return 0

    real = B.load()
    B_ARGS = real.ps_fit_step.argtypes
    monkeypatch.setattr(B, "load", lambda: types.SimpleNamespace(ps_fit_step=call))
    monkeypatch.setattr(B, "_stream", lambda s: None)
    B.ps_fit_step(5, B.PsFrame(), B.PsSettings(), B.PsFitBuffers(), True, lr, 0.9, 0.999, 1e-8, 1e-4, step)
    assert calls[0][0] == 5 and calls[0][5] == lr and calls[0][10] == 3
