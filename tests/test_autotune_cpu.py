"""The autotuner's trials: every schedule it times is a launch of its own. Entries that act on no
kernel of the network, or that the library clamps to the default, would be timed against an equal
launch and chosen by noise."""

import types

import numpy as np
import pytest

import synth
from paper_2602_19959_gb300 import autotune as T, pvf as P

torch = pytest.importorskip("torch")


@pytest.fixture
def trials(monkeypatch):
    """tune() with launches that cost nothing: the schedules that it times."""
    class Finder:
        def __init__(self, *args, **kw):
            pass

        def close(self):
            pass

    monkeypatch.setattr(P, "PVFinder", Finder)
    monkeypatch.setattr(T, "_time_graph", lambda *a: 1.0)
    monkeypatch.setattr(torch.Tensor, "cuda", lambda t: t)
    monkeypatch.setattr(torch, "empty", lambda *a, **kw: None)
    batch = types.SimpleNamespace(n_events=2, features=np.zeros((9, 4), np.float32), offsets=np.array([0, 2, 4], np.int32))

    def run(precision, width):
        _, seen = T.tune(synth.he_weights(0, c0=width), batch, precision=precision)
        return {f: {t[f] for t in seen} - {0} for f in T.FAMILIES}

    return run


@pytest.mark.parametrize("precision", ["fp16", "bf16", "fp8"])
def test_narrow_network(trials, precision):
    tried = trials(precision, 16)
    # one kernel with one CTA per SM runs the encoder
    assert not tried["enc2"] | tried["enc3"] | tried["enc4_up3"]
    # in 16 bits one CTA of dec3_up2 fills an SM and two are dec2_up1's default; e4m3 holds one more
    assert tried["dec3_up2"] == ({1} if precision == "fp8" else set())
    assert tried["dec2_up1"] == ({1, 2} if precision == "fp8" else {1})
    assert tried["dec1_final"] == {1}                     # two are the default
    assert tried["front"] == {1, 2, 3, 4}
    assert tried["tail"] == {1, 2}                        # four are the default


def test_wide_network(trials):
    tried = trials("fp16", 32)
    assert tried["enc2"] == {2, 3}                        # a kernel of its own, four by default
    # one CTA of each of these fills an SM
    assert not any(tried[f] for f in ("enc3", "enc4_up3", "dec3_up2", "dec2_up1", "dec1_final"))


def test_float32_form(trials):
    tried = trials("fp32", 16)
    assert tried["front"] == tried["tail"] == {1}         # two are the default
    assert not any(tried[f] for f in T.FAMILIES if f not in ("front", "tail"))
