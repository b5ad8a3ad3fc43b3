"""The peak finder on logits full of plateaus, ties, edges, infinities and NaN, from a buffer
aligned to 16 and one aligned to 4 bytes, for event counts on both sides of the resident grid:
decisions against the rule stated bin by bin in numpy, centroids in 64 bits (float32 rounding of
z at 300 mm: 1.5e-5 mm; the bound is four times that)."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MAX_PV = 667


def rule(f):
    """(bins, z) of one event: the strict left / non-strict right rule on the logits."""
    thr = np.float32(np.log(0.01 / 0.99))
    keep = f > thr
    with np.errstate(invalid="ignore"):
        for d in range(1, 6):
            keep[d:] &= f[d:] > f[:-d]
            keep[:-d] &= f[:-d] >= f[d:]
    bins = np.nonzero(keep)[0]
    z = []
    for i in bins:
        j = np.arange(max(0, i - 3), min(len(f), i + 4))
        with np.errstate(over="ignore"):
            p = 1.0 / (1.0 + np.exp(-f[j].astype(np.float64)))
        z.append(-100.0 + 0.1 * (i + 0.5 + np.sum(p * (j - i)) / np.sum(p)))
    return bins, np.array(z)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("n", [1, 37, 700])
def test_peaks_against_the_rule(n, offset):
    from paper_2602_19959_gb300 import build, PVFinder
    build()
    rng = np.random.default_rng(17 + n)
    kinds = [rng.integers(-6, 7, (n, 4000)).astype(np.float32),                      # ties everywhere
             rng.normal(0, 120, (n, 4000)).astype(np.float32),                       # saturated sigmoids
             np.where(rng.random((n, 4000)) < 0.2, np.inf, rng.normal(0, 3, (n, 4000))).astype(np.float32),
             np.where(rng.random((n, 4000)) < 0.02, np.nan, rng.normal(0, 3, (n, 4000))).astype(np.float32)]
    kinds[1][:, :6] = 500.0
    kinds[1][:, -3:] = [1.0, 2.0, 3.0]
    kinds[3][:, rng.integers(0, 4000, 5)] = -np.inf
    pv = PVFinder(synth.he_weights(0), precision="fp16", max_events=n, max_pv_per_event=MAX_PV)
    for f in kinds:
        raw = torch.zeros(n * 4000 + offset, device="cuda")
        logit = raw[offset:].view(n, 4000)
        logit.copy_(torch.from_numpy(f))
        z, c = pv.stage_peaks(logit)
        z, c = z.cpu().numpy(), c.cpu().numpy()
        for e in {0, n // 2, n - 1}:
            bins, want = rule(f[e])
            assert c[e] == len(bins)
            np.testing.assert_allclose(z[e, :c[e]], want, rtol=0, atol=6e-5)
    assert pv.device_status() == 0
    pv.close()
