"""FP8 calibration folds every stored activation, and nothing else, into the scales. The fused
encoder runs an event as one, two or four units, by the number of events in a launch, and the
units recompute tiles of their neighbours whose remaining rows hold whatever shared memory held:
the scales must be, bit for bit, those of launches that split no event, whatever ran before."""

import numpy as np
import pytest

import synth
from tests import ref_torch64 as ref

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = 512


@pytest.fixture(scope="module")
def setup():
    from paper_2602_19959_gb300 import build
    build()
    b = synth.generate_standard(N, 1)
    return synth.he_weights(0, bias_std=0.05), torch.from_numpy(b.features).cuda(), np.asarray(b.offsets)


def pick_events(feats, offs, pick):
    """The picked events, gathered: features and offsets of one call."""
    cols = np.concatenate([np.arange(offs[e], offs[e + 1]) for e in pick])
    o = np.concatenate([[0], np.cumsum([offs[e + 1] - offs[e] for e in pick])]).astype(np.int32)
    return feats[:, torch.from_numpy(cols).cuda()].contiguous(), torch.from_numpy(o).cuda()


def leave_other_bits(weights, feats, offs):
    """A large batch of the FP16 form, whose operands lie where the BF16 form's do: f16 bits of
    ordinary activations read as bf16 are huge."""
    from paper_2602_19959_gb300 import PVFinder
    pv = PVFinder(weights, precision="fp16", max_events=N, max_pv_per_event=8)
    pv.infer(feats, torch.from_numpy(offs).cuda())
    torch.cuda.synchronize()
    pv.close()


@pytest.mark.parametrize("n", [1, 16, 64, 100, 160, 320, N])
def test_scales_do_not_depend_on_the_launch(setup, n):
    from paper_2602_19959_gb300 import PVFinder
    weights, feats, offs = setup
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # the same events over and over, in launches of one event per SM, which are not split
    rounds = -(-n // sms)
    whole = PVFinder(weights, precision="bf16", max_events=rounds * sms, chunk_events=sms, max_pv_per_event=8)
    want = whole.calibrate(*pick_events(feats, offs, np.arange(rounds * sms) % n))
    whole.close()
    args = pick_events(feats, offs, np.arange(n))
    for chunk in (0, 128, 16):
        pv = PVFinder(weights, precision="bf16", max_events=n, chunk_events=min(chunk, n), max_pv_per_event=8)
        for _ in range(2):
            leave_other_bits(weights, feats, offs)
            got = pv.calibrate(*args)
            assert np.array_equal(got.view(np.int32), want.view(np.int32)), (chunk, got[:7], want[:7])
        pv.close()


def test_scales_are_the_largest_stored_magnitudes(setup):
    """Against the float64 emulation with bf16 rounding at every stored tensor (which the kernels
    differ from where an fp32 sum rounds to the other neighbour: by less than a bf16 step)."""
    from paper_2602_19959_gb300 import PVFinder
    weights, feats, offs = setup
    n = 16
    args = pick_events(feats, offs, np.arange(n))
    pv = PVFinder(weights, precision="bf16", max_events=n, max_pv_per_event=8)
    leave_other_bits(weights, feats, offs)
    scales = pv.calibrate(*args)
    hist = torch.empty((n, 4000), device="cuda")
    pv.stage_histogram(*args, hist)
    hist = hist.cpu().numpy().astype(np.float64)
    pv.close()
    most = np.zeros(18)
    for e in range(n):
        seen = []

        def q(t):                       # in order: e1, then each layer's weights and its output
            seen.append(float(t.abs().max()))
            return ref.q_bf16(t)

        ref.unet_quantized(weights, hist[e], q)
        most = np.maximum(most, seen)
    e1, e2, e3, e4, u3, d3, u2, d2, u1 = most[0:17:2]
    for slot, want in enumerate((max(e1, u1), max(e2, u2), max(e3, u3), e4, d3, d2)):
        assert abs(448.0 * scales[slot] - want) <= 2.0 ** -7 * want, (slot, 448.0 * scales[slot], want)
