"""The tensor-core front has two shapes (128 or 256 threads, and tracks per pass), by the launch's
size or its schedule, and up to eight blocks share an event where a launch has few: events with
track counts at the edges of warps and passes give the same bits under every shape and share."""

import numpy as np
import pytest

import synth
from tests.test_gpu_front_edges import COUNTS

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def events():
    from paper_2602_19959_gb300 import build
    build()
    rng = np.random.default_rng(12)
    n = sum(COUNTS)
    feats = rng.normal(0.0, 0.1, (9, n)).astype(np.float32)
    feats[2] = np.where(rng.uniform(size=n) < 0.4, rng.uniform(61.0, 69.0, n), rng.uniform(-100.0, 300.0, n))
    feats[2, ::29] = 350.0                                  # dropped tracks
    return torch.from_numpy(feats).cuda(), np.concatenate([[0], np.cumsum(COUNTS)]).astype(np.int32)


def gathered(events, pick):
    feats, offs = events
    cols = np.concatenate([np.arange(offs[e], offs[e + 1]) for e in pick])
    o = np.concatenate([[0], np.cumsum([COUNTS[e] for e in pick])]).astype(np.int32)
    return feats[:, torch.from_numpy(cols).cuda()].contiguous(), torch.from_numpy(o).cuda()


@pytest.mark.parametrize("edge", [0.0, 0.5])
@pytest.mark.parametrize("precision", ["fp16", "bf16"])
def test_both_shapes_give_the_same_histograms(events, precision, edge):
    from paper_2602_19959_gb300 import PVFinder
    w = synth.he_weights(0, bias_std=0.05)
    k = len(COUNTS)
    args = gathered(events, range(k))
    first = None
    for front in (2, 1, 3, 4):                              # 256 threads, then 128
        pv = PVFinder(w, precision=precision, max_events=k, max_pv_per_event=8, boundary_mm=edge, schedule={"front": front})
        out = torch.full((k, 4000), -1.0, device="cuda")
        pv.stage_histogram(*args, out)
        got = out.view(torch.int32)
        first = got if first is None else first
        assert torch.equal(got, first), front
        assert pv.device_status() == 0
        pv.close()


@pytest.mark.parametrize("precision,options", [("fp16", {}), ("bf16", {}), ("fp8", {}), ("fp16", {"boundary_mm": 0.5}),
                                               ("fp16", {"per_interval": True}), ("fp8", {"per_interval": True}),
                                               ("fp16", {"width": 32}), ("fp8", {"width": 32})])
def test_shared_events_give_the_same_logits(events, precision, options):
    from paper_2602_19959_gb300 import PVFinder
    options = dict(options)
    w = synth.he_weights(0, bias_std=0.05, c0=options.pop("width", 16))
    k = len(COUNTS)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    most = sms + k                                          # nothing is shared in a launch of these
    scales = [0.05] * 16 if precision == "fp8" else None
    pv = PVFinder(w, precision=precision, max_events=most, max_pv_per_event=8, fp8_act_scales=scales, **options)

    def run(pick):
        out = torch.empty((len(pick), 4000), device="cuda")
        pv.infer(*gathered(events, pick), logit=out)
        return out.view(torch.int32)

    want = run([e % k for e in range(most)])[:k]
    for m in (1, 2, sms // 16, sms // 8, sms // 4, sms // 2, sms // 2 + 1):
        pick = [(e + k - 1) % k for e in range(m)]          # the largest event first
        assert torch.equal(run(pick), want[pick]), m
    pv.close()
