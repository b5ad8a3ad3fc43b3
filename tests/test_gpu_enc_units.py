"""The fused encoder kernel runs each event as one, two or four units, by the number of events
in the launch: every choice, and every place of an event in a launch, must give bit for bit the
logits the event has alone (which other tests hold against the float64 emulation)."""

import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp16", "bf16", "fp8"])
def test_units_per_event_change_nothing(precision):
    from paper_2602_19959_gb300 import build, PVFinder
    build()
    w = synth.he_weights(0, bias_std=0.05)
    g = torch.Generator("cuda").manual_seed(5)
    # histograms as the front makes them: mostly small values, a few narrow peaks
    hist = torch.rand((8, 4000), generator=g, device="cuda")
    hist[:, ::173] += 40.0
    scales = [0.05] * 16 if precision == "fp8" else None
    most = 4 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    pv = PVFinder(w, precision=precision, max_events=most, max_pv_per_event=8, fp8_act_scales=scales)
    alone = torch.cat([pv.stage_unet(hist[k:k + 1], torch.empty((1, 4000), device="cuda")).clone() for k in range(8)])
    sms = (most - 1) // 4
    for n in (2, 3, sms // 4, sms // 4 + 1, sms // 2, sms // 2 + 1, sms - 1, sms, sms + 1, 2 * sms + 1, most):
        pick = torch.arange(n, device="cuda") % 8
        got = pv.stage_unet(hist[pick].contiguous(), torch.empty((n, 4000), device="cuda"))
        assert torch.equal(got.view(torch.int32), alone[pick].view(torch.int32)), n
    assert pv.device_status() == 0
    pv.close()


@pytest.mark.parametrize("width", [16, 32])
def test_float32_tiles_change_nothing(width):
    """The float32 convolutions take half the positions per tile where every tile then has an SM of
    its own, layer by layer: the same bits at every number of events."""
    from paper_2602_19959_gb300 import build, PVFinder
    build()
    w = synth.he_weights(0, bias_std=0.05, c0=width)
    g = torch.Generator("cuda").manual_seed(6)
    hist = torch.rand((4, 4000), generator=g, device="cuda")
    hist[:, ::173] += 40.0
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    pv = PVFinder(w, precision="fp32", max_events=sms, max_pv_per_event=8)
    alone = torch.cat([pv.stage_unet(hist[k:k + 1], torch.empty((1, 4000), device="cuda")).clone() for k in range(4)])
    per_event = {16, 32}                                    # half tiles per event, by width
    for n in sorted({2, sms} | {sms // p for p in per_event} | {sms // p + 1 for p in per_event}):
        pick = torch.arange(n, device="cuda") % 4
        got = pv.stage_unet(hist[pick].contiguous(), torch.empty((n, 4000), device="cuda"))
        assert torch.equal(got.view(torch.int32), alone[pick].view(torch.int32)), n
    pv.close()
