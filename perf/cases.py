"""Performance cases of the inference library: what its users have it do, through the
public entry points of `paper_2602_19959_gb300.PVFinder`, over the range of event counts,
precisions and options that the configurations, tests and benchmark of this repository use.

Inputs are synthetic collision events with the shape of the paper's workload (standard:
Poisson(5.6) vertices per event, about 155 tracks; uneven: 1 to 12 vertices and a
heavy-tailed background, up to 700 tracks), drawn on the GPU from the seed; weights are the
He-initialised networks the library is used with (no trained checkpoint exists), with small
non-zero biases. `exact` restates the path in 64 bits with plain torch.
"""

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2602_19959_gb300 import PVFinder

N_BINS, N_SLICES = 4000, 40
MAX_PV = 672          # output slots per event: no event can hold more than 667 vertices
UNEVEN_TRACKS = 171   # mean tracks per event of each kind
STANDARD_TRACKS = 155

# what a case leaves out
DEFAULTS = {"entry": "infer", "precision": "fp16", "kind": "standard", "width": 16, "interval": False,
            "boundary_mm": 0.0, "capacity": 0}


def listed():
    return [
        # one collision event, answered at once: an online filter or a monitoring client. Latency.
        {"name": "event_fp16", "events": 1},
        # a batch of the continuous-batching server: the graph captured once per slot with its
        # event count read on the device, at the mean batch of the benchmark's serving run
        {"name": "serving_graph_fp16", "entry": "graph", "events": 121, "kind": "uneven", "capacity": 512},
        # the headline batch of the benchmark, in its headline form
        {"name": "batch_fp16", "events": 1000},
        # bulk processing of stored data: many events of uneven size in one call (no multiple of
        # a power of two or of the SM count)
        {"name": "bulk_uneven_fp16", "events": 15999, "kind": "uneven"},
        # a handful of events at the library's default precision: development, cross-checks
        {"name": "few_fp32", "precision": "fp32", "events": 16},
        # a batch at the default precision: the form every other one is compared with
        {"name": "batch_fp32", "precision": "fp32", "events": 500},
        # the fastest form, with calibrated scales
        {"name": "batch_fp8", "precision": "fp8", "events": 1000},
        # the wide network (32/64/128/256 channels), the paper's larger model
        {"name": "wide_fp16", "width": 32, "events": 250},
        # the per-interval layout: each 10 mm interval through the network on its own
        {"name": "interval_fp16", "interval": True, "events": 500},
        # the histogram alone (validation, sort, FC net), with boundary tracks: studies of the
        # first half, and callers that run their own network behind it
        {"name": "histogram_bf16", "entry": "histogram", "precision": "bf16", "events": 777, "kind": "uneven",
         "boundary_mm": 0.5},
        # the network alone on histograms the caller has
        {"name": "unet_bf16", "entry": "unet", "precision": "bf16", "events": 333},
        # peak finding alone on logits the caller has
        {"name": "peaks", "entry": "peaks", "events": 2500},
    ]


def draw(rng):
    """One more case of the same ranges."""
    entry = rng.choice(["infer", "infer", "infer", "graph", "histogram", "unet", "peaks"])
    precision = rng.choice(["fp16", "fp16", "bf16", "fp8", "fp32"])
    if entry == "graph" and precision == "fp32":
        precision = "bf16"     # captured graphs with a device-side count are of the tensor-core forms
    # the UNet's options
    width, interval = rng.choice([(16, False), (16, False), (16, False), (32, False), (16, True)])
    if entry == "peaks":
        precision, width, interval = "fp16", 16, False
    most = {"fp32": 700}.get(precision, 10000)
    if width == 32:
        most //= 5
    if entry == "graph":
        most = min(most, 1000)
    events = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    case = {"entry": entry, "precision": precision, "events": events, "kind": rng.choice(["standard", "uneven"]),
            "width": width, "interval": interval}
    if entry not in ("unet", "peaks"):
        case["boundary_mm"] = rng.choice([0.0, 0.0, 0.5, round(rng.uniform(0.1, 1.0), 2)])
    if entry == "graph":
        case["capacity"] = events + rng.randrange(0, 200)
    return case


# ------------------------------------------------------------------ inputs

def _events(kind, n, seed):
    """(features float32 [9, n_tracks], offsets int32 [n + 1]) on the GPU."""
    g = torch.Generator("cuda").manual_seed(seed)
    dev = {"device": "cuda"}

    def uniform(shape):
        return torch.rand(shape, generator=g, **dev)

    def normal(shape):
        return torch.randn(shape, generator=g, **dev)

    def poisson(mean, shape):
        return torch.poisson(torch.full(shape, float(mean), **dev), generator=g).long()

    if kind == "standard":
        n_pv = poisson(5.6, (n,)).clamp(min=1)
        n_bkg = poisson(15.0, (n,))
    else:
        n_pv = torch.randint(1, 13, (n,), generator=g, **dev)
        n_bkg = torch.floor(5.0 / (1.0 - uniform((n,))).sqrt()).clamp(max=400.0).long()
    ev_of_pv = torch.repeat_interleave(torch.arange(n, **dev), n_pv)
    z_pv = (45.0 * normal(ev_of_pv.shape)).clamp(-100.0, 300.0)
    n_trk = poisson(25.0, ev_of_pv.shape)
    pv_of_track = torch.repeat_interleave(torch.arange(ev_of_pv.numel(), **dev), n_trk)
    z_sig = z_pv[pv_of_track] + 0.08 * normal(pv_of_track.shape)
    ev_bkg = torch.repeat_interleave(torch.arange(n, **dev), n_bkg)
    z_bkg = -100.0 + 400.0 * uniform(ev_bkg.shape)
    ev = torch.cat([ev_of_pv[pv_of_track], ev_bkg])
    z = torch.cat([z_sig, z_bkg])
    # events contiguous, tracks in random order within each
    order = torch.argsort(ev.double() + uniform(ev.shape).double().clamp(max=0.999))
    ev, z = ev[order], z[order]
    m = z.numel()
    feats = torch.empty((9, m), **dev)
    for k in (0, 1):
        feats[k] = 0.05 * normal((m,))
    feats[2] = z
    for k in (3, 4):
        feats[k] = 0.15 * normal((m,))
    for k in (5, 6, 7):
        feats[k] = 0.05 * torch.exp(0.5 * normal((m,)))
    feats[8] = uniform((m,))
    offsets = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    offsets[1:] = torch.cumsum(torch.bincount(ev, minlength=n), 0).int()
    return feats, offsets


def _shapes(c):
    h = 32
    return {"fc1": ((h, 9), h, 9), "fc2": ((h, h), h, h), "fc3": ((h, h), h, h), "fc4": ((h, h), h, h),
            "fc5": ((h, h), h, h), "fc6": ((100, h), 100, h),
            "enc1": ((c, 1, 5), c, 5), "enc2": ((2 * c, c, 5), 2 * c, 5 * c),
            "enc3": ((4 * c, 2 * c, 5), 4 * c, 10 * c), "enc4": ((8 * c, 4 * c, 5), 8 * c, 20 * c),
            "up3": ((8 * c, 4 * c, 2), 4 * c, 16 * c), "dec3": ((4 * c, 8 * c, 5), 4 * c, 40 * c),
            "up2": ((4 * c, 2 * c, 2), 2 * c, 8 * c), "dec2": ((2 * c, 4 * c, 5), 2 * c, 20 * c),
            "up1": ((2 * c, c, 2), c, 4 * c), "dec1": ((c, 2 * c, 5), c, 10 * c),
            "final": ((1, c, 5), 1, 5 * c)}


def _weights(width):
    """{layer: (W, b)}: He initialisation, biases N(0, 0.05). The network a program has loaded."""
    rng = np.random.default_rng(1234 + width)
    return {name: (rng.normal(0.0, math.sqrt(2.0 / fan_in), shape).astype(np.float32),
                   rng.normal(0.0, 0.05, n_bias).astype(np.float32))
            for name, (shape, n_bias, fan_in) in _shapes(width).items()}


# ------------------------------------------------------------------ the path in 64 bits

def _slices(feats, boundary_mm):
    """(track, slice) pairs each track fills; the decisions are float32 by definition."""
    z = feats[2]
    q = (z + 100.0) / 10.0
    track = torch.nonzero((q >= 0) & (q < N_SLICES) & torch.isfinite(feats).all(0)).reshape(-1)
    s = torch.floor(q[track]).long()
    if boundary_mm > 0.0:
        w = float(np.float32(boundary_mm))
        zr = z[track] - (-100.0 + 10.0 * s.float())
        low = (zr < w) & (s > 0)
        high = ~low & (zr >= float(np.float32(10.0) - np.float32(boundary_mm))) & (s < N_SLICES - 1)
        track, s = torch.cat([track, track[low], track[high]]), torch.cat([s, s[low] - 1, s[high] + 1])
    return track, s


def _histogram64(w, feats, offsets, boundary_mm):
    n = offsets.numel() - 1
    track, s = _slices(feats, boundary_mm)
    x = feats[:, track].double().T.contiguous()
    x[:, 2] -= -100.0 + 10.0 * s.double()
    ev = torch.repeat_interleave(torch.arange(n, device="cuda"), (offsets[1:] - offsets[:-1]).long())[track]
    for k in range(1, 6):
        x = F.leaky_relu(x @ w["fc%d" % k][0].T + w["fc%d" % k][1], 0.01)
    x = F.softplus(x @ w["fc6"][0].T + w["fc6"][1], threshold=50.0)
    hist = torch.zeros((n * N_SLICES, 100), dtype=torch.float64, device="cuda")
    hist.index_add_(0, ev * N_SLICES + s, x)
    return hist.reshape(n, N_BINS)


def _unet64(w, hist, interval):
    """Logits [n, 4000] from histograms [n, 4000], by blocks of events."""
    def conv(x, name):
        return F.conv1d(x, w[name][0], w[name][1], padding=2)

    def up(x, name):
        return F.leaky_relu(F.conv_transpose1d(x, w[name][0], w[name][1], stride=2), 0.01)

    def net(x):
        e1 = F.leaky_relu(conv(x, "enc1"), 0.01)
        e2 = F.leaky_relu(conv(F.max_pool1d(e1, 2), "enc2"), 0.01)
        e3 = F.leaky_relu(conv(F.max_pool1d(e2, 2), "enc3"), 0.01)
        e4 = F.leaky_relu(conv(F.max_pool1d(e3, 2), "enc4"), 0.01)
        d = F.leaky_relu(conv(torch.cat([up(e4, "up3"), e3], 1), "dec3"), 0.01)
        d = F.leaky_relu(conv(torch.cat([up(d, "up2"), e2], 1), "dec2"), 0.01)
        d = F.leaky_relu(conv(torch.cat([up(d, "up1"), e1], 1), "dec1"), 0.01)
        return conv(d, "final")

    out = []
    for h in hist.double().split(100):
        if interval:
            y = net(F.pad(h.reshape(-1, 1, 100), (2, 2)))[:, :, 2:102]
        else:
            y = net(h.reshape(-1, 1, N_BINS))
        out.append(y.reshape(-1, N_BINS))
    return torch.cat(out)


def _weights64(width):
    return {k: tuple(torch.from_numpy(a).double().cuda() for a in v) for k, v in _weights(width).items()}


def _peaks64(logit):
    """(z [n, MAX_PV] with zeros past the count, count [n]): decisions on the float32 logits, centroids in 64 bits."""
    n = logit.shape[0]
    f = F.pad(logit, (5, 5), value=-math.inf)
    peak = logit > float(np.float32(math.log(0.01 / 0.99)))
    for d in range(1, 6):
        peak &= (logit > f[:, 5 - d:5 - d + N_BINS]) & (logit >= f[:, 5 + d:5 + d + N_BINS])
    p = F.pad(torch.sigmoid(logit.double()), (3, 3))
    num = sum(d * p[:, 3 + d:3 + d + N_BINS] for d in range(-3, 4))
    den = sum(p[:, 3 + d:3 + d + N_BINS] for d in range(-3, 4))
    ev, at = torch.nonzero(peak, as_tuple=True)
    z = torch.zeros((n, MAX_PV), dtype=torch.float64, device="cuda")
    slot = torch.cumsum(peak, 1)[ev, at] - 1
    z[ev, slot] = -100.0 + 0.1 * (at + 0.5 + (num / den)[ev, at])
    return z, peak.sum(1).int()


# ------------------------------------------------------------------ the cases

def _input(c, seed):
    """What the entry point of this case reads."""
    n = c["events"]
    if c["entry"] in ("infer", "graph", "histogram"):
        return _events(c["kind"], n, seed)
    w = _weights64(16 if c["entry"] == "peaks" else c["width"])
    if c["entry"] == "unet":
        return (_histogram64(w, *_events(c["kind"], n, seed), 0.0).float(),)
    # logits of a few events through the network, reused at other scales to fill the batch
    base = _unet64(w, _histogram64(w, *_events(c["kind"], min(n, 48), seed), 0.0), False).float()
    g = torch.Generator("cuda").manual_seed(seed + 1)
    pick = torch.randint(0, base.shape[0], (n,), generator=g, device="cuda")
    scale = 0.5 + torch.rand((n, 1), generator=g, device="cuda")
    return ((base[pick] * scale).contiguous(),)


def prepare(case, seed):
    c = {**DEFAULTS, **case}
    n = c["events"]
    args = _input(c, seed)
    weights = _weights(c["width"])
    scales = None
    if c["precision"] == "fp8":
        calib = PVFinder(weights, precision="bf16", max_events=128, max_pv_per_event=8, per_interval=c["interval"])
        scales = calib.calibrate(*_events("standard", 128, 1))
        calib.close()
    pv = PVFinder(weights, precision=c["precision"], max_events=max(n, c["capacity"]), max_pv_per_event=MAX_PV,
                  fp8_act_scales=scales, boundary_mm=c["boundary_mm"], per_interval=c["interval"])
    state = {"case": c, "pv": pv, "args": args}
    if c["entry"] in ("infer", "graph", "peaks"):
        state["z"] = torch.zeros((max(n, c["capacity"]), MAX_PV), device="cuda")
        state["count"] = torch.zeros((max(n, c["capacity"]),), dtype=torch.int32, device="cuda")
    if c["entry"] in ("infer", "unet"):
        state["logit"] = torch.zeros((n, N_BINS), device="cuda")
    if c["entry"] == "histogram":
        state["hist"] = torch.zeros((n, N_BINS), device="cuda")
    if c["entry"] == "graph":
        feats, offsets = args
        slots = torch.full((c["capacity"] + 1,), int(offsets[-1]), dtype=torch.int32, device="cuda")
        slots[:n + 1] = offsets
        state["slots"] = slots
        state["n"] = torch.tensor([n], dtype=torch.int32, device="cuda")
        state["graph"] = pv.capture_graph_dynamic(feats, slots, state["n"], (state["z"], state["count"]))
    return state


def run(state):
    pv, entry = state["pv"], state["case"]["entry"]
    if entry == "infer":
        pv.infer(*state["args"], out=(state["z"], state["count"]), logit=state["logit"])
        return {"z": state["z"], "count": state["count"], "logit": state["logit"]}
    if entry == "graph":
        state["graph"].launch()
        return {"z": state["z"], "count": state["count"]}
    if entry == "histogram":
        return {"hist": pv.stage_histogram(*state["args"], state["hist"])}
    if entry == "unet":
        return {"logit": pv.stage_unet(*state["args"], state["logit"])}
    pv.stage_peaks(*state["args"], out=(state["z"], state["count"]))
    return {"z": state["z"], "count": state["count"]}


def work(case):
    c = {**DEFAULTS, **case}
    n, entry = c["events"], c["entry"]
    tracks = n * (UNEVEN_TRACKS if c["kind"] == "uneven" else STANDARD_TRACKS)
    fc = 2 * 7584 * tracks if entry in ("infer", "graph", "histogram") else 0
    unet = 2 * _unet_macs(c["width"], c["interval"]) * n if entry in ("infer", "graph", "unet") else 0
    reads = {"infer": 36 * tracks + 4 * n, "graph": 36 * tracks + 4 * n, "histogram": 36 * tracks + 4 * n,
             "unet": 4 * N_BINS * n, "peaks": 4 * N_BINS * n}[entry]
    lists = n * (4 + 4 * 200)      # about 200 vertices per event with these weights
    writes = {"infer": lists + 4 * N_BINS * n, "graph": lists, "histogram": 4 * N_BINS * n,
              "unet": 4 * N_BINS * n, "peaks": lists}[entry]
    return {"bytes": reads + writes, "flops": fc + unet}


def _unet_macs(width, interval):
    """Multiply-adds of the UNet on one event's 4000 bins (per-interval: 40 windows of 104)."""
    c, length = width, (40 * 104 if interval else N_BINS)
    conv = (5 * 1 * c * length + 5 * c * 2 * c * length // 2 + 5 * 2 * c * 4 * c * length // 4
            + 5 * 4 * c * 8 * c * length // 8 + 5 * 8 * c * 4 * c * length // 4 + 5 * 4 * c * 2 * c * length // 2
            + 5 * 2 * c * c * length + 5 * c * length)
    up = 2 * 8 * c * 4 * c * length // 8 + 2 * 4 * c * 2 * c * length // 4 + 2 * 2 * c * c * length // 2
    return conv + up


def exact(case, seed):
    c = {**DEFAULTS, **case}
    if c["events"] * (c["width"] // 16) ** 2 > 2500:
        return None
    args = _input(c, seed)
    w = _weights64(c["width"])
    if c["entry"] == "peaks":
        z, count = _peaks64(*args)
        return {"z": z, "count": count}
    if c["entry"] == "unet":
        return {"logit": _unet64(w, *args, c["interval"])}
    if c["entry"] == "graph":
        return None     # vertex lists alone: one decision that falls the other way shifts a list
    hist = _histogram64(w, *args, c["boundary_mm"])
    if c["entry"] == "histogram":
        return {"hist": hist}
    return {"z": None, "count": None, "logit": _unet64(w, hist, c["interval"])}
