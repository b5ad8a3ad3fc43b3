"""The front's FC passes take tracks in tiles (8 or 32 per warp, 256 per chunk, 48 values summed at
a time in the float32 form; 128 or 256 per pass on the tensor cores) and in the float32 form a
cluster of up to eight blocks shares an event by slices where a launch has few: events at the edges
of all of these, their tracks crowded into one slice or spread over all, against the float64 oracle
(the bars of the other histogram tests), and bit for bit the same at every number of events."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

COUNTS = (0, 1, 7, 8, 9, 31, 32, 33, 47, 48, 49, 64, 65, 96, 97, 127, 128, 129, 255, 256, 257, 305, 513, 700)


@pytest.mark.parametrize("edge", [0.0, 0.5])
@pytest.mark.parametrize("crowd", [False, True])
@pytest.mark.parametrize("precision,tol", [("fp32", 1e-4), ("fp16", 4e-3), ("bf16", 3e-2)])
def test_tile_edges_and_shared_events(precision, tol, crowd, edge):
    from paper_2602_19959_gb300 import build, PVFinder
    build()
    w = synth.he_weights(0, bias_std=0.05)
    rng = np.random.default_rng(11)
    n = sum(COUNTS)
    feats = rng.normal(0.0, 0.1, (9, n)).astype(np.float32)
    feats[2] = rng.uniform(61.0, 69.0, n) if crowd else rng.uniform(-100.0, 300.0, n)
    feats[2, ::29] = 350.0                                  # dropped tracks
    offs = np.concatenate([[0], np.cumsum(COUNTS)]).astype(np.int32)
    ref = oracle.infer(w, feats, offs, want_hist=True, nthreads=8, edge_mm=edge)["hist"]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    k = len(COUNTS)
    most = 2 * sms + k
    pv = PVFinder(w, precision=precision, max_events=most, max_pv_per_event=8, boundary_mm=edge)
    f = torch.from_numpy(feats).cuda()

    def run(pick):                                          # the picked events, gathered, as one call
        cols = torch.cat([torch.arange(offs[e], offs[e + 1]) for e in pick]).cuda()
        o = np.concatenate([[0], np.cumsum([COUNTS[e] for e in pick])]).astype(np.int32)
        out = torch.full((len(pick), 4000), -1.0, device="cuda")
        pv.stage_histogram(f[:, cols].contiguous(), torch.from_numpy(o).cuda(), out)
        return out.cpu().numpy()

    got = run(range(k))
    np.testing.assert_array_equal(got == 0, ref == 0)
    assert np.abs(got - ref).max() <= tol * ref.max()
    for m in (1, 2, sms // 4, sms // 4 + 1, sms // 2, sms // 2 + 1, sms, sms + 1, most):
        pick = [(e + k - 1) % k for e in range(m)]          # the largest event first
        assert np.array_equal(run(pick).view(np.int32), got[pick].view(np.int32)), m
    assert pv.device_status() == 0
    pv.close()


def test_track_pointers_of_a_matrix_and_of_its_rows():
    """The addresses taken from a matrix are those of its nine rows, in every form that is taken,
    and what the rows are refused for the matrix is refused for."""
    from paper_2602_19959_gb300.pvf import tracks_struct
    m = torch.zeros((12, 64), device="cuda")
    taken = [m, m[:9], m[1:], m[2:11, 3:40], m[:, :1], m[:, 5:5], m[::1, 7:8], m.int(), m[:1].expand(9, 64),
             m[:, ::64], m.t().contiguous().t()[:, :1], torch.zeros((18, 8), device="cuda")[::2],
             torch.zeros((9, 0), device="cuda"), torch.nn.Parameter(m), m.view(12, 64, 1), m.view(12, 8, 8), m[0]]
    for t in taken:
        a, b = tracks_struct(t), tracks_struct([t[k] for k in range(9)])
        assert a.n_tracks == b.n_tracks and list(a.f) == list(b.f), tuple(t.shape)
    refused = [m.t().contiguous().t(), m[:, ::2], m.half(), m.double(), m.cpu(), m[:8]]
    for t in refused:
        with pytest.raises((ValueError, IndexError)):
            tracks_struct(t)
        with pytest.raises((ValueError, IndexError)):
            tracks_struct([t[k] for k in range(9)])
