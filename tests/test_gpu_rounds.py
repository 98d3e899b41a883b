"""Multi-track top-K rounds, GPU against oracle: events whose extraction ends in different rounds (and empty,
short and malformed ones) in one batch, in one chunk and in several, directly and by graph replay, with
the K best cells per tile and with full votes; the launches of later rounds leave ended events alone."""
import numpy as np
import pytest

from gen import chamber, grid as G
from oracle import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2401_04576_gb300 import apo  # noqa: E402

BINS, LEVELS, TOPK, TRACKS, MIN = [6, 7, 6, 5, 6], 3, 16, 4, 5
PREC, OPREC = [apo.F32, apo.F32, apo.F64, apo.F64], [1, 1, 0, 0]


@pytest.fixture(scope="module")
def batch():
    w, g = chamber.make_wires(), G.make_grid(BINS, LEVELS, TOPK)
    ev = chamber.multi_track_events(19, seed=31, w=w)
    per = [(ev.wire_id[a:b], ev.drift[a:b].copy()) for a, b in zip(ev.offsets[:-1], ev.offsets[1:])]
    per.insert(4, (per[0][0][:0], per[0][1][:0]))     # no hit
    per.insert(11, (per[1][0][:3], per[1][1][:3]))    # too few for a track
    per[14][1][0] = -1.0                              # malformed
    offsets = np.concatenate([[0], np.cumsum([len(a) for a, _ in per])]).astype(np.int32)
    ev = chamber.Events(offsets=offsets, wire_id=np.concatenate([a for a, _ in per]).astype(np.int32),
                        drift=np.concatenate([d for _, d in per]))
    tab = O.Tables(g, w)
    ref = [None if np.any(d < 0) else O.solve_event_multi(tab, a, d, TRACKS, MIN, prec_per_level=OPREC) for a, d in per]
    assert len({r["n_tracks"] for r in ref if r}) >= 3   # extractions end in different rounds
    return w, g, ev, ref


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("chunk", [0, 5])
@pytest.mark.parametrize("full,persistent", [(0, 0), (1, 0), (0, 1)])
def test_rounds_end_apart(batch, full, persistent, chunk, graph):
    w, g, ev, ref = batch
    geom, hits, n = apo.Geometry(g, w), apo.DeviceHits.from_events(ev), int(ev.offsets[-1])
    ht = torch.full((n,), -5, dtype=torch.int32, device="cuda")
    o = apo.solve_opts(precision=PREC, max_tracks=TRACKS, min_votes=MIN, hit_track=ht, use_graph=graph,
                       tune=apo.ApoTune(0, 1, 256, chunk, coarse_full=full, persistent=persistent))
    ws = geom.workspace(ev.n_events, opts=o)
    out = torch.zeros(ev.n_events * TRACKS * apo.TRACK_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    nt = torch.zeros(ev.n_events, dtype=torch.int32, device="cuda")
    for _ in range(2):   # the second pass finds the first one's flags and masks in the workspace
        apo.solve_batch(geom, hits, o, tracks=out, n_tracks=nt, workspace=ws)
        torch.cuda.synchronize()
        t, k, h = apo.tracks_to_numpy(out, ev.n_events, TRACKS), nt.cpu().numpy(), ht.cpu().numpy()
        for e, r in enumerate(ref):
            if r is None:
                assert k[e] == 0 and t[e, 0]["votes"] == apo.APO_EINVAL
                continue
            assert k[e] == r["n_tracks"], e
            for i in range(k[e]):
                assert t[e, i]["votes"] == r["votes"][i]
                assert np.array_equal(t[e, i]["p"], r["p"][i]) and np.array_equal(t[e, i]["w"], r["w"][i])
            assert np.array_equal(h[ev.offsets[e]:ev.offsets[e + 1]], r["hit_track"])
    geom.close()


def test_autotune_leaves_the_accepted_knobs_off(batch):
    w, g, ev, _ = batch
    geom = apo.Geometry(g, w)
    best, ms = apo.autotune(geom, apo.DeviceHits.from_events(ev),
                            apo.solve_opts(precision=PREC, max_tracks=TRACKS, min_votes=MIN))
    assert ms > 0 and best.persistent == 0 and best.coarse_filter == 0
    geom.close()
