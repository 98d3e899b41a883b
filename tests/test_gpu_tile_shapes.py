"""Exact-phase and midpoint-form votes, GPU against oracle, at the level-0 tile shapes where the block
layout can go wrong: fewer (d0, z0) cells than a warp, than hit-mask words or than tan(lambda) bins,
several tiles side by side with a ragged last block, and tiles of two parts; as full votes, as
K best cells per tile and as the max-set schedule's level 0."""
import numpy as np
import pytest

from gen import chamber, grid as G
from oracle import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2401_04576_gb300 import apo  # noqa: E402

OUT = apo.OUTGOING
PRECS = [(apo.F64_EXACT, 4), (apo.F64_EXACT | OUT, 4 | O.OUTGOING), (apo.F64_MID, 3)]
BINS = [[2, 37, 4, 2, 8], [1, 19, 6, 1, 1], [1, 5, 2, 3, 32], [3, 7, 2, 5, 9], [16, 2, 2, 9, 5]]


def _setup(bins, levels, topk):
    w = chamber.make_wires()
    g = G.make_grid(bins, levels, topk)
    # events of more than 32 hits next to short ones
    ev = chamber.multi_track_events(2, seed=sum(bins), w=w)
    return w, g, ev, apo.Geometry(g, w), O.Tables(g, w)


@pytest.mark.parametrize("prec,oprec", PRECS)
@pytest.mark.parametrize("bins", BINS)
def test_full_votes(bins, prec, oprec):
    w, g, ev, geom, tab = _setup(bins, 1, 8)
    got = apo.vote(geom, apo.DeviceHits.from_events(ev), precision=prec).cpu().numpy()
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        np.testing.assert_array_equal(got[e], O.vote_coarse(tab, ev.wire_id[a:b], ev.drift[a:b], oprec))
    geom.close()


@pytest.mark.parametrize("full", [0, 1])
@pytest.mark.parametrize("prec,oprec", PRECS + [(apo.F64, 0), (apo.F32 | OUT, 1 | O.OUTGOING)])
@pytest.mark.parametrize("bins", BINS)
def test_topk_search(bins, prec, oprec, full):
    w, g, ev, geom, tab = _setup(bins, 2, 9)
    o = apo.solve_opts(precision=[prec] * 3, tune=apo.ApoTune(0, 1, 256, 0, coarse_full=full))
    tracks, _ = apo.solve_batch(geom, apo.DeviceHits.from_events(ev), o)
    got = apo.tracks_to_numpy(tracks, ev.n_events)
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        r = O.solve_event(tab, ev.wire_id[a:b], ev.drift[a:b], [oprec] * 3)
        assert got[e, 0]["votes"] == r["votes"]
        assert np.array_equal(got[e, 0]["p"], r["p"]) and np.array_equal(got[e, 0]["w"], r["w"])
    geom.close()


@pytest.mark.parametrize("prec,oprec", PRECS)
@pytest.mark.parametrize("bins", [BINS[0], BINS[3]])
def test_maxset_search(bins, prec, oprec):
    w, g, ev, geom, tab = _setup(bins, 1, 8)
    o = apo.solve_opts(precision=[prec] * 2, schedule=apo.SCHED_MAXSET, max_keep=300, slack=1)
    tracks, _ = apo.solve_batch(geom, apo.DeviceHits.from_events(ev), o)
    got = apo.tracks_to_numpy(tracks, ev.n_events)[:, 0]
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        r = O.solve_event_maxset(tab, ev.wire_id[a:b], ev.drift[a:b], 300, 1, [oprec] * 2)
        assert got[e]["votes"] == r["votes"]
        assert np.array_equal(got[e]["p"], r["p"]) and np.array_equal(got[e]["w"], r["w"])
    geom.close()
