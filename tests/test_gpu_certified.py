"""Votes decided by certified FP32 values, GPU against oracle, at the shapes where the deciding code
can go wrong: level-0 tiles of few cells (several tiles per block) and of two parts, tan(lambda)
bins that straddle 0, one bin and 32; children of a number of kept cells that leaves a block
partly filled; keys whose warp mixes both signs of omega, invalid keys and a partial warp; cells so
wide that no bound decides anything, with more hits than one queue step, so that the queue of
undecided pairs is drained many times."""
import numpy as np
import pytest

from gen import chamber, grid as G
from oracle import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2401_04576_gb300 import apo  # noqa: E402

PRECS = [(apo.F64, 0), (apo.F32, 1), (apo.F64 | apo.OUTGOING, 0 | O.OUTGOING), (apo.F32 | apo.OUTGOING, 1 | O.OUTGOING)]


def _check(geom, tab, ev, grid, level, keys, prec, oprec):
    kt = None if keys is None else torch.as_tensor(keys.view(np.int64), device="cuda")
    got = apo.vote(geom, apo.DeviceHits.from_events(ev), keys=kt, level=level, precision=prec).cpu().numpy()
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        ref = (O.vote_coarse(tab, ev.wire_id[a:b], ev.drift[a:b], oprec) if keys is None else
               O.vote_cells(tab, ev.wire_id[a:b], ev.drift[a:b], level, keys[e], oprec))
        np.testing.assert_array_equal(got[e], ref)


@pytest.mark.parametrize("prec,oprec", PRECS)
@pytest.mark.parametrize("bins", [[2, 37, 4, 2, 8], [1, 19, 6, 1, 1], [1, 5, 2, 3, 32], [16, 3, 2, 16, 7], [3, 2, 2, 43, 5]])
def test_coarse_tiles(bins, prec, oprec):
    w, g = chamber.make_wires(), G.make_grid(bins, 2, 16)
    ev = chamber.multi_track_events(2, seed=sum(bins), w=w)
    geom = apo.Geometry(g, w)
    _check(geom, O.Tables(g, w), ev, g, 0, None, prec, oprec)
    geom.close()


@pytest.mark.parametrize("prec,oprec", PRECS)
@pytest.mark.parametrize("topk", [1, 9, 33])
def test_children_and_keys(topk, prec, oprec):
    w, g = chamber.make_wires(), G.make_grid([4, 9, 6, 3, 5], 3, topk)
    ev = chamber.multi_track_events(2, seed=topk, w=w)
    geom, tab = apo.Geometry(g, w), O.Tables(g, w)
    o = apo.solve_opts(precision=[prec] * 4)
    tracks, _ = apo.solve_batch(geom, apo.DeviceHits.from_events(ev), o)
    got = apo.tracks_to_numpy(tracks, ev.n_events)
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        r = O.solve_event(tab, ev.wire_id[a:b], ev.drift[a:b], [oprec] * 4)
        assert got[e, 0]["votes"] == r["votes"]
        assert np.array_equal(got[e, 0]["p"], r["p"]) and np.array_equal(got[e, 0]["w"], r["w"])
    rng = np.random.default_rng(topk)
    for level in (0, 2):
        n = [int(x) << level for x in g.bins]
        idx = rng.integers(0, n, size=(ev.n_events, 32 * topk + 5, 5))
        keys = np.stack([G.cell_key(i) for i in idx]).astype(np.uint64)
        keys[:, 1::7] |= np.uint64(1023)   # d0 index past the grid: -1 votes
        kt = torch.as_tensor(keys.view(np.int64), device="cuda")
        got = apo.vote(geom, apo.DeviceHits.from_events(ev), keys=kt, level=level, precision=prec).cpu().numpy()
        assert np.all(got[:, 1::7] == -1)
        ok = np.ones(keys.shape[1], bool)
        ok[1::7] = False
        for e in range(ev.n_events):
            a, b = ev.offsets[e], ev.offsets[e + 1]
            ref = O.vote_cells(tab, ev.wire_id[a:b], ev.drift[a:b], level, np.ascontiguousarray(keys[e][ok]), oprec)
            np.testing.assert_array_equal(got[e][ok], ref)
    geom.close()


@pytest.mark.parametrize("prec,oprec", PRECS)
def test_nothing_decidable(prec, oprec):
    w, g = chamber.make_wires(), G.make_grid([16, 2, 2, 16, 3], 1, 8)   # half-turn cells
    ev = chamber.multi_track_events(3, seed=73, w=w)
    assert int(np.diff(ev.offsets).max()) > 40
    geom = apo.Geometry(g, w)
    _check(geom, O.Tables(g, w), ev, g, 0, None, prec, oprec)
    geom.close()
