"""Pairs that no shared bound decides, GPU against oracle: level 0 and bisected cells so wide that a
tile, a tan(lambda) bin or a parent has no bound for most hits (there the FP32 votes are the program's
own, several bins after one prefix)."""
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


@pytest.mark.parametrize("prec,oprec", PRECS)
@pytest.mark.parametrize("bins", [[4, 4, 4, 4, 4], [5, 6, 6, 5, 5], [16, 3, 2, 16, 7], [2, 3, 2, 3, 32]])
def test_wide_cells(bins, prec, oprec):
    w, g = chamber.make_wires(), G.make_grid(bins, 2, 9)
    ev = chamber.multi_track_events(2, seed=sum(bins), w=w)
    geom, tab, hits = apo.Geometry(g, w), O.Tables(g, w), apo.DeviceHits.from_events(ev)
    votes = apo.vote(geom, hits, precision=prec).cpu().numpy()
    tracks, _ = apo.solve_batch(geom, hits, apo.solve_opts(precision=[prec] * 3))
    got = apo.tracks_to_numpy(tracks, ev.n_events)
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        np.testing.assert_array_equal(votes[e], O.vote_coarse(tab, ev.wire_id[a:b], ev.drift[a:b], oprec))
        r = O.solve_event(tab, ev.wire_id[a:b], ev.drift[a:b], [oprec] * 3)
        assert got[e, 0]["votes"] == r["votes"]
        assert np.array_equal(got[e, 0]["p"], r["p"]) and np.array_equal(got[e, 0]["w"], r["w"])
    geom.close()


@pytest.mark.parametrize("prec,oprec", PRECS[2:])
def test_direction_left_open(prec, oprec):
    """Tiles whose bound is too wide for the direction condition of some cells, many bins each."""
    w, g = chamber.make_wires(), G.make_grid([16, 8, 4, 16, 7], 1, 9)
    ev = chamber.single_track_events(2, seed=9, w=w)
    geom, tab = apo.Geometry(g, w), O.Tables(g, w)
    votes = apo.vote(geom, apo.DeviceHits.from_events(ev), precision=prec).cpu().numpy()
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        np.testing.assert_array_equal(votes[e], O.vote_coarse(tab, ev.wire_id[a:b], ev.drift[a:b], oprec))
    geom.close()


@pytest.mark.parametrize("og", [0, apo.OUTGOING])
@pytest.mark.parametrize("bins", [[3, 2, 2, 3, 3], [1, 1, 2, 1, 1], [4, 3, 4, 2, 5]])
def test_fp32_overflow_keeps_fp64_votes(bins, og):
    """Half-turn cells and wires without stereo in every other place: FP32 ends overflow and meet exact
    zeros; the votes are the oracle's and contain the FP64 ones."""
    w, g = chamber.make_wires(), G.make_grid(bins, 2, 2)
    ev = chamber.multi_track_events(3, seed=20, w=w)
    for name in ("tan_tau", "sphi_t", "cphi_t", "t2"):
        getattr(w, name)[::2] = 0.0
    geom, tab, hits = apo.Geometry(g, w), O.Tables(g, w), apo.DeviceHits.from_events(ev)
    v32, v64 = (apo.vote(geom, hits, precision=p | og).cpu().numpy() for p in (apo.F32, apo.F64))
    assert np.all(v32 >= v64)
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        np.testing.assert_array_equal(v32[e], O.vote_coarse(tab, ev.wire_id[a:b], ev.drift[a:b], 1 | og))
        np.testing.assert_array_equal(v64[e], O.vote_coarse(tab, ev.wire_id[a:b], ev.drift[a:b], 0 | og))
    geom.close()
