"""Votes of explicit keys, GPU against oracle, over the ways a warp's 32 keys can lie: one cell's
children, near a track, sorted over all phi0 on one side of omega = 0, on both sides, so wide that no
hit or only some have a bound, with keys outside the grid, and fewer keys than a warp."""
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


def _keys(kind, g, level, par, rng, n):
    nb = np.array([int(b) << level for b in g.bins])
    at = []
    for a in range(5):
        edges = g.lo_edge[a][::1 << (g.levels - level)]
        at.append(int(np.searchsorted(edges, par[a], side="right")) - 1)
    if kind == "children":
        base = np.clip((np.array(at) // 2) + rng.integers(-1, 2, size=(n // 32 + 1, 5)), 0, nb // 2 - 1)
        idx = (2 * base[:, None, :] + ((np.arange(32)[:, None] >> np.arange(5)) & 1)).reshape(-1, 5)[:n]
    elif kind == "near":
        idx = np.clip(np.array(at) + rng.integers(-3, 4, size=(n, 5)), 0, nb - 1)
    else:
        idx = rng.integers(0, nb, size=(n, 5))
        if kind == "one side":   # sorted, omega > 0
            idx[:, 2] = rng.integers(nb[2] // 2, nb[2], size=n)
            idx = idx[np.lexsort(idx.T)]
    return G.cell_key(idx, g).astype(np.uint64)


@pytest.mark.parametrize("prec,oprec", PRECS)
@pytest.mark.parametrize("kind", ["children", "near", "one side", "scattered"])
@pytest.mark.parametrize("bins,levels,level", [([10] * 5, 4, 3), ([5, 6, 6, 5, 5], 2, 1), ([4, 5, 2, 4, 3], 2, 1)])
def test_key_sets(bins, levels, level, kind, prec, oprec):
    w, g = chamber.make_wires(), G.make_grid(bins, levels, 9)
    ev = chamber.multi_track_events(2, seed=sum(bins) + level, w=w)
    geom, tab, hits = apo.Geometry(g, w), O.Tables(g, w), apo.DeviceHits.from_events(ev)
    rng = np.random.default_rng(levels)
    for n in (19, 640):
        keys = np.stack([_keys(kind, g, level, ev.tracks[e][0].params, rng, n) for e in range(ev.n_events)])
        bad = rng.integers(0, n, size=n // 8)
        sent = keys.copy()
        sent[:, bad] |= np.uint64(1023)   # d0 index past the grid
        got = apo.vote(geom, hits, keys=torch.as_tensor(sent.view(np.int64), device="cuda"), level=level,
                       precision=prec).cpu().numpy()
        ok = np.ones(n, bool)
        ok[bad] = False
        assert np.all(got[:, bad] == -1)
        for e in range(ev.n_events):
            a, b = ev.offsets[e], ev.offsets[e + 1]
            ref = O.vote_cells(tab, ev.wire_id[a:b], ev.drift[a:b], level, np.ascontiguousarray(keys[e][ok]), oprec)
            np.testing.assert_array_equal(got[e][ok], ref)
    geom.close()
