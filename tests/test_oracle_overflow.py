"""FP32 overflow in the oracle (CPU): FP32 intervals contain the FP64 ones, so an FP64 vote is an FP32
vote, also where FP32 end points overflow (the phase correction of quarter-turn cells passes 1e39)."""
import numpy as np
import pytest

from gen import chamber, grid as G
from oracle import oracle as O


@pytest.mark.parametrize("og", [0, O.OUTGOING])
def test_fp32_votes_contain_fp64_votes(og):
    w, g = chamber.make_wires(), G.make_grid([4] * 5, 2, 9)
    tab, ev = O.Tables(g, w), chamber.multi_track_events(2, seed=20, w=w)
    keys, over = O.coarse_keys(tab), 0
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        v64, v32 = (O.vote_cells(tab, ev.wire_id[a:b], ev.drift[a:b], 0, keys, p | og) for p in (0, 1))
        assert np.all(v32 >= v64)
        for c in range(0, len(keys), 2):
            cell = O.cell12(g, 0, [int(i) for i in G.coarse_index_to_idx5(c, g.bins)])
            over += sum(np.isinf(O.vote_pair(cell, O.hit9(w, ev.wire_id[i], ev.drift[i]), 1 | og)[1][5:]).any()
                        for i in range(a, b))
    assert over > 0   # some pairs did overflow
