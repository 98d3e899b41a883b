"""The certified FP32 end points (csrc/certified.cuh), compiled as host C++, against the oracle's
FP64 and FP32 end points of G: a parent cell's error bound must hold for the bare end points of
cells inside it, and every decision taken with it must be the oracle's vote.  Grids: the bench's,
ragged ones with the widest cells, the anisotropic one; parents are level-0 tiles (all d0, z0 and
tan(lambda) bins of a phi0 and omega bin) and bisected cells near the generated helices; plus
wires without stereo, d = 0 and cells whose omega reaches 0, where nothing may be decided
wrongly.  The host build uses exact reciprocals and roots; the device's differ from them by the
documented 2^-23 that the bound contains, and the device votes are compared with the oracle's in
the parity tests."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from gen import chamber, grid as G
from oracle import oracle as O

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2401_04576_gb300", "csrc")

SHIM = r"""
#include <cmath>
#include "certified.cuh"
using namespace apo::cert;
static float down(double x) { float f = (float)x; return (double)f > x ? std::nextafter(f, -INFINITY) : f; }
template <int K> static void load(const double *c, const double *h, CellX<K> &cc, HitX<K> &hh) {
    const bool mir = c[7] < 0;
    const int flip[6] = {1, 1, 0, 1, 0, 0};
    X<K> *f = &cc.D;
    for (int a = 0; a < 6; a++)
        f[a] = mir && flip[a] ? mk<K>(-c[2 * a + 1], -c[2 * a]) : mk<K>(c[2 * a], c[2 * a + 1]);
    Sc<K> *s = &hh.x0;
    for (int i = 0; i < 8; i++) s[i] = sc<K>((mir && (i == 1 || i == 3 || i == 6)) ? -down(h[i]) : down(h[i]));
    hh.d = point(sc<K>(down(h[8])));
}
template <int K> static int one(const double *c, const double *h, int og) {
    CellX<K> cc; HitX<K> hh;
    load(c, h, cc, hh);
    const Eval<K> r = eval(cc, hh, true);
    return verdict(r, og != 0, bound(r));
}
extern "C" int single(int k, const double *c, const double *h, int og) {
    return k == 64 ? one<64>(c, h, og) : one<32>(c, h, og);
}
template <int K> static float par(const double *c, const double *h, int og, int *no) {
    CellX<K> cc; HitX<K> hh;
    load(c, h, cc, hh);
    const Eval<K> r = eval(cc, hh);
    const float e = bound(r);
    *no = verdict(r, og != 0, e) == kNo;
    return e;
}
extern "C" float parent(int k, const double *c, const double *h, int og, int *no) {
    return k == 64 ? par<64>(c, h, og, no) : par<32>(c, h, og, no);
}
extern "C" int child(const double *c, const double *h, float e, int og, float *out) {
    CellX<0> cc; HitX<0> hh;
    load(c, h, cc, hh);
    const Eval<0> r = eval(cc, hh);
    out[0] = r.Gp.lo; out[1] = r.Gp.hi; out[2] = r.Gm.lo; out[3] = r.Gm.hi;
    return verdict(r, og != 0, e);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("cert")
    src, so = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-shared", "-fPIC", src, "-o", so], check=True)
    L = C.CDLL(so)
    d8 = C.POINTER(C.c_double)
    L.parent.restype = C.c_float
    L.parent.argtypes = [C.c_int, d8, d8, C.c_int, C.POINTER(C.c_int)]
    L.child.argtypes = [d8, d8, C.c_float, C.c_int, C.POINTER(C.c_float)]
    return L


def _p(a):
    return np.ascontiguousarray(a, np.float64).ctypes.data_as(C.POINTER(C.c_double))


def _span(g, i0, i1):
    c, c1 = O.cell12(g, 0, i0), O.cell12(g, 0, i1)
    for k in (0, 3, 4, 5):
        c[2 * k + 1] = c1[2 * k + 1]
    return c


@pytest.mark.parametrize("og", [0, 1])
@pytest.mark.parametrize("k", [64, 32])
@pytest.mark.parametrize("bins,levels", [([16] * 5, 6), ([2, 256, 16, 2, 8], 5), ([5, 6, 6, 5, 5], 5),
                                         ([7, 6, 8, 5, 9], 2)])
def test_bounds_and_decisions(lib, bins, levels, k, og):
    w, g = chamber.make_wires(), G.make_grid(bins, levels, 64)
    rng = np.random.default_rng(sum(bins) + k)
    ev = chamber.single_track_events(6, seed=17, w=w)
    prec = (0 if k == 64 else 1) | (O.OUTGOING if og else 0)
    decided = undecided = alone = far = 0
    for n in range(500):
        e = int(rng.integers(ev.n_events))
        i = int(rng.integers(ev.offsets[e], ev.offsets[e + 1]))
        h = O.hit9(w, ev.wire_id[i], ev.drift[i])
        if n % 10 == 8:
            h[4:8] = 0.0
        if n % 10 == 9:
            h[8] = 0.0
        if n % 2:   # a level-0 tile
            p, o = int(rng.integers(bins[1])), int(rng.integers(bins[2]))
            P = _span(g, [0, p, o, 0, 0], [bins[0] - 1, p, o, bins[3] - 1, bins[4] - 1])
            kids = [O.cell12(g, 0, [int(rng.integers(bins[0])), p, o, int(rng.integers(bins[3])),
                                    int(rng.integers(bins[4]))]) for _ in range(6)]
        else:       # a kept cell and its children
            lv, par = int(rng.integers(levels)), ev.tracks[e][0].params
            at = []
            for a in range(5):
                edges = g.lo_edge[a][::1 << (levels - lv)]
                j = int(np.searchsorted(edges, par[a], side="right")) - 1 + int(rng.integers(-1, 2))
                at.append(min(max(j, 0), len(edges) - 1))
            P = O.cell12(g, lv, at)
            kids = [O.cell12(g, lv + 1, [2 * at[a] + ((b >> a) & 1) for a in range(5)])
                    for b in rng.choice(32, 6, replace=False)]
        no = C.c_int()
        err = lib.parent(k, _p(P), _p(h), og, C.byref(no))
        if no.value:
            assert O.vote_pair(P, h, prec)[0] == 0
        for c in kids:
            v, ref = O.vote_pair(c, h, prec)
            assert not (no.value and v)
            out = np.zeros(4, np.float32)
            d = lib.child(_p(c), _p(h), C.c_float(err), og, out.ctypes.data_as(C.POINTER(C.c_float)))
            if np.isnan(err):
                assert d == 2
            if ref[4] == 0 and not np.isnan(err):   # evaluated by the oracle
                assert np.abs(out.astype(np.float64) - ref[:4]).max() <= err
            assert d == 2 or d == v
            decided += d != 2
            undecided += d == 2
            d = lib.single(k, _p(c), _p(h), og)   # by its own bound, |delta| > 1 included
            assert d == 2 or d == v
            far += abs(ref[5:]).max() > 1.0 and d != 2
            alone += d == 2
    assert decided > 20 * undecided and undecided >= alone
    if bins == [5, 6, 6, 5, 5] and not og:
        assert far > 0


def test_nothing_is_decided_at_a_guard_or_overflow(lib):
    w, g = chamber.make_wires(), G.make_grid([16] * 5, 6, 64)
    ev = chamber.single_track_events(1, seed=3, w=w)
    h = O.hit9(w, ev.wire_id[0], ev.drift[0])
    no = C.c_int()
    for lo, hi in ((-0.05, 0.05), (0.0, 0.05), (0.2, 1e300)):
        c = O.cell12(g, 0, [3, 4, 12, 5, 6]).copy()
        c[6], c[7] = lo, hi
        assert np.isnan(lib.parent(64, _p(c), _p(h), 0, C.byref(no))) and not no.value
    c = O.cell12(g, 0, [3, 4, 12, 5, 6])
    for drift in (1e38, 1e300, np.inf):
        h[8] = drift
        assert np.isnan(lib.parent(64, _p(c), _p(h), 0, C.byref(no))) and not no.value
