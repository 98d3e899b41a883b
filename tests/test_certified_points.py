"""The point programs' certified FP32 forms (csrc/cert4.cuh, csrc/cert_mid.cuh), compiled as host
C++, against the oracle: with the bound of a range of centres (a group of 2 x 2 x 2 columns and their z0 voxels; a level-0
tile or a kept cell's children) every decision must be the oracle's vote, and in FP64 the end points
of G must lie within the bound of the oracle's.  4-D: the three iterations' voxels, FP64 and FP32,
columns that pass the disk pre-filter anywhere in the grid (hits on either side of the centre, phases
near the jump at 0, negative radicands).  The FP32 reference's column constants are its own values
(reference point at the origin, whose phase is exactly 0)."""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

from gen import chamber, comet, grid as G
from oracle import oracle as O

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2401_04576_gb300", "csrc")

SHIM = r"""
#include <cmath>
#include "cert4.cuh"
#include "cert_mid.cuh"
using namespace apo::cert;
static float down(double x) { float f = (float)x; return (double)f > x ? std::nextafter(f, -INFINITY) : f; }

// ---- 4-D: cc = x_c, y_c, R, |tan(lambda)|, -x_c, -y_c, 1 / |(x_c, y_c)|, phase of the reference point
// (lo / hi pairs for a group of columns); box = x, y, R - R_centre (bound) or R (child), lo / hi ----
template <int K> static X<K> w(double a, double b) {
    X<K> r;
    r.lo = (float)a;
    r.hi = (float)b;
    r.e = 2.f * rnd<K>(mag2(r.lo, r.hi)) + kTiny;
    return r;
}
template <int K> static Bound4 b4(const double *cc, const double *box, const double *z, const double *h) {
    Col4X<X<K>> m;
    Hit4X<X<K>> x;
    X<K> *q = &m.xc, *f = &x.x0;
    for (int i = 0; i < 8; i++) q[i] = w<K>(cc[2 * i], cc[2 * i + 1]);
    m.ion.e *= 2.f;
    for (int i = 0; i < 9; i++) f[i] = w<K>(h[i], h[i]);
    return bound4<K>(m, Box4X<K>{w<K>(box[0], box[1]), w<K>(box[2], box[3]), w<K>(box[4], box[5])}, w<K>(z[0], z[1]),
                     w<K>(z[2], z[3]), x);
}
extern "C" float bound_4d(int k, const double *cc, const double *box, const double *z, const double *h, float *eps) {
    const Bound4 r = k == 64 ? b4<64>(cc, box, z, h) : b4<32>(cc, box, z, h);
    *eps = r.eps;
    return r.e;
}
extern "C" int child_4d(const double *cc, const double *box, const double *z, const double *h, int sign, float e,
                        float eps, float *out) {
    Col4X<Pt> m;
    Hit4X<Pt> x;
    Pt *q = &m.xc, *f = &x.x0, dx, dy;
    for (int i = 0; i < 8; i++) q[i].v = (float)cc[i];
    m.ion.v = 1 / std::sqrt(m.xc.v * m.xc.v + m.yc.v * m.yc.v);
    for (int i = 0; i < 9; i++) f[i].v = (float)h[i];
    const Box4X<0> b{mk<0>(box[0], box[1]), mk<0>(box[2], box[3]), mk<0>(box[4] - cc[2], box[5] - cc[2])};
    bool bad;
    wire4x(m, Pt{(float)z[0]}, x, dx, dy);
    Pre4X<Pt> p = prefix4x(dx, dy, x);
    p.psi = psi4(m, dx, dy, p.iRA, eps, bad);
    p.Rpsi = mul(m.R, p.psi);
    const X<0> A2 = a2_4x<0, Pt>(b, mk<0>(z[1], z[2]), x);
    const Delta4<Pt> d0 = delta4x(p, m.R, m.aL, x.d, x), d1 = delta4x(p, m.R, m.aL, neg(x.d), x);
    const float s = sign > 0 ? -1.f : 1.f;
    const Pt dl[2] = {{std::fma(s, d0.v.v, d0.u.v)}, {std::fma(s, d1.v.v, d1.u.v)}}, L{-s * m.aL.v};
    for (int i = 0; i < 2; i++) {
        const float rad = rad4x(p, m.R, L, i ? neg(x.d) : x.d, dl[i], x).v, r = std::sqrt(rad);
        out[3 * i] = rad;
        out[3 * i + 1] = A2.lo - (r + b.dR.hi) * (r + b.dR.hi);
        out[3 * i + 2] = A2.hi - (r + b.dR.lo) * (r + b.dR.lo);
    }
    return bad ? kUnknown : vote4x(p, m, L, x, A2, b.dR, e, dl);
}

// ---- midpoint form: c = cell12; m = lo / hi of the centres D, sin, cos, W, Z, L ----
static Pt mkn(double a, double, Pt) { return Pt{(float)a}; }
static X<64> mkn(double a, double b, X<64>) { return mk<64>(a, b); }
template <int K, typename N>
static void load(const double *c, const double *m, const double *h, CellX<K> &cc, MidCell<N> &mc, MidHit<N> &hx) {
    const bool mir = c[7] < 0;
    const int fl[6] = {1, 1, 0, 1, 0, 0};
    X<K> *f = &cc.D;
    for (int a = 0; a < 6; a++) f[a] = mir && fl[a] ? mk<K>(-c[2 * a + 1], -c[2 * a]) : mk<K>(c[2 * a], c[2 * a + 1]);
    N *q = &mc.D;
    for (int a = 0; a < 5; a++)
        q[a] = mir && fl[a] ? mkn(-m[2 * a + 1], -m[2 * a], N()) : mkn(m[2 * a], m[2 * a + 1], N());
    mc.R = recip(mc.W);
    N *s = &hx.x0;
    for (int i = 0; i < 9; i++) s[i] = numf<N>((mir && (i == 1 || i == 3 || i == 6)) ? -down(h[i]) : down(h[i]));
}
extern "C" float parent_mid(const double *c, const double *m, const double *h, int *no) {
    CellX<64> cc; MidCell<X<64>> mc; MidHit<X<64>> hx;
    load<64, X<64>>(c, m, h, cc, mc, hx);
    X<64> a, b;
    mid_tail<64, X<64>>(mid_prefix<64, X<64>>(cc, mc, hx), mk<64>(m[10], m[11]), mc, hx, cc.W, a, b);
    const float e = (a.e < 1e30f && b.e < 1e30f) ? 1.01f * fmaxf(a.e, b.e) : NAN;
    *no = decide(a, b, e) == kNo;
    return e;
}
extern "C" int child_mid(const double *c, const double *m, const double *h, float e, float *o) {
    CellX<0> cc; MidCell<Pt> mc; MidHit<Pt> hx;
    load<0, Pt>(c, m, h, cc, mc, hx);
    X<0> a, b;
    mid_tail<0, Pt>(mid_prefix<0, Pt>(cc, mc, hx), Pt{(float)m[10]}, mc, hx, cc.W, a, b);
    o[0] = a.lo; o[1] = a.hi; o[2] = b.lo; o[3] = b.hi;
    return decide(a, b, e);
}
"""

D8, F4 = C.POINTER(C.c_double), C.POINTER(C.c_float)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("certp")
    src, so = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-shared", "-fPIC", src, "-o", so], check=True)
    L = C.CDLL(so)
    L.bound_4d.restype, L.bound_4d.argtypes = C.c_float, [C.c_int, D8, D8, D8, D8, F4]
    L.child_4d.argtypes = [D8, D8, D8, D8, C.c_int, C.c_float, C.c_float, F4]
    L.parent_mid.restype, L.parent_mid.argtypes = C.c_float, [D8, D8, D8, C.POINTER(C.c_int)]
    L.child_mid.argtypes = [D8, D8, D8, C.c_float, F4]
    return L


def _a(x):
    return np.ascontiguousarray(x, np.float64)


def _p(x):
    return x.ctypes.data_as(D8)


def _phase(ox, oy, dx, dy):
    a = math.atan2(ox * dy - oy * dx, ox * dx + oy * dy)
    return a if a >= 0 else a + 2 * math.pi


def _sq(a, b):
    lo, hi = a[0] - b[1], a[1] - b[0]
    return max(0.0, lo, -hi) ** 2, max(-lo, hi) ** 2


@pytest.mark.parametrize("k", [64, 32])
@pytest.mark.parametrize("it", [0, 1, 2])
def test_four_d(lib, it, k):
    w = comet.make_wires()
    ev = comet.events(4, 5, w)
    rng = np.random.default_rng(10 * it + k)
    o = O.four_opts()
    W, N = [o.w[it][a] for a in range(4)], [o.n[it][a] for a in range(4)]
    decided = undecided = 0
    for n in range(250):
        e = int(rng.integers(ev.n_events))
        i = int(rng.integers(ev.offsets[e], ev.offsets[e + 1]))
        h = _a(O.hit9(w, ev.wire_id[i], ev.drift[i]))
        if n % 10 == 9:
            h[8] = 0.0
        if k == 32:   # the program's own FP32 values
            h = _a(h.astype(np.float32))
        lo = [o.glo[a] for a in range(4)]
        if it == 2:
            c = comet.helix_centre(ev.tracks[e][0])
            lo = [c[a] - 0.5 * N[a] * W[a] + 0.002 for a in range(3)] + [-0.5 * N[3] * W[3]]
        boxes = []
        while not boxes:   # a group of 2 x 2 x 2 columns, those that pass
            i0 = [2 * int(rng.integers(N[a] // 2)) for a in range(3)]
            for s in range(8):
                ix = [i0[a] + ((s >> a) & 1) for a in range(3)]
                b = [v for a in range(3) for v in (lo[a] + ix[a] * W[a], lo[a] + (ix[a] + 1) * W[a])]
                if O.four_disk(b) and 0.105 / (0.15 * (b[4] + b[5])) > 1.0 + 1e-5:
                    boxes.append(b)
        ref = (0.0, 0.0) if it == 0 or k == 32 else (0.98 * h[0], 0.97 * h[1])
        cc = []
        for b in boxes:
            x, y, R = (b[0] + b[1]) / 2, (b[2] + b[3]) / 2, (b[4] + b[5]) / 2
            if k == 32:
                x, y, R = [float(np.float32(v)) for v in (x, y, R)]
                aL, ph = O.four_vote_pair(b + [0.0, 0.07], 1, ref, h, prec=1)[1][3], 0.0
            else:
                aL, ph = math.sqrt((0.105 / (0.3 * R)) ** 2 - 1.0), _phase(-x, -y, ref[0] - x, ref[1] - y)
            cc.append([x, y, R, aL, -x, -y, 1.0 / math.hypot(x, y), ph])
        cc, bb = np.array(cc), np.array(boxes)
        group = _a(np.stack([cc.min(0), cc.max(0)], 1).ravel())
        box = _a([bb[:, 0].min(), bb[:, 1].max(), bb[:, 2].min(), bb[:, 3].max(),
                  (bb[:, 4] - cc[:, 2]).min(), (bb[:, 5] - cc[:, 2]).max()])
        z = [lo[3] + j * W[3] for j in range(N[3] + 1)]
        eps = C.c_float()
        zr = _a([(z[0] + z[1]) / 2, (z[-2] + z[-1]) / 2, z[0], z[-1]])
        err = lib.bound_4d(k, _p(group), _p(box), _p(zr), _p(h), C.byref(eps))
        q = int(rng.integers(len(boxes)))
        b, ctr = boxes[q], _a(cc[q])
        for j in rng.choice(N[3], 3, replace=False):
            for sign in (1, -1):
                v, r = O.four_vote_pair(b + [z[j], z[j + 1]], sign, ref, h, prec=0 if k == 64 else 1)
                out = np.zeros(6, np.float32)
                zc = _a([(z[j] + z[j + 1]) / 2, z[j], z[j + 1]])
                d = lib.child_4d(_p(ctr), _p(_a(b)), _p(zc), _p(h), sign, C.c_float(err), eps, out.ctypes.data_as(F4))
                assert d == 2 or (d == v and not math.isnan(err))
                decided += d != 2
                undecided += d == 2
                if k == 32 or d == 2:
                    continue
                xw, yw = sorted([h[0] + z[j + s] * h[5] for s in (0, 1)]), sorted([h[1] - z[j + s] * h[6] for s in (0, 1)])
                sx, sy = _sq(xw, b[0:2]), _sq(yw, b[2:4])
                for s in (0, 1):
                    if out[3 * s] < 1e-5 or (int(r[2]) >> s) & 1:
                        continue
                    g = sorted([(b[4] + r[s]) ** 2, (b[5] + r[s]) ** 2])
                    assert abs(out[3 * s + 1] - (sx[0] + sy[0] - g[1])) <= err
                    assert abs(out[3 * s + 2] - (sx[1] + sy[1] - g[0])) <= err
    assert decided > 10 * undecided


@pytest.mark.parametrize("bins,levels", [([16] * 5, 6), ([5, 6, 6, 5, 5], 5), ([7, 6, 8, 5, 9], 2)])
def test_midpoint(lib, bins, levels):
    w, g = chamber.make_wires(), G.make_grid(bins, levels, 64)
    ev = chamber.single_track_events(6, seed=23, w=w)
    rng = np.random.default_rng(sum(bins))

    def centres(level, i0, i1):
        out = []
        c = [O.cell12(g, level, i) for i in (i0, i1)]
        s = [O.scm2(g, level, i) for i in (i0, i1)]
        for a in range(6):
            v = [s[q][a - 1] if a in (1, 2) else (c[q][2 * a] + c[q][2 * a + 1]) * 0.5 for q in (0, 1)]
            out += [min(v), max(v)]
        return _a(out)

    decided = undecided = 0
    for n in range(400):
        e = int(rng.integers(ev.n_events))
        i = int(rng.integers(ev.offsets[e], ev.offsets[e + 1]))
        h = _a(O.hit9(w, ev.wire_id[i], ev.drift[i]))
        if n % 10 == 8:
            h[4:8] = 0.0
        if n % 10 == 9:
            h[8] = 0.0
        if n % 2:
            p, o, level = int(rng.integers(bins[1])), int(rng.integers(bins[2])), 0
            i0, i1 = [0, p, o, 0, 0], [bins[0] - 1, p, o, bins[3] - 1, bins[4] - 1]
            kids = [[int(rng.integers(bins[0])), p, o, int(rng.integers(bins[3])), int(rng.integers(bins[4]))]
                    for _ in range(6)]
        else:
            lv, par, at = int(rng.integers(levels)), ev.tracks[e][0].params, []
            for a in range(5):
                edges = g.lo_edge[a][::1 << (levels - lv)]
                j = int(np.searchsorted(edges, par[a], side="right")) - 1 + int(rng.integers(-1, 2))
                at.append(min(max(j, 0), len(edges) - 1))
            level, i0, i1 = lv + 1, [2 * v for v in at], [2 * v + 1 for v in at]
            kids = [[2 * at[a] + ((b >> a) & 1) for a in range(5)] for b in rng.choice(32, 6, replace=False)]
        c0, c1 = O.cell12(g, level, i0), O.cell12(g, level, i1)
        P = _a([f(c0[q], c1[q]) for a in range(6) for q, f in ((2 * a, min), (2 * a + 1, max))])
        no = C.c_int()
        err = lib.parent_mid(_p(P), _p(centres(level, i0, i1)), _p(h), C.byref(no))
        for kid in kids:
            c = _a(O.cell12(g, level, kid))
            v, ref = O.vote_pair_mid(c, O.scm2(g, level, kid), h)
            assert not (no.value and v)
            out = np.zeros(4, np.float32)
            d = lib.child_mid(_p(c), _p(centres(level, kid, kid)), _p(h), C.c_float(err), out.ctypes.data_as(F4))
            assert d == 2 or (d == v and not math.isnan(err))
            if ref[4] == 0 and not math.isnan(err):
                assert np.abs(out.astype(np.float64) - ref[:4]).max() <= err
            decided += d != 2
            undecided += d == 2
    assert decided > 20 * undecided
