"""The 4-D search's certified values with FP32 references whose reference point is off the origin (at a
hit, as in iterations 2 and 3): the program's own phase of it is followed in FP32, operation by
operation, and every decision must be the oracle's vote."""
import ctypes as C

import numpy as np
import pytest

from gen import comet
from oracle import oracle as O
from test_certified_points import F4, _a, _p, lib  # noqa: F401

f = np.float32


def _atan(x):
    for _ in range(2):
        x = f(x / f(f(1) + f(np.sqrt(f(f(1) + f(x * x))))))
    y, h = f(x * x), f(f(1) / f(15))
    for k in (13, 11, 9, 7, 5, 3, 1):
        h = f(f(f(1) / f(k)) - f(h * y))
    return f(f(x * h) * f(4))


def _phase(x, y, ref):
    """The FP32 program's phase of the reference point seen from the centre (x, y)."""
    x, y = f(x), f(y)
    ox, oy = f(-x), f(-y)
    on = f(np.sqrt(f(f(ox * ox) + f(oy * oy))))
    dx, dy = f(f(ref[0]) - x), f(f(ref[1]) - y)
    r = f(on * f(np.sqrt(f(f(dx * dx) + f(dy * dy)))))
    sn, cs = f(f(ox * dy) - f(oy * dx)), f(f(ox * dx) + f(oy * dy))
    if cs >= 0:
        ph = f(f(2) * _atan(f(sn / f(r + cs))))
    else:
        ph = f(f(np.copysign(np.pi, sn)) - f(f(2) * _atan(f(sn / f(r - cs)))))
    return float(f(ph + f(2 * np.pi)) if ph < 0 else ph)


@pytest.mark.parametrize("it", [1, 2])
def test_four_d_reference_point(lib, it):  # noqa: F811
    w = comet.make_wires()
    ev = comet.events(4, 6, w)
    rng = np.random.default_rng(it)
    o = O.four_opts()
    W, N = [o.w[it][a] for a in range(4)], [o.n[it][a] for a in range(4)]
    decided = undecided = 0
    for _ in range(250):
        e = int(rng.integers(ev.n_events))
        i, i2 = (int(rng.integers(ev.offsets[e], ev.offsets[e + 1])) for _ in range(2))
        h = _a(_a(O.hit9(w, ev.wire_id[i], ev.drift[i])).astype(f))
        ref = tuple(float(f(v)) for v in O.hit9(w, ev.wire_id[i2], ev.drift[i2])[:2])
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
        cc = []
        for b in boxes:
            x, y, R = (float(f((b[2 * a] + b[2 * a + 1]) / 2)) for a in range(3))
            aL = O.four_vote_pair(b + [0.0, 0.07], 1, ref, h, prec=1)[1][3]
            cc.append([x, y, R, aL, -x, -y, 1.0 / np.hypot(x, y), _phase(x, y, ref)])
        cc, bb = np.array(cc), np.array(boxes)
        group = _a(np.stack([cc.min(0), cc.max(0)], 1).ravel())
        box = _a([bb[:, 0].min(), bb[:, 1].max(), bb[:, 2].min(), bb[:, 3].max(),
                  (bb[:, 4] - cc[:, 2]).min(), (bb[:, 5] - cc[:, 2]).max()])
        z = [lo[3] + j * W[3] for j in range(N[3] + 1)]
        eps = C.c_float()
        err = lib.bound_4d(32, _p(group), _p(box), _p(_a([(z[0] + z[1]) / 2, (z[-2] + z[-1]) / 2, z[0], z[-1]])), _p(h),
                           C.byref(eps))
        q = int(rng.integers(len(boxes)))
        for j in rng.choice(N[3], 3, replace=False):
            for sign in (1, -1):
                v, _ = O.four_vote_pair(boxes[q] + [z[j], z[j + 1]], sign, ref, h, prec=1)
                d = lib.child_4d(_p(_a(cc[q])), _p(_a(boxes[q])), _p(_a([(z[j] + z[j + 1]) / 2, z[j], z[j + 1]])), _p(h),
                                 sign, C.c_float(err), eps, np.zeros(6, f).ctypes.data_as(F4))
                assert d == 2 or d == v
                decided += d != 2
                undecided += d == 2
    assert decided > 10 * undecided
