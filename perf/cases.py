"""The work this framework is used for, as cases that can be timed and compared.

Each case is a dict of plain values.  `prepare` makes its inputs and the plan a program
keeps (geometry, workspace, options), `run` is one pass through the public entry points of
paper_2401_04576_gb300.apo, `work` what a pass cannot do without, and `exact` the result of
the FP64 searches in plain 64-bit torch, where that is affordable.

Events are those of gen/chamber.py and gen/comet.py.  The chamber of gen/chamber.py maps
onto itself under rotations by 45 degrees (every layer has a multiple of 8 wires), so a
pool of simulated tracks gives eight times as many events at the cost of the pool.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from gen import chamber, comet, grid as G
from paper_2401_04576_gb300 import apo

POOL = 96            # simulated tracks behind one case's events
SYMMETRY = 8         # the chamber's rotations by 45 degrees


def listed():
    aniso = {"bins": "2,256,16,2,8", "levels": 5, "topk": 64}
    return [
        # the smallest call: one event from host buffers, as an online trigger would ask
        {"name": "event_f64", "kind": "event", "events": 1, "bins": "10,10,10,10,10", "levels": 4, "topk": 16,
         "precision": "f64"},
        # the headline search: every level in sound FP64 intervals (one and a quarter chunks)
        {"name": "batch_f64", "kind": "search", "events": 320, "bins": "16,16,16,16,16", "levels": 6, "topk": 64,
         "precision": "f64"},
        # the production form of the same search: FP32 levels 0-4, FP64 on the last two
        {"name": "batch_mixed", "kind": "search", "events": 1024, "bins": "16,16,16,16,16", "levels": 6, "topk": 64,
         "precision": "mixed", "full": True},
        # recovering the helix: whole maximum-vote groups with the direction condition
        {"name": "recover_mixed", "kind": "recover", "events": 160, "precision": "mixed", "max_keep": 32768,
         "slack": 0, **aniso},
        # the same for one event in FP64, the per-event path
        {"name": "recover_event_f64", "kind": "recover", "events": 1, "precision": "f64", "max_keep": 32768,
         "slack": 0, **aniso},
        # uneven multi-track events with noise, up to 5 tracks, one persistent launch
        {"name": "multi_topk", "kind": "multi", "events": 1000, "bins": "10,10,10,10,10", "levels": 6, "topk": 64,
         "precision": "mixed", "tracks": 5, "persistent": True},
        # the same events with the max-set schedule, which separates the tracks
        {"name": "multi_maxset", "kind": "multi_maxset", "events": 24, "precision": "mixed", "max_keep": 32768,
         "slack": 6, "tracks": 5, **aniso},
        # a burst of events through the continuous-batching server
        {"name": "serve_burst", "kind": "serve", "events": 200, "bins": "10,10,10,10,10", "levels": 6, "topk": 64,
         "precision": "mixed", "tracks": 5, "batch_events": 64, "slots": 8},
        # the paper's own 4-D search of conversion electrons, in both precisions
        {"name": "paper4d_f32", "kind": "paper4d", "events": 48, "precision": "f32"},
        {"name": "paper4d_f64", "kind": "paper4d", "events": 2, "precision": "f64"},
        # one bisection step driven by hand on a ragged grid: vote, refine, vote the children
        {"name": "step_f64", "kind": "step", "events": 37, "bins": "7,6,8,5,9", "levels": 2, "topk": 33,
         "precision": "f64", "outgoing": True},
        # the paper's midpoint form as a batched search
        {"name": "batch_midpoint", "kind": "search", "events": 24, "bins": "16,16,16,16,16", "levels": 6, "topk": 64,
         "precision": "mid"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: any of the kinds above with sizes over its range."""
    kind = rng.choice(["event", "search", "search", "recover", "multi", "multi_maxset", "serve", "paper4d", "step"])
    if kind == "paper4d":
        prec = rng.choice(["f32", "f64"])
        return {"kind": kind, "events": _log_int(rng, 1, 48) if prec == "f32" else rng.randint(1, 2),
                "precision": prec}
    if kind in ("recover", "multi_maxset"):
        phi = rng.randint(96, 256)
        c = {"kind": kind, "bins": f"2,{phi},{2 * rng.randint(5, 8)},{rng.randint(2, 3)},{rng.randint(6, 9)}",
             "levels": rng.randint(4, 5), "topk": 64, "precision": rng.choice(["f64", "mixed"]),
             "max_keep": _log_int(rng, 2048, 32768)}
        if kind == "recover":
            return {**c, "events": _log_int(rng, 1, 48), "slack": rng.randint(0, 1)}
        return {**c, "events": _log_int(rng, 1, 6), "slack": rng.randint(1, 6), "tracks": rng.randint(2, 5)}
    if kind in ("event", "multi", "serve"):
        c = {"kind": kind, "bins": f"{rng.randint(7, 11)},{rng.randint(9, 13)},{2 * rng.randint(4, 6)},"
             f"{rng.randint(7, 11)},{rng.randint(8, 12)}", "levels": rng.randint(3, 6), "topk": _log_int(rng, 9, 64),
             "precision": rng.choice(["f64", "mixed"])}
        if kind == "event":
            return {**c, "events": _log_int(rng, 1, 5)}
        c = {**c, "precision": "mixed", "tracks": rng.randint(2, 5)}
        if kind == "multi":
            n = _log_int(rng, 7, 1000)
            return {**c, "events": n, "persistent": n >= 500}
        return {**c, "events": _log_int(rng, 3, 200), "batch_events": rng.randint(16, 64), "slots": rng.randint(2, 8)}
    bins = [rng.randint(5, 16), rng.randint(6, 16), 2 * rng.randint(3, 8), rng.randint(5, 16), rng.randint(5, 16)]
    cells = int(np.prod(bins))
    c = {"kind": kind, "bins": ",".join(map(str, bins)), "levels": rng.randint(2, 6), "topk": _log_int(rng, 9, 64)}
    if kind == "step":
        return {**c, "events": _log_int(rng, 1, 48), "precision": rng.choice(["f64", "f32"]),
                "outgoing": rng.random() < 0.5}
    prec = rng.choice(["f64", "mixed", "mid"])
    most = {"f64": 320, "mixed": 1024, "mid": 96}[prec]
    return {**c, "events": min(most, _log_int(rng, 2, max(3, most * 2 ** 20 // max(cells, 2 ** 18)))),
            "precision": prec, "full": rng.random() < 0.5}


# ---- inputs --------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _wires():
    return chamber.make_wires()


@functools.lru_cache(maxsize=None)
def _comet_wires():
    return comet.make_wires()


def _grid(case):
    return G.make_grid([int(b) for b in case["bins"].split(",")], case["levels"], case["topk"])


def _pool(n, rng):
    """(wires, drifts) of n simulated tracks of at least six hits."""
    w, out = _wires(), []
    while len(out) < n:
        hits = chamber.simulate_track(chamber.draw_track(rng), w, rng)
        if len(hits) >= 6:
            out.append((np.array([h.wire for h in hits]), np.array([h.drift for h in hits])))
    return out


def _rotated(wire, turns):
    """The wires reached by turning the chamber by 45 degrees `turns` times."""
    layer = _wires().layer
    n = np.bincount(layer)
    first = np.concatenate([[0], np.cumsum(n)[:-1]])
    a = layer[wire]
    return first[a] + (wire - first[a] + turns * (n[a] // SYMMETRY)) % n[a]


def _events(case, seed):
    rng = np.random.default_rng([seed, case["events"]])
    w, n_ev = _wires(), case["events"]
    multi = case["kind"] in ("multi", "multi_maxset", "serve")
    pool = _pool(min(POOL * (1 if multi or n_ev <= POOL * SYMMETRY else 2), n_ev * (3 if multi else 1)), rng)
    per = []
    for e in range(n_ev):
        if not multi:   # every event another track, or another turn of it
            wire, drift = pool[e % len(pool)]
            wire = _rotated(wire, (e // len(pool) + e) % SYMMETRY)
        else:           # 1-5 tracks; 10-30 % of the hits are noise
            found = {}
            for _ in range(int(rng.integers(1, 6))):
                tw, td = pool[int(rng.integers(len(pool)))]
                for a, d in zip(_rotated(tw, int(rng.integers(SYMMETRY))), td):
                    found[int(a)] = min(float(d), found.get(int(a), np.inf))
            occ = rng.uniform(0.1, 0.3)
            n_noise = int(round(occ / (1.0 - occ) * len(found)))
            free = np.setdiff1d(np.arange(w.n), np.fromiter(found, int))
            noise = rng.choice(free, size=n_noise, replace=False)
            wire = np.concatenate([np.fromiter(found, int), noise])
            drift = np.concatenate([np.fromiter(found.values(), float), rng.uniform(0.0, w.half_cell[noise])])
        order = np.argsort(wire)
        per.append((wire[order], drift[order]))
    offsets = np.concatenate([[0], np.cumsum([len(a) for a, _ in per])]).astype(np.int32)
    return chamber.Events(offsets=offsets, wire_id=np.concatenate([a for a, _ in per]).astype(np.int32),
                          drift=np.concatenate([d for _, d in per]))


def _precision(case):
    """The precision code of each level: mixed is FP64 on the last one (max-set) or two."""
    lv, p = case["levels"], case["precision"]
    out = apo.OUTGOING if case["kind"] in ("recover", "multi_maxset") else 0
    if p == "mixed":
        n64 = 1 if out else min(2, lv)
        return [apo.F32 | out] * (lv + 1 - n64) + [apo.F64 | out] * n64
    return [{"f64": apo.F64, "f32": apo.F32, "mid": apo.F64_MID}[p] | out] * (lv + 1)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    if kind == "paper4d":
        ev = comet.events(case["events"], seed, _comet_wires())
        st["chamber"] = apo.Chamber4(_comet_wires())
        st["hits"] = apo.DeviceHits.from_events(ev)
        st["opts"] = apo.four_opts(precision=apo.F32 if case["precision"] == "f32" else apo.F64)
        st["ws"] = st["chamber"].workspace(ev.n_events, st["opts"])
        st["selected"] = torch.zeros(ev.n_events * apo.HIT_CAP, dtype=torch.uint8, device="cuda")
        return st
    ev = _events(case, seed)
    g = apo.Geometry(_grid(case), _wires())
    st["ev"], st["geom"] = ev, g
    if kind == "step":
        st["hits"] = apo.DeviceHits.from_events(ev)
        st["ws"] = g.workspace(ev.n_events)
        st["precision"] = _precision(case)[0] | (apo.OUTGOING if case["outgoing"] else 0)
        return st
    kw = {"precision": _precision(case)}
    if kind in ("multi", "multi_maxset", "serve"):
        kw.update(max_tracks=case["tracks"], min_votes=6)
    if kind in ("recover", "multi_maxset"):
        kw.update(schedule=apo.SCHED_MAXSET, max_keep=case["max_keep"], slack=case["slack"])
    if kind in ("multi", "multi_maxset"):   # one buffer for any number of hits
        st["hit_track"] = kw["hit_track"] = torch.zeros(ev.n_events * apo.HIT_CAP, dtype=torch.int32, device="cuda")
    if kind == "multi":
        kw["tune"] = apo.ApoTune(0, 1, 256, 0, persistent=int(case["persistent"]))
    if case.get("full"):
        kw["tune"] = apo.ApoTune(0, 1, 256, 0, coarse_full=1)
    o = st["opts"] = apo.solve_opts(**kw)
    if kind == "serve":
        st["server"] = apo.Server(g, o, batch_events=case["batch_events"], max_slots=case["slots"])
    elif kind == "event":
        st["ws"] = torch.empty(apo.host_workspace_bytes(g, ev.n_events, len(ev.wire_id), o), dtype=torch.uint8,
                               device="cuda")
    else:
        st["hits"] = apo.DeviceHits.from_events(ev)
        st["ws"] = g.workspace(ev.n_events, opts=o)
        st["tracks"] = torch.zeros(ev.n_events * int(o.max_tracks) * apo.TRACK_DTYPE.itemsize, dtype=torch.uint8,
                                   device="cuda")
        st["n_tracks"] = torch.zeros(ev.n_events, dtype=torch.int32, device="cuda")
    return st


# ---- one pass ------------------------------------------------------------------------

def run(st):
    kind = st["kind"]
    if kind == "paper4d":
        out, selected = apo.solve4(st["chamber"], st["hits"], st["opts"], selected=st["selected"], workspace=st["ws"])
        rec = out.view(torch.float64).view(-1, 12)
        return {"values": rec[:, :10], "counts": out.view(torch.int32).view(-1, 24)[:, 20:], "selected": selected}
    if kind == "step":
        votes = apo.vote(st["geom"], st["hits"], precision=st["precision"], workspace=st["ws"])
        kept, kept_votes, children = apo.refine(st["geom"], st["hits"], votes, workspace=st["ws"])
        child_votes = apo.vote(st["geom"], st["hits"], keys=children, level=1, precision=st["precision"],
                               workspace=st["ws"])
        return {"votes": votes, "kept": kept, "kept_votes": kept_votes, "children": children,
                "child_votes": child_votes}
    if kind == "event":
        ev = st["ev"]
        tracks, n = apo.solve_batch_host(st["geom"], ev.offsets, ev.wire_id, ev.drift, st["opts"],
                                         workspace=st["ws"])
        return {"p": tracks["p"], "w": tracks["w"], "votes": tracks["votes"], "n_tracks": n}
    if kind == "serve":
        ev, srv = st["ev"], st["server"]
        for e in range(ev.n_events):
            a, b = ev.offsets[e], ev.offsets[e + 1]
            if srv.submit(ev.wire_id[a:b], ev.drift[a:b], e) != apo.APO_OK:
                raise RuntimeError("the server's queue is full")
        srv.drain()
        done = sorted(srv.poll(ev.n_events), key=lambda r: r[0])
        tr = np.stack([t for _, t, _ in done])
        return {"p": tr["p"], "w": tr["w"], "votes": tr["votes"], "n_tracks": np.array([n for _, _, n in done]),
                "ids": np.array([i for i, _, _ in done])}
    tracks, n = apo.solve_batch(st["geom"], st["hits"], st["opts"], tracks=st["tracks"], n_tracks=st["n_tracks"],
                                workspace=st["ws"])
    rec = tracks.view(torch.float64).view(-1, 11)
    out = {"p": rec[:, :5], "w": rec[:, 5:10], "counts": tracks.view(torch.int32).view(-1, 22)[:, 20:],
           "n_tracks": n}
    if "hit_track" in st:
        out["hit_track"] = st["hit_track"]
    return out


# ---- what a pass cannot do without ----------------------------------------------------

def work(case):
    """Hits in, results out; one addition per (cell, hit) pair that gets a vote or none.  The
    interval program is not counted: one proof can decide many pairs."""
    ne, kind = case["events"], case["kind"]
    if kind == "paper4d":
        hits = 40 * ne
        o = apo.four_opts()
        voxels = sum(int(np.prod([o.n[k][a] for a in range(4)], dtype=np.int64)) for k in range(3))
        return {"bytes": 13 * hits + 4 * (ne + 1) + 3 * 96 * ne, "flops": 2 * voxels * hits}
    per = 37 if kind in ("multi", "multi_maxset", "serve") else 10
    cells = int(np.prod([int(b) for b in case["bins"].split(",")], dtype=np.int64))
    nb = 12 * per * ne + 4 * (ne + 1)
    if kind == "step":
        k = case["topk"]
        return {"bytes": nb + ne * (4 * cells + 12 * k + (8 + 4) * 32 * k), "flops": per * ne * (cells + 32 * k)}
    tracks = case.get("tracks", 1)
    return {"bytes": nb + ne * (4 + 88 * tracks) + (4 * per * ne if "tracks" in case else 0),
            "flops": per * ne * (cells + 32 * case["topk"] * case["levels"])}


# ---- 64-bit results in plain torch ------------------------------------------------------
# Intervals are pairs of tensors, evaluated round to nearest: the end points differ from the
# directed ones by a few units of the last place, so a vote could only differ where an end
# point is that close to zero.

def _add(a, b):
    return a[0] + b[0], a[1] + b[1]


def _sub(a, b):
    return a[0] - b[1], a[1] - b[0]


def _neg(a):
    return -a[1], -a[0]


def _mul(a, b):
    p = (a[0] * b[0], a[0] * b[1], a[1] * b[0], a[1] * b[1])
    return torch.minimum(torch.minimum(p[0], p[1]), torch.minimum(p[2], p[3])), \
        torch.maximum(torch.maximum(p[0], p[1]), torch.maximum(p[2], p[3]))


def _sqr(a):
    n = torch.clamp(torch.maximum(a[0], -a[1]), min=0.0)
    m = torch.maximum(-a[0], a[1])
    return n * n, m * m


def _scale(a, k):
    return a[0] * k, a[1] * k


def _sqrt(a):
    return torch.sqrt(torch.clamp(a[0], min=0.0)), torch.sqrt(torch.clamp(a[1], min=0.0))


def _recip(a):
    return 1.0 / a[1], 1.0 / a[0]


def _clamp1(a):
    return torch.clamp(a[0], -1.0, 1.0), torch.clamp(a[1], -1.0, 1.0)


def _atan(x):
    for _ in range(2):
        x = _mul(x, _recip(_add((1.0, 1.0), _sqrt(_add((1.0, 1.0), _sqr(x))))))
    y = _sqr(x)
    h = (torch.full_like(y[0], 1 / 15),) * 2
    for k in range(6, -1, -1):
        h = _sub((1 / (2 * k + 1),) * 2, _mul(h, y))
    rem = torch.maximum(-x[0], x[1]) ** 17 / 17
    a = _mul(x, h)
    return 4 * (a[0] - rem), 4 * (a[1] + rem)


def _sincos(d):
    m = torch.maximum(-d[0], d[1])
    y = _sqr(d)
    s = _mul(d, _sub((1.0, 1.0), _scale(y, 1 / 6)))
    c = _sub((1.0, 1.0), _scale(y, 0.5))
    r5, r4, big = m ** 5 / 120, m ** 4 / 24, m > 1.0
    s, c = _clamp1((s[0] - r5, s[1] + r5)), _clamp1((c[0] - r4, c[1] + r4))
    lo, hi = -torch.ones_like(m), torch.ones_like(m)
    return (torch.where(big, lo, s[0]), torch.where(big, hi, s[1])), \
        (torch.where(big, lo, c[0]), torch.where(big, hi, c[1]))


def _vote(cell, hit, outgoing):
    """Votes (0 / 1) of interval cells (d0, sin phi0, cos phi0, omega, z0, tan lambda) for one
    hit (x0, y0, sin phis, cos phis, tan tau, sphi tan tau, cphi tan tau, tan^2 tau, d)."""
    one = (1.0, 1.0)
    mir = cell[3][1] < 0
    sign = torch.where(mir, -1.0, 1.0)

    def flip(a):
        return torch.where(mir, -a[1], a[0]), torch.where(mir, -a[0], a[1])

    D, S, C, W, Z, L = flip(cell[0]), flip(cell[1]), cell[2], flip(cell[3]), cell[4], cell[5]
    x0, y0, sph, cph, t, spt, cpt, t2, d = [(torch.as_tensor(v),) * 2 for v in hit]
    y0, cph, cpt = [(v[0] * sign,) * 2 for v in (y0, cph, cpt)]
    Xw, Yw = _add(x0, _mul(Z, spt)), _sub(y0, _mul(Z, cpt))
    wt, wn = _add(_mul(Xw, C), _mul(Yw, S)), _sub(_mul(Yw, C), _mul(Xw, S))
    V = _sub(wn, D)
    Xt, Xn = _mul(wt, W), _sub(_mul(V, W), one)
    N = _sqrt(_add(_sqr(Xt), _sqr(Xn)))
    G0 = _add(_mul(W, _sqr(wt)), _mul(V, _sub(Xn, one)))
    den = _sub(N, Xn)
    guard = (N[0] <= 0) | (den[0] <= 0) | (W[0] <= 0)
    psi = _scale(_atan(_mul(Xt, _recip(den))), 2.0)
    E1, E2 = _add(_mul(C, cph), _mul(S, sph)), _sub(_mul(C, sph), _mul(S, cph))
    rsA, rcA = _add(_mul(Xt, E1), _mul(Xn, E2)), _sub(_mul(Xt, E2), _mul(Xn, E1))
    Ni = _recip(N)
    sPA, cPA = _clamp1(_mul(rsA, Ni)), _clamp1(_mul(rcA, Ni))
    cos2, sin2 = _clamp1(_sub(_sqr(cPA), _sqr(sPA))), _clamp1(_scale(_mul(sPA, cPA), 2.0))
    dW, Nh, L2 = _mul(d, W), _scale(_sqr(Ni), 0.5), _sqr(L)
    inner = _sub(_add(_mul(psi, _sub(one, cos2)), _mul(sin2, _sqr(psi))), _mul(sin2, _sqr(dW)))
    P1e = _neg(_mul(_mul(L, _mul(psi, sPA)), Ni))
    P1o = _neg(_mul(_mul(L, _mul(cPA, dW)), Ni))
    P2e = _mul(_mul(inner, L2), Nh)
    P2o = _mul(_mul(_add(_scale(_mul(_mul(psi, cos2), L2), 2.0),
                         _mul(sin2, _add(N, _mul(L2, _add(one, N))))), dW), Nh)
    de, do = _add(_mul(P1e, t), _mul(P2e, t2)), _add(_mul(P1o, t), _mul(P2o, t2))
    dP, dM = _add(de, do), _sub(de, do)
    sd, cd = _sincos((torch.minimum(dP[0], dM[0]), torch.maximum(dP[1], dM[1])))
    sP = _clamp1(_add(_mul(sPA, cd), _mul(cPA, sd)))
    cP = _clamp1(_sub(_mul(cPA, cd), _mul(sPA, sd)))
    t2x = _scale(t, 2.0)
    u2 = _add(_add(_add(one, _mul(t2x, _mul(L, sP))), _mul(L2, t2)), _mul(_sqr(cP), t2))
    guard = guard | (u2[0] <= 0)
    Q = _mul(d, _recip(_sqrt(u2)))
    Qct, LQ = _mul(_mul(cP, t), Q), _mul(L, Q)
    LQrsA, a2, a5 = _mul(LQ, rsA), _mul(W, _sqr(Q)), _mul(W, _sqr(_mul(LQ, t)))
    R = _recip(W)
    vote = guard
    for dl, op, a1 in ((dP, _sub, _scale(Q, 2.0)), (dM, _add, _neg(_scale(Q, 2.0)))):
        zS = op(_mul(_mul(_add(psi, dl), R), L), Qct)
        rct = op(_mul(zS, rcA), LQrsA)
        A = _sub(_sub(_sub(_add(a1, a2), _mul(t2x, rct)), _mul(W, _sqr(_mul(zS, t)))), a5)
        Gv = _sub(G0, A)
        vote = vote | ((Gv[0] <= 0) & (Gv[1] >= 0))
    if outgoing:
        vote = vote & ~(wt[1] < 0)
    return vote


def _counts(g, level, idx, hits, outgoing, chunk=1 << 19):
    """Votes of the cells idx (n, 5) at `level`, in pieces that stay in cache."""
    dev, out = idx.device, []
    edges = [[torch.as_tensor(e, device=dev) for e in (g.lo_edge[a], g.hi_edge[a])] for a in range(5)]
    rows = torch.as_tensor(g.sincos, device=dev)[int(g.sincos_offset[level]):]
    sh = g.levels - level
    for part in idx.split(chunk):
        iv = [(edges[a][0][part[:, a] << sh], edges[a][1][((part[:, a] + 1) << sh) - 1]) for a in range(5)]
        r = rows[part[:, 1]]
        cell = (iv[0], (r[:, 0], r[:, 1]), (r[:, 2], r[:, 3]), iv[2], iv[3], iv[4])
        v = torch.zeros(part.shape[0], dtype=torch.int64, device=dev)
        for h in hits:
            v += _vote(cell, h, outgoing)
        out.append(v)
    return torch.cat(out)


def _linear(idx, g, level):
    lin = torch.zeros_like(idx[:, 0])
    for a in range(4, -1, -1):
        lin = lin * (int(g.bins[a]) << level) + idx[:, a]
    return lin


def _search(case, g, hits, dev):
    """(p, w) of one event's search in 64 bits: top-K or whole maximum-vote groups."""
    maxset = case["kind"] == "recover"
    bits = torch.stack([(torch.arange(32, device=dev) >> a) & 1 for a in range(5)], 1)
    j = torch.arange(g.n_coarse(), device=dev)
    cols = []
    for a in range(5):
        cols.append(j % int(g.bins[a]))
        j = j // int(g.bins[a])
    idx = torch.stack(cols, 1)
    for level in range(g.levels + 1):
        v = _counts(g, level, idx, hits, maxset)
        top = int(v.max())
        if level == g.levels or (maxset and int((v == top).sum()) > case["max_keep"]):
            break
        if maxset:
            least = max(top - case["slack"], min(top, 1))
            while int((v >= least).sum()) > case["max_keep"]:
                least += 1
            kept = idx[v >= least]
        else:
            order = torch.argsort(_linear(idx, g, level))
            order = order[torch.argsort(-v[order], stable=True)]
            kept = idx[order[:g.topk]]
        idx = (2 * kept[:, None, :] + bits).reshape(-1, 5)
    best = idx[v == top]
    p, w = [], []
    for a in range(5):
        lo, hi = g.cell_edges(level, a, best[:, a].cpu().numpy())
        p.append(float(np.mean((lo + hi) * 0.5)))
        w.append(float((hi.max() - lo.min()) * 0.5))
    return p, w


def _exact5(case, seed):
    g, w, ev = _grid(case), _wires(), _events(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    table = np.stack([w.x0, w.y0, w.sin_phis, w.cos_phis, w.tan_tau, w.sphi_t, w.cphi_t, w.t2], 1)
    p, wd = [], []
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        hits = np.concatenate([table[ev.wire_id[a:b]], ev.drift[a:b, None]], 1)
        r = _search(case, g, hits.tolist(), dev)
        p.append(r[0])
        wd.append(r[1])
    return np.array(p), np.array(wd)


def _phase(m, dx, dy):
    """Phase of (dx, dy) seen from the centre, from the direction of the origin, in [0, 2 pi)."""
    return torch.remainder(torch.atan2(m["ox"] * dy - m["oy"] * dx, m["ox"] * dx + m["oy"] * dy), 2 * math.pi)


def _centre(xc, yc, R, o, ref):
    ratio = o.p_gev / (0.3 * o.b_tesla * R)
    m = {"x": xc, "y": yc, "R": R, "ox": -xc, "oy": -yc, "valid": ratio > 1}
    m["L"] = torch.sqrt(torch.clamp(ratio * ratio - 1, min=0.0))
    m["ref"] = _phase(m, ref[0] - xc, ref[1] - yc)
    return m


def _vote4(m, sign, box, zc, hit):
    """Votes of boxes (x, y, R, z0 intervals; centre m, zc) for one hit and sign of tan lambda."""
    x0, y0, sph, cph, t, spt, cpt, t2, d = hit
    L, R = sign * m["L"], m["R"]
    dx, dy = x0 + zc * spt - m["x"], y0 - zc * cpt - m["y"]
    A2 = dx * dx + dy * dy
    RA = torch.sqrt(A2)
    cA, sA = dx * sph - dy * cph, dx * cph + dy * sph
    sPA, cPA, cos2, sin2 = sA / RA, cA / RA, (cA * cA - sA * sA) / A2, 2 * sA * cA / A2
    psi = _phase(m, dx, dy) - m["ref"]
    zA = L * R * psi
    xw = _add((x0, x0), _mul(box[3], (torch.as_tensor(spt),) * 2))
    yw = _sub((y0, y0), _mul(box[3], (torch.as_tensor(cpt),) * 2))
    near = _add(_sqr(_sub(xw, box[0])), _sqr(_sub(yw, box[1])))
    vote = torch.zeros_like(A2, dtype=torch.bool)
    for ds in (d, -d):
        phi1 = -(zA * sPA + L * ds * cPA) / RA
        phi2 = (L * R * zA - L * zA * (R - 2 * ds) * cos2
                + (zA * zA + ds * (RA + L * L * (R + RA - ds))) * sin2) / (2 * A2)
        dl = phi1 * t + phi2 * t2
        sP, cP = sPA * torch.cos(dl) + cPA * torch.sin(dl), cPA * torch.cos(dl) - sPA * torch.sin(dl)
        q = ds / torch.sqrt(1 + 2 * t * L * sP + L * L * t2 + cP * cP * t2)
        zS = L * R * (psi + dl) - q * cP * t
        rad = (R + q) ** 2 - 2 * (zS * cA - L * q * sA) * t - (zS * t) ** 2 - (L * q * t) ** 2
        dax = torch.sqrt(torch.clamp(rad, min=0.0)) - R
        gap = _sub(near, _sqr((box[2][0] + dax, box[2][1] + dax)))
        vote |= (rad < 0) | ((gap[0] <= 0) & (gap[1] >= 0))
    return vote


def _iteration4(o, k, lo, ref, sign, hits, dev):
    """(vmax, value, error) of one sign's accumulator on iteration k's grid at corner lo."""
    n, w = [int(o.n[k][a]) for a in range(4)], [float(o.w[k][a]) for a in range(4)]
    ax = [lo[a] + torch.arange(n[a] + 1, device=dev, dtype=torch.float64) * w[a] for a in range(4)]
    col = torch.stack([x.reshape(-1) for x in torch.meshgrid(*[torch.arange(c, device=dev) for c in n[:3]],
                                                              indexing="ij")], 1)
    box = [(ax[a][col[:, a]], ax[a][col[:, a] + 1]) for a in range(3)]
    rd = (torch.as_tensor(-o.disk_radius), torch.as_tensor(o.disk_radius))
    disk = _sub(_add(_sqr(box[0]), _sqr(box[1])), _sqr(_add(box[2], rd)))
    Rc = (box[2][0] + box[2][1]) / 2
    keep = (disk[0] <= 0) & (disk[1] >= 0) & (o.p_gev / (0.3 * o.b_tesla * Rc) > 1)
    col, box = col[keep], [(a[keep], b[keep]) for a, b in box]
    m = _centre((box[0][0] + box[0][1]) / 2, (box[1][0] + box[1][1]) / 2, Rc[keep], o, ref)
    votes = torch.zeros((n[3], col.shape[0]), dtype=torch.int32, device=dev)
    for iz in range(n[3]):
        z = (ax[3][iz], ax[3][iz + 1])
        for h in hits:
            votes[iz] += _vote4(m, sign, [*box, z], (z[0] + z[1]) / 2, h)
    top = int(votes.max())
    iz, c = torch.nonzero(votes == top, as_tuple=True)
    idx = torch.cat([col[c], iz[:, None]], 1).double()
    mean, first, last = idx.mean(0).tolist(), idx.amin(0).tolist(), idx.amax(0).tolist()
    value = [float(lo[a]) + w[a] * (mean[a] + 0.5) for a in range(4)]
    return top, value, [w[a] * (last[a] + 1 - first[a]) / 2 for a in range(4)]


def _after4(o, k, est, ref, sign, hits, dev):
    """Hit finding around an estimate; the next reference point and grid corner."""
    val, err = est[1], est[2]
    box = [(torch.tensor([val[a] - o.hit_factor * err[a]], dtype=torch.float64, device=dev),
            torch.tensor([val[a] + o.hit_factor * err[a]], dtype=torch.float64, device=dev)) for a in range(4)]
    c = [(b[0] + b[1]) / 2 for b in box]
    m = _centre(c[0], c[1], c[2], o, ref)
    sel = [h for h in hits if bool(_vote4(m, sign, box, c[3], h))] if bool(m["valid"]) else []
    dist = [abs(math.hypot(h[0] - val[0], h[1] - val[1]) - val[2]) for h in sel]
    new = (sel[int(np.argmin(dist))][0], sel[int(np.argmin(dist))][1]) if sel else ref
    if k == 0:
        return sel, new, [float(o.glo[a]) for a in range(4)]
    f64 = functools.partial(torch.tensor, dtype=torch.float64, device=dev)
    m = {"ox": f64(-val[0]), "oy": f64(-val[1])}
    turn = float(_phase(m, f64(new[0] - val[0]), f64(new[1] - val[1]))
                 - _phase(m, f64(ref[0] - val[0]), f64(ref[1] - val[1])))
    ratio = o.p_gev / (0.3 * o.b_tesla * val[2])
    L = sign * math.sqrt(max(ratio * ratio - 1.0, 0.0))
    mid = [val[0], val[1], val[2], val[3] + L * val[2] * turn]
    return sel, new, [mid[a] - o.n[k + 1][a] * o.w[k + 1][a] / 2 for a in range(4)]


def _exact4(case, seed):
    w, ev = _comet_wires(), comet.events(case["events"], seed, _comet_wires())
    o = apo.four_opts()
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    table = np.stack([w.x0, w.y0, w.sin_phis, w.cos_phis, w.tan_tau, w.sphi_t, w.cphi_t, w.t2], 1)
    rows = []
    for e in range(ev.n_events):
        a, b = ev.offsets[e], ev.offsets[e + 1]
        every = np.concatenate([table[ev.wire_id[a:b]], ev.drift[a:b, None]], 1).tolist()
        start = (every, (0.0, 0.0), [float(o.glo[i]) for i in range(4)])
        state = {1: start, -1: start}
        for k in range(3):   # the last iteration has a box, reference point and hits per sign
            est = {s: _iteration4(o, k, state[s][2], state[s][1], s, state[s][0], dev) for s in (1, -1)}
            sign = 1 if est[1][0] >= est[-1][0] else -1
            ref = state[sign][1]
            rows.append(est[sign][1] + est[sign][2] + list(ref))
            if k == 0:
                nxt = _after4(o, k, est[sign], ref, sign, every, dev)
                state = {1: nxt, -1: nxt}
            elif k == 1:
                state = {s: _after4(o, k, est[s], ref, s, every, dev) for s in (1, -1)}
    return np.array(rows)


def exact(case, seed):
    """The estimates of the FP64 searches of a few events.  Mixed-precision searches keep
    other cells by definition, so their estimates have no 64-bit value; counts and keys are
    whole numbers."""
    kind = case["kind"]
    if case["precision"] != "f64" or case["events"] > 2:
        return None
    if kind == "paper4d":
        return {"values": _exact4(case, seed), "counts": None, "selected": None}
    if kind == "event":
        p, w = _exact5(case, seed)
        return {"p": p[:, None, :], "w": w[:, None, :], "votes": None, "n_tracks": None}
    if kind == "recover":
        p, w = _exact5(case, seed)
        return {"p": p, "w": w, "counts": None, "n_tracks": None}
    return None
