// Voting with certified FP32 decisions (certified.cuh, cert_mid.cuh) on the device data layout: the
// votes of the FP64 (K = 64) or outward FP32 (K = 32) interval program or of the midpoint form,
// most of them decided by bare FP32 values and one error bound per (parent cell, hit).
#pragma once
#include "cert_mid.cuh"
#include "certified.cuh"
#include "kernels.cuh"

namespace apo {

// The program whose votes K decides: 64 and 32 as above, kMid the midpoint form (FP64).
constexpr int kMid = 1;
template <int K> struct RefOf { using T = double; };
template <> struct RefOf<32> { using T = float; };

// The reference's sign and guard tests of a cell: its precision's omega interval.  Returns
// whether the cell is mirrored (omega < 0); *guard: omega reaches 0, every hit votes.
template <int K> __device__ __forceinline__ bool omega_sign(IV<double> W, bool *guard) {
    const IV<typename RefOf<K>::T> w = to_prec<typename RefOf<K>::T>(W);
    const bool mir = lt0(w.hi);
    *guard = mir ? false : !gt0(w.lo);
    return mir;
}

template <int Q> __device__ __forceinline__ cert::X<Q> cx(IV<double> a) { return cert::mk<Q>(a.lo, a.hi); }
template <int Q> __device__ __forceinline__ cert::X<Q> cxm(IV<double> a, bool mir) {
    return mir ? cert::mk<Q>(-a.hi, -a.lo) : cert::mk<Q>(a.lo, a.hi);
}
template <int Q> __device__ __forceinline__ cert::CellX<Q> cert_cell(const Cell<double> &c, bool mir) {
    return cert::CellX<Q>{cxm<Q>(c.D, mir), cxm<Q>(c.S0, mir), cx<Q>(c.C0), cxm<Q>(c.W, mir), cx<Q>(c.Z), cx<Q>(c.L)};
}
template <int Q> __device__ __forceinline__ cert::HitX<Q> cert_hit(const void *rec, bool mir) {
    const HitRecF &r = *reinterpret_cast<const HitRecF *>(rec);
    cert::HitX<Q> h;
    h.x0 = cert::sc<Q>(r.lo[0]);
    h.y0 = cert::sc<Q>(mir ? -r.lo[1] : r.lo[1]);
    h.sph = cert::sc<Q>(r.lo[2]);
    h.cph = cert::sc<Q>(mir ? -r.lo[3] : r.lo[3]);
    h.t = cert::sc<Q>(r.lo[4]);
    h.spt = cert::sc<Q>(r.lo[5]);
    h.cpt = cert::sc<Q>(mir ? -r.lo[6] : r.lo[6]);
    h.t2 = cert::sc<Q>(r.lo[7]);
    h.d = cert::point(cert::sc<Q>(r.lo[8]));
    return h;
}

__device__ __forceinline__ IV<double> hull2(IV<double> a, IV<double> b) { return {mn(a.lo, b.lo), mx(a.hi, b.hi)}; }
// the smallest box around cells [i0, i1] of axis a (edges ascend along an axis)
__device__ __forceinline__ IV<double> edge_span(const DevGeom &g, int a, int level, int i0, int i1) {
    return hull2(edge(g, a, level, i0), edge(g, a, level, i1));
}

// A box of cells (a parent) as the evaluations take it: FP32 ends of the mirrored D, S0, C0, W, Z
// and of L, and (midpoint form) the range of its phi0 centres' sin / cos (the other centres lie in
// the box).  Made once per box and kept in shared memory: conversions from FP64 run on its pipe.
struct CertBox {
    float2 v[6], sc[2];
    int mir, guard;
};
template <int K> __device__ __forceinline__ CertBox cert_box(const Cell<double> &c, IV<double> Sc, IV<double> Cc) {
    CertBox b;
    bool guard;
    const bool mir = omega_sign<K>(c.W, &guard);
    auto f = [](cert::X<0> x) { return make_float2(x.lo, x.hi); };
    b.v[0] = f(cxm<0>(c.D, mir));
    b.v[1] = f(cxm<0>(c.S0, mir));
    b.v[2] = f(cx<0>(c.C0));
    b.v[3] = f(cxm<0>(c.W, mir));
    b.v[4] = f(cx<0>(c.Z));
    b.v[5] = f(cx<0>(c.L));
    b.sc[0] = f(cxm<0>(Sc, mir));
    b.sc[1] = f(cx<0>(Cc));
    b.mir = mir;
    b.guard = guard;
    return b;
}
// The box of cells [i0, i1] per axis at `level` (ends included).
template <int K>
__device__ __forceinline__ CertBox cert_span(const DevGeom &g, int level, const int (&i0)[5], const int (&i1)[5]) {
    double s0 = 0.0, c0 = 0.0, s1 = 0.0, c1 = 0.0;
    if constexpr (K == kMid) {
        sincos_phi0_centre(g, level, i0[1], s0, c0);
        sincos_phi0_centre(g, level, i1[1], s1, c1);
    }
    return cert_box<K>(Cell<double>{edge_span(g, 0, level, i0[0], i1[0]),
                                    hull2(sin_phi0(g, level, i0[1]), sin_phi0(g, level, i1[1])),
                                    hull2(cos_phi0(g, level, i0[1]), cos_phi0(g, level, i1[1])),
                                    edge_span(g, 2, level, i0[2], i1[2]), edge_span(g, 3, level, i0[3], i1[3]),
                                    edge_span(g, 4, level, i0[4], i1[4])},
                       IV<double>{mn(s0, s1), mx(s0, s1)}, IV<double>{mn(c0, c1), mx(c0, c1)});
}
template <int Q> __device__ __forceinline__ cert::X<Q> xf(float2 a) {   // ends rounded from FP64
    cert::X<Q> r;
    r.lo = a.x;
    r.hi = a.y;
    r.e = Q ? cert::rnd<Q>(cert::mag2(a.x, a.y)) + cert::kTiny : 0.f;
    return r;
}

// Axis quantity q (0 .. 5: d0, sin phi0, cos phi0, omega, z0, tan(lambda)) of a cell with index i on
// that axis, in FP32.
__device__ __forceinline__ float2 axis_float(const DevGeom &g, int level, int q, int i) {
    const IV<double> v = q == 0 ? edge(g, 0, level, i) : q == 1 ? sin_phi0(g, level, i) : q == 2 ? cos_phi0(g, level, i)
                       : q == 3 ? edge(g, 2, level, i) : q == 4 ? edge(g, 3, level, i) : edge(g, 4, level, i);
    return make_float2((float)v.lo, (float)v.hi);
}
// The box around the two cells v[0], v[1] per quantity.  No omega cell holds 0 (apo_geometry_create);
// an omega that FP32 rounds to 0, or a box over both signs, leaves its reciprocal without a bound.
__device__ __forceinline__ CertBox float_box(const float2 (&v)[2][6]) {
    CertBox b;
    b.mir = v[0][3].y < 0.f && v[1][3].y < 0.f;
    b.guard = 0;
#pragma unroll
    for (int q = 0; q < 6; q++) {
        const float lo = fminf(v[0][q].x, v[1][q].x), hi = fmaxf(v[0][q].y, v[1][q].y);
        b.v[q] = b.mir && (q == 0 || q == 1 || q == 3) ? make_float2(-hi, -lo) : make_float2(lo, hi);
    }
    return b;
}

// The test of one hit on a box: -1 when no cell inside it gets the hit's vote, else the error bound
// its cells share (NaN: they cannot be decided by one).  own: the box is one cell; -2 when it votes.
// Not inlined: its registers stay out of the callers' loops, and one copy stays in the instruction
// cache.
template <int K>
__device__ __noinline__ float box_error(const CertBox *b, const void *rec, bool outgoing, bool own = false) {
    constexpr int Q = K == kMid ? 64 : K;
    if (b->guard) return NAN;
    const cert::CellX<Q> c{xf<Q>(b->v[0]), xf<Q>(b->v[1]), xf<Q>(b->v[2]), xf<Q>(b->v[3]), xf<Q>(b->v[4]), xf<Q>(b->v[5])};
    const cert::HitX<Q> hx = cert_hit<Q>(rec, b->mir);
    if constexpr (K == kMid) {
        using N = cert::X<64>;
        const cert::MidHit<N> h{cert::point(hx.x0), cert::point(hx.y0), cert::point(hx.sph), cert::point(hx.cph),
                                cert::point(hx.t), cert::point(hx.spt), cert::point(hx.cpt), cert::point(hx.t2), hx.d};
        const cert::MidCell<N> m{c.D, xf<64>(b->sc[0]), xf<64>(b->sc[1]), c.W, c.Z, cert::recip(c.W)};
        N Gp, Gm;
        cert::mid_tail<64, N>(cert::mid_prefix<64, N>(c, m, h), c.L, m, h, c.W, Gp, Gm);
        // 1 %: the FP64 program's own distance from the real values
        const float e = (Gp.e < 1e30f && Gm.e < 1e30f) ? 1.01f * fmaxf(Gp.e, Gm.e) : NAN;
        return cert::decide(Gp, Gm, e) == cert::kNo ? -1.f : e;
    } else {
        const cert::Eval<K> x = cert::eval(c, hx, own);
        const float e = cert::bound(x);
        const int v = cert::verdict(x, outgoing, e);
        return v == cert::kNo ? -1.f : (own && v == cert::kYes ? -2.f : e);
    }
}
// Whether no cell inside the box with its tan(lambda) ends replaced by L gets the hit's vote, for an
// error bound e of the box (the bound holds for every box inside it, so bare end points do).
template <int K>
__device__ __noinline__ bool box_refuses(const CertBox *b, float2 L, const void *rec, float e, bool outgoing) {
    if (b->guard) return false;
    const cert::CellX<0> c{xf<0>(b->v[0]), xf<0>(b->v[1]), xf<0>(b->v[2]), xf<0>(b->v[3]), xf<0>(b->v[4]), xf<0>(L)};
    const cert::HitX<0> hx = cert_hit<0>(rec, b->mir);
    if constexpr (K == kMid) {
        using N = cert::X<0>;
        const cert::MidHit<N> h{cert::point(hx.x0), cert::point(hx.y0), cert::point(hx.sph), cert::point(hx.cph),
                                cert::point(hx.t), cert::point(hx.spt), cert::point(hx.cpt), cert::point(hx.t2), hx.d};
        const cert::MidCell<N> m{c.D, xf<0>(b->sc[0]), xf<0>(b->sc[1]), c.W, c.Z, cert::recip(c.W)};
        N Gp, Gm;
        cert::mid_tail<0, N>(cert::mid_prefix<0, N>(c, m, h), c.L, m, h, c.W, Gp, Gm);
        return cert::decide(Gp, Gm, e) == cert::kNo;
    } else {
        return cert::verdict(cert::eval(c, hx), outgoing, e) == cert::kNo;
    }
}

// The FP32 program's votes of one hit for the cells c with tan(lambda) cells l0 + bit, bits of `mask`;
// they share its tan(lambda)-free part.  rec: the staged FP32 record.
static __device__ __noinline__ uint32_t program_f32(const DevGeom &g, const Cell<double> &c, int level, int l0, uint32_t mask,
                                             const void *rec) {
    Cell<float> x{to_prec<float>(c.D), to_prec<float>(c.S0), to_prec<float>(c.C0),
                  to_prec<float>(c.W), to_prec<float>(c.Z), IV<float>{0.f, 0.f}};
    Hit<float> h = load_hit<float>(rec);
    if (mirror_cell(x)) mirror_hit(h);
    if (le0(x.W.lo)) return mask;
    const IV<float> R = recip(x.W);
    const Pre<float> p = prefix(x, h, g.k);
    if (p.novote) return 0u;
    if (p.guard) return mask;
    uint32_t yes = 0;
#pragma unroll 1
    while (mask) {
        const int b = __ffs(mask) - 1;
        mask &= mask - 1;
        if (tail(p, to_prec<float>(edge(g, 4, level, l0 + b)), h, R, x.W, g.k)) yes |= 1u << b;
    }
    return yes;
}

// The direction condition of a cell and hit as the program (T) tests it: true when it refuses the vote.
template <typename T> __device__ __noinline__ bool upstream(const Cell<double> &c, const void *rec) {
    Cell<T> x{to_prec<T>(c.D), to_prec<T>(c.S0), to_prec<T>(c.C0), to_prec<T>(c.W), to_prec<T>(c.Z), IV<T>{T(0), T(0)}};
    Hit<T> h = load_hit<T>(rec);
    if (mirror_cell(x)) mirror_hit(h);
    const IV<T> Xw = add(h.x0, mul(x.Z, h.spt)), Yw = sub(h.y0, mul(x.Z, h.cpt));
    return lt0(add(mul(Xw, x.C0), mul(Yw, x.S0)).hi);
}
// The same where its certified test may be undecided: kYes or kNo.  Left open, every tan(lambda) bin of the
// pair would be undecided, and one lane would evaluate them all (level 0 with the direction condition, 256
// events of 16^5 cells, FP32: 8.0 -> 4.8 ms with this and the votes above; one event 0.39 -> 0.12 ms).
template <int K>
__device__ __forceinline__ int settle_direction(int dir, const Cell<double> &c, const HitRecD *hd, const void *hf) {
    if constexpr (K != kMid) {
        if (dir == cert::kUnknown)
            dir = upstream<typename RefOf<K>::T>(c, K == 64 ? static_cast<const void *>(hd) : hf) ? cert::kNo : cert::kYes;
    }
    return dir;
}

// Hits no parent could decide for a cell, one by one: FP64 with `own` (the parent had no bound) by the
// cell's own evaluation with errors first, then the reference program; FP32 by the program at once, which
// costs no more than an evaluation with errors.  mask: tan(lambda) cells l0 + bit
// in question; returns those that vote.  Not inlined: about one pair in 10^4 comes here, and its
// registers stay out of the callers' loops.
template <int K>
__device__ __noinline__ uint32_t resolve(const DevGeom &g, int level, int d, int p, int w, int z, int l0,
                                         uint32_t mask, bool own, const HitRecD *hd, const void *hf) {
    Cell<double> c{edge(g, 0, level, d), sin_phi0(g, level, p), cos_phi0(g, level, p), edge(g, 2, level, w),
                   edge(g, 3, level, z), {0.0, 0.0}};
    uint32_t yes = 0;
    if constexpr (K == kMid) {   // the midpoint form's own evaluation
        MidCentre m;
        sincos_phi0_centre(g, level, p, m.S0, m.C0);
        m.D = pt::centre(c.D);
        m.W = pt::centre(c.W);
        m.Z = pt::centre(c.Z);
        while (mask) {
            const int b = __ffs(mask) - 1;
            mask &= mask - 1;
            if (mid_vote_pair(c, m, pt::centre(edge(g, 4, level, l0 + b)), load_hit<double>(hd))) yes |= 1u << b;
        }
        return yes;
    } else if constexpr (K == 32) {
        return program_f32(g, c, level, l0, mask, hf);
    } else {
        const IV<double> L0 = edge(g, 4, level, l0);
        c.L = L0;
        CertBox box = cert_box<K>(c, L0, L0);
        while (mask) {
            const int b = __ffs(mask) - 1;
            mask &= mask - 1;
            c.L = edge(g, 4, level, l0 + b);
            int v = cert::kUnknown;
            if (own) {
                box.v[5] = make_float2((float)c.L.lo, (float)c.L.hi);
                const float e = box_error<K>(&box, hf, g.k.outgoing != 0, true);
                v = e == -1.f ? cert::kNo : (e == -2.f ? cert::kYes : cert::kUnknown);
            }
            if (v == cert::kUnknown) v = vote_pair<double>(c, load_hit<double>(hd), g.k) ? cert::kYes : cert::kNo;
            if (v == cert::kYes) yes |= 1u << b;
        }
        return yes;
    }
}

// The reference's own evaluation of one pair, out of the callers' registers.
template <typename T>
__device__ __noinline__ bool vote_reference(const DevGeom &g, const Cell<double> &c, const Hit<T> &h) {
    const Cell<T> ct{to_prec<T>(c.D), to_prec<T>(c.S0), to_prec<T>(c.C0),
                     to_prec<T>(c.W), to_prec<T>(c.Z), to_prec<T>(c.L)};
    return vote_pair<T>(ct, h, g.k);
}

// The vote of a staged hit for one cell (not mirrored), by the pair's own bound.
template <int K>
__device__ __forceinline__ bool vote_single(const DevGeom &g, const Cell<double> &c, const HitRecD *hd,
                                            const HitRecF *hf) {
    using T = typename RefOf<K>::T;
    bool guard;
    const bool mir = omega_sign<K>(c.W, &guard);
    if (guard) return true;
    const cert::Eval<K> x = cert::eval(cert_cell<K>(c, mir), cert_hit<K>(hf, mir), true);
    const int v = cert::verdict(x, g.k.outgoing != 0, cert::bound(x));
    if (v != cert::kUnknown) return v == cert::kYes;
    const void *rec = K == 64 ? static_cast<const void *>(hd) : static_cast<const void *>(hf);
    return vote_reference<T>(g, c, load_hit<T>(rec));
}

// The FP64 vote of a staged hit for one cell with its drift widened to [max(rd(d - width), 0),
// ru(d + width)] (the hit finding), by the pair's own bound.  Not inlined (see resolve).
template <int K = 64>
__device__ __noinline__ bool vote_widened(const DevGeom &g, const Cell<double> &c, const HitRecD *hd,
                                             double width) {
    Hit<double> h = load_hit<double>(hd);
    const double d = h.d.lo, dlo = __dsub_rd(d, width);
    h.d = {gt0(dlo) ? dlo : 0.0, __dadd_ru(d, width)};
    bool guard;
    const bool mir = omega_sign<64>(c.W, &guard);
    if (guard) return true;
    cert::HitX<64> hx;
    const IV<double> *f = &h.x0;
    cert::Sc<64> *s = &hx.x0;
#pragma unroll
    for (int i = 0; i < 8; i++)
        s[i] = cert::sc<64>(__double2float_rd((mir && (i == 1 || i == 3 || i == 6)) ? -f[i].lo : f[i].lo));
    hx.d = cx<64>(h.d);
    const cert::Eval<64> x = cert::eval(cert_cell<64>(c, mir), hx, true);
    const int v = cert::verdict(x, g.k.outgoing != 0, cert::bound(x));
    if (v != cert::kUnknown) return v == cert::kYes;
    return vote_reference<double>(g, c, h);
}

// A warp's undecided (lane, hit) pairs, resolved by its lanes together once 32 are waiting and at
// the end.  Every lane calls push in step, so no atomics and no block barrier are needed (a block's
// queue behind barriers cost a quarter of the voting kernels' time).
struct WarpQueue {
    uint32_t id[64];     // lane (or pair, below 256) | hit << 8 | own << 16
    uint32_t mask[64];   // tan(lambda) bits in question, then those that vote
    // n: entries held (below 32 on entry), the same in every lane; returns their new number
    __device__ __forceinline__ int push(int n, int lane, int h, bool own, uint32_t m) {
        return push(n, lane, lane, h, own, m);
    }
    __device__ __forceinline__ int push(int n, int pair, int lane, int h, bool own, uint32_t m) {
        const unsigned b = __ballot_sync(0xffffffffu, m != 0u);
        if (m) {
            const int s = n + __popc(b & ((1u << lane) - 1u));
            id[s] = (uint32_t)pair | ((uint32_t)h << 8) | (own ? 1u << 16 : 0u);
            mask[s] = m;
        }
        return n + __popc(b);
    }
    // each(pair, hit, own, mask) for all n entries, one per lane
    template <typename Each> __device__ __forceinline__ void drain(int n, int lane, Each each) {
        __syncwarp();
        for (int i = lane; i < n; i += 32)
            each((int)(id[i] & 255u), (int)((id[i] >> 8) & 255u), (id[i] >> 16) != 0u, mask[i]);
        __syncwarp();
    }
    // resolves all n entries (solve(lane, hit, own, mask) -> voting bits) and gives every lane its
    // own (take(bits))
    template <typename Solve, typename Take>
    __device__ __forceinline__ void drain(int n, int lane, Solve solve, Take take) {
        __syncwarp();
        for (int i = lane; i < n; i += 32)
            mask[i] = solve((int)(id[i] & 255u), (int)((id[i] >> 8) & 255u), (id[i] >> 16) != 0u, mask[i]);
        __syncwarp();
        for (int i = 0; i < n; i++)
            if ((int)(id[i] & 255u) == lane) take(mask[i]);
        __syncwarp();
    }
};

// The vote of one tan(lambda) interval for a prefix and error bound e.
__device__ __forceinline__ int cert_tail(const cert::PreX<0> &p, cert::X<0> L, const cert::HitX<0> &h,
                                         cert::X<0> R, cert::X<0> W, float e) {
    cert::X<0> Gp, Gm;
    cert::tail(p, L, h, R, W, Gp, Gm);
    return cert::decide(Gp, Gm, e);
}

// The direction condition for a prefix: kNo refuses every vote, kUnknown leaves it open.
__device__ __forceinline__ int cert_direction(const cert::PreX<0> &p, bool outgoing, float e) {
    if (!outgoing) return cert::kYes;
    return p.wt.hi < -e ? cert::kNo : (p.wt.hi >= e ? cert::kYes : cert::kUnknown);
}

// One cell's evaluation per program: what a thread keeps of its cell, the tan(lambda)-free part per
// hit, and one tan(lambda) cell's vote with the parent's error bound e.  L: the cell's end points,
// or (midpoint form) its centre in .x.
template <int K> struct Prog {
    struct CellT { cert::CellX<0> c; cert::X<0> R; };
    using HitT = cert::HitX<0>;
    using Pre = cert::PreX<0>;
    static __device__ __forceinline__ CellT cell(const DevGeom &, int, int, const Cell<double> &c, bool mir) {
        const cert::CellX<0> x = cert_cell<0>(c, mir);
        return CellT{x, cert::recip(x.W)};
    }
    // from FP32 ends (not mirrored) of its cells per axis
    static __device__ __forceinline__ CellT cell(const float2 (&v)[2][6], const int (&bit)[4], bool mir) {
        auto f = [&](int q, int a, bool flip) {
            const float2 x = v[bit[a]][q];
            return flip ? cert::X<0>{-x.y, -x.x, 0.f} : cert::X<0>{x.x, x.y, 0.f};
        };
        const cert::CellX<0> x{f(0, 0, mir), f(1, 1, mir), f(2, 1, false), f(3, 2, mir), f(4, 3, false), {0.f, 0.f, 0.f}};
        return CellT{x, cert::recip(x.W)};
    }
    static __device__ __forceinline__ float2 tanl(IV<double> L) { return make_float2((float)L.lo, (float)L.hi); }
    static __device__ __forceinline__ HitT hit(const void *rec, bool mir) { return cert_hit<0>(rec, mir); }
    static __device__ __forceinline__ Pre prefix(const CellT &c, const HitT &h) { return cert::prefix(c.c, h); }
    static __device__ __forceinline__ int direction(const Pre &p, bool outgoing, float e) {
        return cert_direction(p, outgoing, e);
    }
    static __device__ __forceinline__ int vote(const Pre &p, float2 L, const CellT &c, const HitT &h, float e) {
        return cert_tail(p, cert::X<0>{L.x, L.y, 0.f}, h, c.R, c.c.W, e);
    }
};
template <> struct Prog<kMid> {
    struct CellT { cert::CellX<0> c; cert::MidCell<cert::Pt> m; };
    using HitT = cert::MidHit<cert::Pt>;
    using Pre = cert::MidPreX<0, cert::Pt>;
    static __device__ __forceinline__ CellT cell(const DevGeom &g, int level, int p, const Cell<double> &c, bool mir) {
        double s, co;
        sincos_phi0_centre(g, level, p, s, co);
        const float sg = mir ? -1.f : 1.f, W = sg * (float)pt::centre(c.W);
        return CellT{cert_cell<0>(c, mir), {{sg * (float)pt::centre(c.D)}, {sg * (float)s}, {(float)co}, {W},
                                            {(float)pt::centre(c.Z)}, {cert::rcp_a(W)}}};
    }
    static __device__ __forceinline__ float2 tanl(IV<double> L) { return make_float2((float)pt::centre(L), 0.f); }
    static __device__ __forceinline__ HitT hit(const void *rec, bool mir) {
        const cert::HitX<0> h = cert_hit<0>(rec, mir);
        return HitT{{h.x0.v}, {h.y0.v}, {h.sph.v}, {h.cph.v}, {h.t.v}, {h.spt.v}, {h.cpt.v}, {h.t2.v}, {h.d.lo}};
    }
    static __device__ __forceinline__ Pre prefix(const CellT &c, const HitT &h) {
        return cert::mid_prefix<0, cert::Pt>(c.c, c.m, h);
    }
    static __device__ __forceinline__ int direction(const Pre &, bool, float) { return cert::kYes; }
    static __device__ __forceinline__ int vote(const Pre &p, float2 L, const CellT &c, const HitT &h, float e) {
        cert::X<0> Gp, Gm;
        cert::mid_tail<0, cert::Pt>(p, cert::Pt{L.x}, c.m, h, c.c.W, Gp, Gm);
        return cert::decide(Gp, Gm, e);
    }
};

// Bit-sliced vote counters: bit l of plane q is bit q of counter l (counts <= 256: 9 planes);
// adding a mask of votes is a ripple-carry add.
struct VotePlanes {
    uint32_t pl[9];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int q = 0; q < 9; q++) pl[q] = 0u;
    }
    __device__ __forceinline__ void add(uint32_t m) {
#pragma unroll
        for (int q = 0; q < 9; q++) {
            const uint32_t c = pl[q] & m;
            pl[q] ^= m;
            m = c;
        }
    }
    __device__ __forceinline__ int get(int l) const {
        int v = 0;
#pragma unroll
        for (int q = 0; q < 9; q++) v |= (int)((pl[q] >> l) & 1u) << q;
        return v;
    }
};

}  // namespace apo
