// The midpoint form (APO_F64_MID, vote_program.cuh) in plain FP32 with a certified distance to
// the FP64 evaluation: the point part at the voxel's centre on Pt or, for a range of centres, on
// X<64>; the interval G0 over the voxel.  A range of centres encloses every centre in it and the
// joined voxel every voxel, so a parent's G encloses its children's: where it excludes 0 no child
// votes, although the form itself says nothing about children.
#pragma once
#include "cert_point.cuh"

namespace apo {
namespace cert {

template <typename N> struct MidCell { N D, S0, C0, W, Z, R; };   // the mirrored centre, R = 1 / W
template <typename N> struct MidHit { N x0, y0, sph, cph, t, spt, cpt, t2, d; };   // mirrored with its cell
// Names as PreX (certified.cuh).
template <int K, typename N> struct MidPreX { X<K> G0; N psi, N_, sPA, cPA, rsA, rcA, sin2, A1, B1, A2, B2, pc2, tt; };

// atan without remainder, as the program's (two reductions, through x^15)
APO_CERT Pt atan_pt(Pt x) {
    float v = x.v;
#pragma unroll
    for (int i = 0; i < 2; i++) v = v * rcp_a(1.f + sqrt_a(fmaf(v, v, 1.f)));
    const float y = v * v;
    float h = (float)(1.0 / 15);
    h = fmaf(-h, y, (float)(1.0 / 13));
    h = fmaf(-h, y, (float)(1.0 / 11));
    h = fmaf(-h, y, (float)(1.0 / 9));
    h = fmaf(-h, y, (float)(1.0 / 7));
    h = fmaf(-h, y, (float)(1.0 / 5));
    h = fmaf(-h, y, (float)(1.0 / 3));
    h = fmaf(-h, y, 1.f);
    return {4.f * v * h};
}
// the interval form's enclosure holds it: its remainder only widens the range
template <int K> APO_CERT X<K> atan_pt(X<K> x) { return atanx(x); }

// c: the mirrored voxel (its W also serves G below); m: its centre(s)
template <int K, typename N>
APO_CERT MidPreX<K, N> mid_prefix(const CellX<K> &c, const MidCell<N> &m, const MidHit<N> &h) {
    MidPreX<K, N> p;
    {   // G0 = rho ((R^Ax)^2 - R^2) over the voxel
        const X<K> Xw = add(mul(c.Z, ivp(h.spt)), ivp(h.x0)), Yw = sub(ivp(h.y0), mul(c.Z, ivp(h.cpt)));
        const X<K> wt = add(mul(Xw, c.C0), mul(Yw, c.S0));
        const X<K> V = sub(sub(mul(Yw, c.C0), mul(Xw, c.S0)), c.D);
        p.G0 = add(mul_pp(c.W, sqr(wt)), mul(V, add1(mul_nn(V, c.W), -2.f)));
    }
    const N Xw = add(h.x0, mul(m.Z, h.spt)), Yw = sub(h.y0, mul(m.Z, h.cpt));
    const N wt = add(mul(Xw, m.C0), mul(Yw, m.S0));
    const N V = sub(sub(mul(Yw, m.C0), mul(Xw, m.S0)), m.D);
    const N Xt = mul(wt, m.W), Xn = add1(mul(V, m.W), -1.f);
    p.N_ = sqrtx(add(sqr(Xt), sqr(Xn)));
    p.psi = scl(atan_pt(mul(Xt, recip(sub(p.N_, Xn)))), 2.f);
    const N E1 = add(mul(m.C0, h.cph), mul(m.S0, h.sph)), E2 = sub(mul(m.C0, h.sph), mul(m.S0, h.cph));
    p.rsA = add(mul(Xt, E1), mul(Xn, E2));
    p.rcA = sub(mul(Xt, E2), mul(Xn, E1));
    const N Ninv = recip(p.N_);
    p.sPA = mul(p.rsA, Ninv);
    p.cPA = mul(p.rcA, Ninv);
    const N cos2 = sub(sqr(p.cPA), sqr(p.sPA));
    p.sin2 = scl(mul(p.sPA, p.cPA), 2.f);
    const N dW = mul(h.d, m.W), Nt2 = mul(scl(sqr(Ninv), 0.5f), h.t2);
    p.A1 = neg(mul(mul(p.psi, p.sPA), Ninv));
    p.B1 = neg(mul(mul(p.cPA, dW), Ninv));
    p.A2 = mul(sub(add(mul(p.psi, add1(neg(cos2), 1.f)), mul(p.sin2, sqr(p.psi))), mul(p.sin2, sqr(dW))), Nt2);
    p.B2 = mul(dW, Nt2);
    p.pc2 = scl(mul(p.psi, cos2), 2.f);
    p.tt = mul(h.t, h.t);
    return p;
}

// G of both drift signs for the centre's tan(lambda) L; W the voxel's interval
template <int K, typename N>
APO_CERT void mid_tail(const MidPreX<K, N> &p, N L, const MidCell<N> &m, const MidHit<N> &h, X<K> W, X<K> &Gp, X<K> &Gm) {
    const N L2 = sqr(L), Lt = mul(L, h.t), Lt2 = mul(L2, h.t2);
    const N de = add(mul(p.A1, Lt), mul(p.A2, L2));
    const N dod = add(mul(p.B1, Lt), mul(add(mul(p.pc2, L2), mul(p.sin2, add(p.N_, mul(L2, add1(p.N_, 1.f))))), p.B2));
    const N RL = mul(m.R, Lt);
#pragma unroll
    for (int sg = 0; sg < 2; sg++) {
        const N dl = sg ? sub(de, dod) : add(de, dod);
        N sd, cd;
        sincos4(dl, sd, cd);
        const N sP = add(mul(p.sPA, cd), mul(p.cPA, sd)), cP = sub(mul(p.cPA, cd), mul(p.sPA, sd));
        const N u2 = add(add(add1(mul(scl(Lt, 2.f), sP), 1.f), Lt2), mul(sqr(cP), h.t2));
        const N Q = mul(h.d, recip(sqrtx(u2)));
        const N cz = mul(mul(cP, p.tt), Q), LQt = mul(Lt, Q);
        const N zL = mul(add(p.psi, dl), RL);
        const N zt = sg ? add(zL, cz) : sub(zL, cz);
        const N zr = mul(zt, p.rcA), LQr = mul(LQt, p.rsA);
        const N Y = scl(sg ? add(zr, LQr) : sub(zr, LQr), 2.f);
        const N a1 = sg ? neg(scl(Q, 2.f)) : scl(Q, 2.f);
        const N A = add(sub(a1, Y), mul(m.W, sub(sub(sqr(Q), sqr(zt)), sqr(LQt))));
        const N dax = mul(A, recip(add1(sqrtx(add1(mul(m.W, A), 1.f)), 1.f)));
        const X<K> x = ivp(dax);
        const X<K> G = sub(p.G0, add(scl(x, 2.f), mul_pp(W, sqr(x))));
        if (sg) Gm = G;
        else Gp = G;
    }
}

}  // namespace cert
}  // namespace apo
