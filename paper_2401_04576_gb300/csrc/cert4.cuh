// The 4-D search's vote (fourd.cuh) in plain FP32 with a certified distance to its evaluation in
// FP64 (K = 64) or FP32 (K = 32): the radicand of d^Ax and the interval G = A2 - (R_v + d^Ax)^2 of a
// voxel.  Every step of the program has its step here with the same operands (products are
// regrouped, a quotient is a product with an approximate reciprocal), so the bound's roundings
// cover the program's own as well.
#pragma once
#include "cert_point.cuh"

namespace apo {
namespace cert {

// One column's centre: point constants (from the FP64 centre) and the direction of the origin.
template <typename N> struct Col4X { N xc, yc, R, aL, ox, oy, ion, psi_ref; };   // ion = 1 / on
template <typename N> struct Hit4X { N x0, y0, sph, cph, t, spt, cpt, t2, d; };

// z0- and sign-free quantities of one (centre, hit)
template <typename N> struct Pre4X { N RA, iRA, cA, sA, sPA, cPA, cos2, sin2, psi, Rpsi, iA2; };

constexpr float kTwoPi = 6.2831853f, kPi = 3.14159265f;
// 2 atan(x), 0 <= |x| <= 1: one half-angle reduction, the series through x^15 (|x| <= 0.4143
// there: truncation below 1e-7).  With angle4's steps, in units of 2^-24: 5.5 before x, 5.5 x 1.42 in
// the reduction, 3.5 x pi / 2 in the series, 5 from pi: below 1.5e-6.
template <int K> struct AngleErr { static constexpr float v = 1.5e-6f; };
// and the FP32 program's own: in the same units 10 before x, 3.5 in each reduction, 5 in the series,
// all x pi / 2, 2 from pi: below 2.3e-6
template <> struct AngleErr<32> { static constexpr float v = 3.8e-6f; };
APO_CERT float twice_atan(float x) {
    x = x * rcp_a(1.f + sqrt_a(fmaf(x, x, 1.f)));
    const float y = x * x;
    float h = (float)(1.0 / 15);
    h = fmaf(-h, y, (float)(1.0 / 13));
    h = fmaf(-h, y, (float)(1.0 / 11));
    h = fmaf(-h, y, (float)(1.0 / 9));
    h = fmaf(-h, y, (float)(1.0 / 7));
    h = fmaf(-h, y, (float)(1.0 / 5));
    h = fmaf(-h, y, (float)(1.0 / 3));
    h = fmaf(-h, y, 1.f);
    return 4.f * x * h;
}
// the angle of (cs, sn) / r in (-pi, pi] for r = |(cs, sn)|, as the program's half-angle form
APO_CERT float angle4(float sn, float cs, float ir) {
    const float s = sn * ir, c = cs * ir;
    const float a = twice_atan(s * rcp_a(1.f + fabsf(c)));
    return c >= 0.f ? a : copysignf(kPi, s) - a;
}

// psi of a child: its phase from the direction of the origin, in [0, 2 pi), less the reference's.
// Undecided (bad) where the phase is within eps of the jump at 0.
APO_CERT Pt psi4(const Col4X<Pt> &m, Pt dx, Pt dy, Pt iRA, float eps, bool &bad) {
    const float sn = m.ox.v * dy.v - m.oy.v * dx.v, cs = m.ox.v * dx.v + m.oy.v * dy.v;
    float ph = angle4(sn, cs, m.ion.v * iRA.v);
    bad = !(fabsf(ph) > eps);
    if (ph < 0.f) ph += kTwoPi;
    return {ph - m.psi_ref.v};
}
// The phases of a range of wire points (dx, dy) and centres: the middle's +- the largest turn; eps: the error
// a child's phase can have, (e_sn + e_cs) / r + AngleErr and the roundings of 2 pi and the sum.
struct Turn4 { float ph, turn, eps; };
template <int K> APO_CERT Turn4 turn4(const Col4X<X<K>> &m, X<K> dx, X<K> dy, X<K> iRA) {
    const X<K> sn = sub(mul(m.ox, dy), mul(m.oy, dx)), cs = add(mul(m.ox, dx), mul(m.oy, dy));
    const X<K> ir = mul(m.ion, iRA);
    const float mx = 0.5f * (dx.lo + dx.hi), my = 0.5f * (dy.lo + dy.hi);
    const float ux = 0.5f * (m.ox.lo + m.ox.hi), uy = 0.5f * (m.oy.lo + m.oy.hi);
    Turn4 r;
    r.ph = angle4(ux * my - uy * mx, ux * mx + uy * my, rcp_a(sqrt_a(ux * ux + uy * uy) * sqrt_a(mx * mx + my * my)));
    const float hx = dx.hi - mx + 2.f * dx.e, hy = dy.hi - my + 2.f * dy.e;
    const float kx = m.ox.hi - ux + 2.f * m.ox.e, ky = m.oy.hi - uy + 2.f * m.oy.e;
    // each vector's turn; below 1 rad it is under 1.1 chord / radius
    r.turn = 1.6f * (sqrt_a(hx * hx + hy * hy) * M(iRA) + sqrt_a(kx * kx + ky * ky) * M(m.ion));
    const float least = ir.lo - 2.f * ir.e;   // 1 / r's own relative error turns the angle by at most that
    r.eps = when(least > 0.f, ((sn.e + cs.e) * M(ir) + ir.e / least + 8.f * Unit<K>::u + AngleErr<K>::v) * 1.01f);
    return r;
}

template <typename N> APO_CERT void wire4x(const Col4X<N> &m, N z, const Hit4X<N> &h, N &dx, N &dy) {
    dx = sub(add(h.x0, mul(z, h.spt)), m.xc);
    dy = sub(sub(h.y0, mul(z, h.cpt)), m.yc);
}
// all but psi and Rpsi
template <typename N> APO_CERT Pre4X<N> prefix4x(N dx, N dy, const Hit4X<N> &h) {
    Pre4X<N> p;
    p.RA = sqrtx(add(sqr(dx), sqr(dy)));
    p.iRA = recip(p.RA);
    p.cA = sub(mul(dx, h.sph), mul(dy, h.cph));
    p.sA = add(mul(dx, h.cph), mul(dy, h.sph));
    p.sPA = mul(p.sA, p.iRA);
    p.cPA = mul(p.cA, p.iRA);
    p.iA2 = scl(sqr(p.iRA), 0.5f);   // 1 / (2 A2)
    p.cos2 = scl(mul(sub(sqr(p.cA), sqr(p.sA)), p.iA2), 2.f);
    p.sin2 = scl(mul(mul(p.sA, p.cA), p.iA2), 4.f);
    return p;
}

// The phase correction of one drift sign (ds = +-d), even and odd in tan(lambda) = L = +-aL: for L it
// is u - v, for -L it is u + v.
template <typename N> struct Delta4 { N u, v; };
template <typename N> APO_CERT Delta4<N> delta4x(const Pre4X<N> &p, N R, N L, N ds, const Hit4X<N> &h) {
    const N zA = mul(L, p.Rpsi), Lz = mul(L, zA), L2 = sqr(L);
    const N f1 = add(mul(zA, p.sPA), mul(mul(L, ds), p.cPA));            // -Phi1 RA
    const N f2 = add(sub(mul(R, Lz), mul(mul(Lz, sub(R, scl(ds, 2.f))), p.cos2)),
                     mul(add(sqr(zA), mul(ds, add(p.RA, mul(L2, sub(add(R, p.RA), ds))))), p.sin2));
    return Delta4<N>{mul(mul(f2, p.iA2), h.t2), mul(mul(f1, p.iRA), h.t)};
}
// (R + d^Ax)^2: the radicand of Eq. (defdiAX_b) for a phase correction dl
template <typename N> APO_CERT N rad4x(const Pre4X<N> &p, N R, N L, N ds, N dl, const Hit4X<N> &h) {
    N sd, cd;
    sincos4(dl, sd, cd);
    const N sP = add(mul(p.sPA, cd), mul(p.cPA, sd)), cP = sub(mul(p.cPA, cd), mul(p.sPA, sd));
    const N Lt = mul(L, h.t);
    const N u2 = add(add(add1(mul(scl(Lt, 2.f), sP), 1.f), mul(sqr(L), h.t2)), mul(sqr(cP), h.t2));
    const N q = mul(ds, rsqrtx(u2));
    const N zt = mul(sub(mul(L, mul(R, add(p.psi, dl))), mul(mul(q, cP), h.t)), h.t);   // z^St t
    const N Lqt = mul(q, Lt);
    const N ct = sub(mul(zt, p.cA), mul(Lqt, p.sA));                                     // c^tau t
    return sub(sub(sub(sqr(add(R, q)), scl(ct, 2.f)), sqr(zt)), sqr(Lqt));
}

// The voxel's intervals: x_c, y_c, and R_v - R about the centre's R (each at most dR)
template <int K> struct Box4X { X<K> X_, Y_, dR; };
template <int K, typename N>
APO_CERT X<K> a2_4x(const Box4X<K> &b, X<K> Z, const Hit4X<N> &h) {
    const X<K> xw = add(ivp(h.x0), mul(Z, ivp(h.spt))), yw = sub(ivp(h.y0), mul(Z, ivp(h.cpt)));
    return add(sqr(sub(xw, b.X_)), sqr(sub(yw, b.Y_)));
}

struct Bound4 { float e, eps; };   // of G and of the radicand; of a phase (e NaN: undecidable)

// The errors of every child of some columns and one hit: centres m, z and voxels b, Z (ranges), both signs of
// tan(lambda) and of the drift (one evaluation over their hulls: the errors grow with magnitudes).
// G = A2 - (s + dR)^2 with s = sqrt(rad): its error is e_A2 + e_rad (1 + dR / s), at most
// e_A2 + 2 e_rad where s >= dR, and the roundings of s, of d^Ax = s - R, of the sum and of the
// square on both sides: 10 units of 2^-23 of the square.
template <int K>
APO_CERT Bound4 bound4(const Col4X<X<K>> &m, const Box4X<K> &b, X<K> z, X<K> Z, const Hit4X<X<K>> &h) {
    X<K> dx, dy;
    wire4x(m, z, h, dx, dy);
    Pre4X<X<K>> p = prefix4x(dx, dy, h);
    const Turn4 tr = turn4<K>(m, dx, dy, p.iRA);
    const X<K> A2 = a2_4x<K, X<K>>(b, Z, h);
    X<K> L = m.aL, ds = h.d;
    L.lo = -L.hi;
    ds.lo = -ds.hi;
    // the range of phases in [0, 2 pi), in two parts when it holds the jump at 0
    const float w = tr.turn + 2.f * tr.eps;
    const bool pos = tr.ph + w > 0.f, neg_ = tr.ph - w < 0.f;
    float e = 0.f;
    for (int s = 0; s < 2; s++) {
        if (!(s ? neg_ : pos)) continue;
        X<K> ph;
        ph.lo = s ? tr.ph - w + kTwoPi : fmaxf(tr.ph - w, 0.f);
        ph.hi = s ? fminf(tr.ph + w, 0.f) + kTwoPi : tr.ph + w;
        ph.e = tr.eps + rnd<K>(4.f * kTwoPi);
        p.psi = sub(ph, m.psi_ref);
        p.Rpsi = mul(m.R, p.psi);
        const Delta4<X<K>> dl = delta4x(p, m.R, L, ds, h);   // L and ds hold both signs
        const X<K> rad = rad4x(p, m.R, L, ds, sub(dl.u, dl.v), h);
        const float mr = M(rad), md = M(b.dR);
        const float x = A2.e + 2.f * rad.e + 10.f * Unit<K>::ua * (mr + md * md) + 2.f * rnd<K>(M(A2)) + 4.f * b.dR.e;
        e = x < 1e30f ? fmaxf(e, x) : INFINITY;
    }
    const bool ok = tr.turn < 1.f && tr.eps < 1e-2f && e < 1e30f;
    // 1 %: FP32 constants and what regrouping moves between roundings
    return Bound4{ok ? e * 1.01f : NAN, tr.eps};
}

// One voxel and sign of tan(lambda), L = +-aL: kYes / kNo / kUnknown (either drift sign; a negative
// radicand guards, and votes); dl: its phase corrections for the drift signs + and -.
APO_CERT int vote4x(const Pre4X<Pt> &p, const Col4X<Pt> &m, Pt L, const Hit4X<Pt> &h, X<0> A2, X<0> dR, float e,
                    const Pt (&dl)[2]) {
    const float md = mag2(dR.lo, dR.hi), least = fmaxf(4.f * e, 1.01f * md * md);
    bool yes = false, no = true;
#pragma unroll
    for (int sg = 0; sg < 2; sg++) {
        const float rad = rad4x(p, m.R, L, sg ? neg(h.d) : h.d, dl[sg], h).v;
        const float s = sqrt_a(rad), a = s + dR.lo, c = s + dR.hi;   // s >= |dR|: both ends >= 0
        const float lo = A2.lo - c * c, hi = A2.hi - a * a;
        const bool in = rad > least;
        yes = yes || rad < -e || (in && lo <= -e && hi >= e);
        no = no && in && (lo > e || hi < -e);
    }
    return yes ? kYes : (no ? kNo : kUnknown);
}

}  // namespace cert
}  // namespace apo
