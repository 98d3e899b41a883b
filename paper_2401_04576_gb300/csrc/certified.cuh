// The interval vote program in plain FP32 with a certified distance to the reference
// evaluation, so that a vote of the FP64 program can be decided without FP64 arithmetic.
//
// The FP64 program (vote_program.cuh) maps the end points of its operand intervals to the end
// points of G by sums, products (min / max over end-point products), quotients and square
// roots, each rounded outward.  Here the same end points are followed in FP32, rounded to
// nearest, and every quantity carries one number e >= 0 with
//       |lo - lo_ref| <= e   and   |hi - hi_ref| <= e,
// lo_ref / hi_ref being the end points of the FP64 program on the same cell and hit.  Min, max
// and clamps are 1-Lipschitz; a product's error is |a| e_b + |b| e_a plus the roundings of both
// sides; a root's or quotient's uses the smallest argument possible.  With G's end points and e:
// lo <= -e and hi >= e proves that the FP64 program votes, lo > e or hi < -e that it does not;
// otherwise the pair is undecided and the FP64 program itself is evaluated.  The votes are
// therefore those of the FP64 program, whatever the size of e.
//
// e can be shared: every bound below grows with the magnitudes of the operands and with 1 / the
// smallest divisor or radicand, and interval operations are inclusion-isotonic, so the e of a
// cell holds for every cell inside it.  One evaluation with errors on a parent cell
// (K = 64) serves all its children, which run the bare end points (K = 0): about the cost of
// an FP32 program without directed rounding.  Magnitudes are taken as max(|lo|, |hi|) + 2 e,
// which bounds the child's reference value (parent's reference + nothing, so mag + e) and the
// child's FP32 value (another e).
//
// A guard of the program (divisor or radicand reaching 0), an angle beyond the series' range,
// an overflow or an operand out of range make e NaN or infinite, which decides nothing.
//
// Compiles as host C++ too (the bounds are checked against the oracle's end points there).
#pragma once
#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define APO_CERT __device__ __forceinline__
#else
#define APO_CERT inline
#endif

namespace apo {
namespace cert {

#ifdef __CUDACC__
// Documented maximum relative error 2^-23 each (PTX ISA, rcp / sqrt .approx.f32)
APO_CERT float rcp_a(float x) { float r; asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }
APO_CERT float sqrt_a(float x) { float r; asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }
// (rsqrt: 2^-22.9)
APO_CERT float rsqrt_a(float x) { float r; asm("rsqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }
APO_CERT float min3(float a, float b, float c) { float r; asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c)); return r; }
APO_CERT float max3(float a, float b, float c) { float r; asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c)); return r; }
#else
APO_CERT float rcp_a(float x) { return 1.0f / x; }
APO_CERT float sqrt_a(float x) { return std::sqrt(x); }
APO_CERT float rsqrt_a(float x) { return 1.0f / std::sqrt(x); }
APO_CERT float min3(float a, float b, float c) { return fminf(fminf(a, b), c); }
APO_CERT float max3(float a, float b, float c) { return fmaxf(fmaxf(a, b), c); }
#endif

// Rounding of one operation, both sides together, relative to the result's magnitude: FP32 to
// nearest (2^-24) and the reference's directed rounding, 2^-52 in FP64 (K = 64) or 2^-23 in FP32
// (K = 32); about 1 % of margin covers the roundings of e itself.  kUA: the same for the
// approximate reciprocal and root (2^-23 here).
template <int K> struct Unit { static constexpr float u = 6.0e-8f, ua = 1.3e-7f; };
template <> struct Unit<32> { static constexpr float u = 1.81e-7f, ua = 2.6e-7f; };
constexpr float kTiny = 1.2e-38f;   // FP32 underflow of a product (2^-149) and of its error terms

// An interval's end points and their error (K = 0: e is unused)
template <int K> struct X { float lo, hi, e; };
template <int K> struct Sc { float v, e; };   // a number (a hit's constant)

APO_CERT float mag2(float lo, float hi) { return fmaxf(fabsf(lo), fabsf(hi)); }
template <int K> APO_CERT float M(X<K> a) { return mag2(a.lo, a.hi) + 2.f * a.e; }
template <int K> APO_CERT float M(Sc<K> a) { return fabsf(a.v) + 2.f * a.e; }
// rounding of a result of magnitude up to m (infinite before m itself could overflow)
template <int K> APO_CERT float rnd(float m) { return (m * 4.f) * (Unit<K>::u * 0.25f); }
// closes an operation: e so far from the operands, + the rounding of the result r
template <int K> APO_CERT X<K> fin(float lo, float hi, float e) {
    X<K> r;
    r.lo = lo;
    r.hi = hi;
    r.e = K ? e + rnd<K>(mag2(lo, hi) + 2.f * e) : 0.f;
    return r;
}
template <int K> APO_CERT X<K> mk(double lo, double hi) {
    X<K> r;
    r.lo = (float)lo;
    r.hi = (float)hi;
    r.e = K ? rnd<K>(mag2(r.lo, r.hi)) + kTiny : 0.f;
    return r;
}
// a hit's constant from its FP32 value rounded down: within 2^-23 of the FP64 value and of both
// ends of the FP32 program's interval
template <int K> APO_CERT Sc<K> sc(float v) {
    Sc<K> r;
    r.v = v;
    r.e = K ? 2.f * rnd<K>(fabsf(v)) + kTiny : 0.f;
    return r;
}
template <int K> APO_CERT X<K> point(Sc<K> s) { X<K> r; r.lo = r.hi = s.v; r.e = s.e; return r; }
template <int K> APO_CERT Sc<K> neg(Sc<K> a) { a.v = -a.v; return a; }
template <int K> APO_CERT Sc<K> smul(Sc<K> a, Sc<K> b) {
    Sc<K> r;
    r.v = a.v * b.v;
    r.e = K ? M(a) * b.e + M(b) * a.e + rnd<K>(fabsf(r.v) + 2.f * (M(a) * b.e + M(b) * a.e)) + kTiny : 0.f;
    return r;
}
template <int K> APO_CERT X<K> neg(X<K> a) { X<K> r; r.lo = -a.hi; r.hi = -a.lo; r.e = a.e; return r; }
template <int K> APO_CERT X<K> scl(X<K> a, float s) {   // s a power of two, s > 0
    X<K> r;
    r.lo = a.lo * s;
    r.hi = a.hi * s;
    r.e = a.e * s;
    return r;
}
template <int K> APO_CERT X<K> add(X<K> a, X<K> b) { return fin<K>(a.lo + b.lo, a.hi + b.hi, K ? a.e + b.e : 0.f); }
template <int K> APO_CERT X<K> sub(X<K> a, X<K> b) { return fin<K>(a.lo - b.hi, a.hi - b.lo, K ? a.e + b.e : 0.f); }
template <int K> APO_CERT X<K> add1(X<K> a, float c) { return fin<K>(a.lo + c, a.hi + c, a.e); }      // a + c, c exact
template <int K> APO_CERT X<K> rsub1(float c, X<K> a) { return fin<K>(c - a.hi, c - a.lo, a.e); }     // c - a

template <int K, typename A, typename B> APO_CERT float perr(A a, B b) {   // a product's propagated error
    return K ? M(a) * b.e + M(b) * a.e + kTiny : 0.f;
}
template <int K> APO_CERT X<K> mul(X<K> a, X<K> b) {
    const float p = a.lo * b.lo, q = a.lo * b.hi, r = a.hi * b.lo, s = a.hi * b.hi;
    return fin<K>(min3(p, q, fminf(r, s)), max3(p, q, fmaxf(r, s)), perr<K>(a, b));
}
// b >= 0 in the reference (its structure), both >= 0, b <= 0
template <int K> APO_CERT X<K> mul_nn(X<K> a, X<K> b) {
    return fin<K>(fminf(a.lo * b.lo, a.lo * b.hi), fmaxf(a.hi * b.lo, a.hi * b.hi), perr<K>(a, b));
}
template <int K> APO_CERT X<K> mul_pp(X<K> a, X<K> b) { return fin<K>(a.lo * b.lo, a.hi * b.hi, perr<K>(a, b)); }
// times a number (S = 1: known to be >= 0)
template <int S, int K> APO_CERT X<K> muls(X<K> a, Sc<K> s) {
    const float p = a.lo * s.v, q = a.hi * s.v;
    if (S > 0) return fin<K>(p, q, perr<K>(a, s));
    return fin<K>(fminf(p, q), fmaxf(p, q), perr<K>(a, s));
}
// (ends of a s) + c for numbers s, c: the sum's rounding and the product's
template <int K> APO_CERT X<K> axpc(X<K> a, Sc<K> s, Sc<K> c) {
    const float p = fmaf(a.lo, s.v, c.v), q = fmaf(a.hi, s.v, c.v);
    return fin<K>(fminf(p, q), fmaxf(p, q), K ? perr<K>(a, s) + rnd<K>(M(a) * M(s)) + c.e : 0.f);
}
template <int K> APO_CERT X<K> sqr(X<K> a) {
    const float m = fmaxf(-a.lo, a.hi), n = max3(0.f, a.lo, -a.hi);
    return fin<K>(n * n, m * m, K ? 2.f * M(a) * a.e + kTiny : 0.f);
}
template <int K> APO_CERT X<K> clamp1(X<K> a) {
    X<K> r;
    r.lo = fmaxf(a.lo, -1.f);
    r.hi = fminf(a.hi, 1.f);
    r.e = a.e;
    return r;
}
// an error that holds only under a condition (else nothing is decided)
APO_CERT float when(bool ok, float e) { return ok ? e : INFINITY; }
// 1 / b, b > 0
template <int K> APO_CERT X<K> recip(X<K> b) {
    X<K> r;
    r.lo = rcp_a(b.hi);
    r.hi = rcp_a(b.lo);
    r.e = 0.f;
    if (K) {
        const float x = b.lo - 2.f * b.e;                 // smallest divisor on either side
        const float h = 1.001f / x;
        r.e = when(x > 0.f, b.e * h * h + Unit<K>::ua * h + kTiny);
    }
    return r;
}
// sqrt(x), x > 0
template <int K> APO_CERT X<K> sqrtx(X<K> a) {
    X<K> r;
    r.lo = sqrt_a(a.lo);
    r.hi = sqrt_a(a.hi);
    r.e = 0.f;
    if (K) {
        const float x = a.lo - 2.f * a.e;
        r.e = when(x > 0.f, 0.5005f * a.e / sqrt_a(x) + Unit<K>::ua * 1.001f * sqrt_a(M(a)) + kTiny);
    }
    return r;
}

// atan as in the program: two half-angle reductions, the series through x^15, the remainder,
// times 4.  With M(x) <= 1/2 after the reductions (y <= 1/4) every Horner value is positive, so
// its lower end goes with y.hi and its upper end with y.lo; the error of the series value is
// at most sum_j y^j (h_{j+1} e_y + 2.25 U c_j) <= 0.4 e_y + 2.6 U with c_j = 1 / (2 j + 1).
template <int K> APO_CERT X<K> atanx(X<K> x) {
#pragma unroll
    for (int i = 0; i < 2; i++) x = mul_nn(x, recip(add1(sqrtx(add1(sqr(x), 1.f)), 1.f)));
    const X<K> y = sqr(x);
    X<K> h;
    h.lo = h.hi = (float)(1.0 / 15);
    const float c[7] = {1.f, (float)(1.0 / 3), (float)(1.0 / 5), (float)(1.0 / 7), (float)(1.0 / 9), (float)(1.0 / 11),
                        (float)(1.0 / 13)};
#pragma unroll
    for (int j = 6; j >= 0; j--) {
        const float lo = fmaf(-h.hi, y.hi, c[j]), hi = fmaf(-h.lo, y.lo, c[j]);
        h.lo = lo;
        h.hi = hi;
    }
    h.e = K ? when(M(x) <= 0.5f && y.e <= 1e-3f, 0.4f * y.e + 2.6f * Unit<K>::u) : 0.f;
    const X<K> a = mul_nn(x, h);
    // remainder |x|^17 / 17: derivative |x|^16 <= 2^-16, value below 4.5e-7 with 25 roundings
    const float m = fmaxf(-x.lo, x.hi), m2 = m * m, m4 = m2 * m2, m8 = m4 * m4;
    const float rem = m8 * m8 * (m * (float)(1.0 / 17));
    return scl(fin<K>(a.lo - rem, a.hi + rem, K ? a.e + 2e-5f * x.e + 6e-12f : 0.f), 4.f);
}

// sin and cos as in the program: series and remainder for |d| <= 1, else [-1, 1].  A box whose d may
// pass 1 has cells on either side and no bound; a single cell (own) is certainly beyond where its
// magnitude is by more than the error.
template <int K> APO_CERT void sincosx(X<K> d, X<K> &s, X<K> &c, bool own) {
    if (K && own && mag2(d.lo, d.hi) - 2.f * d.e > 1.f) {
        s.lo = c.lo = -1.f;
        s.hi = c.hi = 1.f;
        s.e = c.e = 0.f;
        return;
    }
    const X<K> y = sqr(d);
    const float c6 = (float)(1.0 / 6);
    X<K> S;
    S.lo = fmaf(-y.hi, c6, 1.f);
    S.hi = fmaf(-y.lo, c6, 1.f);
    S.e = K ? 0.17f * y.e + 2.5f * Unit<K>::u : 0.f;
    const float m = fmaxf(-d.lo, d.hi), m2 = m * m, m4 = m2 * m2;
    const float r5 = m4 * m * (float)(1.0 / 120), r4 = m4 * (float)(1.0 / 24);
    float e5 = 0.f, e4 = 0.f;
    const float Md = M(d), Md2 = Md * Md;
    if (K) {   // d/dm of the remainders, and 8 roundings of their value
        e5 = Md2 * Md2 * (d.e * 0.042f + 8.f * Unit<K>::u * 0.0084f) + kTiny;
        e4 = Md2 * Md * (d.e * 0.167f + 8.f * Unit<K>::u * 0.042f) + kTiny;
        e5 = when(Md <= 1.f, e5);
    }
    const X<K> ds = mul_nn(d, S);
    s = clamp1(fin<K>(ds.lo - r5, ds.hi + r5, K ? ds.e + e5 : 0.f));
    const float clo = fmaf(-0.5f, y.hi, 1.f), chi = fmaf(-0.5f, y.lo, 1.f);
    c = clamp1(fin<K>(clo - r4, chi + r4, K ? 0.5f * y.e + rnd<K>(1.f) + e4 : 0.f));
}

template <int K> struct CellX { X<K> D, S0, C0, W, Z, L; };           // mirrored, W > 0
template <int K> struct HitX { Sc<K> x0, y0, sph, cph, t, spt, cpt, t2; X<K> d; };   // mirrored with its cell

// The tan(lambda)-free part.  Interval products and sums are associative and products with a
// number distribute over sums, so factors free of tan(lambda) are gathered here (the reference
// multiplies them in one by one): the end points are the same real numbers, and the roundings
// of either order stay within the bound.  wt: the direction condition's quantity;
// A1 = -psi sin(Phi^Ax) / N and B1 = -(d rho) cos(Phi^Ax) / N (times L t: the even / odd parts of
// Phi1 t); A2 = inner t^2 / (2 N^2) (times L^2); B2 = d rho t^2 / (2 N^2); pc2 = 2 psi cos 2Phi^Ax.
template <int K> struct PreX {
    X<K> wt, G0, psi, N, sPA, cPA, rsA, rcA, sin2, A1, B1, A2, B2, pc2;
    Sc<K> tt;   // t t
};

template <int K> APO_CERT PreX<K> prefix(const CellX<K> &c, const HitX<K> &h) {
    PreX<K> p;
    const X<K> Xw = axpc(c.Z, h.spt, h.x0);
    const X<K> Yw = axpc(c.Z, neg(h.cpt), h.y0);
    const X<K> wt = add(mul(Xw, c.C0), mul(Yw, c.S0));
    const X<K> wn = sub(mul(Yw, c.C0), mul(Xw, c.S0));
    p.wt = wt;
    const X<K> V = sub(wn, c.D);
    const X<K> Xt = mul_nn(wt, c.W);
    const X<K> Xn = add1(mul_nn(V, c.W), -1.f);
    p.N = sqrtx(add(sqr(Xt), sqr(Xn)));
    p.G0 = add(mul_pp(c.W, sqr(wt)), mul(V, add1(Xn, -1.f)));
    p.psi = scl(atanx(mul_nn(Xt, recip(sub(p.N, Xn)))), 2.f);
    const X<K> E1 = add(muls<0>(c.C0, h.cph), muls<0>(c.S0, h.sph));
    const X<K> E2 = sub(muls<0>(c.C0, h.sph), muls<0>(c.S0, h.cph));
    p.rsA = add(mul(Xt, E1), mul(Xn, E2));
    p.rcA = sub(mul(Xt, E2), mul(Xn, E1));
    const X<K> Ninv = recip(p.N);
    p.sPA = clamp1(mul_nn(p.rsA, Ninv));
    p.cPA = clamp1(mul_nn(p.rcA, Ninv));
    const X<K> cos2 = clamp1(sub(sqr(p.cPA), sqr(p.sPA)));
    p.sin2 = clamp1(scl(mul(p.sPA, p.cPA), 2.f));
    const X<K> dW = mul_pp(h.d, c.W);
    const X<K> Nt2 = muls<1>(scl(mul_pp(Ninv, Ninv), 0.5f), h.t2);
    p.A1 = neg(mul_nn(mul(p.psi, p.sPA), Ninv));
    p.B1 = neg(mul_nn(mul_nn(p.cPA, dW), Ninv));
    p.A2 = mul_nn(sub(add(mul_nn(p.psi, rsub1(1.f, cos2)), mul_nn(p.sin2, sqr(p.psi))),
                      mul_nn(p.sin2, mul_pp(dW, dW))), Nt2);
    p.B2 = mul_pp(dW, Nt2);
    p.pc2 = scl(mul(p.psi, cos2), 2.f);
    p.tt = smul(h.t, h.t);
    return p;
}

// The rest for one tan(lambda) interval L (R = 1 / W): G of both drift signs,
// G = G0 - a2 + a5 + 2 (z t rcA -+ L Q t rsA) + W (z t)^2 -+ 2 Q with z = z^St - z_ref.
// One copy for every sign of L and t: copies with the signs known take two minima less in six
// products, but then a voting loop outgrows the instruction cache (level 0 of 1024 events, FP32:
// 41.3 ms with three copies).
template <int K>
APO_CERT void tail(const PreX<K> &p, X<K> L, const HitX<K> &h, X<K> R, X<K> W, X<K> &Gp, X<K> &Gm, bool own = false) {
    const X<K> L2 = sqr(L), Lt = muls<0>(L, h.t);
    const X<K> de = add(mul(p.A1, Lt), mul_nn(p.A2, L2));
    const X<K> NL = add(p.N, mul_pp(L2, add1(p.N, 1.f)));
    const X<K> dod = add(mul(p.B1, Lt), mul_nn(add(mul_nn(p.pc2, L2), mul_nn(p.sin2, NL)), p.B2));
    const X<K> dP = add(de, dod), dM = sub(de, dod);
    X<K> dh, sd, cd;
    dh.lo = fminf(dP.lo, dM.lo);
    dh.hi = fmaxf(dP.hi, dM.hi);
    dh.e = K ? dP.e + (dM.e - dM.e) + fmaxf(dM.e - dP.e, 0.f) : 0.f;   // the larger; NaN / inf kept
    sincosx(dh, sd, cd, own);
    // cos(delta) > 0 for |delta| <= 1, as where only bare end points are evaluated
    const X<K> sP = clamp1(add(K ? mul(p.sPA, cd) : mul_nn(p.sPA, cd), mul(p.cPA, sd)));
    const X<K> cP = clamp1(sub(K ? mul(p.cPA, cd) : mul_nn(p.cPA, cd), mul(p.sPA, sd)));
    const X<K> u2 = add(add(add1(mul(sP, scl(Lt, 2.f)), 1.f), muls<1>(L2, h.t2)), muls<1>(sqr(cP), h.t2));
    const X<K> Q = mul_pp(h.d, recip(sqrtx(u2)));
    const X<K> cz = mul_nn(cP, muls<1>(Q, p.tt));                      // t (cos Phi) t q
    const X<K> LQt = mul_nn(Lt, Q), LQr = mul(p.rsA, LQt);
    const X<K> a2 = mul_pp(W, mul_pp(Q, Q)), a5 = mul_pp(W, sqr(LQt));
    const X<K> base = add(sub(p.G0, a2), a5);
    const X<K> Q2 = scl(Q, 2.f);
#pragma unroll
    for (int sg = 0; sg < 2; sg++) {
        const X<K> zL = mul(mul_nn(add(p.psi, sg ? dM : dP), R), Lt);
        const X<K> zt = sg ? add(zL, cz) : sub(zL, cz);
        const X<K> zr = mul(zt, p.rcA);
        const X<K> Y = scl(sg ? add(zr, LQr) : sub(zr, LQr), 2.f);
        const X<K> a4 = mul_pp(W, sqr(zt));
        X<K> G = add(add(sg ? add(base, Q2) : sub(base, Q2), Y), a4);
        // the FP32 reference rounds sums in another order: four partial sums, each at most
        // the sum of all terms' magnitudes
        if (K == 32) G.e += 4.f * rnd<K>(M(p.G0) + M(a2) + M(a5) + M(Q2) + M(Y) + M(a4));
        if (sg) Gm = G;
        else Gp = G;
    }
}

enum : int { kNo = 0, kYes = 1, kUnknown = 2 };

template <int K> APO_CERT int decide(X<K> Gp, X<K> Gm, float e) {
    if ((Gp.lo <= -e && Gp.hi >= e) || (Gm.lo <= -e && Gm.hi >= e)) return kYes;
    return ((Gp.lo > e || Gp.hi < -e) && (Gm.lo > e || Gm.hi < -e)) ? kNo : kUnknown;
}

// One evaluation: the cell's G and direction quantity.  own: a single cell, not a box of cells whose
// bound is wanted
template <int K> struct Eval { X<K> Gp, Gm, wt; };
template <int K> APO_CERT Eval<K> eval(const CellX<K> &c, const HitX<K> &h, bool own = false) {
    Eval<K> r;
    const PreX<K> p = prefix(c, h);
    tail(p, c.L, h, recip(c.W), c.W, r.Gp, r.Gm, own);
    r.wt = p.wt;
    return r;
}
// The one error the children use for all three tests; NaN when nothing can be decided.
template <int K> APO_CERT float bound(const Eval<K> &r) {
    return (r.Gp.e < 1e30f && r.Gm.e < 1e30f && r.wt.e < 1e30f) ? fmaxf(fmaxf(r.Gp.e, r.Gm.e), r.wt.e) : NAN;
}
// The vote of a whole evaluation with error bound e (its own cell's or a parent's)
template <int K> APO_CERT int verdict(const Eval<K> &r, bool outgoing, float e) {
    if (outgoing) {
        if (r.wt.hi < -e) return kNo;
        if (!(r.wt.hi >= e)) return kUnknown;
    }
    return decide(r.Gp, r.Gm, e);
}

}  // namespace cert
}  // namespace apo
