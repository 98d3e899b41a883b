// Point programs in plain FP32 with certified errors (certified.cuh): the same program text runs on
// Pt, one FP32 number, or on X<64>, a range of numbers with the error that holds for each of them.
//
// The reference of a point program is a number as well, not an interval, so any algebraically
// equal form may be evaluated: the FP64 program's own distance from the real value has the same
// bound with 2^-52 for 2^-24, far inside the margin, where its series are followed term by term or
// are long enough to count as exact.
#pragma once
#include "certified.cuh"

namespace apo {
namespace cert {

struct Pt { float v; };
APO_CERT Pt add(Pt a, Pt b) { return {a.v + b.v}; }
APO_CERT Pt sub(Pt a, Pt b) { return {a.v - b.v}; }
APO_CERT Pt mul(Pt a, Pt b) { return {a.v * b.v}; }
APO_CERT Pt neg(Pt a) { return {-a.v}; }
APO_CERT Pt scl(Pt a, float s) { return {a.v * s}; }
APO_CERT Pt add1(Pt a, float c) { return {a.v + c}; }
APO_CERT Pt sqr(Pt a) { return {a.v * a.v}; }
APO_CERT Pt recip(Pt a) { return {rcp_a(a.v)}; }
APO_CERT Pt sqrtx(Pt a) { return {sqrt_a(a.v)}; }
APO_CERT Pt rsqrtx(Pt a) { return {rsqrt_a(a.v)}; }
template <int K> APO_CERT X<K> rsqrtx(X<K> a) { return recip(sqrtx(a)); }   // two units for rsqrt's one
template <typename N> APO_CERT N numf(float v);            // from a hit's value rounded down
template <> APO_CERT Pt numf<Pt>(float v) { return {v}; }
template <> APO_CERT X<64> numf<X<64>>(float v) { return point(sc<64>(v)); }
APO_CERT X<0> ivp(Pt a) { X<0> r; r.lo = r.hi = a.v; r.e = 0.f; return r; }
template <int K> APO_CERT X<K> ivp(X<K> a) { return a; }

// sin d and cos d by the FP64 program's polynomials (through d^9 / d^10).  Error for |d| <= 1.5
// (y <= 2.25): slopes in y below 0.2 and 0.55, at most 9 roundings of values below 2.2.
APO_CERT void sincos4(Pt d, Pt &s, Pt &c) {
    const float y = d.v * d.v;
    float p = fmaf(y, 1.f / 362880, -1.f / 5040);
    p = fmaf(y, p, 1.f / 120);
    p = fmaf(y, p, -1.f / 6);
    s.v = d.v * fmaf(y, p, 1.f);
    float q = fmaf(y, -1.f / 3628800, 1.f / 40320);
    q = fmaf(y, q, -1.f / 720);
    q = fmaf(y, q, 1.f / 24);
    q = fmaf(y, q, -0.5f);
    c.v = fmaf(y, q, 1.f);
}
template <int K> APO_CERT void sincos4(X<K> d, X<K> &s, X<K> &c) {
    const X<K> y = sqr(d);
    X<K> S;   // 1 - y/6 <= S <= 1 - y/6 + y^2/120, and for cos likewise
    S.lo = 1.f - y.hi * (float)(1.0 / 6);
    S.hi = 1.f - y.lo * (float)(1.0 / 6) + y.hi * y.hi * (float)(1.0 / 120);
    S.e = when(M(d) <= 1.5f, 0.2f * y.e + 20.f * Unit<K>::u);
    s = mul(d, S);
    c.lo = 1.f - y.hi * 0.5f;
    c.hi = 1.f - y.lo * 0.5f + y.hi * y.hi * (float)(1.0 / 24);
    c.e = when(M(d) <= 1.5f, 0.55f * y.e + 20.f * Unit<K>::u);
}

}  // namespace cert
}  // namespace apo
