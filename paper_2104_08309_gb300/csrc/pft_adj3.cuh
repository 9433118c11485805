// pft_adj3.cuh -- the 3D pair adjoint of the vertex gradients, two faces per thread in paired FP32
// instructions.
//
// The face term J = -s exp(i mu) Z of a (Q, face) pair (pft_pairs.cuh), weight gt, differentiated in
// reverse mode into the 12 record fields.  Bound: the FP32 lanes (65 / 74 / 83 / 115 operations a pair in
// the four series forms below), two of them per issue slot.  A thread holds faces 2t and 2t + 1 of its
// block, field by field as float2, and takes one Q point at a time, its fields broadcast (doubling them in
// shared memory, 48 B a record, ran 2-3 % slower: 5.82 against 5.69 ms on 81,920 faces x 32,768 Q; two Q
// points of one face per thread took 168-182 registers and ran slower than scalar code: 11.7 against 9.3
// ms).  The compensated sums, touched once per tile, live in shared memory.  Where a warp's phases need the edge sum, a
// thread's faces take it in scalar code, one after the other.  Blocks of few faces hold one a thread (pair_span).
#pragma once

#include "pft_pairs.cuh"

namespace pft {

// Q record of the adjoints: Q in FP32, the weight gt and -Im gt.
struct __align__(16) QRec {
  float qx, qy, qz, gr, gi, ngi, pad0, pad1;
};
static_assert(sizeof(QRec) == 32, "Q record is two float4");

// Z = zr + i zi (zi = G_re, zr = -G_im = t r) and its derivatives in P and in t = a0 a1 (a0 + a1) = -T, for the
// series k <= 7 (FORM 0), k <= 9 (1), k <= 11 (2) and k <= 17 (3): the coefficients of face_series,
// face_series_k9, face_series_long and face_series_xlong.
template <int FORM, class V>
__device__ __forceinline__ void series_grad(V t, V P, V& zr, V& zi, V& zr_P, V& zr_t, V& zi_P, V& zi_t) {
  const V t2 = vmul(t, t);
  if constexpr (FORM == 0) {
    zi = vfma(P, vs<V>(-2.48015873e-5f), vs<V>(1.38888889e-3f));
    zi = vfma(P, zi, vs<V>(-4.16666667e-2f));
    zi = vfma(P, zi, vs<V>(0.5f));
    zi = vfma(t2, vs<V>(-2.48015873e-5f), zi);
    zi_P = vfma(P, vfma(P, vs<V>(-7.44047619e-5f), vs<V>(2.77777778e-3f)), vs<V>(-4.16666667e-2f));
    zi_t = vmul(t, vs<V>(-4.96031746e-5f));
    const V r = vfma(P, vfma(P, vs<V>(-8.26719577e-6f), vs<V>(3.96825397e-4f)), vs<V>(-8.33333333e-3f));
    zr = vmul(t, r);
    zr_P = vmul(t, vfma(P, vs<V>(-1.653439154e-5f), vs<V>(3.96825397e-4f)));
    zr_t = r;
  } else if constexpr (FORM == 1) {
    V A0 = vfma(P, vs<V>(2.755731922e-07f), vs<V>(-2.480158730e-05f));
    A0 = vfma(P, A0, vs<V>(1.388888889e-03f));
    A0 = vfma(P, A0, vs<V>(-4.166666667e-02f));
    A0 = vfma(P, A0, vs<V>(0.5f));
    const V A2 = vfma(P, vs<V>(8.267195767e-07f), vs<V>(-2.480158730e-05f));
    zi = vfma(t2, A2, A0);
    V dA = vfma(P, vs<V>(1.1022927688e-06f), vs<V>(-7.44047619e-05f));
    dA = vfma(P, dA, vs<V>(2.777777778e-03f));
    dA = vfma(P, dA, vs<V>(-4.166666667e-02f));
    zi_P = vfma(t2, vs<V>(8.267195767e-07f), dA);
    zi_t = vmul(vadd(t, t), A2);
    V D1 = vfma(P, vs<V>(1.002084335e-07f), vs<V>(-8.267195767e-06f));
    D1 = vfma(P, D1, vs<V>(3.968253968e-04f));
    D1 = vfma(P, D1, vs<V>(-8.333333333e-03f));
    const V r = vfma(t2, vs<V>(2.505210839e-08f), D1);
    zr = vmul(t, r);
    V dD = vfma(P, vs<V>(3.006253005e-07f), vs<V>(-1.6534391534e-05f));
    dD = vfma(P, dD, vs<V>(3.968253968e-04f));
    zr_P = vmul(t, dD);
    zr_t = vfma(t2, vs<V>(5.010421678e-08f), r);
  } else if constexpr (FORM == 2) {
    V A = vfma(P, vs<V>(-2.087675588e-9f), vs<V>(2.75573192e-7f));
    A = vfma(P, A, vs<V>(-2.48015873e-5f));
    A = vfma(P, A, vs<V>(1.38888889e-3f));
    A = vfma(P, A, vs<V>(-4.16666667e-2f));
    A = vfma(P, A, vs<V>(0.5f));
    V B = vfma(P, vs<V>(-1.252605397e-8f), vs<V>(8.26719577e-7f));
    B = vfma(P, B, vs<V>(-2.48015873e-5f));
    zi = vfma(t2, B, A);
    V dA = vfma(P, vs<V>(-1.043837794e-8f), vs<V>(1.102292768e-6f));
    dA = vfma(P, dA, vs<V>(-7.44047619e-5f));
    dA = vfma(P, dA, vs<V>(2.77777778e-3f));
    dA = vfma(P, dA, vs<V>(-4.16666667e-2f));
    const V dB = vfma(P, vs<V>(-2.505210794e-8f), vs<V>(8.26719577e-7f));
    zi_P = vfma(t2, dB, dA);
    zi_t = vmul(vadd(t, t), B);
    V D = vfma(P, vs<V>(-8.029522047e-10f), vs<V>(1.002084318e-7f));
    D = vfma(P, D, vs<V>(-8.26719577e-6f));
    D = vfma(P, D, vs<V>(3.96825397e-4f));
    D = vfma(P, D, vs<V>(-8.33333333e-3f));
    const V E = vfma(P, vs<V>(-6.423617749e-10f), vs<V>(2.505210794e-8f));
    const V r = vfma(t2, E, D);
    zr = vmul(t, r);
    V dD = vfma(P, vs<V>(-3.211808819e-9f), vs<V>(3.006252954e-7f));
    dD = vfma(P, dD, vs<V>(-1.653439154e-5f));
    dD = vfma(P, dD, vs<V>(3.96825397e-4f));
    zr_P = vmul(t, vfma(t2, vs<V>(-6.423617749e-10f), dD));
    zr_t = vfma(vadd(t2, t2), E, r);
  } else {
    // the derivative in P of a polynomial that Horner evaluates comes along: d = d P + v before v = v P + c
    auto row = [&](V& v, V& d, float c) {
      d = vfma(P, d, v);
      v = vfma(P, v, vs<V>(c));
    };
    const V tt = vadd(t2, t2);
    {   // G_re = A0 + t2 (A2 + t2 A4)
      V v = vfma(P, vs<V>(2.342881045e-15f), vs<V>(-2.389738666e-13f)), d = vs<V>(2.342881045e-15f);   // A4
      row(v, d, 1.147074560e-11f);
      V w = vfma(P, vs<V>(3.280033463e-15f), vs<V>(-7.169215999e-13f)), e = vs<V>(3.280033463e-15f);   // A2
      row(w, e, 1.147074560e-10f);
      row(w, e, -1.252605419e-08f);
      row(w, e, 8.267195767e-07f);
      row(w, e, -2.480158730e-05f);
      const V A24 = vfma(t2, v, w), dA24 = vfma(t2, d, e);
      zi_t = vmul(vadd(t, t), vfma(t2, v, A24));              // 2 t (A2 + 2 t2 A4)
      V u = vfma(P, vs<V>(1.561920697e-16f), vs<V>(-4.779477332e-14f)), g = vs<V>(1.561920697e-16f);   // A0
      row(u, g, 1.147074560e-11f);
      row(u, g, -2.087675699e-09f);
      row(u, g, 2.755731922e-07f);
      row(u, g, -2.480158730e-05f);
      row(u, g, 1.388888889e-03f);
      row(u, g, -4.166666667e-02f);
      row(u, g, 0.5f);
      zi = vfma(t2, A24, u);
      zi_P = vfma(t2, dA24, g);
    }
    {   // r = D1 + t2 (D3 + t2 D5), zr = t r
      const V v = vfma(P, vs<V>(4.932381148e-17f), vs<V>(-2.811457254e-15f));   // D5
      V w = vfma(P, vs<V>(2.877222336e-16f), vs<V>(-5.622914509e-14f)), e = vs<V>(2.877222336e-16f);   // D3
      row(w, e, 7.647163732e-12f);
      row(w, e, -6.423617535e-10f);
      row(w, e, 2.505210839e-08f);
      const V D35 = vfma(t2, v, w), dD35 = vfma(t2, vs<V>(4.932381148e-17f), e);
      const V twice = vfma(t2, v, D35);                        // D3 + 2 t2 D5
      V u = vfma(P, vs<V>(6.576508197e-17f), vs<V>(-1.968020078e-14f)), g = vs<V>(6.576508197e-17f);   // D1
      row(u, g, 4.588298239e-12f);
      row(u, g, -8.029521918e-10f);
      row(u, g, 1.002084335e-07f);
      row(u, g, -8.267195767e-06f);
      row(u, g, 3.968253968e-04f);
      row(u, g, -8.333333333e-03f);
      const V r = vfma(t2, D35, u);
      zr = vmul(t, r);
      zr_P = vmul(t, vfma(t2, dD35, g));
      zr_t = vfma(tt, twice, r);                               // d/dt (t r) = r + 2 t2 (D3 + 2 t2 D5)
    }
  }
}

// Adds the record adjoints of one Q and the thread's faces F (12 fields, Face32's order) to a.  The
// adjoints of q0, q1 and N are kept negated there (adj_sign): the products come out that way.
__device__ __forceinline__ constexpr float adj_sign(int k) { return k < 3 ? 1.f : -1.f; }

template <int FORM, class V>
__device__ __forceinline__ void series_adj(const QRec& Q, V mu, V a0, V a1, V s1, V m, V s, V (&a)[12]) {
  const V P = vfma(a0, a0, m), t = vmul(a0, m);   // m = a1 (a0 + a1)
  V zr, zi, zr_P, zr_t, zi_P, zi_t;
  series_grad<FORM>(t, P, zr, zi, zr_P, zr_t, zi_P, zi_t);
  V sm, cm;
  sincos_v(mu, sm, cm);
  const V p = vfma(vs<V>(Q.gr), cm, vmul(vs<V>(Q.gi), sm));     // conj(gt) exp(i mu) = p + i q
  const V q = vfma(vs<V>(Q.gr), sm, vmul(vs<V>(Q.ngi), cm));
  const V nq = vmul(q, vs<V>(-1.0f));
  const V nsb = vfma(p, zr, vmul(nq, zi));        // -dc/ds = Re((p + i q) Z), c = Re(conj(gt) J)
  const V mub = vmul(s, vfma(p, zi, vmul(q, zr)));   // dc/dmu = s Im((p + i q) Z)
  const V ps = vmul(s, p), ns = vmul(s, nq);      // -dc = ps dzr + ns dzi
  const V nP = vfma(ps, zr_P, vmul(ns, zi_P)), nT = vfma(ps, zr_t, vmul(ns, zi_t));
  // dP = e0 da0 + e1 da1, dt = a1 e0 da0 + a0 e1 da1, e0 = 2 a0 + a1, e1 = 2 a1 + a0
  const V n0 = vmul(vadd(a0, s1), vfma(nT, a1, nP)), n1 = vmul(vadd(a1, s1), vfma(nT, a0, nP));
  const V qx = vs<V>(Q.qx), qy = vs<V>(Q.qy), qz = vs<V>(Q.qz);
  a[0] = vfma(mub, qx, a[0]);
  a[1] = vfma(mub, qy, a[1]);
  a[2] = vfma(mub, qz, a[2]);
  a[3] = vfma(n0, qx, a[3]);
  a[4] = vfma(n0, qy, a[4]);
  a[5] = vfma(n0, qz, a[5]);
  a[6] = vfma(n1, qx, a[6]);
  a[7] = vfma(n1, qy, a[7]);
  a[8] = vfma(n1, qz, a[8]);
  a[9] = vfma(nsb, qx, a[9]);
  a[10] = vfma(nsb, qy, a[10]);
  a[11] = vfma(nsb, qz, a[11]);
}

}  // namespace pft
