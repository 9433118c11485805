// pft_f64.cuh -- per-pair arithmetic of the FP64 comparison path.
//
// Bound: the FP64 pipe (2 fused multiply-adds a clock and SM on GB300, 1/64 of the FP32 lanes), so a
// pair costs the FP64 instructions it issues; table loads, integer work and the warp votes are hidden
// behind them.  Library sincos (about 40 FP64 operations for both), a 17-term series for every face
// and sin(u)/u with a division came to 210 operations per (Q, face) pair; the forms below take about
// 65 in the series and 150 in the edge sum, and 40 per (Q, segment) pair instead of 71.
#pragma once

#include "pft_kernels.cuh"

namespace pft {

// sin and cos of 2 pi k / 256, k = 0 .. 255, each correctly rounded; the quarter wave is written out.
struct TrigTable { double2 v[256]; };   // (sin, cos)
constexpr double kQuarterSin[65] = {
    0.0, 0.024541228522912288, 0.049067674327418015, 0.07356456359966743,
    0.0980171403295606, 0.1224106751992162, 0.14673047445536175, 0.17096188876030122,
    0.19509032201612828, 0.2191012401568698, 0.2429801799032639, 0.26671275747489837,
    0.2902846772544624, 0.31368174039889146, 0.33688985339222005, 0.35989503653498817,
    0.3826834323650898, 0.40524131400498986, 0.4275550934302821, 0.4496113296546066,
    0.47139673682599764, 0.49289819222978404, 0.5141027441932218, 0.5349976198870973,
    0.5555702330196022, 0.5758081914178453, 0.5956993044924334, 0.6152315905806268,
    0.6343932841636455, 0.6531728429537768, 0.6715589548470184, 0.6895405447370669,
    0.7071067811865476, 0.7242470829514669, 0.7409511253549591, 0.7572088465064846,
    0.773010453362737, 0.7883464276266062, 0.8032075314806449, 0.8175848131515837,
    0.8314696123025452, 0.8448535652497071, 0.8577286100002721, 0.8700869911087115,
    0.881921264348355, 0.8932243011955153, 0.9039892931234433, 0.9142097557035307,
    0.9238795325112867, 0.9329927988347388, 0.9415440651830208, 0.9495281805930367,
    0.9569403357322088, 0.9637760657954398, 0.970031253194544, 0.9757021300385286,
    0.9807852804032304, 0.9852776423889412, 0.989176509964781, 0.99247953459871,
    0.9951847266721969, 0.9972904566786902, 0.9987954562051724, 0.9996988186962042,
    1.0};
constexpr double sin256(int k) {   // sin(2 pi k / 256), 0 <= k
  const int m = k & 255, q = m & 127, s = q <= 64 ? q : 128 - q;
  return m < 128 ? kQuarterSin[s] : -kQuarterSin[s];
}
constexpr TrigTable make_trig() {
  TrigTable t{};
  for (int k = 0; k < 256; ++k) {
    t.v[k].x = sin256(k);
    t.v[k].y = sin256(k + 64);
  }
  return t;
}
static __device__ const TrigTable kTrig = make_trig();

// sin and cos of x: x = k 2 pi/256 + r, |r| <= pi/256, with 2 pi/256 as a sum of two doubles (Cody and
// Waite), the table for k and Taylor polynomials for r (left out: below 1e-17).  Table and last
// rounding: about 1 ulp of 1.  |x| >= 1e9, infinities and NaN take the library's.
constexpr double kStep = 0.02454369260617026, kStepLo = 9.567553118338697e-19, kInvStep = 40.74366543152521;
constexpr double kRound = 6755399441055744.0;   // 1.5 * 2^52: adding it rounds to an integer
struct Reduced { double r, r2, sn, cs; };       // remainder, its square, table entry
__device__ __forceinline__ bool trig_range(double x) {   // |x| < 1e9, on the integer pipe
  return (__double2hiint(x) & 0x7fffffff) < 0x41cdcd65;
}
__device__ __forceinline__ Reduced trig_reduce(double x) {
  const double t = fma(x, kInvStep, kRound), k = t - kRound;
  const double2 e = kTrig.v[__double2loint(t) & 255];
  const double r = fma(-k, kStepLo, fma(-k, kStep, x));
  return Reduced{r, r * r, e.x, e.y};
}
__device__ __forceinline__ double trig_sin_r(const Reduced& a) {   // sin r
  return fma(a.r * a.r2, fma(a.r2, 1.0 / 120.0, -1.0 / 6.0), a.r);
}
__device__ __forceinline__ double trig_cosm1_r(const Reduced& a) {   // cos r - 1
  return a.r2 * fma(a.r2, fma(a.r2, -1.0 / 720.0, 1.0 / 24.0), -0.5);
}
__device__ __forceinline__ void sincos64(double x, double& sn, double& cs) {
  if (trig_range(x)) {
    const Reduced a = trig_reduce(x);
    const double s = trig_sin_r(a), c = trig_cosm1_r(a);
    sn = fma(a.cs, s, fma(a.sn, c, a.sn));
    cs = fma(-a.sn, s, fma(a.cs, c, a.cs));
  } else {
    sincos(x, &sn, &cs);
  }
}
__device__ __forceinline__ double sin64(double x) {
  if (trig_range(x)) {
    const Reduced a = trig_reduce(x);
    return fma(a.cs, trig_sin_r(a), fma(a.sn, trig_cosm1_r(a), a.sn));
  }
  return sin(x);
}

constexpr double fact(int n) { return n < 2 ? 1.0 : n * fact(n - 1); }
// Coefficients are forced to compile time (a recursive function called in an unrolled loop is not).
template <int N> struct SincCoef {   // of u^(2N)
  static constexpr double v = (N & 1) ? -1.0 / fact(2 * N + 1) : 1.0 / fact(2 * N + 1);
};
template <int N>
__device__ __forceinline__ double sinc_horner(double p, double v) {   // down to N = 0
  p = fma(p, v, SincCoef<N>::v);
  if constexpr (N > 0) return sinc_horner<N - 1>(p, v);
  else return p;
}

// sinc(u) = sin(u)/u for N values: the Taylor polynomial through u^22 where u^2 <= 4 (left out: 1e-18),
// the quotient beyond, evaluated only in warps where some lane needs it (warp-converged callers).
template <int N>
__device__ __forceinline__ void sinc64(const double (&u)[N], double (&S)[N]) {
  bool big = false;
#pragma unroll
  for (int l = 0; l < N; ++l) {
    const double v = u[l] * u[l];
    S[l] = sinc_horner<10>(SincCoef<11>::v, v);
    big = big || (__double2hiint(u[l]) & 0x7fffffff) >= 0x40000000;   // |u| >= 2 (or NaN)
  }
  if (__any_sync(0xffffffffu, big)) {
#pragma unroll
    for (int l = 0; l < N; ++l)
      if ((__double2hiint(u[l]) & 0x7fffffff) >= 0x40000000) S[l] = sin64(u[l]) / u[l];
  }
}

// 2D: the term -i w sinc(u) exp(i ph) of Eq. 6 (half the cross product; see pft_pairs.cuh).
__device__ __forceinline__ void seg_pair64(double qx, double qy, const Seg64& s, double& re, double& im) {
  const double ph = fma(qx, s.mx, qy * s.my);
  const double u[1] = {fma(qx, s.hx, qy * s.hy)};
  const double w = fma(qx, s.hy, -qy * s.hx);
  double S[1], sn, cs;
  sinc64(u, S);
  sincos64(ph, sn, cs);
  const double ws = w * S[0];
  re = fma(ws, sn, re);
  im = fma(-ws, cs, im);
}

// G from its series (pft_pairs.cuh), terms k <= K: the coefficient of P^i T^j is (-1)^(k/2)
// C(i+j, i)/(k+2)!, k = 2i + 3j; Horner in P for every power of T, then in T^2.
constexpr double series_coef(int i, int j) {
  const double c = fact(i + j) / (fact(i) * fact(j)) / fact(2 * i + 3 * j + 2);
  return ((2 * i + 3 * j) & 2) ? -c : c;
}
template <int I, int J> struct SeriesCoef { static constexpr double v = series_coef(I, J); };
template <int I, int J>
__device__ __forceinline__ double series_horner(double r, double P) {   // down to P^0
  r = fma(r, P, SeriesCoef<I, J>::v);
  if constexpr (I > 0) return series_horner<I - 1, J>(r, P);
  else return r;
}
template <int K, int J>
__device__ __forceinline__ double series_row(double P) {
  constexpr int top = (K - 3 * J) / 2;
  if constexpr (top > 0) return series_horner<top - 1, J>(SeriesCoef<top, J>::v, P);
  else return SeriesCoef<0, J>::v;
}
template <int K, int J>
__device__ __forceinline__ double series_rows(double P, double T2) {   // rows J, J + 2, ...
  const double a = series_row<K, J>(P);
  if constexpr (3 * (J + 2) <= K) return fma(T2, series_rows<K, J + 2>(P, T2), a);
  else return a;
}
template <int K>
__device__ __forceinline__ void series64(double P, double T, double& zr, double& zi) {   // Z = i G
  const double T2 = T * T;
  zi = series_rows<K, 0>(P, T2);
  zr = -T * series_rows<K, 1>(P, T2);
}
// The shortest form whose terms left out stay below 3e-17 (|G| <= 1/2) for every P up to the warp's
// largest (high words of doubles, which order as unsigned integers for P >= 0; NaN above all).  The
// longest, k <= 19, reaches P = 2.27: the path's series end at tau = 3, P = 9/4.
constexpr uint32_t kHi9 = 0x3f982a56u, kHi11 = 0x3fb98db6u, kHi13 = 0x3fd29a09u, kHi15 = 0x3fe55d97u,
                   kHi17 = 0x3ff4e4f9u;   // 0.0236, 0.0998, 0.2906, 0.6677, 1.306

// 3D face term, as face_common / face_series / face_edge of pft_pairs.cuh: the series when every lane's
// P is below p_hi, else the edge sum (a lane below p_lo then takes the shortest series).
__device__ __forceinline__ void face_pair64(double qx, double qy, double qz, const Face64& f, double p_hi, double p_lo,
                                            double& re, double& im) {
  const double mu = fma(qx, f.gx, fma(qy, f.gy, qz * f.gz));
  const double a0 = fma(qx, f.q0x, fma(qy, f.q0y, qz * f.q0z));
  const double a1 = fma(qx, f.q1x, fma(qy, f.q1y, qz * f.q1z));
  const double s = fma(qx, f.nx, fma(qy, f.ny, qz * f.nz));
  const double s1 = a0 + a1, p1 = a0 * a1;
  const double P = fma(s1, s1, -p1), T = -p1 * s1;
  const uint32_t wmax = __reduce_max_sync(0xffffffffu, (uint32_t)__double2hiint(P) & 0x7fffffffu);
  double zr, zi;
  if (wmax < (uint32_t)__double2hiint(p_hi)) {
    if (wmax < kHi9) series64<9>(P, T, zr, zi);
    else if (wmax < kHi11) series64<11>(P, T, zr, zi);
    else if (wmax < kHi13) series64<13>(P, T, zr, zi);
    else if (wmax < kHi15) series64<15>(P, T, zr, zi);
    else if (wmax < kHi17) series64<17>(P, T, zr, zi);
    else series64<19>(P, T, zr, zi);
  } else {
    const double Xx = fma(f.ny, qz, -f.nz * qy), Xy = fma(f.nz, qx, -f.nx * qz), Xz = fma(f.nx, qy, -f.ny * qx);
    const double x2 = fma(Xx, Xx, fma(Xy, Xy, Xz * Xz));
    const double b0 = fma(f.q0x, Xx, fma(f.q0y, Xy, f.q0z * Xz));
    const double b1 = fma(f.q1x, Xx, fma(f.q1y, Xy, f.q1z * Xz));
    const double w[3] = {b1 - b0, fma(-2.0, b1, -b0), fma(2.0, b0, b1)};
    const double h0 = 0.5 * a0, h1 = 0.5 * a1;
    const double u[3] = {h1 - h0, fma(-2.0, h1, -h0), fma(2.0, h0, h1)};
    double S[3], sp[3], cp[3];
    sinc64(u, S);
    sincos64(-h0, sp[1], cp[1]);   // psi_1 = -h0, psi_2 = -h1, psi_0 = h0 + h1
    sincos64(-h1, sp[2], cp[2]);
    cp[0] = fma(cp[1], cp[2], -sp[1] * sp[2]);
    sp[0] = -fma(sp[1], cp[2], cp[1] * sp[2]);
    double sr = 0.0, si = 0.0;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      const double ws = w[l] * S[l];
      sr = fma(ws, cp[l], sr);
      si = fma(ws, sp[l], si);
    }
    const double inv = x2 > 0.0 ? 1.0 / x2 : 0.0;
    zr = sr * inv;
    zi = si * inv;
    if (P < p_lo) series64<9>(P, T, zr, zi);   // p_lo = (0.05)^2/4 at most
  }
  double sm, cm;
  sincos64(mu, sm, cm);
  const double c = -s * cm, d = -s * sm;   // -s exp(i mu) = c + i d
  re = fma(c, zr, fma(-d, zi, re));
  im = fma(c, zi, fma(d, zr, im));
}

}  // namespace pft
