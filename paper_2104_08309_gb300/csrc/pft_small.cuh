// pft_small.cuh -- the small-|Q| pass of the 3D transforms (|Q| r_max < 1/4), shared by the
// forward call and the Q-gradient.
//
// There S0(Q) = sum over the signed tetrahedra (c, p0, p1, p2) of det sum_k i^k h_k(x)/(k+3)!,
// x_j = Q.(p_j - c), is a power series in Q: with |x_j| < 1/4 the terms past k = 12 are below
// 5e-19 of sum |det|/6.  Two ways to it:
//  * kSmallDirect listed Q points or fewer: each evaluated over the faces, (Q point, face chunk)
//    units spread over the grid, the chunk sums added in order by the finishing kernel;
//  * more: the series' coefficients (moments of the shape, one per monomial of degree <= 12, 455
//    of them) are summed over the faces once, and every small Q point evaluates the polynomial.
// Line between them: a directly evaluated point costs about 70 FP64 operations a face and the moments
// about 900 with lanes to spare, so they break even near 30 points (on 20,480 faces 32 points take
// 75 us at the FP64 rate, the moments 60).  A curve of 2,928 points on
// 20,480 faces, 1,220 of them small: the call took 5,267 us with one block per point and 17 terms,
// 352 us with the moments.
// Both run in FP64, except that monomials of degree >= 8, which together stay below 1.1e-10 of
// the result, are summed in compensated FP32 (an error below 2e-17 of it).
#pragma once

#include "pft_kernels.cuh"

namespace pft {

constexpr int kMomK = 12;                 // highest degree kept
constexpr int kMomLo = 7;                 // degrees 0 .. 7 in FP64, 8 .. 12 in FP32
constexpr int mom_count(int k) { return (k + 1) * (k + 2) * (k + 3) / 6; }   // monomials of degree <= k
constexpr int kMomN = mom_count(kMomK);   // 455
constexpr int kMomN64 = mom_count(kMomLo);   // 120
constexpr int kMomN32 = kMomN - kMomN64;  // 335
// Monomial x^a y^b z^c of degree k = a + b + c, s = b + c: index mom_count(k - 1) + s (s + 1)/2 + c.

// Scratch of the pass (it lies over the records, which are no longer needed):
// the summed moments (kMomN doubles), then per block kMomN64 doubles and kMomN32 float pairs;
// the direct sums lie over the same bytes.
constexpr size_t kMomHead = 4096;         // kMomN doubles, rounded up
constexpr size_t kMomPart = 3840;         // kMomN64 * 8 + kMomN32 * 8 = 3640, rounded up
constexpr int kMomFaces = 32;             // faces of one batch (one per lane)
constexpr int kDirectChunks = 64;         // face chunks of a directly evaluated Q point at most
static_assert(kMomN * 8 <= kMomHead && kMomN64 * 8 + kMomN32 * 8 <= kMomPart, "moment scratch");

inline int64_t small3_blocks(int64_t nf, int sms) {
  return std::max<int64_t>(1, std::min<int64_t>(sms, (nf + kMomFaces - 1) / kMomFaces));
}
__host__ __device__ inline int64_t small3_chunks(int64_t nf) {   // face chunks per Q point, >= 256 faces each
  const int64_t c = (nf + 255) / 256;
  return c < 1 ? 1 : (c < kDirectChunks ? c : kDirectChunks);
}
// Bytes of scratch the pass needs for nf faces.
inline size_t small3_bytes(int64_t nf, int sms) {
  return kMomHead + std::max((size_t)small3_blocks(nf, sms) * kMomPart,
                             (size_t)(kSmallDirect * small3_chunks(nf)) * 8 * sizeof(double));
}

// The direct series of one tetrahedron (c, p0, p1, p2): its corner phases x and the monomials'
// coefficients 1/(k+3)!, terms through kMomK.
__device__ __forceinline__ void tetra_series(const double (&x)[3], double& re, double& im) {
  simplex_series<3, 3, kMomK>(x, re, im);
}

// S0(Q) from the moments m (already holding (-1)^(k/2)/(k+3)! and the scale of the coordinates):
// Horner in x for every y^b z^c, even and odd powers apart (the even degrees are the real part).
// With GRAD also the derivatives in the scaled Q, g[d] = (re, im).
template <bool GRAD>
__device__ __forceinline__ void mom_eval(const double* m, double x, double y, double z, double& re, double& im,
                                         double (&g)[3][2]) {
  const double x2 = x * x;
  double ev = 0.0, od = 0.0;
  double gx[2] = {0.0, 0.0}, gy[2] = {0.0, 0.0}, gz[2] = {0.0, 0.0};   // [0] even degrees, [1] odd
  double yp = 1.0;   // y^b over the outer loop, z^c over the inner one
  double dyp = 0.0;  // b y^(b-1)
  for (int b = 0; b <= kMomK; ++b) {
    double w = yp, dwy = dyp, zc1 = 0.0, zp = 1.0;   // y^b z^c, its derivatives
    for (int c = 0; b + c <= kMomK; ++c) {
      const int s = b + c, row = s * (s + 1) / 2 + c;
      // p[0] + x p[1] = sum_a M[a + s] x^a;  d[.] its derivative in x
      double p0 = 0.0, p1 = 0.0, d0 = 0.0, d1 = 0.0;
      for (int a = kMomK - s; a >= 0; --a) {
        const int k = a + s;
        const double M = m[k * (k + 1) * (k + 2) / 6 + row];
        if (a & 1) {
          p1 = fma(p1, x2, M);
          if (GRAD) d1 = fma(d1, x2, (double)a * M);        // x^(a-1), a - 1 even
        } else {
          p0 = fma(p0, x2, M);
          if (GRAD && a > 0) d0 = fma(d0, x2, (double)a * M);   // x^(a-1), a - 1 odd
        }
      }
      // degree parity of p0 is that of s
      const double e = (s & 1) ? x * p1 : p0, o = (s & 1) ? p0 : x * p1;
      ev = fma(w, e, ev);
      od = fma(w, o, od);
      if (GRAD) {
        // derivative in x: a odd -> d1 (even powers), a even -> x d0; they keep their terms' degrees
        const double dxe = (s & 1) ? d1 : x * d0, dxo = (s & 1) ? x * d0 : d1;
        gx[0] = fma(w, dxe, gx[0]);
        gx[1] = fma(w, dxo, gx[1]);
        const double dwz = yp * zc1;
        gy[0] = fma(dwy, e, gy[0]);
        gy[1] = fma(dwy, o, gy[1]);
        gz[0] = fma(dwz, e, gz[0]);
        gz[1] = fma(dwz, o, gz[1]);
        zc1 = fma(zc1, z, zp);          // (c + 1) z^c from c z^(c-1) and z^c
        zp *= z;
        dwy = dyp * zp;
        w = yp * zp;
      } else {
        w *= z;
      }
    }
    if (GRAD) dyp = fma(dyp, y, yp);
    yp *= y;
  }
  re = ev;
  im = od;
  if (GRAD) {
    for (int t = 0; t < 2; ++t) { g[0][t] = gx[t]; g[1][t] = gy[t]; g[2][t] = gz[t]; }
  }
}

// Bytes by which the scratch exceeds the records of a pft3d_mesh call (part of its workspace size).
size_t small3_growth(int64_t n_faces, int64_t n_q, const pft_options* opts);

// pft_small.cu.  q = NULL: only the moments (nothing for h->small_q_count <= kSmallDirect).
cudaError_t launch_small3(const float* v, int64_t nv, const int32_t* f, int64_t nf, const double* q, WsHeader* h,
                          const double* mparts, int n_measure, void* scratch, cudaStream_t st);

// The vertex adjoint.  The small-|Q| points' share of dL/dv is the shape derivative of the integral of
// Phi(r) = Re sum_Q conj(g_Q) e^{iQ.r}, for corner k of a face N times the face average of lambda_k Phi.
// With few points each is evaluated in turn (corner_adj); with more than kSmallAdjoint of them Phi is
// summed once into a polynomial in r - c (degree <= 12: the terms past it are below 1e-17), and every
// face integrates that by Gauss quadrature of the order its size needs.
constexpr int kSmallAdjoint = 24;
constexpr int kPhiLo = 8;                  // degrees 0 .. 8 in FP64; 9 .. 12, below 1.1e-11, in FP32
constexpr int kPhiBlocks = 64;             // blocks that sum Phi's coefficients
struct PhiPoly {
  double c64[mom_count(kPhiLo)];
  float c32[kMomN - mom_count(kPhiLo)];    // in units of scale
  double scale;                            // the largest coefficient (0: Phi vanishes)
};
constexpr size_t kPhiHead = 4096;
static_assert(sizeof(PhiPoly) <= kPhiHead, "Phi's coefficients");
inline size_t small_adjoint_bytes(int64_t nf) {
  return kPhiHead + sizeof(double) * (kMomN * (size_t)kPhiBlocks + 3 * (size_t)std::max<int64_t>(nf, 1));
}
inline const double* small_adjoint_faces(const void* scratch) {   // [nf][3]: face averages of lambda_k Phi
  return reinterpret_cast<const double*>(static_cast<const char*>(scratch) + kPhiHead) + kMomN * (size_t)kPhiBlocks;
}
// Two launches; they do nothing for h->small_q_count <= kSmallAdjoint.
cudaError_t launch_small_adjoint3(const float* v, int64_t nv, const int32_t* f, int64_t nf, const double* q,
                                  const double* g, int64_t n_q, WsHeader* h, void* scratch, cudaStream_t st);

}  // namespace pft
