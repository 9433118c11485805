// pft_small.cuh -- the small-|Q| pass of the 3D transforms (|Q| r_max < 1/4), shared by the
// forward call and the Q-gradient.
//
// There S0(Q) = sum over the signed tetrahedra (c, p0, p1, p2) of det sum_k i^k h_k(x)/(k+3)!,
// x_j = Q.(p_j - c), is a power series in Q: with |x_j| < 1/4 the terms past k = 12 are below
// 5e-19 of sum |det|/6.  Three ways to it:
//  * kSmallDirect listed Q points or fewer: each evaluated over the faces, (Q point, face chunk)
//    units spread over the grid, the chunk sums added in order by the finishing kernel;
//  * more: the series' coefficients (moments of the shape, one per monomial of degree <= 12, 455
//    of them) are summed over the faces once, and every small Q point evaluates the polynomial.
//  * of a shape of few faces the finishing kernel sums each point over the faces itself (small_few).
// Line between the first two: a directly evaluated point costs about 70 FP64 operations a face and the moments
// about 900 with lanes to spare, so they break even near 30 points (on 20,480 faces 32 points take
// 75 us at the FP64 rate, the moments 102).  A curve of 2,928 points on
// 20,480 faces, 1,220 of them small: the call took 5,267 us with one block per point and 17 terms,
// 233 us with the moments (k_small3 102 us, the polynomials in k_finalize3d 25 us).
// Both run in FP64, except that monomials of degree >= 8, which together stay below 1.1e-10 of sum |det|/6,
// are evaluated in FP32 and summed there in compensated pairs (some 16 roundings of 2^-24 on that: about
// 1e-16 of sum |det|/6, what FP64 roundings of the other terms amount to).
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

// Up to kFewFaces faces, k_finalize3d's warps take a small point's faces 32 at a time and k_small3 has only
// the volume to do: 120 FP64 instructions a point and 32 faces, 6.6 ns of the chip, against 25 us and more for
// the moments (a batch, its block's sums and their hand-over) and a block for only 32 faces where k_small3
// sums directly.  Calls with all points small, through k_small3 / so: 12 faces x 20 Q 131 / 30 us, x 300 68 / 34,
// x 3,000 86 / 53; 80 faces x 40 Q 64 / 35 us, x 300 67 / 37; past the line 80 x 3,000 84.
constexpr int64_t kFewFaces = 256;
__host__ __device__ inline bool small_few(uint32_t count, int64_t nf) {
  return nf <= kFewFaces && (int64_t)count * ((nf + 31) / 32) <= 3000;
}

// The Q-gradient: points evaluated one by one in blocks of their own (k_qsmall_part; 22 ns of the chip a point
// and 32 faces, 30 ns a point besides), where that is less than the 30 us that the moments add.  Calls with all
// points small, moments / direct: 12 faces x 40 Q 85 / 56 us, 80 x 300 95 / 74, 320 x 40 114 / 86; past the line 320
// x 300 112 / 148 (with 17 terms), 1,280 x 40 105 / 111.
__host__ __device__ inline bool qsmall_direct(uint32_t count, int64_t nf) {
  return count <= (uint32_t)kSmallDirect || (int64_t)count * (nf + 48) <= 40000;
}

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

// Corners of face m relative to c; false (and zeros) for an index out of range.
__device__ __forceinline__ bool corners(const float* v, int64_t nv, const int32_t* f, int64_t m, const double* c,
                                        double (&P)[3][3]) {
  const int32_t id[3] = {f[3 * m], f[3 * m + 1], f[3 * m + 2]};
  const bool ok = id[0] >= 0 && id[1] >= 0 && id[2] >= 0 && id[0] < nv && id[1] < nv && id[2] < nv;
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int d = 0; d < 3; ++d) P[k][d] = ok ? (double)v[3 * (int64_t)id[k] + d] - c[d] : 0.0;
  return ok;
}
__device__ __forceinline__ double det3(const double (&P)[3][3]) {
  return P[0][0] * (P[1][1] * P[2][2] - P[1][2] * P[2][1]) + P[0][1] * (P[1][2] * P[2][0] - P[1][0] * P[2][2]) +
         P[0][2] * (P[1][0] * P[2][1] - P[1][1] * P[2][0]);
}

// The direct series of one tetrahedron (c, p0, p1, p2): its corner phases x and the monomials'
// coefficients 1/(k+3)!, terms through kMomK.
__device__ __forceinline__ void tetra_series(const double (&x)[3], double& re, double& im) {
  simplex_series<3, 3, kMomK>(x, re, im);
}

// The summed moments' order: by b, then c downwards, then a upwards, so that an evaluation walks them.
__host__ __device__ constexpr int mom_pos(int a, int b, int c) {
  int n = 0;
  for (int j = 0; j < b; ++j) n += (kMomK + 1 - j) * (kMomK + 2 - j) / 2;
  const int r = kMomK - b - c;
  return n + r * (r + 1) / 2 + a;
}

// S0(Q) from the summed moments m (already holding (-1)^(k/2)/(k+3)! and the scale of the coordinates), by
// one warp (all lanes pass the same scaled Q and get the result): lane 2b + e takes the rows y^b z^c with
// c of parity e, Horner in x and z^2, the even degrees (the real part) and the odd ones apart.  With GRAD
// also the derivatives in the scaled Q, g[d] = (re, im).  One thread per point ran one long dependent
// chain of FP64 operations: 95 us for 1,220 points, 149 us for 190 with GRAD.
template <bool GRAD>
__device__ __forceinline__ void mom_eval(const double* m, double x, double y, double z, double& re, double& im,
                                         double (&g)[3][2]) {
  const int lane = threadIdx.x & 31, b = lane >> 1, par = lane & 1;
  const double x2 = x * x, z2 = z * z;
  double v[2] = {0.0, 0.0}, vx[2] = {0.0, 0.0}, vz[2] = {0.0, 0.0};   // [0] even degrees, [1] odd
  if (b <= kMomK) {
    const int top = kMomK - b, first = top - ((top ^ par) & 1);   // the largest c of this parity
    const double* row = m + mom_pos(0, b, top);
    for (int c = first; c >= 0; c -= 2) {
      const int n = top - c;                                  // the row's highest power of x
      const double* w = row + n * (n + 1) / 2;
      double p0 = 0.0, p1 = 0.0, d0 = 0.0, d1 = 0.0;   // sums over even a of M x^a; odd, less an x; a M x^(a-1)
#pragma unroll 2
      for (int a = n & ~1; a >= 0; a -= 2) {
        const double M = w[a], N = a < n ? w[a + 1] : 0.0;
        p1 = fma(p1, x2, N);
        p0 = fma(p0, x2, M);
        if (GRAD) {
          d1 = fma(d1, x2, (double)(a + 1) * N);
          if (a > 0) d0 = fma(d0, x2, (double)a * M);
        }
      }
      const bool odd = (b + c) & 1;   // terms of degree parity e have a of parity e ^ (b + c)
      p1 *= x;
      d0 *= x;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const bool q = (e == 1) != odd;
        if (GRAD) {   // d/dz of sum z^c: Horner in z^2 for c z^(c-1), less a z where c is odd (c = 0: nothing)
          vz[e] = c > 1 || par ? fma(vz[e], z2, (double)c * (q ? p1 : p0)) : vz[e];
          vx[e] = fma(vx[e], z2, q ? d1 : d0);
        }
        v[e] = fma(v[e], z2, q ? p1 : p0);
      }
    }
  }
  // z^par, y^b and their derivatives; c z^(c-1) = z^(par - 1 + 2j): par odd needs no factor, even one z
  double yb = 1.0, dy = 0.0;
  for (int j = 0; j < b; ++j) {
    dy = fma(dy, y, yb);
    yb *= y;
  }
  const double zp = par ? z : 1.0;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    g[0][e] = GRAD ? yb * zp * vx[e] : 0.0;
    g[1][e] = GRAD ? dy * zp * v[e] : 0.0;
    g[2][e] = GRAD ? yb * (par ? 1.0 : z) * vz[e] : 0.0;
    v[e] *= yb * zp;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      v[e] += __shfl_xor_sync(0xffffffffu, v[e], o);
      if (GRAD)
#pragma unroll
        for (int d = 0; d < 3; ++d) g[d][e] += __shfl_xor_sync(0xffffffffu, g[d][e], o);
    }
  }
  re = v[0];
  im = v[1];
}

// Bytes of a pft3d_mesh workspace that pft3d_mesh_noalloc's limit does not count.
size_t uncounted_bytes(int64_t n_faces, int64_t n_q, const pft_options* opts);

// pft_small.cu.  q = NULL: the moments for the Q-gradient, where qsmall_direct does not hold.
cudaError_t launch_small3(const float* v, int64_t nv, const int32_t* f, int64_t nf, const double* q, WsHeader* h,
                          const double* mparts, int n_measure, void* scratch, cudaStream_t st);

// The vertex adjoint.  The small-|Q| points' share of dL/dv is the shape derivative of the integral of
// Phi(r) = Re sum_Q conj(g_Q) e^{iQ.r}, for corner k of a face N times the face average of lambda_k Phi.
// With few points each is evaluated in turn (corner_adj); with more than kSmallAdjoint of them Phi is
// summed once into a polynomial in r - c (degree <= 12: the terms past it are below 1e-17), and every
// face integrates that by Gauss quadrature of the order its size needs.
constexpr int kSmallAdjoint = 24;
constexpr int kPhiLo = 7;                  // degrees 0 .. 7 in FP64; 8 .. 12, below 4e-10, in FP32
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
