// pft_small.cu -- k_small3: the sums over the faces that the small-|Q| points of a 3D call need
// (see pft_small.cuh), and the volume for Q = 0.
#include <algorithm>

#include "pft_small.cuh"

namespace pft {
namespace {

constexpr int kNT = 512, kNW = kNT / 32;

// (s, c) of row s (s + 1)/2 + c, for every row of a degree's monomials
struct RowTable { unsigned char s[91], c[91]; };
constexpr RowTable make_rows() {
  RowTable t{};
  int i = 0;
  for (int s = 0; s <= kMomK; ++s)
    for (int c = 0; c <= s; ++c, ++i) {
      t.s[i] = (unsigned char)s;
      t.c[i] = (unsigned char)c;
    }
  return t;
}
__constant__ RowTable kRows = make_rows();

constexpr int rows_of(int k) { return (k + 1) * (k + 2) / 2; }
constexpr int slots_of(int k) { return (rows_of(k) + kNW - 1) / kNW; }
// accumulator slots of the degrees lo .. k - 1
constexpr int slot_base(int lo, int k) {
  int n = 0;
  for (int d = lo; d < k; ++d) n += slots_of(d);
  return n;
}
constexpr int kSlots64 = slot_base(0, kMomLo + 1);            // 12
constexpr int kSlots32 = slot_base(kMomLo + 1, kMomK + 1);    // 23

struct Sum64 {
  double v;
  __device__ void init() { v = 0.0; }
  __device__ void add(double a, double b) { v = fma(a, b, v); }
};
struct Sum32 {
  CAcc v;
  __device__ void init() { v.init(); }
  __device__ void add(float a, float b) { v.add(a * b); }
};

// One batch of 32 faces, one per lane, over the block's warps: the coefficients of h_k(x0, x1, x2) as
// polynomials in Q, x_j = Q.p_j, degree by degree.  The complete homogeneous polynomials obey
//   H_j[k] = H_{j-1}[k] + x_j H_j[k-1]   (nodes 0 .. j, H_{-1}[k] = 0 for k > 0, H[0] = 1),
// so the coefficient of a monomial takes one fused multiply-add per node and per neighbour of the
// degree below (same row, row of y, row of z).  A warp holds whole monomials (the neighbours are
// then warp-uniform) and a lane one face; two levels of the three nodes' coefficients live in
// shared memory.  det times the last node's coefficient of the degrees KLO .. KHI is summed.
template <class T, class Sum, int KLO, int KHI>
__device__ __forceinline__ void batch(const T (&P)[3][3], T det, T* buf, Sum* acc, int lane, int warp) {
  constexpr int W = rows_of(KHI) * 32;     // one level of one node
#pragma unroll
  for (int k = 0; k <= KHI; ++k) {
    T* cur = buf + (k & 1) * 3 * W;
    const T* old = buf + ((k & 1) ^ 1) * 3 * W;
#pragma unroll
    for (int i = 0; i < slots_of(k); ++i) {
      const int m = warp + kNW * i;
      if (m < rows_of(k)) {
        T H;
        if (k == 0) {
          H = (T)1;
          cur[lane] = H;
          cur[W + lane] = H;
          cur[2 * W + lane] = H;
        } else {
          const int s = kRows.s[m], c = kRows.c[m], ny = (s - 1) * s / 2 + c;
          H = (T)0;
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const T* o = old + j * W;
            if (s < k) H = fma(P[j][0], o[m * 32 + lane], H);
            if (c < s) H = fma(P[j][1], o[ny * 32 + lane], H);
            if (c > 0) H = fma(P[j][2], o[(ny - 1) * 32 + lane], H);
            if (k < KHI) cur[j * W + m * 32 + lane] = H;
          }
        }
        if (k >= KLO) acc[slot_base(KLO, k < KLO ? KLO : k) + i].add(det, H);
      }
    }
    __syncthreads();
  }
}

__device__ __forceinline__ double wsum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  return x;
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

// dynamic shared memory: two levels of three nodes' coefficients, then the lanes' FP64 sums
constexpr size_t kBuf64 = 2 * 3 * (size_t)rows_of(kMomLo) * 32 * sizeof(double);
constexpr size_t kBuf32 = 2 * 3 * (size_t)rows_of(kMomK) * 32 * sizeof(float);
constexpr size_t kRed = (size_t)kMomN64 * 33 * sizeof(double);
constexpr size_t cmax(size_t a, size_t b) { return a > b ? a : b; }
constexpr size_t kShared = cmax(cmax(kBuf64, kBuf32), kRed);

// The last block to finish adds the blocks' partial moments (in block order) and scales them:
// (-1)^(k/2)/(k+3)!, the sign of i^k = (-1)^(k/2) (1 or i).
__device__ void sum_moments(const char* parts, int nb, double r3, double* out) {
  for (int t = threadIdx.x; t < kMomN; t += kNT) {
    int k = 0;
    while (mom_count(k) <= t) ++k;
    double s = 0.0;
    if (t < kMomN64) {
      for (int b = 0; b < nb; ++b) s += reinterpret_cast<const double*>(parts + b * kMomPart)[t];
    } else {
      CAcc a;
      a.init();
      for (int b = 0; b < nb; ++b) {
        const float2 p = reinterpret_cast<const float2*>(parts + b * kMomPart + kMomN64 * 8)[t - kMomN64];
        a.add(p.x);
        a.lo += p.y;
      }
      s = ((double)a.hi + (double)a.lo) * r3;
    }
    double w = 1.0;
    for (int j = 2; j <= k + 3; ++j) w /= (double)j;
    out[t] = (k & 2) ? -s * w : s * w;
  }
}

// Bound: the moments are FP64 work (876 fused multiply-adds a face in FP64, 3,600 in FP32, at 2
// and 128 a clock and SM), so a batch of 32 faces is paced by the FP64 pipe (about 9 us a batch and
// SM); one batch a block and round, one block of 16 warps per SM.
__global__ void __launch_bounds__(kNT) k_small3(const float* __restrict__ v, int64_t nv,
                                                const int32_t* __restrict__ f, int64_t nf,
                                                const double* __restrict__ q, WsHeader* h,
                                                const double* __restrict__ mparts, int n_measure, char* scratch) {
  extern __shared__ __align__(16) char sh[];
  __shared__ double red[kNW][2];
  __shared__ int last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (blockIdx.x == 0 && mparts != nullptr) {   // the volume, for Q = 0: a fixed-order sum
    double s = 0.0;
    for (int b = threadIdx.x; b < n_measure; b += kNT) s += mparts[b];
    s = wsum(s);
    if (lane == 0) red[warp][0] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      s = 0.0;
      for (int w = 0; w < kNW; ++w) s += red[w][0];
      h->measure = s;
    }
    __syncthreads();
  }
  const uint32_t count = h->small_q_count;
  if (count == 0) return;
  const double c[3] = {h->center[0], h->center[1], h->center[2]};
  char* parts = scratch + kMomHead;
  if (count <= (uint32_t)kSmallDirect) {
    if (q == nullptr) return;
    const int64_t nch = small3_chunks(nf), per = (nf + nch - 1) / nch;
    for (int64_t u = blockIdx.x; u < (int64_t)count * nch; u += gridDim.x) {
      const int64_t i = h->small_list[u / nch], m0 = (u % nch) * per, m1 = min(nf, m0 + per);
      const double Q[3] = {q[3 * i], q[3 * i + 1], q[3 * i + 2]};
      double re = 0.0, im = 0.0;
      for (int64_t m = m0 + threadIdx.x; m < m1; m += kNT) {
        double P[3][3];
        if (!corners(v, nv, f, m, c, P)) continue;
        const double x[3] = {Q[0] * P[0][0] + Q[1] * P[0][1] + Q[2] * P[0][2],
                             Q[0] * P[1][0] + Q[1] * P[1][1] + Q[2] * P[1][2],
                             Q[0] * P[2][0] + Q[1] * P[2][1] + Q[2] * P[2][2]};
        const double det = det3(P);
        double sr, si;
        tetra_series(x, sr, si);
        re = fma(det, sr, re);
        im = fma(det, si, im);
      }
      re = wsum(re);
      im = wsum(im);
      if (lane == 0) { red[warp][0] = re; red[warp][1] = im; }
      __syncthreads();
      if (threadIdx.x < 2) {
        double s = 0.0;
        for (int w = 0; w < kNW; ++w) s += red[w][threadIdx.x];
        reinterpret_cast<double*>(parts)[2 * u + threadIdx.x] = s;
      }
      __syncthreads();
    }
    return;
  }
  const float rmax = __uint_as_float(h->rmax_bits);
  const double inv = rmax > 0.f ? 1.0 / (double)rmax : 0.0;   // coordinates in units of r_max
  Sum64 a64[kSlots64];
  Sum32 a32[kSlots32];
#pragma unroll
  for (int i = 0; i < kSlots64; ++i) a64[i].init();
#pragma unroll
  for (int i = 0; i < kSlots32; ++i) a32[i].init();
  const int64_t batches = (nf + kMomFaces - 1) / kMomFaces;
  for (int64_t b = blockIdx.x; b < batches; b += gridDim.x) {
    const int64_t m = b * kMomFaces + lane;
    double P[3][3], det = 0.0;
    if (m < nf) {
      corners(v, nv, f, m, c, P);
      det = det3(P);
    } else {
      for (int k = 0; k < 3; ++k)
        for (int d = 0; d < 3; ++d) P[k][d] = 0.0;
    }
    float Pf[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        P[k][d] *= inv;
        Pf[k][d] = (float)P[k][d];
      }
    // det in units of r_max^3 in FP32 (it could leave the FP32 range otherwise); scaled back below
    const float detf = (float)(det * inv * inv * inv);
    batch<double, Sum64, 0, kMomLo>(P, det, reinterpret_cast<double*>(sh), a64, lane, warp);
    batch<float, Sum32, kMomLo + 1, kMomK>(Pf, detf, reinterpret_cast<float*>(sh), a32, lane, warp);
  }
  // lanes -> one sum per monomial: through shared memory in FP64 (33 doubles a row: no conflicts),
  // by compensated shuffles in FP32
  char* mine = parts + (size_t)blockIdx.x * kMomPart;
  double* rb = reinterpret_cast<double*>(sh);
#pragma unroll
  for (int k = 0; k <= kMomLo; ++k)
#pragma unroll
    for (int i = 0; i < slots_of(k); ++i) {
      const int m = warp + kNW * i;
      if (m < rows_of(k)) rb[(mom_count(k - 1) + m) * 33 + lane] = a64[slot_base(0, k) + i].v;
    }
  __syncthreads();
  {
    const int t = threadIdx.x >> 2, part = threadIdx.x & 3;   // four threads a monomial, 8 lanes each
    double s = 0.0;
    if (t < kMomN64)
      for (int l = 0; l < 8; ++l) s += rb[t * 33 + 8 * part + l];
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (t < kMomN64 && part == 0) reinterpret_cast<double*>(mine)[t] = s;
  }
#pragma unroll
  for (int k = kMomLo + 1; k <= kMomK; ++k)
#pragma unroll
    for (int i = 0; i < slots_of(k); ++i) {
      const int m = warp + kNW * i;
      if (m < rows_of(k)) {
        CAcc a = a32[slot_base(kMomLo + 1, k) + i].v;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float hi = __shfl_xor_sync(0xffffffffu, a.hi, o), lo = __shfl_xor_sync(0xffffffffu, a.lo, o);
          a.add(hi);
          a.lo += lo;
        }
        if (lane == 0) reinterpret_cast<float2*>(mine + kMomN64 * 8)[mom_count(k - 1) + m - kMomN64] = make_float2(a.hi, a.lo);
      }
    }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&h->ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  sum_moments(parts, (int)gridDim.x, (double)rmax * (double)rmax * (double)rmax, reinterpret_cast<double*>(scratch));
}

// ---------------------------------------------------------------------------
// Vertex adjoint: Phi's coefficients, then its face averages.
// ---------------------------------------------------------------------------

// Coefficient of (r')^alpha, r' = (r - c)/r_max, Q' = Q r_max, k = |alpha|:
//   Re(i^k sum_Q conj(g) e^{iQ.c} Q'^alpha) / alpha!.
// Each block takes a run of Q points in order, picks the small ones (in order: the sum is
// reproducible) and adds them one thread per monomial; the last block adds the blocks.
constexpr int kPhiQ = 16;   // points of one round
__global__ void __launch_bounds__(kNT) k_phi(const double* __restrict__ q, const double* __restrict__ g, int64_t n_q,
                                             WsHeader* h, char* scratch) {
  __shared__ int list[kNT];
  __shared__ int wcount[kNW];
  __shared__ double pw[kPhiQ][3][kMomK + 1], wt[kPhiQ][2];
  __shared__ double wmax[kNW];
  __shared__ int last;
  if (h->small_q_count <= (uint32_t)kSmallAdjoint) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = threadIdx.x;
  const float rmaxf = __uint_as_float(h->rmax_bits);
  const double rmax = (double)rmaxf;
  int k = 0, a = 0, b = 0, c = 0;
  if (t < kMomN) {
    while (mom_count(k) <= t) ++k;
    const int m = t - k * (k + 1) * (k + 2) / 6, s = kRows.s[m];
    c = kRows.c[m];
    b = s - c;
    a = k - s;
  }
  double acc = 0.0;
  const int64_t per = (n_q + gridDim.x - 1) / gridDim.x, q0 = blockIdx.x * per, q1 = min(n_q, q0 + per);
  for (int64_t base = q0; base < q1; base += kNT) {
    const int64_t i = base + t;
    bool small = false;
    if (i < q1) {
      const double q2 = q_norm2(q[3 * i], q[3 * i + 1], q[3 * i + 2]);
      small = q2 == 0.0 || small_q(q2, rmaxf);
    }
    const unsigned bal = __ballot_sync(0xffffffffu, small);
    if (lane == 0) wcount[warp] = __popc(bal);
    __syncthreads();
    int before = 0, n = 0;
    for (int w = 0; w < kNW; ++w) {
      if (w < warp) before += wcount[w];
      n += wcount[w];
    }
    if (small) list[before + __popc(bal & ((1u << lane) - 1u))] = t;
    __syncthreads();
    for (int e0 = 0; e0 < n; e0 += kPhiQ) {
      const int cnt = min(kPhiQ, n - e0);
      if (t < 3 * cnt) {
        const double x = q[3 * (base + list[e0 + t / 3]) + t % 3] * rmax;
        double p = 1.0;
        for (int j = 0; j <= kMomK; ++j) {
          pw[t / 3][t % 3][j] = p;
          p *= x;
        }
      } else if (t >= 64 && t < 64 + cnt) {
        const int64_t iq = base + list[e0 + t - 64];
        double sn, cs;
        sincos(q[3 * iq] * h->center[0] + q[3 * iq + 1] * h->center[1] + q[3 * iq + 2] * h->center[2], &sn, &cs);
        const double gr = g[2 * iq], gi = g[2 * iq + 1];
        wt[t - 64][0] = gr * cs + gi * sn;
        wt[t - 64][1] = gr * sn - gi * cs;
      }
      __syncthreads();
      if (t < kMomN)
        for (int e = 0; e < cnt; ++e) acc = fma(wt[e][k & 1] * pw[e][0][a], pw[e][1][b] * pw[e][2][c], acc);
      __syncthreads();
    }
  }
  double* parts = reinterpret_cast<double*>(scratch + kPhiHead);
  if (t < kMomN) parts[(size_t)blockIdx.x * kMomN + t] = acc;
  __threadfence();
  __syncthreads();
  if (t == 0) last = atomicAdd(&h->ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  PhiPoly* out = reinterpret_cast<PhiPoly*>(scratch);
  double sum = 0.0;
  if (t < kMomN) {
    for (unsigned u = 0; u < gridDim.x; ++u) sum += parts[(size_t)u * kMomN + t];
    // Re(i w) = -Im w: the sign of i^k over the real (k even) or imaginary (k odd) part
    double w = ((k + 1) & 2) ? -1.0 : 1.0;
    for (int j = 2; j <= a; ++j) w /= (double)j;
    for (int j = 2; j <= b; ++j) w /= (double)j;
    for (int j = 2; j <= c; ++j) w /= (double)j;
    sum *= w;
  }
  double mx = fabs(sum);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) wmax[warp] = mx;
  __syncthreads();
  mx = wmax[0];
  for (int w = 1; w < kNW; ++w) mx = fmax(mx, wmax[w]);
  if (t < mom_count(kPhiLo)) out->c64[t] = sum;
  else if (t < kMomN) out->c32[t - mom_count(kPhiLo)] = mx > 0.0 ? (float)(sum / mx) : 0.f;
  if (t == 0) out->scale = mx;
}

// Sum over degrees KLO .. KHI of C_alpha x^a y^b z^c (coefficients of degree k from C + (mom_count(k-1)
// - mom_count(KLO-1))), Horner in each variable.
template <class T, int KLO, int KHI>
__device__ __forceinline__ T poly3(const T* C, T x, T y, T z) {
  T r = (T)0;
  for (int b = KHI; b >= 0; --b) {
    T rz = (T)0;
    for (int c = KHI - b; c >= 0; --c) {
      const int s = b + c, row = s * (s + 1) / 2 + c, alo = KLO > s ? KLO - s : 0;
      T rx = (T)0;
      for (int a = KHI - s; a >= alo; --a) {
        const int k = a + s;
        rx = fma(rx, x, C[k * (k + 1) * (k + 2) / 6 - mom_count(KLO - 1) + row]);
      }
      for (int a = alo; a > 0; --a) rx *= x;
      rz = fma(rz, z, rx);
    }
    r = fma(r, y, rz);
  }
  return r;
}

// Gauss-Legendre nodes and weights on [0, 1], n = 3 .. 8 (Abramowitz & Stegun, table 25.4).
__constant__ double kGlX[6][8] = {
    {0.1127016653792583, 0.5, 0.8872983346207417},
    {0.06943184420297371, 0.33000947820757187, 0.6699905217924281, 0.9305681557970262},
    {0.04691007703066802, 0.23076534494715845, 0.5, 0.7692346550528415, 0.9530899229693319},
    {0.03376524289842403, 0.16939530676686776, 0.38069040695840156, 0.6193095930415985, 0.8306046932331322,
     0.9662347571015759},
    {0.0254460438286207, 0.12923440720030277, 0.2970774243113014, 0.5, 0.7029225756886985, 0.8707655927996972,
     0.9745539561713793},
    {0.019855071751231912, 0.10166676129318664, 0.2372337950418355, 0.4082826787521751, 0.5917173212478248,
     0.7627662049581645, 0.8983332387068134, 0.9801449282487681}};
__constant__ double kGlW[6][8] = {
    {0.27777777777777778, 0.44444444444444444, 0.27777777777777778},
    {0.17392742256872679, 0.3260725774312732, 0.3260725774312732, 0.17392742256872679},
    {0.11846344252809464, 0.23931433524968315, 0.28444444444444444, 0.23931433524968315, 0.11846344252809464},
    {0.08566224618958514, 0.18038078652406936, 0.23395696728634552, 0.23395696728634552, 0.18038078652406936,
     0.08566224618958514},
    {0.06474248308443487, 0.13985269574463843, 0.19091502525255935, 0.20897959183673465, 0.19091502525255935,
     0.13985269574463843, 0.06474248308443487},
    {0.05061426814518853, 0.11119051722668721, 0.15685332293894344, 0.18134189168918083, 0.18134189168918083,
     0.15685332293894344, 0.11119051722668721, 0.05061426814518853}};
// n points integrate a polynomial times u lambda_k exactly up to degree D = 2n - 3 (collapsed
// coordinates); a face whose phases about its centroid stay below kGlY[n - 3] has its terms of degree
// D + 1 below 1e-17: y^(D+1)/(D+1)!.  n = 8 is exact for all 12 degrees.
__constant__ float kGlY[5] = {1.2e-4f, 4.4e-3f, 2.8e-2f, 9.0e-2f, 0.20f};

// One warp per face, one quadrature point per lane and round: r = p0 + u ((p1 - p0) + w (p2 - p1)),
// lambda = (1 - u, u (1 - w), u w), element u du dw.
__global__ void __launch_bounds__(256) k_phi_faces(const float* __restrict__ v, int64_t nv,
                                                   const int32_t* __restrict__ f, int64_t nf,
                                                   const WsHeader* __restrict__ h, const char* __restrict__ scratch,
                                                   double* __restrict__ out) {
  __shared__ PhiPoly phi;
  if (h->small_q_count <= (uint32_t)kSmallAdjoint) return;
  for (int t = threadIdx.x; t < (int)(sizeof(PhiPoly) / 4); t += 256)
    reinterpret_cast<uint32_t*>(&phi)[t] = reinterpret_cast<const uint32_t*>(scratch)[t];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const float rmax = __uint_as_float(h->rmax_bits);
  const double inv = rmax > 0.f ? 1.0 / (double)rmax : 0.0;
  const double c[3] = {h->center[0], h->center[1], h->center[2]};
  for (int64_t m = blockIdx.x * 8 + (threadIdx.x >> 5); m < nf; m += (int64_t)gridDim.x * 8) {
    double P[3][3];
    corners(v, nv, f, m, c, P);
    float far = 0.f;   // the largest distance of a corner from the centroid, in units of r_max
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int d = 0; d < 3; ++d) P[k][d] *= inv;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float d2 = 0.f;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float e = (float)(P[k][d] - (P[0][d] + P[1][d] + P[2][d]) * (1.0 / 3.0));
        d2 = fmaf(e, e, d2);
      }
      far = fmaxf(far, d2);
    }
    const float y = (float)kTauSmallQ * 1.001f * sqrtf(far);
    int n = 3;
    while (n < 8 && !(y < kGlY[n - 3])) ++n;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int p = lane; p < n * n; p += 32) {
      const int iu = p / n, iw = p - iu * n;
      const double u = kGlX[n - 3][iu], w = kGlX[n - 3][iw];
      double r[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) r[d] = fma(u, fma(w, P[2][d] - P[1][d], P[1][d] - P[0][d]), P[0][d]);
      double val = poly3<double, 0, kPhiLo>(phi.c64, r[0], r[1], r[2]);
      val = fma(phi.scale, (double)poly3<float, kPhiLo + 1, kMomK>(phi.c32, (float)r[0], (float)r[1], (float)r[2]), val);
      val *= kGlW[n - 3][iu] * kGlW[n - 3][iw] * u;
      const double uw = u * w;
      s0 = fma(1.0 - u, val, s0);
      s1 = fma(u - uw, val, s1);
      s2 = fma(uw, val, s2);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (lane == 0) {
      out[3 * m] = s0;
      out[3 * m + 1] = s1;
      out[3 * m + 2] = s2;
    }
  }
}

}  // namespace

cudaError_t launch_small_adjoint3(const float* v, int64_t nv, const int32_t* f, int64_t nf, const double* q,
                                  const double* g, int64_t n_q, WsHeader* h, void* scratch, cudaStream_t st) {
  char* s = static_cast<char*>(scratch);
  k_phi<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(kPhiBlocks, (n_q + 63) / 64)), kNT, 0, st>>>(q, g, n_q, h, s);
  if (cudaError_t e = cudaGetLastError()) return e;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(8 * 152, (nf + 7) / 8));
  k_phi_faces<<<(unsigned)grid, 256, 0, st>>>(v, nv, f, nf, h, s, const_cast<double*>(small_adjoint_faces(s)));
  return cudaGetLastError();
}

cudaError_t launch_small3(const float* v, int64_t nv, const int32_t* f, int64_t nf, const double* q, WsHeader* h,
                          const double* mparts, int n_measure, void* scratch, cudaStream_t st) {
  int dev = 0, sms = 1;
  if (cudaError_t e = cudaGetDevice(&dev)) return e;
  if (cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) return e;
  if (cudaError_t e = cudaFuncSetAttribute(k_small3, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kShared)) return e;
  k_small3<<<(unsigned)small3_blocks(nf, sms), kNT, kShared, st>>>(v, nv, f, nf, q, h, mparts, n_measure,
                                                                  static_cast<char*>(scratch));
  return cudaGetLastError();
}

}  // namespace pft
