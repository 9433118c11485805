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
constexpr int kGW = kNW / 2;   // warps that sum the FP64 degrees; the others sum the FP32 ones
constexpr int slots_of(int k) { return (rows_of(k) + kGW - 1) / kGW; }
// accumulator slots of the degrees lo .. k - 1
constexpr int slot_base(int lo, int k) {
  int n = 0;
  for (int d = lo; d < k; ++d) n += slots_of(d);
  return n;
}
constexpr int kSlots64 = slot_base(0, kMomLo + 1);            // 19
constexpr int kSlots32 = slot_base(kMomLo + 1, kMomK + 1);    // 44

// 1/n!
struct InvFact { double v[16]; };
constexpr InvFact make_inv_fact() {
  InvFact t{};
  double f = 1.0;
  for (int n = 0; n < 16; ++n) {
    if (n > 1) f *= n;
    t.v[n] = 1.0 / f;
  }
  return t;
}
__constant__ InvFact kInvFact = make_inv_fact();

// Accumulators of a thread: one per slot in FP64; in FP32 the slot's 32 faces are added by shuffles and
// lane slot % 32 keeps the sum (44 compensated sums a thread would not fit the registers).
struct Sum64 {
  double v[kSlots64];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < kSlots64; ++i) v[i] = 0.0;
  }
  __device__ __forceinline__ void add(int slot, double a, double b, int) { v[slot] = fma(a, b, v[slot]); }
};
struct Sum32 {
  CAcc v[(kSlots32 + 31) / 32];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int i = 0; i < (kSlots32 + 31) / 32; ++i) v[i].init();
  }
  __device__ __forceinline__ void add(int slot, float a, float b, int lane) {
    float x = a * b;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == slot % 32) v[slot / 32].add(x);
  }
};
// Barrier of one half of the block (id 1: the FP64 warps, 2: the FP32 warps).
__device__ __forceinline__ void half_sync(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kGW * 32) : "memory"); }
// Barrier of the whole block for code where the halves are in different branches: __syncthreads() there would be
// two barriers of the source, reached on a condition that is not the same for the block.
__device__ __forceinline__ void both_sync() { asm volatile("bar.sync 3, %0;" ::"n"(kNT) : "memory"); }

// One batch of 32 faces, one per lane, over kGW warps: the coefficients of h_k(x0, x1, x2) as
// polynomials in Q, x_j = Q.p_j, degree by degree.  The complete homogeneous polynomials obey
//   H_j[k] = H_{j-1}[k] + x_j H_j[k-1]   (nodes 0 .. j, H_{-1}[k] = 0 for k > 0, H[0] = 1),
// so the coefficient of a monomial takes one fused multiply-add per node and per neighbour of the
// degree below (same row, row of y, row of z).  A warp holds whole monomials (the neighbours are
// then warp-uniform) and a lane one face; two levels of the three nodes' coefficients live in
// shared memory.  det times the last node's coefficient of the degrees KLO .. KHI is summed.
template <class T, class Sum, int KLO, int KHI, int K = 0>
__device__ __forceinline__ void batch(const T (&P)[3][3], T det, T* buf, Sum& acc, int lane, int warp, int id) {
  constexpr int W = rows_of(KHI - 1) * 32;     // one level of one node
  constexpr int S = slots_of(K), base = slot_base(KLO, K < KLO ? KLO : K);
  T* cur = buf + (K & 1) * 3 * W;
  const T* old = buf + ((K & 1) ^ 1) * 3 * W;
  T H[S][3];   // read the level below first, write this one after: loads are not held up by stores
#pragma unroll
  for (int i = 0; i < S; ++i) {
    const int m = warp + kGW * i;
    if (K == 0) {
      H[i][0] = H[i][1] = H[i][2] = (T)1;
    } else if (m < rows_of(K)) {
      const int s = kRows.s[m], c = kRows.c[m], ny = (s - 1) * s / 2 + c;
      T h = (T)0;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const T* o = old + j * W;
        if (s < K) h = fma(P[j][0], o[m * 32 + lane], h);
        if (c < s) h = fma(P[j][1], o[ny * 32 + lane], h);
        if (c > 0) h = fma(P[j][2], o[(ny - 1) * 32 + lane], h);
        H[i][j] = h;
      }
    }
  }
  if constexpr (K >= KLO) {
#pragma unroll
    for (int i = 0; i < S; ++i)
      if (warp + kGW * i < rows_of(K)) acc.add(base + i, det, H[i][2], lane);
  }
  if (K < KHI) {
#pragma unroll
    for (int i = 0; i < S; ++i) {
      const int m = warp + kGW * i;
      if (m < rows_of(K))
#pragma unroll
        for (int j = 0; j < 3; ++j) cur[j * W + m * 32 + lane] = H[i][j];
    }
  }
  half_sync(id);
  if constexpr (K < KHI) batch<T, Sum, KLO, KHI, K + 1>(P, det, buf, acc, lane, warp, id);
}

__device__ __forceinline__ double wsum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  return x;
}

// dynamic shared memory: two levels of three nodes' coefficients in FP64 (then the lanes' sums) and FP32
constexpr size_t kBuf64 = 2 * 3 * (size_t)rows_of(kMomLo - 1) * 32 * sizeof(double);
constexpr size_t kBuf32 = 2 * 3 * (size_t)rows_of(kMomK - 1) * 32 * sizeof(float);
constexpr size_t kRed = (size_t)kMomN64 * 33 * sizeof(double);
constexpr size_t kHalf64 = kBuf64 > kRed ? kBuf64 : kRed;
constexpr size_t kShared = kHalf64 + kBuf32;

// The last block to finish adds the blocks' partial moments (in a fixed order) and scales them:
// (-1)^(k/2)/(k+3)!, the sign of i^k = (-1)^(k/2) (1 or i).
__device__ void sum_moments(const char* parts, int nb, double r3, double* out) {
  constexpr int kBatch = 20;
  const int part = threadIdx.x & 3;   // four threads a moment
  for (int t = threadIdx.x >> 2; t < ((kMomN + 7) & ~7); t += kNT / 4) {   // whole warps
    double s = 0.0;
    CAcc a;
    a.init();
    const bool wide = t < kMomN64;
    const char* p = parts + (wide ? 8 * t : 8 * min(t, kMomN - 1));   // the float pairs follow the doubles
    for (int b0 = part; b0 < nb; b0 += 4 * kBatch) {   // kBatch loads in flight
      double x[kBatch];
#pragma unroll
      for (int j = 0; j < kBatch; ++j)
        x[j] = b0 + 4 * j < nb ? *reinterpret_cast<const double*>(p + (size_t)(b0 + 4 * j) * kMomPart) : 0.0;
      if (wide) {
#pragma unroll
        for (int j = 0; j < kBatch; ++j) s += x[j];
      } else {
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {   // a float pair (zeros past the end)
          a.add(__int_as_float(__double2loint(x[j])));
          a.lo += __int_as_float(__double2hiint(x[j]));
        }
      }
    }
    if (!wide) s = ((double)a.hi + (double)a.lo) * r3;
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (part != 0 || t >= kMomN) continue;
    int k = 0;
    while (mom_count(k) <= t) ++k;
    const int m = t - k * (k + 1) * (k + 2) / 6, sr = kRows.s[m], c = kRows.c[m];
    const double w = kInvFact.v[k + 3];
    out[mom_pos(k - sr, sr - c, c)] = (k & 2) ? -s * w : s * w;
  }
}

// Bound: the moments are FP64 work (876 fused multiply-adds a face in FP64, 3,600 in FP32, at 2
// and 128 a clock and SM): 7 us of the FP64 pipe for a batch of 32 faces, where a round takes 18 (the 13 levels'
// barriers and their first loads from shared memory).  One block
// of 16 warps per SM, half of them on the FP64 degrees and half on the FP32 ones of the same faces, so
// that the FP32 work and the short first levels' latencies hide behind the other half.  20,480 faces
// (5 rounds): 102 us; with all 16 warps on one type after the other 148 us.
__global__ void __launch_bounds__(kNT) k_small3(const float* __restrict__ v, int64_t nv,
                                                const int32_t* __restrict__ f, int64_t nf,
                                                const double* __restrict__ q, WsHeader* h,
                                                const double* __restrict__ mparts, int n_measure, char* scratch) {
  extern __shared__ __align__(16) char sh[];
  __shared__ double red[kNW][2];
  __shared__ double face64[2][10][32];
  __shared__ float face32[2][10][32];
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
  if (count == 0 || (q != nullptr ? small_few(count, nf) : qsmall_direct(count, nf))) return;
  const double c[3] = {h->center[0], h->center[1], h->center[2]};
  char* parts = scratch + kMomHead;
  if (q != nullptr && count <= (uint32_t)kSmallDirect) {
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
  const int64_t batches = (nf + kMomFaces - 1) / kMomFaces;
  char* mine = parts + (size_t)blockIdx.x * kMomPart;
  // One warp prepares a batch for all (its conversions and determinants are FP64 work): coordinates in
  // units of r_max and det, component by component, for the FP64 half and (det in units of r_max^3: it
  // could leave the FP32 range otherwise; scaled back at the end) for the FP32 half.
  auto load = [&](int64_t b, int slot) {
    const int64_t m = b * kMomFaces + lane;
    double P[3][3], det = 0.0;
    if (m < nf) {
      corners(v, nv, f, m, c, P);
      det = det3(P);
    } else {
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int d = 0; d < 3; ++d) P[k][d] = 0.0;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double x = P[k][d] * inv;
        face64[slot][3 * k + d][lane] = x;
        face32[slot][3 * k + d][lane] = (float)x;
      }
    face64[slot][9][lane] = det;
    face32[slot][9][lane] = (float)(det * inv * inv * inv);
  };
  constexpr int kLoader = kNW - 1;   // a warp of the FP32 half loads a batch ahead
  if (warp == kLoader) load(blockIdx.x, 0);
  __syncthreads();
  if (warp < kGW) {
    Sum64 a64;
    a64.init();
    double* buf = reinterpret_cast<double*>(sh);
    int slot = 0;
    for (int64_t b = blockIdx.x; b < batches; b += gridDim.x, slot ^= 1) {
      double P[3][3];
#pragma unroll
      for (int k = 0; k < 9; ++k) P[k / 3][k % 3] = face64[slot][k][lane];
      batch<double, Sum64, 0, kMomLo>(P, face64[slot][9][lane], buf, a64, lane, warp, 1);
      both_sync();
    }
    // lanes -> one sum per monomial through shared memory (33 doubles a row: no bank conflicts)
#pragma unroll
    for (int k = 0; k <= kMomLo; ++k)
#pragma unroll
      for (int i = 0; i < slots_of(k); ++i) {
        const int m = warp + kGW * i;
        if (m < rows_of(k)) buf[(mom_count(k - 1) + m) * 33 + lane] = a64.v[slot_base(0, k) + i];
      }
    half_sync(1);
    const int t = threadIdx.x >> 1, part = threadIdx.x & 1;   // two threads a monomial, 16 lanes each
    double s = 0.0;
    if (t < kMomN64)
      for (int l = 0; l < 16; ++l) s += buf[t * 33 + 16 * part + l];
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (t < kMomN64 && part == 0) reinterpret_cast<double*>(mine)[t] = s;
  } else {
    Sum32 a32;
    a32.init();
    float* buf = reinterpret_cast<float*>(sh + kHalf64);
    int slot = 0;
    for (int64_t b = blockIdx.x; b < batches; b += gridDim.x, slot ^= 1) {
      if (warp == kLoader && b + gridDim.x < batches) load(b + gridDim.x, slot ^ 1);
      float P[3][3];
#pragma unroll
      for (int k = 0; k < 9; ++k) P[k / 3][k % 3] = face32[slot][k][lane];
      batch<float, Sum32, kMomLo + 1, kMomK>(P, face32[slot][9][lane], buf, a32, lane, warp - kGW, 2);
      both_sync();
    }
#pragma unroll
    for (int k = kMomLo + 1; k <= kMomK; ++k)
#pragma unroll
      for (int i = 0; i < slots_of(k); ++i) {
        const int m = warp - kGW + kGW * i, slot = slot_base(kMomLo + 1, k) + i;
        if (m < rows_of(k) && lane == slot % 32)
          reinterpret_cast<float2*>(mine + kMomN64 * 8)[mom_count(k - 1) + m - kMomN64] =
              make_float2(a32.v[slot / 32].hi, a32.v[slot / 32].lo);
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
#pragma unroll 32
    for (unsigned u = 0; u < gridDim.x; ++u) sum += parts[(size_t)u * kMomN + t];
    // Re(i w) = -Im w: the sign of i^k over the real (k even) or imaginary (k odd) part
    sum *= (((k + 1) & 2) ? -kInvFact.v[a] : kInvFact.v[a]) * (kInvFact.v[b] * kInvFact.v[c]);
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
#pragma unroll
  for (int b = KHI; b >= 0; --b) {
    asm volatile("" ::: "memory");   // keeps the coefficients' loads of one b together (fewer spills)
    T rz = (T)0;
#pragma unroll
    for (int c = KHI - b; c >= 0; --c) {
      const int s = b + c, row = s * (s + 1) / 2 + c, alo = KLO > s ? KLO - s : 0;
      T rx = (T)0;
#pragma unroll
      for (int a = KHI - s; a >= 0; --a) {
        const int k = a + s;
        rx = a >= alo ? fma(rx, x, C[k * (k + 1) * (k + 2) / 6 - mom_count(KLO - 1) + row]) : rx * x;
      }
      rz = fma(rz, z, rx);
    }
    r = fma(r, y, rz);
  }
  return r;
}

// Quadrature on a triangle (barycentric l1, l2 and weight; the weights add to 1/2).  For faces whose
// phases about their centroid stay below kPhiNear, Dunavant's rule of degree 8 (Int. J. Numer. Methods
// Eng. 21, 1985), 16 points: lambda_k times the terms of degree <= 7 of Phi, the next being below
// kPhiNear^8/8! = 1e-17.  For larger faces n x n Gauss-Legendre points (Abramowitz & Stegun, table 25.4)
// in collapsed coordinates r = p0 + u ((p1 - p0) + w (p2 - p1)), element u du dw: degree 2n - 3 of Phi,
// n = 8 exact for all 12 degrees.
constexpr float kPhiNear = 0.028f;
__constant__ float kPhiFar[2] = {9.0e-2f, 0.20f};   // n = 6, 7: y^(2n-2)/(2n-2)! = 1e-17
struct Rule16 { double l1[16], l2[16], w[16]; };
constexpr Rule16 make_rule16() {
  Rule16 r{};
  int n = 0;
  auto put = [&](double l1, double l2, double w) {
    r.l1[n] = l1;
    r.l2[n] = l2;
    r.w[n] = 0.5 * w;
    ++n;
  };
  put(1.0 / 3, 1.0 / 3, 0.14431560767778717);
  const double a[3] = {0.4592925882927232, 0.1705693077517602, 0.05054722831703098};
  const double w[3] = {0.09509163426728462, 0.10321737053471824, 0.03245849762319808};
  for (int k = 0; k < 3; ++k) {
    put(a[k], a[k], w[k]);
    put(1.0 - 2.0 * a[k], a[k], w[k]);
    put(a[k], 1.0 - 2.0 * a[k], w[k]);
  }
  const double b = 0.2631128296346381, c = 0.008394777409957605, d = 1.0 - b - c;
  const double p[6][2] = {{b, c}, {c, b}, {b, d}, {d, b}, {c, d}, {d, c}};
  for (int k = 0; k < 6; ++k) put(p[k][0], p[k][1], 0.027230314174434993);
  return r;
}
__constant__ Rule16 kRule16 = make_rule16();
__constant__ double kGlX[3][8] = {
    {0.03376524289842403, 0.16939530676686776, 0.38069040695840156, 0.6193095930415985, 0.8306046932331322,
     0.9662347571015759},
    {0.0254460438286207, 0.12923440720030277, 0.2970774243113014, 0.5, 0.7029225756886985, 0.8707655927996972,
     0.9745539561713793},
    {0.019855071751231912, 0.10166676129318664, 0.2372337950418355, 0.4082826787521751, 0.5917173212478248,
     0.7627662049581645, 0.8983332387068134, 0.9801449282487681}};
__constant__ double kGlW[3][8] = {
    {0.08566224618958514, 0.18038078652406936, 0.23395696728634552, 0.23395696728634552, 0.18038078652406936,
     0.08566224618958514},
    {0.06474248308443487, 0.13985269574463843, 0.19091502525255935, 0.20897959183673465, 0.19091502525255935,
     0.13985269574463843, 0.06474248308443487},
    {0.05061426814518853, 0.11119051722668721, 0.15685332293894344, 0.18134189168918083, 0.18134189168918083,
     0.15685332293894344, 0.11119051722668721, 0.05061426814518853}};

// Half a warp per face, one quadrature point per lane and round.  Bound: FP64, about 170 operations a
// point (a warp's instruction takes 16 cycles of the SM's pipe).  5,120 faces: 57 us (a warp per face
// with 25 Gauss points each: 100 us).
__global__ void __launch_bounds__(256, 2) k_phi_faces(const float* __restrict__ v, int64_t nv,
                                                      const int32_t* __restrict__ f, int64_t nf,
                                                      const WsHeader* __restrict__ h,
                                                      const char* __restrict__ scratch, double* __restrict__ out) {
  __shared__ PhiPoly phi;
  if (h->small_q_count <= (uint32_t)kSmallAdjoint) return;
  for (int t = threadIdx.x; t < (int)(sizeof(PhiPoly) / 4); t += 256)
    reinterpret_cast<uint32_t*>(&phi)[t] = reinterpret_cast<const uint32_t*>(scratch)[t];
  __syncthreads();
  const int lane = threadIdx.x & 15;
  const float rmax = __uint_as_float(h->rmax_bits);
  const double inv = rmax > 0.f ? 1.0 / (double)rmax : 0.0;
  const double c[3] = {h->center[0], h->center[1], h->center[2]};
  // the two halves of a warp run the same rounds (the shuffles take the whole warp)
  for (int64_t m0 = blockIdx.x * 16; m0 < nf; m0 += (int64_t)gridDim.x * 16) {
    const int64_t m = m0 + (threadIdx.x >> 4);
    double P[3][3];
    corners(v, nv, f, min(m, nf - 1), c, P);
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
    const bool near = y < kPhiNear;
    const int n = y < kPhiFar[0] ? 6 : (y < kPhiFar[1] ? 7 : 8), points = near ? 16 : n * n;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int p = lane; p < points; p += 16) {
      double l1, l2, w;
      if (near) {
        l1 = kRule16.l1[p];
        l2 = kRule16.l2[p];
        w = kRule16.w[p];
      } else {
        const int iu = p / n, iw = p - iu * n;
        const double u = kGlX[n - 6][iu], t = kGlX[n - 6][iw];
        w = kGlW[n - 6][iu] * kGlW[n - 6][iw] * u;
        l2 = u * t;
        l1 = u - l2;
      }
      double r[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) r[d] = fma(l1, P[1][d] - P[0][d], fma(l2, P[2][d] - P[0][d], P[0][d]));
      double val = poly3<double, 0, kPhiLo>(phi.c64, r[0], r[1], r[2]);
      val = fma(phi.scale, (double)poly3<float, kPhiLo + 1, kMomK>(phi.c32, (float)r[0], (float)r[1], (float)r[2]), val);
      val *= w;
      s1 = fma(l1, val, s1);
      s2 = fma(l2, val, s2);
      s0 += val;   // lambda_0 = 1 - l1 - l2
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (lane == 0 && m < nf) {
      out[3 * m] = s0 - s1 - s2;
      out[3 * m + 1] = s1;
      out[3 * m + 2] = s2;
    }
  }
}

}  // namespace

cudaError_t launch_small_adjoint3(const float* v, int64_t nv, const int32_t* f, int64_t nf, const double* q,
                                  const double* g, int64_t n_q, WsHeader* h, void* scratch, cudaStream_t st) {
  char* s = static_cast<char*>(scratch);
  k_phi<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(kPhiBlocks, (n_q + 7) / 8)), kNT, 0, st>>>(q, g, n_q, h, s);
  if (cudaError_t e = cudaGetLastError()) return e;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(16 * device_sms(), (nf + 15) / 16));
  k_phi_faces<<<(unsigned)grid, 256, 0, st>>>(v, nv, f, nf, h, s, const_cast<double*>(small_adjoint_faces(s)));
  return cudaGetLastError();
}

cudaError_t launch_small3(const float* v, int64_t nv, const int32_t* f, int64_t nf, const double* q, WsHeader* h,
                          const double* mparts, int n_measure, void* scratch, cudaStream_t st) {
  const int sms = device_sms();
  if (cudaError_t e = cudaFuncSetAttribute(k_small3, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kShared)) return e;
  k_small3<<<(unsigned)small3_blocks(nf, sms), kNT, kShared, st>>>(v, nv, f, nf, q, h, mparts, n_measure,
                                                                  static_cast<char*>(scratch));
  return cudaGetLastError();
}

}  // namespace pft
