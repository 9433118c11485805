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

// dynamic shared memory: two levels of three nodes' coefficients (FP32: 12 * 91 * 2 ...)
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

}  // namespace

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
