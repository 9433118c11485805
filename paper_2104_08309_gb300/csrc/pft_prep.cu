// pft_prep.cu -- input validation, centring, segment/face records, the finalize
// pass (fixed-order FP64 split sum, 1/|Q|^2, translation phase, Q = 0 limit) and
// the FP64 small-|Q| pass.
#include <algorithm>

#include "pft_small.cuh"

namespace pft {

namespace {


template <typename T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  return x;
}

// Fixed-order block sum (tree within warps, then warp 0 over the warp sums).
template <int NT>
__device__ double block_sum(double x, double* sh) {
  x = warp_sum(x);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = x;
  __syncthreads();
  double r = 0.0;
  if (wid == 0) {
    r = (lane < NT / 32) ? sh[lane] : 0.0;
    r = warp_sum(r);
  }
  __syncthreads();
  return r;   // valid in thread 0
}

__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

__device__ __forceinline__ void load_center(const WsHeader* h, int dim, double* c) {
  for (int k = 0; k < dim; ++k)
    c[k] = 0.5 * ((double)ord2f(h->bbox_enc[k]) + (double)ord2f(h->bbox_enc[3 + k]));
}

__global__ void k_init_header(WsHeader* h) {
  uint32_t* w = reinterpret_cast<uint32_t*>(h);
  for (int i = threadIdx.x; i < (int)(sizeof(WsHeader) / 4); i += blockDim.x) w[i] = 0u;
  __syncthreads();
  if (threadIdx.x < 3) h->bbox_enc[threadIdx.x] = 0xffffffffu;   // min slots start above every code
}

template <int D>
__global__ void k_bbox(const float* __restrict__ v, int64_t n, WsHeader* h) {
  float mn[D], mx[D];
#pragma unroll
  for (int c = 0; c < D; ++c) { mn[c] = __int_as_float(0x7f800000); mx[c] = -mn[c]; }
  bool bad = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int c = 0; c < D; ++c) {
      float x = v[i * D + c];
      if (!isfinite(x)) { bad = true; continue; }
      mn[c] = fminf(mn[c], x);
      mx[c] = fmaxf(mx[c], x);
    }
  }
#pragma unroll
  for (int c = 0; c < D; ++c) {
    mn[c] = -warp_max(-mn[c]);
    mx[c] = warp_max(mx[c]);
  }
  const bool any_bad = __any_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0) {
    for (int c = 0; c < D; ++c) {
      if (mn[c] <= mx[c]) {
        atomicMin(&h->bbox_enc[c], f2ord(mn[c]));
        atomicMax(&h->bbox_enc[3 + c], f2ord(mx[c]));
      }
    }
    if (any_bad) set_status(&h->status, ST_NONFINITE);
  }
}

// Few vertices: the header reset and the bounding box in one block, the rest of the grid zeroing an
// optional array (one launch instead of two to four; a launch costs a small call more than the work).
constexpr int kStartT = 1024;
// The line: 16 rounds of the block take 3.5 us in 2D, where 20,000 vertices take 2.8 us in k_bbox's blocks and 1.3 us
// in the reset before it, and a launch more.
constexpr int64_t kStartVerts = 16384;
template <int D>
__global__ void __launch_bounds__(kStartT) k_start(const float* __restrict__ v, int64_t n, WsHeader* h,
                                                   int32_t* __restrict__ zero, int64_t n_zero) {
  __shared__ float red[2][D][kStartT / 32];
  if (blockIdx.x > 0) {
    for (int64_t i = (int64_t)(blockIdx.x - 1) * kStartT + threadIdx.x; i < n_zero; i += (int64_t)(gridDim.x - 1) * kStartT)
      zero[i] = 0;
    return;
  }
  float mn[D], mx[D];
#pragma unroll
  for (int c = 0; c < D; ++c) { mn[c] = __int_as_float(0x7f800000); mx[c] = -mn[c]; }
  bool bad = false;
  for (int64_t i = threadIdx.x; i < n; i += kStartT) {
#pragma unroll
    for (int c = 0; c < D; ++c) {
      const float x = v[i * D + c];
      if (!isfinite(x)) { bad = true; continue; }
      mn[c] = fminf(mn[c], x);
      mx[c] = fmaxf(mx[c], x);
    }
  }
  if (threadIdx.x < (int)(sizeof(WsHeader) / 4)) reinterpret_cast<uint32_t*>(h)[threadIdx.x] = 0u;
#pragma unroll
  for (int c = 0; c < D; ++c) {
    mn[c] = -warp_max(-mn[c]);
    mx[c] = warp_max(mx[c]);
    if ((threadIdx.x & 31) == 0) { red[0][c][threadIdx.x >> 5] = mn[c]; red[1][c][threadIdx.x >> 5] = mx[c]; }
  }
  const bool any_bad = __syncthreads_or(bad);
  if (threadIdx.x < 32) {
    if (threadIdx.x < 3) {   // above every code, as for an axis without a finite coordinate
      h->bbox_enc[threadIdx.x] = 0xffffffffu;
      h->bbox_enc[3 + threadIdx.x] = 0u;
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < D; ++c) {
      const float lo = -warp_max(-red[0][c][threadIdx.x]), hi = warp_max(red[1][c][threadIdx.x]);
      if (threadIdx.x == 0 && lo <= hi) {
        h->bbox_enc[c] = f2ord(lo);
        h->bbox_enc[3 + c] = f2ord(hi);
      }
    }
    if (threadIdx.x == 0 && any_bad) h->status = ST_NONFINITE;
  }
}

__global__ void k_zero_i32(int32_t* p, int64_t n) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) p[i] = 0;
}

// 2D: one thread per vertex j builds the segment j -> next(j) of its loop.
template <bool FP64>
__global__ void __launch_bounds__(kPrepThreads) k_prep2d(const float* __restrict__ v, int64_t nv,
                                                         const int64_t* __restrict__ off, int64_t nl, WsHeader* h,
                                                         void* items, double* partials) {
  __shared__ double sh[kPrepThreads / 32];
  const int64_t j = blockIdx.x * (int64_t)kPrepThreads + threadIdx.x;
  double c[2];
  load_center(h, 2, c);
  if (j <= nl) {   // offset validation (one thread per entry)
    bool ok = true;
    if (j == 0) ok = (off[0] == 0);
    if (j == nl) ok = ok && (off[nl] == nv);
    if (j < nl) ok = ok && (off[j] <= off[j + 1]);
    if (!ok) set_status(&h->status, ST_OFFSETS);
  }
  double area = 0.0;
  float rm = 0.0f;
  if (j < nv) {
    // loop l with off[l] <= j < off[l+1]: last l whose start is <= j
    int64_t lo = 0, hi = nl;   // search in off[0..nl-1]
    while (lo + 1 < hi) {
      int64_t mid = (lo + hi) >> 1;
      if (off[mid] <= j) lo = mid; else hi = mid;
    }
    int64_t s0 = off[lo], s1 = off[lo + 1];
    int64_t k = (j + 1 < s1) ? j + 1 : s0;
    if (k < 0 || k >= nv || j < s0 || j >= s1) {
      set_status(&h->status, ST_OFFSETS);
      k = j;
    }
    double x0 = (double)v[2 * j] - c[0], y0 = (double)v[2 * j + 1] - c[1];
    double x1 = (double)v[2 * k] - c[0], y1 = (double)v[2 * k + 1] - c[1];
    double mx = 0.5 * (x0 + x1), my = 0.5 * (y0 + y1), hx = 0.5 * (x1 - x0), hy = 0.5 * (y1 - y0);
    area = 0.5 * (x0 * y1 - x1 * y0);
    rm = __double2float_ru(sqrt(x0 * x0 + y0 * y0));
    if (FP64) {
      reinterpret_cast<Seg64*>(items)[j] = Seg64{mx, my, hx, hy};
    } else {
      reinterpret_cast<Seg32*>(items)[j] =
          Seg32{(float)mx, (float)my, (float)hx, (float)hy};
    }
  }
  double s = block_sum<kPrepThreads>(area, sh);
  float m = warp_max(rm);
  if ((threadIdx.x & 31) == 0) atomicMax(&h->rmax_bits, __float_as_uint(m));
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
  if (blockIdx.x == 0 && threadIdx.x == 0) { h->center[0] = c[0]; h->center[1] = c[1]; h->center[2] = 0.0; }
}

// 3D: one thread per face.  Bound: FP64 arithmetic (about 80 operations a face), so the blocks are small
// (kPrep3Threads) and the faces spread over all SMs: 256 threads a block, with three FP64 divisions and a
// square root a face, took 13 us for 320 faces as for 20,480.  deg != NULL: counts the corners at each
// vertex (for the vertex adjoint's gather).
template <bool FP64>
__global__ void __launch_bounds__(kPrep3Threads) k_prep3d(const float* __restrict__ v, int64_t nv,
                                                          const int32_t* __restrict__ f, int64_t nf, WsHeader* h,
                                                          void* items, double* partials, int64_t pair_faces,
                                                          int32_t* __restrict__ deg) {
  __shared__ double sh[kPrep3Threads / 32];
  const int64_t m = blockIdx.x * (int64_t)kPrep3Threads + threadIdx.x;
  double c[3];
  load_center(h, 3, c);
  double vol = 0.0;
  float rm = 0.0f;
  if (m < nf) {
    const int32_t i0 = f[3 * m], i1 = f[3 * m + 1], i2 = f[3 * m + 2];
    double g[3] = {0, 0, 0}, q0[3] = {0, 0, 0}, q1[3] = {0, 0, 0}, N[3] = {0, 0, 0};
    bool paired_ok = true;   // a face of a pair: the pair's first edges must be (a, b) and (b, a)
    if (m < pair_faces) {
      const int64_t a = m & ~(int64_t)1;
      paired_ok = f[3 * a] == f[3 * (a + 1) + 1] && f[3 * a + 1] == f[3 * (a + 1)];
    }
    if (i0 < 0 || i1 < 0 || i2 < 0 || i0 >= nv || i1 >= nv || i2 >= nv) {
      set_status(&h->status, ST_INDEX);   // the face is skipped (all-zero record contributes 0)
    } else if (!paired_ok) {
      set_status(&h->status, ST_PAIRS);   // both faces of the pair are skipped
    } else {
      double P[3][3];
      const int32_t id[3] = {i0, i1, i2};
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (deg != nullptr) atomicAdd(&deg[id[k]], 1);
#pragma unroll
        for (int d = 0; d < 3; ++d) P[k][d] = (double)v[3 * (int64_t)id[k] + d] - c[d];
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        g[d] = (P[0][d] + P[1][d] + P[2][d]) * (1.0 / 3.0);
        q0[d] = P[0][d] - g[d];
        q1[d] = P[1][d] - g[d];
      }
      double e1[3] = {P[1][0] - P[0][0], P[1][1] - P[0][1], P[1][2] - P[0][2]};
      double e2[3] = {P[2][0] - P[0][0], P[2][1] - P[0][1], P[2][2] - P[0][2]};
      N[0] = e1[1] * e2[2] - e1[2] * e2[1];
      N[1] = e1[2] * e2[0] - e1[0] * e2[2];
      N[2] = e1[0] * e2[1] - e1[1] * e2[0];
      vol = (P[0][0] * (P[1][1] * P[2][2] - P[1][2] * P[2][1]) + P[0][1] * (P[1][2] * P[2][0] - P[1][0] * P[2][2]) +
             P[0][2] * (P[1][0] * P[2][1] - P[1][1] * P[2][0])) * (1.0 / 6.0);
      double r2 = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) r2 = fmax(r2, P[k][0] * P[k][0] + P[k][1] * P[k][1] + P[k][2] * P[k][2]);
      // an upper bound of the radius: square root in FP32, both steps rounded up (a square beyond the
      // FP32 range keeps FP64's root)
      rm = r2 < 1e38 && r2 > 1e-30 ? __fsqrt_ru(__double2float_ru(r2)) : __double2float_ru(sqrt(r2));
    }
    if (FP64) {
      reinterpret_cast<Face64*>(items)[m] = Face64{g[0], g[1], g[2], q0[0], q0[1], q0[2], q1[0], q1[1], q1[2],
                                                   N[0], N[1], N[2]};
    } else {
      reinterpret_cast<Face32*>(items)[m] =
          Face32{(float)g[0], (float)g[1], (float)g[2],
                 (float)q0[0], (float)q0[1], (float)q0[2], (float)q1[0], (float)q1[1], (float)q1[2],
                 (float)N[0], (float)N[1], (float)N[2]};
    }
  }
  double s = block_sum<kPrep3Threads>(vol, sh);
  float mm = warp_max(rm);
  if ((threadIdx.x & 31) == 0) atomicMax(&h->rmax_bits, __float_as_uint(mm));
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
  if (blockIdx.x == 0 && threadIdx.x == 0) { h->center[0] = c[0]; h->center[1] = c[1]; h->center[2] = c[2]; }
}

// Planar polygon faces (CSR) -> triangles that tile each face with signed areas (exact for
// any planar simple polygon, convex or not), so that the triangle path computes the same
// integral.  The split is by recursive halving: the chain p_i .. p_j closed by its diagonal
// is the triangle (p_i, p_m, p_j), m = (i + j)/2, plus the chains p_i .. p_m and p_m .. p_j,
// starting from p_0 .. p_{n-1}; triangles are numbered in pre-order.  The diagonals' terms
// cancel between neighbouring triangles only up to rounding, and this split keeps their
// total length near perimeter x log2(n) where a fan from p_0 has n - 3 diagonals as long as
// the face (a 65,536-gon's fan loses about 3 decimal digits).
//
// One thread per triangle: triangle t belongs to the face m with off[m] - 2m <= t <
// off[m+1] - 2(m+1), found by bisection, and the pre-order walk from the root finds its
// corners in at most log2(n) + 1 steps.  The first n_faces threads also check the offsets;
// a triangle that would fall outside its face (only with malformed offsets) is written
// degenerate (0, 0, 0), contributes nothing, and sets ST_OFFSETS.
__device__ __forceinline__ void halving_triangle(int64_t n, int64_t t, int64_t& a, int64_t& b, int64_t& c) {
  int64_t i = 0, j = n - 1;
  for (int step = 0; step < 64; ++step) {
    const int64_t m = (i + j) >> 1;
    if (t == 0 || j - i < 2) { a = i; b = m; c = j; return; }
    t -= 1;
    const int64_t nl = m - i - 1 > 0 ? m - i - 1 : 0;   // triangles of the chain i .. m
    if (t < nl) j = m;
    else { t -= nl; i = m; }
  }
  a = b = c = 0;
}

__global__ void k_fan3d(const int32_t* __restrict__ idx, int64_t n_idx, const int64_t* __restrict__ off,
                        int64_t n_faces, int32_t* __restrict__ tris, int64_t n_tris, WsHeader* h) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < n_faces) {
    const int64_t a = off[t], b = off[t + 1];
    if (b - a < 3 || (t == 0 && a != 0) || (t == n_faces - 1 && b != n_idx)) set_status(&h->status, ST_OFFSETS);
  }
  if (t >= n_tris) return;
  int64_t lo = 0, hi = n_faces - 1;   // the largest m with off[m] - 2m <= t
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (off[mid] - 2 * mid <= t) lo = mid;
    else hi = mid - 1;
  }
  const int64_t base = off[lo], n = off[lo + 1] - base;
  const int64_t k = t - (base - 2 * lo);          // this face's triangle number, 0 .. n - 3
  int32_t i0 = 0, i1 = 0, i2 = 0;
  if (base >= 0 && n >= 3 && k >= 0 && k < n - 2 && base + n <= n_idx) {
    int64_t a, b, c;
    halving_triangle(n, k, a, b, c);
    i0 = idx[base + a];
    i1 = idx[base + b];
    i2 = idx[base + c];
  } else {
    set_status(&h->status, ST_OFFSETS);
  }
  tris[3 * t] = i0;
  tris[3 * t + 1] = i1;
  tris[3 * t + 2] = i2;
}

// Finalize: out(Q) = exp(iQ.c) * scale / |Q|^2 * sum_splits partial (fixed order, FP64), at the
// caller's Q: the FP32 pair sums ran at Q rounded to float in coordinates centred on the bounding
// box, where that moves them by ~1e-7 of |S|; in the phase Q.c the same rounding would move the
// result by |c| times it, which for a shape far from the origin is not small.
__device__ __forceinline__ void finish(const double (&Q)[3], double re, double im, const WsHeader* h,
                                       double* __restrict__ out) {
  const double ph = Q[0] * h->center[0] + Q[1] * h->center[1] + Q[2] * h->center[2];
  double sp, cp;
  sincos(ph, &sp, &cp);
  out[0] = re * cp - im * sp;
  out[1] = re * sp + im * cp;
}
__device__ __forceinline__ void split_sum(const double2* __restrict__ partial, int ks, int64_t n_q, int64_t i,
                                          double k, double& re, double& im) {
  re = 0.0;
  im = 0.0;
#pragma unroll 8
  for (int s = 0; s < ks; ++s) {
    const double2 p = partial[(int64_t)s * n_q + i];
    re += p.x;
    im += p.y;
  }
  re *= k;
  im *= k;
}

__global__ void k_finalize2d(const double* __restrict__ q, int64_t n_q, const double2* __restrict__ partial,
                             int ks, WsHeader* h, const double* __restrict__ mparts, int nm, int32_t* small_list,
                             double* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n_q) return;
  const double Q[3] = {q[2 * i], q[2 * i + 1], 0.0};
  const double q2 = q_norm2(Q[0], Q[1], Q[2]);
  if (q2 == 0.0) {
    double s = 0.0;
    for (int b = 0; b < nm; ++b) s += mparts[b];
    out[2 * i] = s;
    out[2 * i + 1] = 0.0;
    return;
  }
  if (small_q(q2, __uint_as_float(h->rmax_bits))) {
    small_list[atomicAdd(&h->small_q_count, 1u)] = (int32_t)i;
    return;
  }
  double re, im;
  split_sum(partial, ks, n_q, i, 2.0 / q2, re, im);   // records hold half edge vectors
  finish(Q, re, im, h, out + 2 * i);
}

// 3D: small-|Q| points (as k_fwd listed them) take their sum from k_small3's results, or over the faces of a
// small mesh.  A block finishes per_block = 2 .. 256 points (a power of two), one per thread; those that need
// the moments' polynomial, or the (point, 32 faces) of a direct sum, are dealt to its warps.  With fewer points than threads, 256 / per_block lanes of a warp add a point's chunk
// sums side by side (in a fixed order): one thread per point walked 640 chunks in 50 us for 1,000 points
// (81,920 faces x 1,000 Q at 640 chunks: the call 237 us, 166 us so).
constexpr int kFinT = 256;
constexpr int kFewPts = 32;   // points of one round of the direct sums
__global__ void __launch_bounds__(kFinT) k_finalize3d(const float* __restrict__ v, int64_t nv,
                                                      const int32_t* __restrict__ f, int64_t nf,
                                                      const double* __restrict__ q, int64_t n_q,
                                                      const double2* __restrict__ partial, int ks,
                                                      const WsHeader* __restrict__ h,
                                                      const int32_t* __restrict__ small,
                                                      const char* __restrict__ scratch, double* __restrict__ out,
                                                      int per_block) {
  __shared__ double mom[kMomN];
  __shared__ double at[kFinT][3];   // a point's Q (scaled, for the moments), then its result
  __shared__ double few_sums[kFewPts * (kFewFaces / 32)][2];
  __shared__ int list[kFinT];
  __shared__ int n_list;
  __shared__ double sums[kFinT / 2][2];
  __shared__ bool need[kFinT / 2];
  const int t = threadIdx.x;
  const int64_t i = blockIdx.x * (int64_t)per_block + t;
  const bool mine = t < per_block && i < n_q;
  const float rmax = __uint_as_float(h->rmax_bits);
  const bool few = small_few(h->small_q_count, nf), direct = !few && h->small_q_count <= (uint32_t)kSmallDirect;
  double Q[3] = {0.0, 0.0, 0.0}, q2 = 0.0;
  bool is_small = false;
  if (mine) {
    for (int d = 0; d < 3; ++d) Q[d] = q[3 * i + d];
    q2 = q_norm2(Q[0], Q[1], Q[2]);
    is_small = q2 != 0.0 && small_q(q2, rmax);
  }
  if (!direct) {   // uniform
    if (t == 0) n_list = 0;
    if (__syncthreads_or(is_small)) {
      const double unit = few ? 1.0 : (double)rmax;
      if (is_small) {
        for (int d = 0; d < 3; ++d) at[t][d] = Q[d] * unit;
        list[atomicAdd(&n_list, 1)] = t;   // their order is immaterial
      }
      if (!few)
        for (int j = t; j < kMomN; j += kFinT) mom[j] = reinterpret_cast<const double*>(scratch)[j];
      __syncthreads();
      if (few) {
        const double c[3] = {h->center[0], h->center[1], h->center[2]};
        const int ng = (int)((nf + 31) / 32);
        for (int e0 = 0; e0 < n_list; e0 += kFewPts) {   // uniform
          const int cnt = min(kFewPts, n_list - e0);
          for (int u = t >> 5; u < cnt * ng; u += kFinT / 32) {
            const int l = list[e0 + u / ng], m = (u % ng) * 32 + (t & 31);
            double P[3][3], re = 0.0, im = 0.0;
            if (m < nf && corners(v, nv, f, m, c, P)) {
              double x[3];
              for (int k = 0; k < 3; ++k) x[k] = at[l][0] * P[k][0] + at[l][1] * P[k][1] + at[l][2] * P[k][2];
              const double det = det3(P);
              tetra_series(x, re, im);
              re *= det;
              im *= det;
            }
            re = warp_sum(re);
            im = warp_sum(im);
            if ((t & 31) == 0) {
              few_sums[u][0] = re;
              few_sums[u][1] = im;
            }
          }
          __syncthreads();
          if (t < 2 * cnt) {
            double s = 0.0;
            for (int k = 0; k < ng; ++k) s += few_sums[(t >> 1) * ng + k][t & 1];
            at[list[e0 + (t >> 1)]][t & 1] = s;
          }
          __syncthreads();
        }
      } else {
        for (int e = t >> 5; e < n_list; e += kFinT / 32) {
          const int l = list[e];
          double re, im, g[3][2];
          mom_eval<false>(mom, at[l][0], at[l][1], at[l][2], re, im, g);
          __syncwarp();
          if ((t & 31) == 0) {
            at[l][0] = re;
            at[l][1] = im;
          }
        }
        __syncthreads();
      }
    }
  }
  const int lanes = ks > 16 ? kFinT / per_block : 1;   // uniform; up to 16 chunks are two rounds of loads anyway
  if (lanes > 1) {
    if (t < per_block) need[t] = mine && q2 != 0.0 && !is_small;
    __syncthreads();
    const int p = t / lanes;
    double a = 0.0, b = 0.0;
    if (need[p]) {
      const double2* row = partial + blockIdx.x * (int64_t)per_block + p;
#pragma unroll 4
      for (int s = t % lanes; s < ks; s += lanes) {
        const double2 x = row[(int64_t)s * n_q];
        a += x.x;
        b += x.y;
      }
    }
    for (int o = lanes / 2; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (t % lanes == 0) {
      sums[p][0] = a;
      sums[p][1] = b;
    }
    __syncthreads();
  }
  if (!mine) return;
  if (q2 == 0.0) {
    out[2 * i] = h->measure;
    out[2 * i + 1] = 0.0;
    return;
  }
  double re = 0.0, im = 0.0;
  if (!is_small && lanes > 1) {
    const double k = 1.0 / q2;
    re = sums[t][0] * k;
    im = sums[t][1] * k;
  } else if (!is_small) {
    split_sum(partial, ks, n_q, i, 1.0 / q2, re, im);
  } else if (direct) {
    const int64_t nch = small3_chunks(nf);
    const double* p = reinterpret_cast<const double*>(scratch + kMomHead) + 2 * nch * small[i];
    for (int64_t c = 0; c < nch; ++c) {
      re += p[2 * c];
      im += p[2 * c + 1];
    }
  } else {
    re = at[t][0];
    im = at[t][1];
  }
  finish(Q, re, im, h, out + 2 * i);
}

constexpr int kSmallThreads = 256;

// Small |Q| in 2D: fan of signed triangles (c, p_j, p_{j+1}).
__global__ void __launch_bounds__(kSmallThreads) k_smallq2d(const float* __restrict__ v, int64_t nv,
                                                            const int64_t* __restrict__ off, int64_t nl,
                                                            const double* __restrict__ q, const WsHeader* h,
                                                            const int32_t* list, double* __restrict__ out) {
  __shared__ double sh[kSmallThreads / 32];
  const uint32_t count = h->small_q_count;
  const double c[2] = {h->center[0], h->center[1]};
  for (uint32_t e = blockIdx.x; e < count; e += gridDim.x) {
    const int64_t i = list[e];
    double Q[2];
    for (int d = 0; d < 2; ++d) Q[d] = q[2 * i + d];   // the caller's Q (FP64 series)
    double re = 0.0, im = 0.0;
    for (int64_t j = threadIdx.x; j < nv; j += kSmallThreads) {
      int64_t lo = 0, hi = nl;
      while (lo + 1 < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (off[mid] <= j) lo = mid; else hi = mid;
      }
      int64_t s0 = off[lo], s1 = off[lo + 1];
      int64_t k = (j + 1 < s1) ? j + 1 : s0;
      if (k < 0 || k >= nv) continue;
      const double x0 = (double)v[2 * j] - c[0], y0 = (double)v[2 * j + 1] - c[1];
      const double x1 = (double)v[2 * k] - c[0], y1 = (double)v[2 * k + 1] - c[1];
      const double x[2] = {Q[0] * x0 + Q[1] * y0, Q[0] * x1 + Q[1] * y1};
      double sr, si;
      simplex_series<2, 2, 16>(x, sr, si);
      const double det = x0 * y1 - x1 * y0;
      re += det * sr;
      im += det * si;
    }
    re = block_sum<kSmallThreads>(re, sh);
    im = block_sum<kSmallThreads>(im, sh);
    if (threadIdx.x == 0) {
      double sp, cp;
      sincos(Q[0] * c[0] + Q[1] * c[1], &sp, &cp);
      out[2 * i] = re * cp - im * sp;
      out[2 * i + 1] = re * sp + im * cp;
    }
  }
}

}  // namespace

cudaError_t launch_init_header(WsHeader* h, cudaStream_t st) {
  k_init_header<<<1, 64, 0, st>>>(h);
  return cudaGetLastError();
}

cudaError_t launch_start(const float* v, int64_t n, int dim, WsHeader* h, cudaStream_t st, int* launches,
                         int32_t* zero, int64_t n_zero) {
  if (n <= kStartVerts) {
    const unsigned grid = 1 + (unsigned)std::min<int64_t>(256, (n_zero + kStartT - 1) / kStartT);
    if (dim == 2) k_start<2><<<grid, kStartT, 0, st>>>(v, n, h, zero, n_zero);
    else k_start<3><<<grid, kStartT, 0, st>>>(v, n, h, zero, n_zero);
    ++*launches;
    return cudaGetLastError();
  }
  if (cudaError_t e = launch_init_header(h, st)) return e;
  const int blocks = (int)std::min<int64_t>(1024, (n + 255) / 256);
  if (dim == 2) k_bbox<2><<<blocks, 256, 0, st>>>(v, n, h);
  else k_bbox<3><<<blocks, 256, 0, st>>>(v, n, h);
  *launches += 2;
  if (n_zero > 0) {
    k_zero_i32<<<(unsigned)((n_zero + 255) / 256), 256, 0, st>>>(zero, n_zero);
    ++*launches;
  }
  return cudaGetLastError();
}

cudaError_t launch_prep2d(const float* v, int64_t nv, const int64_t* off, int64_t nl, WsHeader* h, void* segs,
                          bool fp64, double* partials, int nblk, cudaStream_t st) {
  // at least enough threads to validate all nl + 1 offsets
  const int need = prep_blocks(std::max<int64_t>(nv, nl + 1));
  if (need != nblk) return cudaErrorInvalidValue;
  if (fp64) k_prep2d<true><<<nblk, kPrepThreads, 0, st>>>(v, nv, off, nl, h, segs, partials);
  else k_prep2d<false><<<nblk, kPrepThreads, 0, st>>>(v, nv, off, nl, h, segs, partials);
  return cudaGetLastError();
}

cudaError_t launch_prep3d(const float* v, int64_t nv, const int32_t* f, int64_t nf, WsHeader* h, void* faces,
                          bool fp64, double* partials, int nblk, cudaStream_t st, int64_t pair_faces, int32_t* deg) {
  if (nblk != prep3_blocks(nf)) return cudaErrorInvalidValue;
  if (fp64) k_prep3d<true><<<nblk, kPrep3Threads, 0, st>>>(v, nv, f, nf, h, faces, partials, pair_faces, deg);
  else k_prep3d<false><<<nblk, kPrep3Threads, 0, st>>>(v, nv, f, nf, h, faces, partials, pair_faces, deg);
  return cudaGetLastError();
}

cudaError_t launch_fan3d(const int32_t* idx, int64_t n_idx, const int64_t* off, int64_t n_faces, int32_t* tris,
                         int64_t n_tris, WsHeader* h, cudaStream_t st) {
  const int64_t n = std::max(n_tris, n_faces);
  const int64_t blocks = std::max<int64_t>(1, (n + 255) / 256);
  if (blocks > INT32_MAX) return cudaErrorInvalidValue;
  k_fan3d<<<(unsigned)blocks, 256, 0, st>>>(idx, n_idx, off, n_faces, tris, n_tris, h);
  return cudaGetLastError();
}

// Points per block of the finishing kernels: few enough that a small call's FP64 arithmetic (the phase's
// sincos, the small-|Q| polynomial) spreads over all SMs.
static int finish_points(int64_t n_q, int least) {
  int n = 256;
  while (n > least && n_q < (int64_t)n * 256) n /= 2;
  return n;
}

cudaError_t launch_finalize2d(const double* q, int64_t n_q, const double2* partial, int k_splits, WsHeader* h,
                              const double* mparts, int nm, int32_t* small_list, double* out, cudaStream_t st) {
  const int nt = finish_points(n_q, 32);
  k_finalize2d<<<(unsigned)((n_q + nt - 1) / nt), nt, 0, st>>>(q, n_q, partial, k_splits, h, mparts, nm, small_list,
                                                              out);
  return cudaGetLastError();
}

cudaError_t launch_finalize3d(const float* v, int64_t nv, const int32_t* f, int64_t nf, const double* q, int64_t n_q,
                              const double2* partial, int k_splits, const WsHeader* h, const int32_t* small,
                              const void* scratch, double* out, cudaStream_t st) {
  // side-by-side chunk sums take a warp's lanes a point at most, so 8 points or more
  const int per = finish_points(n_q, nf <= kFewFaces && k_splits <= 16 ? 2 : 8);
  k_finalize3d<<<(unsigned)((n_q + per - 1) / per), kFinT, 0, st>>>(v, nv, f, nf, q, n_q, partial, k_splits, h, small,
                                                                   static_cast<const char*>(scratch), out, per);
  return cudaGetLastError();
}

cudaError_t launch_smallq2d(const float* v, int64_t nv, const int64_t* off, int64_t nl, const double* q,
                            const WsHeader* h, const int32_t* list, double* out, cudaStream_t st) {
  k_smallq2d<<<device_sms(), kSmallThreads, 0, st>>>(v, nv, off, nl, q, h, list, out);
  return cudaGetLastError();
}

}  // namespace pft
