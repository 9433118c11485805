// pft_fwd.cu -- the hot loop: every (Q, segment) or (Q, face) pair of the
// divergence-theorem sum.
//
// Mapping: each thread owns R Q points in registers; a block covers NT*R Q
// points and one chunk of the segments/faces (blockIdx.y, split-K).  Segment or
// face records stream through shared memory in tiles moved by bulk copies
// (cp.async.bulk, TMA) into a STAGES-deep ring guarded by mbarriers; one thread
// issues the copies, every thread reads each record as a broadcast.  Sums are
// per thread and in a fixed order: FP32 within a tile, error-free (TwoSum)
// compensation across tiles; the per-chunk partials are added in FP64 by the
// finalize kernel.  No atomics on data, so results are deterministic.
#include <atomic>

#include "pft_pairs.cuh"

namespace pft {
namespace {

// ---------------------------------------------------------------------------
// The main kernel: bulk-copy ring of record tiles, R Q points per thread.
//
// Ring protocol (no block-wide barrier inside the loop): full[s] completes when
// the bulk copy of the tile in slot s has landed (expect_tx by the issuing
// thread).  When a warp has finished reading slot s its lane 0 increments
// done[s]; the warp that brings the count to the number of warps resets it and
// issues the copy of the tile kStages further on into the same slot.  So no
// warp ever waits for a particular other warp: the slowest warp gates a slot's
// refill, and the others may run up to kStages - 1 tiles ahead.  Every wait is
// bounded and every stop decision is warp-uniform; a wait that gives up sets
// ST_TIMEOUT and the block stops early, after letting copies in flight land.
// ---------------------------------------------------------------------------
// 3D: whether Q point i (x: its coordinates as float) belongs to the small-|Q| pass (Q = 0 included),
// and, if `list`, its entry in that pass's list.  Such points take no part in the pair sum (their place
// in a warp's largest P is immaterial: it is the smallest).  The FP32 test settles all but those near
// or below the bound and those that leave the FP32 range on the way: the finishing kernel asks in FP64 alone,
// and reads a place in the list for every point that it finds small.
template <class QT>
__device__ __forceinline__ bool list_small(const double* __restrict__ q, int64_t i, const QT (&x)[3], float rmax,
                                           WsHeader* h, int32_t* __restrict__ small, bool list) {
  const float fx = (float)x[0] * rmax, fy = (float)x[1] * rmax, fz = (float)x[2] * rmax;
  const float x2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
  if (x2 > 1.01f * (float)(kTauSmallQ * kTauSmallQ) && x2 <= 3.402823466e38f) return false;
  const double q2 = q_norm2(q[i * 3], q[i * 3 + 1], q[i * 3 + 2]);
  const bool is_small = q2 == 0.0 || small_q(q2, rmax);
  if (is_small && q2 != 0.0 && list) {
    const uint32_t e = atomicAdd(&h->small_q_count, 1u);
    small[i] = (int32_t)e;
    if (e < (uint32_t)kSmallDirect) h->small_list[e] = (int32_t)i;
  }
  return is_small;
}

template <class Pol, int R, int NT>
__global__ void __launch_bounds__(NT, kMinBlocks<Pol, R, NT>) k_fwd(const typename Pol::Item* __restrict__ items, int64_t n_items,
                                            int64_t per_split, const double* __restrict__ q, int64_t n_q,
                                            Thr th, double2* __restrict__ partial, WsHeader* h,
                                            int32_t* __restrict__ small, const int32_t* __restrict__ qperm) {
  using Item = typename Pol::Item;
  using QT = typename Pol::QT;
  constexpr int TILE = Pol::kTile;
  constexpr int D = Pol::kDim;
  constexpr int NW = NT / 32;
  __shared__ __align__(128) Item ring[kStages * TILE];
  __shared__ __align__(8) uint64_t full[kStages];
  __shared__ int done[kStages];
  __shared__ int issued;

  const int64_t i0 = (int64_t)blockIdx.y * per_split;
  const int64_t n = max((int64_t)0, min(per_split, n_items - i0));
  const int ntiles = (int)((n + TILE - 1) / TILE);
  const Item* src = items + i0;

  // slot qbase + r NT holds Q point qperm[slot] (the caller's index; without qperm the slot itself)
  QT qr[R][3];
  const int64_t qbase = (int64_t)blockIdx.x * (NT * R) + threadIdx.x;
  bool live = D == 2;   // 3D: some point of this thread needs the pair sum (|Q| r_max >= 1/4)
  const float rmax = D == 3 ? __uint_as_float(h->rmax_bits) : 0.f;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t iq = qbase + (int64_t)r * NT;
#pragma unroll
    for (int d = 0; d < 3; ++d) qr[r][d] = (QT)0;
    if (iq < n_q) {
      const int64_t src = qperm ? (int64_t)qperm[iq] : iq;
#pragma unroll
      for (int d = 0; d < D; ++d) qr[r][d] = (QT)q[src * D + d];
      if constexpr (D == 3) live = !list_small(q, src, qr[r], rmax, h, small, blockIdx.y == 0) || live;
    }
  }
  live = __any_sync(0xffffffffu, live);
  typename Pol::template Acc<R> acc;
  acc.init();

  auto issue = [&](int t) {
    const int s = t % kStages;
    const int64_t cnt = min((int64_t)TILE, n - (int64_t)t * TILE);
    const uint32_t bytes = (uint32_t)(cnt * (int64_t)sizeof(Item));
    mbar_arrive_expect_tx(&full[s], bytes);
    bulk_g2s(ring + s * TILE, src + (int64_t)t * TILE, bytes, &full[s]);
    atomicAdd(&issued, 1);
  };
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      done[s] = 0;
    }
    issued = 0;
    fence_mbar_init();
  }
  if (!__syncthreads_or(live)) return;
  if (threadIdx.x == 0)
    for (int t = 0; t < min(kStages, ntiles); ++t) issue(t);

  bool ok = true;
  for (int t = 0; t < ntiles; ++t) {
    const int s = t % kStages;
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full[s], (uint32_t)((t / kStages) & 1)))) { ok = false; break; }
    const int cnt = (int)min((int64_t)TILE, n - (int64_t)t * TILE);
    if (live) Pol::template tile<R>(ring + s * TILE, cnt, qr, acc, th, i0 + (int64_t)t * TILE);
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
      __threadfence_block();                       // this warp's reads of slot s come first
      if (atomicAdd(&done[s], 1) == NW - 1) {      // last warp out of slot s refills it
        atomicExch(&done[s], 0);
        if (t + kStages < ntiles) {
          fence_proxy_async_smem();
          issue(t + kStages);
        }
      }
    }
  }
  if (!ok) set_status(&h->status, ST_TIMEOUT);
  __syncthreads();   // reached by every thread: stop decisions above are per warp, never inside a warp
  if (threadIdx.x == 0) {   // no copy may still be writing into the ring when the block exits
    const int m = issued;
    for (int u = max(0, m - kStages); u < m; ++u)
      (void)mbar_wait_bounded(&full[u % kStages], (uint32_t)((u / kStages) & 1));
  }
  if (!ok) return;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t iq = qbase + (int64_t)r * NT;
    if (iq < n_q) partial[(int64_t)blockIdx.y * n_q + (qperm ? (int64_t)qperm[iq] : iq)] = acc.get(r);
  }
}

// ---------------------------------------------------------------------------
// Short launches of the 3D FP32 path (few faces x Q points: k_fwd would run a block or a few, each
// walking its 128-face tiles alone, ~1,000 cycles a face).  A block takes one tile and one of k_fwd's
// groups of 128 Q points (the 32 lanes x 4 points of a warp there, on which the branch of a face is
// decided), and its 8 warps evaluate the tile's faces side by side, 4 faces at a time each.  The tile's
// FP32 sums run in k_fwd's order all the same: every warp keeps its faces' terms in registers and
// adds them to the sums that the warp before it passes on through shared memory, so the results are
// those of k_fwd bit for bit.
// ---------------------------------------------------------------------------
constexpr int kGrpWarps = 8, kGrpFaces = 4;   // faces a warp holds at a time
using GrpV = typename QPack<4>::V;

// Hand-over between two warps: the giver arrives, the taker waits (named barrier of their 64 threads).
__device__ __forceinline__ void give(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void take(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }

__global__ void __launch_bounds__(kGrpWarps * 32, 2) k_fwd_group(const Face32* __restrict__ faces, int64_t n_faces,
                                                                 const double* __restrict__ q, int64_t n_q, Thr th,
                                                                 double2* __restrict__ partial, WsHeader* h,
                                                                 int32_t* __restrict__ small) {
  constexpr int R = 4, N = QPack<R>::N, TILE = Pol3F32::kTile;
  __shared__ __align__(16) Face32 rec[TILE];
  __shared__ GrpV sums[2][N][32];   // the running (re, im) sums of the 128 points
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i0 = (int64_t)blockIdx.y * TILE;
  const int cnt = (int)min((int64_t)TILE, n_faces - i0);
  // group g of k_fwd's block b: points b 512 + 128 r + 32 g + lane
  const int64_t qbase = (int64_t)(blockIdx.x >> 2) * 512 + (blockIdx.x & 3) * 32 + lane;
  float qr[R][3];
  bool live = false;
  const float rmax = __uint_as_float(h->rmax_bits);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t iq = qbase + (int64_t)r * 128;
    float x[3] = {0.f, 0.f, 0.f};
    if (iq < n_q) {
#pragma unroll
      for (int d = 0; d < 3; ++d) x[d] = (float)q[iq * 3 + d];
      live = !list_small(q, iq, x, rmax, h, small, blockIdx.y == 0 && warp == 0) || live;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) qr[r][d] = x[d];
  }
  if (!__syncthreads_or(live)) return;   // (every warp holds the same points)
  for (int t = threadIdx.x; t < cnt * 3; t += kGrpWarps * 32)
    reinterpret_cast<float4*>(rec)[t] = reinterpret_cast<const float4*>(faces + i0)[t];
  __syncthreads();
  GrpV qv[N][3];
  QPack<R>::pack<3>(qr, qv);
  const int passes = (cnt + kGrpWarps * kGrpFaces - 1) / (kGrpWarps * kGrpFaces);
  for (int p = 0; p < passes; ++p) {
    GrpV c[kGrpFaces][N], d[kGrpFaces][N], zr[kGrpFaces][N], zi[kGrpFaces][N];
    const int f0 = (p * kGrpWarps + warp) * kGrpFaces;
#pragma unroll
    for (int k = 0; k < kGrpFaces; ++k) {
      if (f0 + k < cnt) {   // warp-uniform
        const float4* t = reinterpret_cast<const float4*>(rec + f0 + k);
        const float4 A = t[0], B = t[1], C = t[2];
        FaceQ<R> f;
        f.load(qv, A, B, C);
        GrpV S0[N];
        if (f.wmax < th.hi) f.series(th, zr[k], zi[k]);
        else f.template edge<false>(th, qv, A, B, C, zr[k], zi[k], S0);
#pragma unroll
        for (int j = 0; j < N; ++j) face_weight(f.mu[j], f.s[j], c[k][j], d[k][j]);
      }
    }
    GrpV tre[N], tim[N];
    if (p + warp > 0) {
      take(1 + warp);
#pragma unroll
      for (int j = 0; j < N; ++j) { tre[j] = sums[0][j][lane]; tim[j] = sums[1][j][lane]; }
    } else {
#pragma unroll
      for (int j = 0; j < N; ++j) { tre[j] = vs<GrpV>(0.f); tim[j] = vs<GrpV>(0.f); }
    }
#pragma unroll
    for (int k = 0; k < kGrpFaces; ++k)
      if (f0 + k < cnt) {
#pragma unroll
        for (int j = 0; j < N; ++j) face_add(c[k][j], d[k][j], zr[k][j], zi[k][j], tre[j], tim[j]);
      }
    if (p + 1 < passes || warp + 1 < kGrpWarps) {
#pragma unroll
      for (int j = 0; j < N; ++j) { sums[0][j][lane] = tre[j]; sums[1][j][lane] = tim[j]; }
      give(1 + (warp + 1) % kGrpWarps);
    } else {
      Acc32<R> acc;
      acc.init();
#pragma unroll
      for (int r = 0; r < R; ++r) {
        acc.re[r].add(el(tre, r));
        acc.im[r].add(el(tim, r));
        const int64_t iq = qbase + (int64_t)r * 128;
        if (iq < n_q) partial[(int64_t)blockIdx.y * n_q + iq] = acc.get(r);
      }
    }
  }
}

template <class Pol, int R, int NT>
cudaError_t launch_one(const FwdLaunch& L, const void* items, int64_t n_items, const double* q, int64_t n_q,
                       Thr th, double2* partial, WsHeader* h, int32_t* small, cudaStream_t st,
                       const int32_t* qperm) {
  dim3 grid((unsigned)L.q_tiles, (unsigned)L.k_splits);
  k_fwd<Pol, R, NT><<<grid, NT, 0, st>>>(static_cast<const typename Pol::Item*>(items), n_items, L.per_split, q,
                                         n_q, th, partial, h, small, qperm);
  return cudaGetLastError();
}

template <class Pol, int R, int NT>
int occupancy_one() {
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_fwd<Pol, R, NT>, NT, 0) != cudaSuccess) return 1;
  return b > 0 ? b : 1;
}

// Dispatch over the instantiated configurations (FP64 paths keep R <= 2).
template <class Pol, class F>
cudaError_t dispatch(int r, int nt, F&& f) {
  constexpr bool kBig = sizeof(typename Pol::QT) == 4;
#define PFT_CASE(RR, NN) \
  if (r == RR && nt == NN) return f.template operator()<Pol, RR, NN>();
  PFT_CASE(1, 128) PFT_CASE(2, 128) PFT_CASE(1, 256) PFT_CASE(2, 256)
  if constexpr (kBig) {
    PFT_CASE(4, 128) PFT_CASE(8, 128) PFT_CASE(4, 256) PFT_CASE(8, 256)
  }
#undef PFT_CASE
  return cudaErrorInvalidConfiguration;
}

// The paired-face policy: the FP32 launch shapes with R <= 4.
template <class F>
cudaError_t dispatch_pairs(int r, int nt, F&& f) {
#define PFT_CASE(RR, NN) \
  if (r == RR && nt == NN) return f.template operator()<Pol3F32Pair, RR, NN>();
  PFT_CASE(1, 128) PFT_CASE(2, 128) PFT_CASE(4, 128) PFT_CASE(1, 256) PFT_CASE(2, 256) PFT_CASE(4, 256)
#undef PFT_CASE
  return cudaErrorInvalidConfiguration;
}

struct LaunchF {
  const FwdLaunch& L; const void* items; int64_t n_items; const double* q; int64_t n_q; Thr th;
  double2* partial; WsHeader* h; int32_t* small; cudaStream_t st; const int32_t* qperm;
  template <class Pol, int R, int NT>
  cudaError_t operator()() const {
    return launch_one<Pol, R, NT>(L, items, n_items, q, n_q, th, partial, h, small, st, qperm);
  }
};

struct OccF {
  int* out;
  template <class Pol, int R, int NT>
  cudaError_t operator()() const { *out = occupancy_one<Pol, R, NT>(); return cudaSuccess; }
};

}  // namespace

cudaError_t launch_fwd(int dim, bool fp64, const FwdLaunch& L, const void* items, int64_t n_items, const double* q,
                       int64_t n_q, float tau, double2* partial, WsHeader* h, int32_t* small, cudaStream_t st,
                       int64_t pair_faces, const int32_t* qperm) {
  // the FP64 path keeps its series (through k = 16) for P < 9/4, where it truncates below 1e-14
  if (fp64) tau = fminf(tau, 3.0f);
  const float tau_lo = fminf(tau, kTauLo);
  const Thr th{0.25f * tau * tau, 0.25f * tau_lo * tau_lo, tau > 1.0f ? 1 : 0, tau > 3.0f ? 1 : 0,
               dim == 3 && !fp64 ? pair_faces : 0};
  LaunchF f{L, items, n_items, q, n_q, th, partial, h, small, st, qperm};
  if (L.group) {
    k_fwd_group<<<dim3((unsigned)L.q_tiles, (unsigned)L.k_splits), kGrpWarps * 32, 0, st>>>(
        static_cast<const Face32*>(items), n_items, q, n_q, th, partial, h, small);
    return cudaGetLastError();
  }
  if (dim == 2) return fp64 ? dispatch<Pol2F64>(L.r, L.nt, f) : dispatch<Pol2F32>(L.r, L.nt, f);
  if (!fp64 && th.pair_end > 0) return dispatch_pairs(L.r, L.nt, f);
  return fp64 ? dispatch<Pol3F64>(L.r, L.nt, f) : dispatch<Pol3F32>(L.r, L.nt, f);
}

constexpr int kDevices = 64;   // devices whose properties are remembered

int device_sms() {
  static std::atomic<int> known[kDevices];   // 0: not asked yet
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  if (dev >= 0 && dev < kDevices && (sms = known[dev].load(std::memory_order_relaxed)) > 0) return sms;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 1;
  if (dev >= 0 && dev < kDevices) known[dev].store(sms, std::memory_order_relaxed);
  return sms;
}

int fwd_blocks_per_sm(int dim, bool fp64, int r, int nt, bool pairs) {
  static std::atomic<int> known[kDevices][64];   // 0: not asked yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
  std::atomic<int>* slot = nullptr;
  if (dev >= 0 && dev < kDevices) {
    const int lr = r == 1 ? 0 : (r == 2 ? 1 : (r == 4 ? 2 : 3));
    slot = &known[dev][((((dim - 2) * 2 + fp64) * 2 + pairs) * 2 + (nt == 256)) * 4 + lr];
    if (const int b = slot->load(std::memory_order_relaxed)) return b;
  }
  int b = 1;
  OccF f{&b};
  cudaError_t e;
  if (dim == 2) e = fp64 ? dispatch<Pol2F64>(r, nt, f) : dispatch<Pol2F32>(r, nt, f);
  else if (!fp64 && pairs) e = dispatch_pairs(r, nt, f);
  else e = fp64 ? dispatch<Pol3F64>(r, nt, f) : dispatch<Pol3F32>(r, nt, f);
  if (e != cudaSuccess) return 1;
  if (slot) slot->store(b, std::memory_order_relaxed);
  return b;
}

int fwd_tile(int dim, bool fp64) {
  if (dim == 2) return fp64 ? Pol2F64::kTile : Pol2F32::kTile;
  return fp64 ? Pol3F64::kTile : Pol3F32::kTile;
}

}  // namespace pft
