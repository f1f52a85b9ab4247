// kf_fit.cu -- track-fit kernels: one thread per track, state and covariance
// in registers, structure-of-arrays global layout (coalesced 128-byte warp
// transactions per component).
//
// Track fitting is the branch-free part of Kalman-filter tracking (Cerati et
// al., Sec. 2): with the hit set fixed, every track runs propagate + update
// over the layers.  Forms:
//   fit_fused_kernel        all layers in one launch, the track held in
//                           registers (kf_fit, kf_fit_fused, kf_fit_noalloc;
//                           fit_mixed_kernel: the mixed-precision form);
//   fit_gather_kernel       the same over the hits a build chose (kf_refit);
//   fit_layer_stage_kernel  one layer step over the whole batch (kf_fit with
//                           kf_tuning.fit_stage replays one launch per layer
//                           from a captured CUDA graph), each warp's next 32
//                           tracks copied into shared memory by 2-D tensor
//                           copies while it computes the current ones
//                           (bitwise equal);
//   fit_f64_kernel          the plain FP64 form, launched per event and per
//                           layer.
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "kf_internal.h"
#include "kf_math.cuh"
#include "kf_tma.cuh"

namespace kfi {

constexpr int kFitThreads = 128;
// Resident warps per SM of the fused fit: 24 (80 registers, no spills).  The
// layers' arithmetic is bound by instruction issue and register reads, not by
// memory: 1.444 ms for 4M tracks x 10 layers against 1.472 at 20 warps.
constexpr int kFitWarpsPerSM = 24;
// with the table of events, or gathered hits, the registers go over 80
constexpr int kFitTableBlocksPerSM = 5;
constexpr int kNewtonF32 = 12;  // iteration cap of the safeguarded Newton solve
constexpr int kNewtonF64 = 16;
constexpr int kF64MinBlock = 32;

// Positive-definiteness of the rank-5 covariance: Cholesky of P C P^T where P
// maps to (t . pos, z, px, py, pz), t the transverse tangent of the cylinder
// at the track position (the radial direction is exactly singular after a
// surface propagation).
template <typename T>
__device__ __forceinline__ bool pd5(const T p[6], const T C[21]) {
  using kf::sym;
  const T r = kf::sqrt_t(p[0] * p[0] + p[1] * p[1]);
  const T t0 = r > T(0) ? -p[1] / r : T(0), t1 = r > T(0) ? p[0] / r : T(1);
  T M[5][5];
  M[0][0] = t0 * t0 * C[sym(0, 0)] + T(2) * t0 * t1 * C[sym(1, 0)] + t1 * t1 * C[sym(1, 1)];
#pragma unroll
  for (int j = 1; j < 5; ++j) {
    const int cj = j + 1;  // z, px, py, pz
    M[j][0] = t0 * C[sym(0, cj)] + t1 * C[sym(1, cj)];
#pragma unroll
    for (int k = 1; k <= j; ++k) M[j][k] = C[sym(cj, k + 1)];
  }
  T L[5][5];
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    T d = M[j][j];
#pragma unroll
    for (int k = 0; k < j; ++k) d -= L[j][k] * L[j][k];
    if (!(d > T(0))) return false;
    L[j][j] = kf::sqrt_t(d);
    const T inv = T(1) / L[j][j];
#pragma unroll
    for (int i = j + 1; i < 5; ++i) {
      T v = M[i][j];
#pragma unroll
      for (int k = 0; k < j; ++k) v -= L[i][k] * L[j][k];
      L[i][j] = v * inv;
    }
  }
  return true;
}

// One propagate + (optional) update step of one track.  Returns the status
// bits raised; writes chi2 (-1 when no update).  UPD64: S^-1 and the
// covariance downdate in FP64 (single-precision state only).
template <typename T, int NEWTON, bool EXT, bool UPD64 = false>
__device__ __forceinline__ int32_t track_step(T p[6], T lo[3], T C[21], T a, T R, T x_x0, T mass, bool has_hit,
                                              T m0, T m1, T m2, T v0, T v1, T v2, T& chi2) {
  chi2 = T(-1);
  const int st = kf::propagate<T, NEWTON, EXT>(p, lo, C, a, R);
  if (st) return st;
  if (x_x0 > T(0)) kf::scatter(p, lo, C, x_x0, mass);
  if (!has_hit) return kf::ST_NO_HIT;
  T r0, r1, r2;
  kf::residual<T, EXT>(p, lo, m0, m1, m2, r0, r1, r2);
  if constexpr (UPD64) {
    chi2 = kf::kalman_update_f64(p, lo, C, r0, r1, r2, v0, v1, v2);
  } else {
    T Si[6];
    kf::inverse_S(C, v0, v1, v2, Si);
    chi2 = kf::chi2_of(r0, r1, r2, Si);
    kf::kalman_update<T, EXT>(p, lo, C, Si, r0, r1, r2, v0, v1, v2);
  }
  return 0;
}

// The step of track i given its inputs; writes its outputs.
__device__ __forceinline__ void fit_layer_track(const FitLayerArgs& A, int64_t i, int32_t st, float p[6], float lo[3],
                                                float C[21], int8_t q, bool has_hit, float m0, float m1, float m2) {
  const int64_t n = A.n;
  if (st & KF_ST_STOPPED) {  // stopped at an earlier layer: nothing to do
    if (A.chi2) A.chi2[i] = -1.f;
    return;
  }
  const float a = A.a_scale * float(q);
  float chi2;
  const int32_t raised =
      track_step<float, kNewtonF32, true>(p, lo, C, a, A.R, A.x_x0, A.mass, has_hit, m0, m1, m2, A.v0, A.v1, A.v2,
                                          chi2);
  const bool stopped = (raised & KF_ST_STOPPED) != 0;
  if (!stopped || A.first) {
#pragma unroll
    for (int c = 0; c < 6; ++c) A.out_par[c * n + i] = p[c];
#pragma unroll
    for (int c = 0; c < 3; ++c) A.out_lo[c * n + i] = lo[c];
#pragma unroll
    for (int c = 0; c < 21; ++c) A.out_cov[c * n + i] = C[c];
  }
  if (A.chi2) A.chi2[i] = chi2;
  st |= raised;
  if ((A.last || stopped) && !pd5(p, C)) st |= KF_ST_NOT_PD;
  if (A.first || raised || A.last) A.status[i] = st;
}

// ---------------------------------------------------------------------------
// Staged form of the layer step (kf_tuning.fit_stage = 1): the same step per
// track, but the 33 float rows a track reads (state, position low parts,
// covariance, hit) arrive in shared memory by tensor copies.  Each warp walks
// tiles of 32 tracks; lane 0 issues four 2-D tensor copies (boxes of 32 tracks
// x 6, 3, 21 and 3 rows) for the warp's next tile into the other half of a
// double buffer while the warp computes the current tile, so a tile's loads
// are in flight during the previous tile's arithmetic without holding
// registers.  Completion is tracked by one mbarrier per buffer; every wait is
// bounded (a wait that gives up marks the warp's remaining tracks with
// KF_ST_DEVICE_TIMEOUT).  Requires n, begin and count multiples of 32 and
// 16-byte aligned rows (stage_layout_ok); kf_fit takes the fused launch otherwise.
constexpr int kStageTile = 32;                 // tracks per warp tile
constexpr int kStageThreads = 64;              // two warps per block
constexpr int kStageBlocksPerSM = 12;          // 24 warps per SM
constexpr uint32_t kStageWaitLimit = 1u << 22; // bounded mbarrier polls

struct StageTile {  // one buffer: rows of 32 tracks, each box 128-byte aligned
  float par[6][kStageTile];
  float lo[3][kStageTile];
  float cov[21][kStageTile];
  float hit[3][kStageTile];
};
static_assert(sizeof(StageTile) % 128 == 0, "box alignment");
constexpr size_t kStageSmem = size_t(kStageThreads / 32) * 2 * sizeof(StageTile) + 64;

__device__ __forceinline__ void tensor_g2s_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void stage_issue(const FitStageMaps& M, bool has_lo, StageTile& T, uint64_t* bar, int x,
                                            uint32_t bytes) {
  mbar_arrive_expect_tx(bar, bytes);
  tensor_g2s_2d(T.par, &M.par, x, 0, bar);
  if (has_lo) tensor_g2s_2d(T.lo, &M.lo, x, 0, bar);
  tensor_g2s_2d(T.cov, &M.cov, x, 0, bar);
  tensor_g2s_2d(T.hit, &M.hit, x, 0, bar);
}

__global__ void __launch_bounds__(kStageThreads, kStageBlocksPerSM)
    fit_layer_stage_kernel(const FitLayerArgs A, const __grid_constant__ FitStageMaps M) {
  extern __shared__ __align__(128) unsigned char stage_smem[];
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  StageTile* buf = reinterpret_cast<StageTile*>(stage_smem) + 2 * wib;
  uint64_t* bar = reinterpret_cast<uint64_t*>(stage_smem + size_t(kStageThreads / 32) * 2 * sizeof(StageTile)) + 2 * wib;
  const int64_t n_tiles = A.count / kStageTile;
  const int64_t nwarps = int64_t(gridDim.x) * (kStageThreads / 32);
  int64_t t = int64_t(blockIdx.x) * (kStageThreads / 32) + wib;
  if (t >= n_tiles) return;  // the whole warp
  const bool has_lo = A.in_lo != nullptr;
  const uint32_t bytes = uint32_t(sizeof(float)) * kStageTile * (6 + 21 + 3 + (has_lo ? 3 : 0));
  // Test hook (kf_test_stage_fault): the copies of the batch's tile
  // A.skip_tile are never issued, so the wait for it runs out; A.wait_limit
  // (0: the normal limit) bounds the waits for staged input.  The drain wait
  // before the block exits always keeps the normal limit.
  // lane 0: bit b set while the pending phase of buffer b has copies in flight
  uint32_t armed = 0;
  if (lane == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_init_fence();
    if (A.begin / kStageTile + t != A.skip_tile) {
      stage_issue(M, has_lo, buf[0], &bar[0], int(A.begin + t * kStageTile), bytes);
      armed = 1u;
    }
  }
  __syncwarp();
  uint32_t ph0 = 0, ph1 = 0;
  bool failed = false;
  for (int s = 0; t < n_tiles; t += nwarps, s ^= 1) {
    const int64_t i = A.begin + t * kStageTile + lane;
    if (failed) {  // an earlier wait gave up: flag the remaining tracks
      A.status[i] = (A.first ? 0 : A.status[i]) | KF_ST_DEVICE_TIMEOUT;
      continue;
    }
    // the next tile into the other buffer (its previous tile was read by every
    // lane before the __syncwarp that closed the last iteration)
    const int64_t tn = t + nwarps;
    if (tn < n_tiles && lane == 0 && A.begin / kStageTile + tn != A.skip_tile) {
      fence_proxy_async_smem();
      stage_issue(M, has_lo, buf[s ^ 1], &bar[s ^ 1], int(A.begin + tn * kStageTile), bytes);
      armed |= 1u << (s ^ 1);
    }
    // per-track inputs outside the tile, loaded while the copies land
    const int32_t st = A.first ? 0 : A.status[i];
    const int8_t q = A.charge[i];
    const bool has_hit = A.valid ? A.valid[i] != 0 : true;
    const bool ok = __all_sync(
        0xffffffffu, mbar_wait_bounded(&bar[s], s ? ph1 : ph0, A.wait_limit ? A.wait_limit : kStageWaitLimit));
    if (!ok) {  // the phase stays pending: waited for once more below
      failed = true;
      A.status[i] = st | KF_ST_DEVICE_TIMEOUT;
      continue;
    }
    if (s)
      ph1 ^= 1u;
    else
      ph0 ^= 1u;
    armed &= ~(1u << s);
    const StageTile& T = buf[s];
    float p[6], lo[3], C[21];
#pragma unroll
    for (int c = 0; c < 6; ++c) p[c] = T.par[c][lane];
#pragma unroll
    for (int c = 0; c < 3; ++c) lo[c] = has_lo ? T.lo[c][lane] : 0.f;
#pragma unroll
    for (int c = 0; c < 21; ++c) C[c] = T.cov[c][lane];
    const float m0 = T.hit[0][lane], m1 = T.hit[1][lane], m2 = T.hit[2][lane];
    __syncwarp();  // every lane has read buffer s before lane 0 may refill it
    fit_layer_track(A, i, st, p, lo, C, q, has_hit, m0, m1, m2);
  }
  // Copies still in flight land before the block's memory is released.  Should
  // this bounded wait give up too, the block exits with a copy in flight into
  // shared memory that a later block on the SM may already use: the damage is
  // not confined to this warp's tracks, which is why a KF_ST_DEVICE_TIMEOUT on
  // any track invalidates every result of the call (documented in kf.h).
  if (failed && lane == 0) {
    if (armed & 1u) mbar_wait_bounded(&bar[0], ph0, kStageWaitLimit);
    if (armed & 2u) mbar_wait_bounded(&bar[1], ph1, kStageWaitLimit);
  }
}

// The hits of one track, layer after layer: get(l, ..) is called for l = 0, 1,
// .. in turn and returns whether layer l has a hit.
// From the fit's own arrays [L][3][n], valid [L][n] or null.
struct ArrayHits {
  const float* xyz;
  const uint8_t* valid;
  int64_t n, i;
  __device__ __forceinline__ bool get(int l, float& m0, float& m1, float& m2) {
    const float* h = xyz + int64_t(l) * 3 * n;
    m0 = h[i];
    m1 = h[n + i];
    m2 = h[2 * n + i];
    return valid ? valid[int64_t(l) * n + i] != 0 : true;
  }
};

// Of a built track (kf_refit): the seeding layers from the seed's own hits,
// the building layers by the ids the build chose, looked up in the raw hits of
// the seed's event.  The lookups are two dependent loads, so the hit of the
// next layer is fetched, and the id of the one after it, before a layer's
// arithmetic.
struct GatherHits {
  const RefitGatherArgs& G;
  int64_t i;
  int e;
  int32_t id;             // of the layer after the next
  float nx, ny, nz;       // the next layer's hit
  bool nok;

  __device__ __forceinline__ GatherHits(const RefitGatherArgs& g, int64_t track) : G(g), i(track) {
    int lo = 0, hi = G.E - 1;  // the event: seed_off[e] <= i < seed_off[e + 1]
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (G.seed_off[mid] <= i)
        lo = mid;
      else
        hi = mid - 1;
    }
    e = lo;
    id = id_of(0);
    fetch(0);
  }
  __device__ __forceinline__ int32_t id_of(int l) const {
    const int b = l - G.Ls;
    return b >= 0 && b < G.Lb ? G.hit_idx[int64_t(b) * G.n + i] : -1;
  }
  // the hit of layer l (its id in `id`) into nx .. nok, and the id of layer l + 1
  __device__ __forceinline__ void fetch(int l) {
    const int64_t n = G.n;
    nx = ny = nz = 0.f;
    nok = false;
    if (l < G.Ls) {
      const float* s = G.seed_xyz + int64_t(l) * 3 * n;
      nx = s[i];
      ny = s[n + i];
      nz = s[2 * n + i];
      nok = G.seed_valid ? G.seed_valid[int64_t(l) * n + i] != 0 : true;
    } else if (id >= 0) {
      const int64_t* seg = G.seg_off + int64_t(e) * G.Lb + (l - G.Ls);
      const int64_t h = seg[0] + id;
      if (h < seg[1] && h >= 0 && h < G.n_hits) {
        nx = G.hit_xyz[h];
        ny = G.hit_xyz[G.n_hits + h];
        nz = G.hit_xyz[2 * G.n_hits + h];
        nok = true;
      }
    }
    id = id_of(l + 1);
  }
  __device__ __forceinline__ bool get(int l, float& m0, float& m1, float& m2) {
    m0 = nx;
    m1 = ny;
    m2 = nz;
    const bool ok = nok;
    if (l + 1 < G.Ls + G.Lb) fetch(l + 1);
    return ok;
  }
};

// All layers of track i of the arrays of E (FitFusedArgs itself, or one
// event of a table: the same field names), with the layers and constants of A
// and the hits of H.
template <bool UPD64, class EV, class HITS>
__device__ __forceinline__ void fused_track(const EV& E, const FitFusedArgs& A, int64_t i, HITS H) {
  const int64_t n = E.n;
  {
    float p[6], lo[3], C[21];
#pragma unroll
    for (int c = 0; c < 6; ++c) p[c] = E.in_par[c * n + i];
#pragma unroll
    for (int c = 0; c < 3; ++c) lo[c] = E.in_lo ? E.in_lo[c * n + i] : 0.f;
#pragma unroll
    for (int c = 0; c < 21; ++c) C[c] = E.in_cov[c * n + i];
    const float a = A.a_scale * float(E.charge[i]);
    int32_t st = 0;
    for (int l = 0; l < A.n_layers; ++l) {
      float chi2 = -1.f;
      if (!(st & KF_ST_STOPPED)) {
        float m0, m1, m2;
        const bool has_hit = H.get(l, m0, m1, m2);
        st |= track_step<float, kNewtonF32, true, UPD64>(p, lo, C, a, A.R[l], A.x_x0[l], A.mass, has_hit, m0, m1, m2,
                                                         A.v0, A.v1, A.v2, chi2);
      }
      if (E.chi2) E.chi2[int64_t(l) * n + i] = chi2;
    }
    if (!pd5(p, C)) st |= KF_ST_NOT_PD;
#pragma unroll
    for (int c = 0; c < 6; ++c) E.out_par[c * n + i] = p[c];
    if (E.out_lo) {
#pragma unroll
      for (int c = 0; c < 3; ++c) E.out_lo[c * n + i] = lo[c];
    }
#pragma unroll
    for (int c = 0; c < 21; ++c) E.out_cov[c * n + i] = C[c];
    if (E.status) E.status[i] = st;
  }
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS, kFitWarpsPerSM * 32 / THREADS) fit_fused_kernel(const FitFusedArgs A) {
  chain_begin();
  const int64_t i = int64_t(blockIdx.x) * THREADS + threadIdx.x;
  if (i < A.n) fused_track<false>(A, A, i, ArrayHits{A.hits, A.valid, A.n, i});
}

// The mixed-precision form (kf_fit_mixed).
__global__ void __launch_bounds__(kFitThreads, 1) fit_mixed_kernel(const FitFusedArgs A) {
  const int64_t i = int64_t(blockIdx.x) * kFitThreads + threadIdx.x;
  if (i < A.n) fused_track<true>(A, A, i, ArrayHits{A.hits, A.valid, A.n, i});
}

// The re-fit of built tracks: the fused fit over gathered hits (A's hit arrays
// are not used).  A pass that gathers them into arrays first took 18 us of the
// 79 us re-fit of 128 000 tracks over 10 layers.
__global__ void __launch_bounds__(kFitThreads, kFitTableBlocksPerSM)
    fit_gather_kernel(const FitFusedArgs A, const RefitGatherArgs G) {
  chain_begin();
  const int64_t i = int64_t(blockIdx.x) * kFitThreads + threadIdx.x;
  if (i < A.n) fused_track<false>(A, A, i, GatherHits(G, i));
}

// The fused fit of several events in one launch (the events a serving
// iteration prepares): thread t fits track t - table[q].begin of event q,
// the last with table[q].begin <= t; the arithmetic of fit_fused_kernel.
__global__ void __launch_bounds__(kFitThreads, kFitTableBlocksPerSM)
    fit_fused_table_kernel(const FitFusedArgs A, const FitEvent* table, int n_events, int64_t n_total) {
  chain_begin();
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n_total; t += stride) {
    int q = 0;
    while (q + 1 < n_events && table[q + 1].begin <= t) ++q;
    const FitEvent& E = table[q];
    const int64_t i = t - E.begin;
    fused_track<false>(E, A, i, ArrayHits{E.hits, E.valid, E.n, i});
  }
}

// Plain FP64 form: the same arithmetic in double, no position pair, one
// thread per track of one event, one launch per event and layer.
__global__ void __launch_bounds__(kFitThreads) fit_f64_kernel(const FitF64Args A) {
  const int64_t n = A.n;
  const int64_t i = A.begin + int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= A.end) return;
  int32_t st = A.first ? 0 : A.status[i];
  if (st & KF_ST_STOPPED) {
    if (A.chi2) A.chi2[i] = -1.0;
    return;
  }
  double p[6], lo[3] = {0, 0, 0}, C[21];
  for (int c = 0; c < 6; ++c) p[c] = A.in_par[c * n + i];
  for (int c = 0; c < 21; ++c) C[c] = A.in_cov[c * n + i];
  const double a = A.a_scale * double(A.charge[i]);
  const bool has_hit = A.valid ? A.valid[i] != 0 : true;
  double chi2;
  const int32_t raised = track_step<double, kNewtonF64, false>(
      p, lo, C, a, A.R, A.x_x0, A.mass, has_hit, double(A.hit[i]), double(A.hit[n + i]), double(A.hit[2 * n + i]), A.v0,
      A.v1, A.v2, chi2);
  const bool stopped = (raised & KF_ST_STOPPED) != 0;
  if (!stopped || A.first) {
    for (int c = 0; c < 6; ++c) A.out_par[c * n + i] = p[c];
    for (int c = 0; c < 21; ++c) A.out_cov[c * n + i] = C[c];
  }
  if (A.chi2) A.chi2[i] = chi2;
  st |= raised;
  if ((A.last || stopped) && !pd5(p, C)) st |= KF_ST_NOT_PD;
  if (A.first || raised || A.last) A.status[i] = st;
}

static bool stage_aligned(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool stage_layout_ok(const kf_tracks* seeds, const kf_track_hits* hits, const kf_tracks* out) {
  if (seeds->n % kStageTile || seeds->n > (int64_t(1) << 31) - 1) return false;
  const float* const in[] = {seeds->par, seeds->par_lo, seeds->cov, hits->xyz};
  for (const float* p : in)
    if (!stage_aligned(p)) return false;
  if (hits->n_layers > 1)  // the layers after the first read the outputs
    for (const float* p : {out->par, out->par_lo, out->cov})
      if (!stage_aligned(p)) return false;
  return true;
}

// Tensor maps of a layer step for fit_layer_stage_kernel: 2-D views (x =
// track, y = row) of the input state, position low parts, covariance and the
// layer's hits, boxes of 32 tracks x all rows.  False when the layout does not
// allow them (rows not 16-byte aligned, sizes not multiples of 32) or the
// driver's encoder is unavailable.
bool make_stage_maps(const FitLayerArgs& a, FitStageMaps* m) {
  if (a.n % kStageTile || a.begin % kStageTile || a.count % kStageTile || a.count <= 0) return false;
  if (a.n > (int64_t(1) << 31) - 1) return false;
  for (const float* p : {a.in_par, a.in_cov, a.hit, a.in_lo})
    if (!stage_aligned(p)) return false;
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  });
  if (!encode) return false;
  auto map2d = [&](CUtensorMap* t, const float* base, uint32_t rows) {
    const cuuint64_t dims[2] = {cuuint64_t(a.n), rows};
    const cuuint64_t strides[1] = {cuuint64_t(a.n) * sizeof(float)};
    const cuuint32_t box[2] = {kStageTile, rows};
    const cuuint32_t estr[2] = {1, 1};
    return encode(t, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  std::memset(m, 0, sizeof(*m));
  return map2d(&m->par, a.in_par, 6) && (!a.in_lo || map2d(&m->lo, a.in_lo, 3)) && map2d(&m->cov, a.in_cov, 21) &&
         map2d(&m->hit, a.hit, 3);
}

cudaError_t launch_fit_layer_stage(const FitLayerArgs& a, const FitStageMaps& m, int num_sms, cudaStream_t st) {
  const int64_t tiles = a.count / kStageTile;
  const int64_t need = (tiles + kStageThreads / 32 - 1) / (kStageThreads / 32);
  const int grid = int(std::max<int64_t>(1, std::min<int64_t>(need, int64_t(num_sms) * kStageBlocksPerSM)));
  cudaError_t e = cudaFuncSetAttribute(fit_layer_stage_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(kStageSmem));
  if (e != cudaSuccess) return e;
  fit_layer_stage_kernel<<<grid, kStageThreads, kStageSmem, st>>>(a, m);
  return cudaGetLastError();
}

cudaError_t launch_fit_fused_table(const FitFusedArgs& a, const FitEvent* table, int n_events, int64_t n_total,
                                   cudaStream_t st) {
  if (n_total <= 0) return cudaSuccess;
  const int grid = int((n_total + kFitThreads - 1) / kFitThreads);
  return launch_chained(fit_fused_table_kernel, grid, kFitThreads, 0, st, a, table, n_events, n_total);
}

cudaError_t launch_fit_fused(const FitFusedArgs& a, int block, cudaStream_t st) {
  if (a.n <= 0) return cudaSuccess;
  // blocks of 32 for small batches, to spread their warps over the SMs, made no
  // difference (18.43 us for 1 000 tracks x 10 layers either way)
  const int grid = int((a.n + block - 1) / block);
  return block == 64 ? launch_chained(fit_fused_kernel<64>, grid, 64, 0, st, a)
                     : launch_chained(fit_fused_kernel<128>, grid, 128, 0, st, a);
}

cudaError_t launch_fit_gather(const FitFusedArgs& a, const RefitGatherArgs& g, cudaStream_t st) {
  if (a.n <= 0) return cudaSuccess;
  fit_gather_kernel<<<int((a.n + kFitThreads - 1) / kFitThreads), kFitThreads, 0, st>>>(a, g);
  return cudaGetLastError();
}

cudaError_t launch_fit_mixed(const FitFusedArgs& a, cudaStream_t st) {
  if (a.n <= 0) return cudaSuccess;
  fit_mixed_kernel<<<int((a.n + kFitThreads - 1) / kFitThreads), kFitThreads, 0, st>>>(a);
  return cudaGetLastError();
}

// Threads per block: as many as spread the event over all SMs, 32 to 128.  The
// FP64 pipe serves under two lanes a cycle and SM, so an event's few warps side
// by side on one SM wait for each other while other SMs idle.
cudaError_t launch_fit_f64(const FitF64Args& a, int num_sms, cudaStream_t st) {
  const int64_t cnt = a.end - a.begin;
  if (cnt <= 0) return cudaSuccess;
  int block = kFitThreads;
  while (block > kF64MinBlock && cnt < int64_t(num_sms) * block) block /= 2;
  const int grid = int((cnt + block - 1) / block);
  fit_f64_kernel<<<grid, block, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace kfi
