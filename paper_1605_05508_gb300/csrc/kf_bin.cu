// kf_bin.cu -- spatial partitioning of hits (and seeds) into directionally
// projective eta x phi bins per layer (Cerati et al., Sec. 3: hits sorted in
// phi within eta bins, phi bins for fast look-up of compatible hits).
//
// A counting sort of every segment (one event on one layer) into the 64 x 256
// bins, either by passes over all points of all segments at once or by one
// block per segment (launch_bin_points), with a final pass that orders each
// bin by id so that the output is deterministic (skipped with
// kf_tuning.bin_unordered: the build's results do not depend on the order of
// the hits inside a bin).  The unordered form can sort by 64 x 512 sub-bins
// instead, each bin two of them, and give the sub-bin starts as well: the
// build's windows then cover half as wide a strip of phi beyond their edges.
#include "kf_bin.cuh"
#include "kf_internal.h"

#include <algorithm>
#include <atomic>
#include <limits>

namespace kfi {

constexpr int kScanThreads = 1024;
static_assert(KF_NBINS % kScanThreads == 0, "bins per thread");  // 16 consecutive bins a thread
constexpr int kPointThreads = 256;
constexpr int64_t kNoLimit = std::numeric_limits<int64_t>::max();  // of a segment's points

// padded shared-memory index of bin b: a thread's 16 (or 32) consecutive
// bins and a warp's 32 threads fall in distinct banks
__device__ __forceinline__ int pad_idx(int b) { return b + (b >> 5); }
constexpr int kScanSmem = (KF_NBINS + KF_NBINS / 32) * int(sizeof(int));
// the sub-bin histogram: one block per SM
constexpr int kFineSmem = (KF_NBINS_FINE + KF_NBINS_FINE / 32) * int(sizeof(int));
static_assert(KF_NBINS_FINE % kScanThreads == 0, "sub-bins per thread");

// Exclusive scan, in place, of the NB counts in cnt (padded layout) by the
// block's kScanThreads threads, each owning NB / kScanThreads consecutive
// bins; returns the total to every thread.  Ends with a barrier.
template <int NB = KF_NBINS>
__device__ __forceinline__ int scan_bins(int* cnt, int* warp_tot) {
  constexpr int kPer = NB / kScanThreads;
  const int tid = threadIdx.x;
  int run = 0;
#pragma unroll
  for (int t = 0; t < kPer; ++t) run += cnt[pad_idx(tid * kPer + t)];
  const int lane = tid & 31, warp = tid >> 5;
  int incl = run;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int w = warp_tot[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += v;
    }
    warp_tot[lane] = w;  // inclusive over warps
  }
  __syncthreads();
  int acc = (incl - run) + (warp > 0 ? warp_tot[warp - 1] : 0);
  const int total = warp_tot[kScanThreads / 32 - 1];
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const int i = pad_idx(tid * kPer + t);
    const int c = cnt[i];
    cnt[i] = acc;
    acc += c;
  }
  __syncthreads();
  return total;
}

// segment s of the request: a table entry, or segment s of the arrays of A
template <bool FINE>
__device__ __forceinline__ BinSegment segment(const BinArgs& A, int s) {
  if (A.table) return A.table[s];
  BinSegment S;
  S.xyz = A.xyz;
  S.stride = A.stride;
  S.p0 = A.seg_off[s];
  S.p1 = min(A.seg_off[s + 1], A.stride);
  S.begin = S.p0;
  S.bin_off = A.bin_off + int64_t(s) * (KF_NBINS + 1);
  S.fine_off = FINE ? A.fine_off + int64_t(s) * (KF_NBINS_FINE + 1) : nullptr;
  S.out_pts = A.out_pts;
  S.out_id = A.out_id;
  return S;
}
// the last segment that begins at or before point g of the launch's points
__device__ __forceinline__ int segment_of(const BinArgs& A, int64_t g) {
  int lo = 0, hi = A.n_seg - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((A.table ? A.table[mid].begin : A.seg_off[mid]) <= g)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// The unordered counting sort of one segment per block, its counts and
// cursors in shared memory (one launch for all segments): (1) every point of
// the segment adds one to its bin's count, (2) the block turns the counts
// into exclusive offsets (written to bin_off) and cursors, (3) every point
// takes the next slot of its bin.  The order inside a bin is that of the
// shared-memory atomics: for kf_tuning.bin_unordered, whose users do not
// depend on it.
// Segment S (number seg) by the whole block, with cnt (KF_NBINS padded ints of
// shared memory) and warp_tot.
// FINE: the counting sort runs over the KF_NBINS_FINE sub-bins (cnt holds
// as many), whose starts go to fine_off, and the bin starts to `off` are
// those of the even sub-bins (a bin is two consecutive sub-bins).
template <bool FINE = false>
__device__ __forceinline__ void bin_one_segment(const BinSegment& S, int32_t* out_seg, int seg, int* cnt,
                                                int* warp_tot) {
  const float* const xyz = S.xyz;
  const int64_t stride = S.stride, p0 = S.p0, p1 = S.p1;
  int32_t* const off = S.bin_off;
  int32_t* const fine_off = S.fine_off;
  float4* const out_pts = S.out_pts;
  int32_t* const out_id = S.out_id;
  constexpr int NB = FINE ? KF_NBINS_FINE : KF_NBINS;
  constexpr int NPHI = FINE ? KF_BIN_PHI_FINE : KF_BIN_PHI;
  const int tid = threadIdx.x;
  for (int b = tid; b < NB; b += kScanThreads) cnt[pad_idx(b)] = 0;
  __syncthreads();
  // the points in batches of kSegBatch a thread, their loads issued together
  constexpr int kSegBatch = 4;
  for (int64_t g0 = p0 + tid; g0 < p1; g0 += int64_t(kScanThreads) * kSegBatch) {
    float x[kSegBatch], y[kSegBatch], z[kSegBatch];
#pragma unroll
    for (int u = 0; u < kSegBatch; ++u) {
      const int64_t g = g0 + int64_t(u) * kScanThreads;
      if (g < p1) {
        x[u] = xyz[g];
        y[u] = xyz[stride + g];
        z[u] = xyz[2 * stride + g];
      }
    }
#pragma unroll
    for (int u = 0; u < kSegBatch; ++u) {
      const int64_t g = g0 + int64_t(u) * kScanThreads;
      if (g < p1) {
        const int b = bin_of<NPHI>(x[u], y[u], z[u]);
        atomicAdd(&cnt[pad_idx(b)], 1);
        // with points out (hits: their ids travel in .w), out_id is scratch:
        // it keeps each point's bin for the second pass
        if (out_pts) out_id[g] = b;
      }
    }
  }
  __syncthreads();
  const int total = scan_bins<NB>(cnt, warp_tot);
  if (tid == 0) off[KF_NBINS] = total;
  if constexpr (FINE) {
    if (tid == 0) fine_off[KF_NBINS_FINE] = total;
    for (int b = tid; b < KF_NBINS_FINE; b += kScanThreads) fine_off[b] = cnt[pad_idx(b)];  // coalesced
    for (int b = tid; b < KF_NBINS; b += kScanThreads) off[b] = cnt[pad_idx(2 * b)];
  } else {
    for (int b = tid; b < KF_NBINS; b += kScanThreads) off[b] = cnt[pad_idx(b)];  // coalesced
  }
  // every start read before the scatter below moves the cursors on
  __syncthreads();
  for (int64_t g0 = p0 + tid; g0 < p1; g0 += int64_t(kScanThreads) * kSegBatch) {
    float x[kSegBatch], y[kSegBatch], z[kSegBatch];
    int bins[kSegBatch];
#pragma unroll
    for (int u = 0; u < kSegBatch; ++u) {
      const int64_t g = g0 + int64_t(u) * kScanThreads;
      if (g < p1) {
        x[u] = xyz[g];
        y[u] = xyz[stride + g];
        z[u] = xyz[2 * stride + g];
        bins[u] = out_pts ? out_id[g] : 0;
      }
    }
#pragma unroll
    for (int u = 0; u < kSegBatch; ++u) {
      const int64_t g = g0 + int64_t(u) * kScanThreads;
      if (g < p1) {
        const int i = int(g - p0);
        if (out_pts) {  // the bin from the first pass; out_id stays scratch
          const int64_t q = p0 + atomicAdd(&cnt[pad_idx(bins[u])], 1);
          out_pts[q] = make_float4(x[u], y[u], z[u], __int_as_float(i));
        } else {
          const int64_t q = p0 + atomicAdd(&cnt[pad_idx(bin_of<NPHI>(x[u], y[u], z[u]))], 1);
          out_id[q] = i;
          if (out_seg) out_seg[q] = seg;
        }
      }
    }
  }
}

// (a segment of more than `limit` points is left to bin_large_count_kernel and
// what follows it, its counts set to zero)
template <bool FINE>
__global__ void __launch_bounds__(kScanThreads) bin_segment_kernel(const BinArgs A, const int64_t limit) {
  chain_begin();
  extern __shared__ int cnt[];  // counts, then cursors (padded layout)
  __shared__ int warp_tot[32];
  const BinSegment S = segment<FINE>(A, int(blockIdx.x));
  if (S.p1 - S.p0 <= limit)
    bin_one_segment<FINE>(S, A.out_seg, int(blockIdx.x), cnt, warp_tot);
  else if (!FINE)
    for (int b = threadIdx.x; b <= KF_NBINS; b += kScanThreads) S.bin_off[b] = 0;
}

// ---------------------------------------------------------------------------
// The passes over all points of all segments at once: a segment of any size
// spreads over the whole GPU.
//   (zero)            the counts, in the bin (or sub-bin) starts' own place
//   bin_count_kernel  every point adds one to its bin's count; the count before
//                     it is its place in the bin, kept with the bin in one word
//   bin_scan_kernel   one block per segment: counts to starts
//   bin_place_kernel  every point to its bin's start plus its place
//   bin_order_kernel  (ordered form) a warp sorts the hits of consecutive bins,
//                     a contiguous run, by id inside each bin
// A point's word between the passes: its bin above its place, or, with the top
// bit set, its position in the segment.  A place of kPlaceMax or more (a bin of
// more than 65 535 hits) does not fit: the count leaves it in the point's own
// entry of the output, and the scan, between the two passes, turns it into a
// position.
constexpr int kPlaceBits = 16;
constexpr uint32_t kPlaceMax = (1u << kPlaceBits) - 1;
constexpr uint32_t kIsPosition = 1u << 31;
static_assert(KF_NBINS_FINE <= 1 << (31 - kPlaceBits), "bin and place in a word");

// kZeroPer bins a thread: with one, the launch of the blocks, about one a
// nanosecond, set the time (21.6 us for the sub-bins of 151 segments; of 151
// segments of 3 000 hits the passes take 41 us by sub-bin and 32 by bin, not 55
// and 39).  With 16 the passes after it were slower when called in a row.
constexpr int kZeroPer = 4;
template <bool FINE>
__global__ void __launch_bounds__(kPointThreads) bin_zero_kernel(const BinArgs A) {
  chain_begin();
  constexpr int kBlocks = (FINE ? KF_NBINS_FINE : KF_NBINS) / (kPointThreads * kZeroPer);
  const BinSegment S = segment<FINE>(A, int(blockIdx.x) / kBlocks);
  int32_t* const c = (FINE ? S.fine_off : S.bin_off) + int(blockIdx.x) % kBlocks * (kPointThreads * kZeroPer);
#pragma unroll
  for (int t = 0; t < kZeroPer; ++t) c[t * kPointThreads + threadIdx.x] = 0;
}

// N points of segment S, q, q + step, .. (those below S.p1), their loads and
// atomics in flight together
template <bool FINE, int N>
__device__ __forceinline__ void count_points(const BinSegment& S, int64_t q, int64_t step) {
  float x[N], y[N], z[N];
  uint32_t place[N];
  int b[N];
#pragma unroll
  for (int t = 0; t < N; ++t)
    if (q + t * step < S.p1) {
      x[t] = S.xyz[q + t * step];
      y[t] = S.xyz[S.stride + q + t * step];
      z[t] = S.xyz[2 * S.stride + q + t * step];
    }
#pragma unroll
  for (int t = 0; t < N; ++t)
    if (q + t * step < S.p1) {
      b[t] = bin_of<FINE ? KF_BIN_PHI_FINE : KF_BIN_PHI>(x[t], y[t], z[t]);
      place[t] = uint32_t(atomicAdd((FINE ? S.fine_off : S.bin_off) + b[t], 1));
    }
#pragma unroll
  for (int t = 0; t < N; ++t)
    if (q + t * step < S.p1) {
      if (place[t] >= kPlaceMax) S.out_pts[q + t * step].x = __uint_as_float(place[t]);
      S.out_id[q + t * step] = int(uint32_t(b[t]) << kPlaceBits | min(place[t], kPlaceMax));
    }
}
template <bool FINE, int N>
__device__ __forceinline__ void place_points(const BinSegment& S, int64_t q, int64_t step) {
  float x[N], y[N], z[N];
  uint32_t w[N];
#pragma unroll
  for (int t = 0; t < N; ++t)
    if (q + t * step < S.p1) {
      w[t] = uint32_t(S.out_id[q + t * step]);
      x[t] = S.xyz[q + t * step];
      y[t] = S.xyz[S.stride + q + t * step];
      z[t] = S.xyz[2 * S.stride + q + t * step];
    }
  int at[N];
#pragma unroll
  for (int t = 0; t < N; ++t)
    if (q + t * step < S.p1)
      at[t] = w[t] & kIsPosition ? int(w[t] & ~kIsPosition)
                                 : (FINE ? S.fine_off : S.bin_off)[w[t] >> kPlaceBits] + int(w[t] & kPlaceMax);
#pragma unroll
  for (int t = 0; t < N; ++t)
    if (q + t * step < S.p1)
      S.out_pts[S.p0 + at[t]] = make_float4(x[t], y[t], z[t], __int_as_float(int(q + t * step - S.p0)));
}

template <bool FINE>
__global__ void __launch_bounds__(kPointThreads) bin_count_kernel(const BinArgs A) {
  chain_begin();
  const int64_t g = int64_t(blockIdx.x) * kPointThreads + threadIdx.x;
  if (g >= A.n_points) return;
  const BinSegment S = segment<FINE>(A, segment_of(A, g));
  const int64_t q = g - S.begin + S.p0;
  if (q >= S.p0 && q < S.p1) count_points<FINE, 1>(S, q, 0);  // (else outside every segment)
}

// Counts of segment S to starts, by the whole block, with cnt (padded) and
// warp_tot in shared memory.
template <bool FINE>
__device__ __forceinline__ void scan_segment(const BinSegment& S, int* cnt, int* warp_tot) {
  constexpr int NB = FINE ? KF_NBINS_FINE : KF_NBINS;
  constexpr int kPer = NB / kScanThreads;
  int32_t* const c = FINE ? S.fine_off : S.bin_off;
  const int tid = threadIdx.x;
  // 16 loads a thread in flight together (coalesced): one after the other they
  // were two thirds of the pass when few segments leave most SMs idle
  bool over = false;  // a bin with places that do not fit their words
#pragma unroll 1
  for (int t0 = 0; t0 < kPer; t0 += 16) {
    int v[16];
#pragma unroll
    for (int t = 0; t < 16; ++t) v[t] = c[(t0 + t) * kScanThreads + tid];
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      cnt[pad_idx((t0 + t) * kScanThreads + tid)] = v[t];
      over |= v[t] > int(kPlaceMax);
    }
  }
  over = __syncthreads_or(over);
  const int total = scan_bins<NB>(cnt, warp_tot);
  if (tid == 0) c[NB] = total;
  for (int b = tid; b < NB; b += kScanThreads) c[b] = cnt[pad_idx(b)];
  if constexpr (FINE) {
    if (tid == 0) S.bin_off[KF_NBINS] = total;
    for (int b = tid; b < KF_NBINS; b += kScanThreads) S.bin_off[b] = cnt[pad_idx(2 * b)];
  }
  if (over)
    for (int64_t q = S.p0 + tid; q < S.p1; q += kScanThreads) {
      const uint32_t w = uint32_t(S.out_id[q]);
      if ((w & kPlaceMax) != kPlaceMax) continue;
      const uint32_t at = uint32_t(cnt[pad_idx(int(w >> kPlaceBits))]) + __float_as_uint(S.out_pts[q].x);
      S.out_id[q] = int(kIsPosition | at);
    }
}
template <bool FINE>
__global__ void __launch_bounds__(kScanThreads) bin_scan_kernel(const BinArgs A) {
  chain_begin();
  extern __shared__ int cnt[];  // counts, then starts (padded layout)
  __shared__ int warp_tot[32];
  scan_segment<FINE>(segment<FINE>(A, int(blockIdx.x)), cnt, warp_tot);
}

template <bool FINE>
__global__ void __launch_bounds__(kPointThreads) bin_place_kernel(const BinArgs A) {
  chain_begin();
  const int64_t g = int64_t(blockIdx.x) * kPointThreads + threadIdx.x;
  if (g >= A.n_points) return;
  const BinSegment S = segment<FINE>(A, segment_of(A, g));
  const int64_t q = g - S.begin + S.p0;
  if (q >= S.p0 && q < S.p1) place_points<FINE, 1>(S, q, 0);
}

// One warp per NB bins of a segment: their hits, ids in any order inside a bin,
// are a contiguous run.  Runs of up to kOrderRun hits are taken whole: loaded
// (coalesced, all in flight), every hit's place found by counting the smaller
// ids of its bin in shared memory, and the moved ones written back.  Of a
// longer run, as many bins as fit are taken at a time; a single bin that does
// not fit goes through order_long_bin, after the others.
constexpr int kOrderRun = 128;
constexpr int kOrderWarps = 4;

// A bin of more than kOrderRun hits, n from `beg` of segment s on, by one warp:
// a radix sort of the ids (stable passes of 7 bits, the counters in shared
// memory, between out_pts[].w and the bin's part of the scratch out_id, whose
// words the passes before are done with), after which every hit is fetched by
// its id.  The time is linear in n: 60 000 hits in some 325 bins take 88 us,
// 5 000 in 25 bins 65; by one lane's insertion sort, the bins of a warp one
// after the other, 5.6 and 9.6 ms, by one a thread a bin 1.1 and 1.7 ms.
constexpr int kDigitBits = 7;
__device__ __forceinline__ void order_long_bin(const BinArgs& A, int s, int beg, int n, int* digits) {
  const int64_t p0 = A.seg_off[s], m = min(A.seg_off[s + 1], A.stride) - p0;
  float4* const pts = A.out_pts + p0 + beg;
  int* const tmp = A.out_id + p0 + beg;
  constexpr int kDigits = 1 << kDigitBits, kAhead = 4;  // ids a lane has in flight
  const int lane = threadIdx.x & 31;
  bool in_tmp = false;  // where the ids are
  for (int shift = 0; shift < 31 && (m - 1) >> shift > 0; shift += kDigitBits) {
    for (int t = lane; t < kDigits; t += 32) digits[t] = 0;
    __syncwarp();
    auto load = [&](int i0, int (&id)[kAhead]) {
#pragma unroll
      for (int t = 0; t < kAhead; ++t) {
        const int i = i0 + 32 * t + lane;
        id[t] = i < n ? (in_tmp ? tmp[i] : __float_as_int(pts[i].w)) : -1;
      }
    };
    for (int i0 = 0; i0 < n; i0 += 32 * kAhead) {
      int id[kAhead];
      load(i0, id);
#pragma unroll
      for (int t = 0; t < kAhead; ++t)
        if (id[t] >= 0) atomicAdd(&digits[(id[t] >> shift) & (kDigits - 1)], 1);
    }
    __syncwarp();
    {  // counts to starts, kDigits / 32 of them a lane
      constexpr int kPer = kDigits / 32;
      int v[kPer], sum = 0;
#pragma unroll
      for (int t = 0; t < kPer; ++t) {
        v[t] = digits[lane * kPer + t];
        sum += v[t];
      }
      int inc = sum;
#pragma unroll
      for (int d = 1; d < 32; d *= 2) {
        const int o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
      }
      int at = inc - sum;
#pragma unroll
      for (int t = 0; t < kPer; ++t) {
        digits[lane * kPer + t] = at;
        at += v[t];
      }
    }
    __syncwarp();
    for (int i0 = 0; i0 < n; i0 += 32 * kAhead) {
      int id[kAhead];
      load(i0, id);
#pragma unroll
      for (int t = 0; t < kAhead; ++t) {
        const int d = id[t] >= 0 ? (id[t] >> shift) & (kDigits - 1) : kDigits;
        const unsigned same = __match_any_sync(0xffffffffu, d);
        const int before = __popc(same & ((1u << lane) - 1u));
        int at = 0;
        if (id[t] >= 0) at = digits[d] + before;
        __syncwarp();
        if (id[t] >= 0) {
          if (before == 0) digits[d] += __popc(same);
          if (in_tmp)
            pts[at].w = __int_as_float(id[t]);
          else
            tmp[at] = id[t];
        }
        __syncwarp();
      }
    }
    in_tmp = !in_tmp;
  }
  for (int i = lane; i < n; i += 32) {
    const int id = in_tmp ? tmp[i] : __float_as_int(pts[i].w);
    const float* const h = A.xyz + p0 + id;
    pts[i] = make_float4(h[0], h[A.stride], h[2 * A.stride], __int_as_float(id));
  }
  __syncwarp();  // the counters are free again
}

// NB bins of segment s from b0 on, by one warp, with ids (kOrderRun) and off (NB
// + 1) in shared memory; LIMIT: unless the segment has more than `limit` hits.
template <int NB, bool LIMIT>
__device__ __forceinline__ void order_bins(const BinArgs& A, int s, int64_t limit, int b0, int* ids, int* off) {
  static_assert(kOrderRun >= 1 << kDigitBits, "ids holds order_long_bin's counters");
  const int lane = threadIdx.x & 31;
  const int32_t* const starts = A.bin_off + int64_t(s) * (KF_NBINS + 1) + b0;
  const int64_t p0 = A.seg_off[s], p1 = LIMIT ? A.seg_off[s + 1] : 0;
  float4* const pts = A.out_pts + p0;
#pragma unroll
  for (int b = lane; b <= NB; b += 32) off[b] = starts[b];
  __syncwarp();
  if (LIMIT && p1 - p0 > limit) return;
  const int end_all = off[NB];
  bool crowded = false;
  for (int bb = 0; bb < NB && off[bb] < end_all;) {
    const int beg = off[bb];
    // the bins bb .. be-1 whose hits fit a run
    int be = bb, above = NB + 1;
    if (end_all - beg <= kOrderRun) be = NB;
    while (above - be > 1) {
      const int mid = (be + above) >> 1;
      if (off[mid] - beg <= kOrderRun)
        be = mid;
      else
        above = mid;
    }
    if (be == bb) {  // one bin alone is too long: below
      crowded = true;
      ++bb;
      continue;
    }
    const int n = off[be] - beg;
    float4 h[kOrderRun / 32];
#pragma unroll
    for (int t = 0; t < kOrderRun / 32; ++t)
      if (lane + 32 * t < n) h[t] = pts[beg + lane + 32 * t];
#pragma unroll
    for (int t = 0; t < kOrderRun / 32; ++t)
      if (lane + 32 * t < n) ids[lane + 32 * t] = __float_as_int(h[t].w);
    __syncwarp();
#pragma unroll
    for (int t = 0; t < kOrderRun / 32; ++t) {
      const int i = lane + 32 * t;
      if (i < n) {
        int lo = bb, hi = be - 1;  // the bin of hit i
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (off[mid] - beg <= i)
            lo = mid;
          else
            hi = mid - 1;
        }
        const int first = off[lo] - beg, last = off[lo + 1] - beg, id = ids[i];
        int at = first;
        for (int u = first; u < last; ++u) at += ids[u] < id ? 1 : 0;
        if (at != i) pts[beg + at] = h[t];
      }
    }
    __syncwarp();  // ids are read before the next run's
    bb = be;
  }
  if (crowded)
    for (int b = 0; b < NB; ++b)
      if (off[b + 1] - off[b] > kOrderRun) order_long_bin(A, s, off[b], off[b + 1] - off[b], ids);
}

// (10 or 11 blocks an SM, as measured: with 10 one segment of 1 500 000 hits takes
// 140 us, not 165, with 11 350 of 20 000 202, not 206; segments of more than
// `limit` hits are left to bin_large_order_kernel)
template <int NB, bool LIMIT>
__global__ void __launch_bounds__(32 * kOrderWarps, NB <= 8 ? 10 : 11)
    bin_order_kernel(const __grid_constant__ BinArgs A, const int64_t limit) {
  chain_begin();
  __shared__ int s_id[kOrderWarps][kOrderRun];
  __shared__ int s_off[kOrderWarps][NB + 1];
  const int warp = threadIdx.x >> 5;
  const int s = int(blockIdx.x) / (KF_NBINS / NB / kOrderWarps);
  const int b0 = (int(blockIdx.x) % (KF_NBINS / NB / kOrderWarps) * kOrderWarps + warp) * NB;
  order_bins<NB, LIMIT>(A, s, limit, b0, s_id[warp], s_off[warp]);
}

// The segments of more than `limit` points of an ordered request whose others
// take a block each: their counts are zeroed by their blocks, then the passes
// above run over their points alone, in three launches.  They cost a request
// without such segments, which the host cannot tell from one with them, 3 to 5
// us.
constexpr int kLargePer = 4;  // points a thread has in flight
constexpr int kLargeUnit = kPointThreads * kLargePer;

// f(s, S, u) for every large segment S (number s), u running over this block's
// share of its units_of(points) units; then done(S, n, units), n the units taken,
// if any.
template <int THREADS, class U, class F, class D>
__device__ __forceinline__ void for_large(const BinArgs& A, int64_t limit, U units_of, F f, D done) {
  constexpr int kAhead = 4, kWords = kAhead * THREADS / 32;  // sizes a thread has in flight
  __shared__ unsigned s_large[kWords];
  const int tid = threadIdx.x;
  int64_t u = blockIdx.x;  // this block's next unit, counted on from segment to segment
  for (int s0 = 0; s0 < A.n_seg; s0 += kAhead * THREADS) {
    bool any = false, large[kAhead];
#pragma unroll
    for (int t = 0; t < kAhead; ++t) {
      const int s = s0 + t * THREADS + tid;
      large[t] = s < A.n_seg && min(A.seg_off[s + 1], A.stride) - A.seg_off[s] > limit;
    }
#pragma unroll
    for (int t = 0; t < kAhead; ++t) {
      const unsigned m = __ballot_sync(0xffffffffu, large[t]);
      if ((tid & 31) == 0) s_large[(t * THREADS + tid) >> 5] = m;
      any |= large[t];
    }
    if (__syncthreads_or(any))
      for (int w = 0; w < kWords; ++w)
        for (unsigned left = s_large[w]; left; left &= left - 1) {
          const int s = s0 + 32 * w + __ffs(left) - 1;
          const BinSegment S = segment<false>(A, s);
          const int64_t units = units_of(S.p1 - S.p0);
          int n = 0;
          for (; u < units; u += gridDim.x, ++n) f(s, S, u);
          u -= units;
          if (n > 0) done(S, n, int(units));
        }
    __syncthreads();  // s_large is read before the next segments'
  }
}

// Count; the block that ends a segment's last unit turns the counts to starts
// (the units done so far are counted in the place of the total).
__global__ void __launch_bounds__(kPointThreads)
    bin_large_count_kernel(const __grid_constant__ BinArgs A, const int64_t limit) {
  chain_begin();
  __shared__ int s_sum[kPointThreads / 32];
  __shared__ int s_done;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for_large<kPointThreads>(
      A, limit, [](int64_t points) { return (points + kLargeUnit - 1) / kLargeUnit; },
      [&](int, const BinSegment& S, int64_t u) {
        count_points<false, kLargePer>(S, S.p0 + u * kLargeUnit + tid, kPointThreads);
      },
      [&](const BinSegment& S, int n, int units) {
        __threadfence();  // this block's counts and words before its units are counted
        __syncthreads();
        if (tid == 0) s_done = atomicAdd(&S.bin_off[KF_NBINS], n) + n;
        __syncthreads();
        if (s_done != units) return;
        __threadfence();
        int carry = 0;
        bool over = false;  // a bin with places that do not fit their words
        for (int b0 = 0; b0 < KF_NBINS; b0 += 4 * kPointThreads) {
          int v[4], sum = 0;
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            v[t] = __ldcg(&S.bin_off[b0 + 4 * tid + t]);
            over |= v[t] > int(kPlaceMax);
            sum += v[t];
          }
          int inc = sum;
#pragma unroll
          for (int d = 1; d < 32; d *= 2) {
            const int o = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += o;
          }
          if (lane == 31) s_sum[warp] = inc;
          __syncthreads();
          int at = carry + inc - sum;
          for (int w = 0; w < kPointThreads / 32; ++w) {
            if (w < warp) at += s_sum[w];
            carry += s_sum[w];
          }
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            S.bin_off[b0 + 4 * tid + t] = at;
            at += v[t];
          }
          __syncthreads();  // s_sum is read before the next bins'
        }
        if (tid == 0) S.bin_off[KF_NBINS] = carry;
        if (__syncthreads_or(over))
          for (int64_t q = S.p0 + tid; q < S.p1; q += kPointThreads) {
            const uint32_t w = uint32_t(__ldcg(&S.out_id[q]));
            if ((w & kPlaceMax) != kPlaceMax) continue;
            const uint32_t place = __float_as_uint(__ldcg(&S.out_pts[q].x));
            S.out_id[q] = int(kIsPosition | (uint32_t(S.bin_off[w >> kPlaceBits]) + place));
          }
      });
}

__global__ void __launch_bounds__(kPointThreads)
    bin_large_place_kernel(const __grid_constant__ BinArgs A, const int64_t limit) {
  chain_begin();
  for_large<kPointThreads>(
      A, limit, [](int64_t points) { return (points + kLargeUnit - 1) / kLargeUnit; },
      [&](int, const BinSegment& S, int64_t u) {
        place_points<false, kLargePer>(S, S.p0 + u * kLargeUnit + int(threadIdx.x), kPointThreads);
      },
      [](const BinSegment&, int, int) {});
}

// As bin_order_kernel, with bins of about a run's worth a warp at each segment's
// own density.
__device__ __forceinline__ int large_bins(int64_t points) {
  return points * 32 <= 2 * int64_t(kOrderRun) * KF_NBINS ? 32 : 8;
}
__global__ void __launch_bounds__(32 * kOrderWarps, 8)
    bin_large_order_kernel(const __grid_constant__ BinArgs A, const int64_t limit) {
  chain_begin();
  __shared__ int s_id[kOrderWarps][kOrderRun];
  __shared__ int s_off[kOrderWarps][33];
  const int warp = threadIdx.x >> 5;
  for_large<32 * kOrderWarps>(
      A, limit, [](int64_t points) { return KF_NBINS / (large_bins(points) * kOrderWarps); },
      [&](int s, const BinSegment& S, int64_t u) {
        const int at = int(u) * kOrderWarps + warp;
        if (large_bins(S.p1 - S.p0) == 32)
          order_bins<32, false>(A, s, kNoLimit, at * 32, s_id[warp], s_off[warp]);
        else
          order_bins<8, false>(A, s, kNoLimit, at * 8, s_id[warp], s_off[warp]);
        __syncwarp();  // off is read before the next unit's
      },
      [](const BinSegment&, int, int) {});
}

constexpr int kMaxDevices = 64;

// a kernel's shared-memory attributes, set once per device (the serving loop
// bins from several threads' calls; setting them again is harmless)
template <class K>
static cudaError_t segment_smem_attrs(K kernel, int smem, std::atomic<bool>* done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < kMaxDevices && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  // the largest shared-memory carveout (a block takes 68 KB, or 135 KB with
  // the sub-bins; its 1024 threads' registers already leave room for one
  // block per SM)
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             int(cudaSharedmemCarveoutMaxShared));
  if (e == cudaSuccess && dev >= 0 && dev < kMaxDevices) done[dev].store(true, std::memory_order_release);
  return e;
}

template <bool FINE>
static cudaError_t launch_bin_wide(const BinArgs& a, cudaStream_t st) {
  static std::atomic<bool> attr_set[kMaxDevices];
  constexpr int smem = FINE ? kFineSmem : kScanSmem;
  cudaError_t e = segment_smem_attrs(bin_scan_kernel<FINE>, smem, attr_set);
  if (e != cudaSuccess) return e;
  const unsigned zero = unsigned(a.n_seg) * ((FINE ? KF_NBINS_FINE : KF_NBINS) / (kPointThreads * kZeroPer));
  const unsigned grid = unsigned((a.n_points + kPointThreads - 1) / kPointThreads);
  e = launch_chained(bin_zero_kernel<FINE>, zero, kPointThreads, 0, st, a);
  if (e == cudaSuccess && grid > 0) e = launch_chained(bin_count_kernel<FINE>, grid, kPointThreads, 0, st, a);
  if (e == cudaSuccess) e = launch_chained(bin_scan_kernel<FINE>, a.n_seg, kScanThreads, smem, st, a);
  if (e == cudaSuccess && grid > 0) e = launch_chained(bin_place_kernel<FINE>, grid, kPointThreads, 0, st, a);
  return e;
}

// a block per segment; those of more than `limit` points (FINE: no limit) by passes of their own
template <bool FINE>
static cudaError_t launch_bin_blocks(const BinArgs& a, int64_t limit, int num_sms, cudaStream_t st) {
  static std::atomic<bool> attr_set[kMaxDevices];
  constexpr int smem = FINE ? kFineSmem : kScanSmem;
  cudaError_t e = segment_smem_attrs(bin_segment_kernel<FINE>, smem, attr_set);
  if (e == cudaSuccess) e = launch_chained(bin_segment_kernel<FINE>, a.n_seg, kScanThreads, smem, st, a, limit);
  if (e != cudaSuccess || limit == kNoLimit) return e;
  e = launch_chained(bin_large_count_kernel, 4 * num_sms, kPointThreads, 0, st, a, limit);
  if (e == cudaSuccess) e = launch_chained(bin_large_place_kernel, 4 * num_sms, kPointThreads, 0, st, a, limit);
  return e;
}

// The form by the costs given at plan_of, the sizes being known here (a request
// served alone mostly has small segments: with the wide passes whatever the size a
// small event's latency was 201 us, not 193).
cudaError_t launch_bin_segment_table(const BinSegment* table, int n, int64_t n_points, int64_t max_points, bool fine,
                                     int num_sms, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  BinArgs a;
  a.table = table;
  a.n_seg = n;
  a.n_points = n_points;
  const double m = 1e-3 * double(max_points), rounds = double((n + num_sms - 1) / num_sms);
  const double blocks = rounds * (fine ? 12.5 + 1.5 * m : 10 + 1.42 * m);
  const double wide = (fine ? 20 + 0.07 * n : 15 + 0.05 * n) + 0.0225e-3 * double(n_points);
  if (blocks <= wide)
    return fine ? launch_bin_blocks<true>(a, kNoLimit, num_sms, st)
                : launch_bin_blocks<false>(a, kNoLimit, num_sms, st);
  return fine ? launch_bin_wide<true>(a, st) : launch_bin_wide<false>(a, st);
}

// Bins a warp of the order pass takes.  A warp's runs follow one another, and
// a warp of few hits costs its launch and its loads all the same, so: about as
// many bins as hold one run at the mean density, as long as every SM has some
// twenty warps.  After the wide passes, whose segments may be of very different
// sizes, no more than 32.  Whole binning, measured with 128, 64, 32 and 8 bins
// a warp: 350 segments of 20 000 hits 207, 202, 227 and 418 us, 1 540 of 1 000
// 124, -, 283 and 861; 7 of 20 000 26.8, -, 21.6 and 23.7; one of 1 500 000
// 1 456, -, 405 and 140.
static cudaError_t launch_bin_order(const BinArgs& a, int num_sms, bool wide, int64_t limit, cudaStream_t st) {
  const auto go = [&](void (*kernel)(BinArgs, int64_t), int nb) {
    return launch_chained(kernel, unsigned(a.n_seg) * unsigned(KF_NBINS / nb / kOrderWarps), 32 * kOrderWarps, 0, st, a,
                          limit);
  };
  const auto fills = [&](int nb) { return int64_t(a.n_seg) * (KF_NBINS / nb) >= int64_t(num_sms) * 20; };
  const auto one_run = [&](int nb) { return a.n_points * nb <= int64_t(a.n_seg) * kOrderRun * KF_NBINS; };
  if (limit != kNoLimit) {  // blocks for a run each, if all hits were in large segments
    const int grid = int(std::min<int64_t>(8 * num_sms, a.n_points / (kOrderRun * kOrderWarps) + 1));
    const cudaError_t e = launch_chained(bin_large_order_kernel, grid, 32 * kOrderWarps, 0, st, a, limit);
    if (e != cudaSuccess) return e;
  }
  const bool all = limit == kNoLimit;
  if (!wide && fills(128) && one_run(128))
    return all ? go(bin_order_kernel<128, false>, 128) : go(bin_order_kernel<128, true>, 128);
  if (!wide && fills(64) && one_run(64))
    return all ? go(bin_order_kernel<64, false>, 64) : go(bin_order_kernel<64, true>, 64);
  if (fills(32)) return all ? go(bin_order_kernel<32, false>, 32) : go(bin_order_kernel<32, true>, 32);
  return go(bin_order_kernel<8, false>, 8);  // (never with a limit: a few segments of over 3 000 hits)
}

// Which form: with m thousand hits in the largest segment and n in all, a block
// per segment takes some 10 + 1.42 m us (by sub-bin 12.5 + 1.5 m), the wide
// passes 15 + 0.05 a segment + 0.0225 n (20 + 0.07 a segment + 0.0225 n).  7
// segments of 20 000: 40 against 18 us, of 3 000 15 against 16; 70 of 12 000 27
// against 36; 350 of 20 000 164 against 190, by sub-bin 186 against 220; 84 uneven
// ones of 43 000 on average (2 000 ... 200 000) 304 against 102.  The sizes are on
// the device, so the rule goes by their mean, as if some segment had several
// times that: blocks for small segments and, up to some 40 000 hits, for more
// segments than SMs.
//
// In the ordered form the segments larger than `limit`, whose block alone would
// take twice as long as all by the wide passes, are taken from the blocks to
// passes of their own.  154 segments, half of 1 500 000 hits in 7 of them: 105 us
// (by blocks alone 195); one of 700 000 hits among 153 of 2 000: 104 (1 240).  A
// request of up to 150 000 hits, which those passes would cost up to a third,
// goes without: at most some 0.25 ms, were all in one segment.  An unordered one
// goes without too (its callers have always had a block a segment there).
struct BinPlan {
  bool wide;
  int64_t limit;
};
static BinPlan plan_of(const BinArgs& a, int num_sms) {
  if (!a.out_pts) return {false, kNoLimit};
  if (a.n_points > int64_t(a.n_seg) * (a.n_seg >= num_sms ? 40000 : 3000)) return {true, kNoLimit};
  const int64_t limit = int64_t((10000 + 100.0 * a.n_seg + 0.045 * double(a.n_points)) / 1.42);
  return {false, !a.unordered && a.n_points > std::max<int64_t>(limit, 150000) ? limit : kNoLimit};
}

cudaError_t launch_bin_points(const BinArgs& a, int num_sms, cudaStream_t st) {
  if (a.n_seg <= 0) return cudaSuccess;
  if (a.fine_off && !a.unordered) return cudaErrorInvalidValue;  // sub-bins only with the unordered binning
  if (a.out_seg && a.out_pts) return cudaErrorInvalidValue;      // segments only with ids
  const BinPlan plan = plan_of(a, num_sms);
  cudaError_t e = plan.wide ? (a.fine_off ? launch_bin_wide<true>(a, st) : launch_bin_wide<false>(a, st))
                            : (a.fine_off ? launch_bin_blocks<true>(a, plan.limit, num_sms, st)
                                          : launch_bin_blocks<false>(a, plan.limit, num_sms, st));
  if (e == cudaSuccess && !a.unordered && a.n_points > 0) e = launch_bin_order(a, num_sms, plan.wide, plan.limit, st);
  return e;
}

}  // namespace kfi

using namespace kfi;

extern "C" int kf_bin_hits(kf_ctx* ctx, const kf_layer_hits* in, kf_layer_hit_bins* out, void* stream) {
  if (!ctx || !in || !out) return KF_EINVAL;
  if (in->n_events < 0 || in->n_layers < 1 || in->first_layer < 0 ||
      in->first_layer + in->n_layers > ctx->cfg.n_layers || in->n_hits < 0)
    return KF_EINVAL;
  if (!in->seg_off || !out->bin_off || (in->n_hits > 0 && (!in->xyz || !out->hits))) return KF_EINVAL;
  if (out->fine_off && !ctx->tune.bin_unordered) return KF_EINVAL;  // sub-bins: unordered binning only
  out->n_events = in->n_events;
  out->n_layers = in->n_layers;
  out->first_layer = in->first_layer;
  out->n_hits = in->n_hits;
  out->seg_off = in->seg_off;
  const int nseg = in->n_events * in->n_layers;
  if (nseg == 0) return KF_OK;
  KF_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  const size_t id_bytes = (size_t(in->n_hits > 0 ? in->n_hits : 1) * sizeof(int32_t) + 255) & ~size_t(255);
  int rc = scratch_reserve(ctx, ctx->s_bin_id, id_bytes);
  if (rc) return rc;
  BinArgs a;
  a.xyz = in->xyz;
  a.stride = in->n_hits;
  a.seg_off = in->seg_off;
  a.n_seg = nseg;
  a.n_points = in->n_hits;
  a.bin_off = out->bin_off;
  a.out_pts = reinterpret_cast<float4*>(out->hits);
  a.out_id = static_cast<int32_t*>(ctx->s_bin_id.ptr);
  a.out_seg = nullptr;
  a.unordered = ctx->tune.bin_unordered;
  a.fine_off = out->fine_off;
  KF_CUDA_TRY(ctx, launch_bin_points(a, ctx->num_sms, static_cast<cudaStream_t>(stream)));
  return KF_OK;
}
