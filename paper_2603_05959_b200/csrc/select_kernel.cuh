// Budgeted selection (Eq. 8) over a thread-block cluster, and the fused per-step kernel that prepares its input: anchor
// flags (Sec. 3.3), activation smoothing (Eq. 6), hybrid priorities (Eq. 7).
//
// A cluster of up to 8 CTAs x 512 threads splits the N candidates into contiguous position ranges, one per CTA, held in
// that CTA's shared memory.  Protected rows get the largest possible key, so "every protected row plus the B - |P| best
// evictable rows" is simply "the B largest keys", ties by position: a row stays if its key is above T, or equal to T and
// its position at most posT, where (T, posT) is the B-th candidate in that order.
//
// What bounds it is latency: under 1 MB is touched, but every step depends on the one before, and a cluster barrier costs
// about a microsecond.  So the usual way to T takes three: one to exchange the groups' ranges (Eq. 7), one after which
// every CTA reads all CTAs' 512-bin histograms of the priorities and finds the bin of the B-th row, one after which every
// CTA reads the few candidates of that bin and ranks them by comparison; the counts that place each CTA's output travel
// with them.  A crowded bin is histogrammed once more in 256 finer ones with the range of keys in each: a stream whose
// frames recur fills its cache with copies of the same scores, and the finer bin then holds nothing but ties, which go by
// position alone (a step of 1374 x 5470 x 16 in stored-score mode, after 10,000 frames that recur: 69.4 us with radix passes
// alone, 58.9 us so).  What is still crowded and not one key takes four 8-bit radix passes,
// a barrier each.  A warp then owns a contiguous range of positions and writes survivors, meta
// and moves with ballots, so that neighbouring lanes write neighbouring words.  (Radix passes for every step, a
// contiguous range per thread, and a separate exchange for the moves took 36 us at 17758 candidates and 18 us at 325.)
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"
#include "score_kernels.cuh"

namespace ovggt {

namespace cg = cooperative_groups;

constexpr int kSelectThreads = 512;   // 512 x 64 registers: half an SM, so a CTA fits beside an attention CTA
constexpr int kSelectWarps = kSelectThreads / 32;
constexpr int kSelectMaxCtas = 8;
static_assert(kSelectMaxCtas == kSumsLists, "a list of key sums per CTA");
constexpr int kSelectBins = kSelectThreads;       // a thread per bin; the last bin holds the protected rows
constexpr int kSelectSubBins = 256;               // of a crowded bin
constexpr int kSelectCtaCands = 64, kSelectAllCands = 256;   // candidates of the threshold bin, per CTA and in all
constexpr uint32_t kKeyProtected = 0xFFFFFFFFu;   // above the key of +inf (0xFF800000)

// The CTAs that share a problem.  A single CTA needs no cluster: its barrier is the block's, which costs a tenth.
template <bool SINGLE>
struct Peers {
  __device__ __forceinline__ static int count() {
    if constexpr (SINGLE) return 1;
    else return (int)cg::this_cluster().num_blocks();
  }
  __device__ __forceinline__ static int rank() {
    if constexpr (SINGLE) return 0;
    else return (int)cg::this_cluster().block_rank();
  }
  __device__ __forceinline__ static void sync() {
    if constexpr (SINGLE) __syncthreads();
    else cg::this_cluster().sync();
  }
  // Before a CTA leaves: nobody reads its shared memory any more.  Orders no memory, so it waits for no stores.
  __device__ __forceinline__ static void leave() {
    if constexpr (!SINGLE) {
      asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    }
  }
  template <typename T>
  __device__ __forceinline__ static T* of(T* p, int r) {   // the same object in CTA r
    if constexpr (SINGLE) return p;
    else return cg::this_cluster().map_shared_rank(p, r);
  }
  static constexpr int kMax = SINGLE ? 1 : kSelectMaxCtas;
};

struct SelectShared {
  union {
    int hist[kSelectBins];     // this CTA's histogram, read by the cluster between the second and the third barrier
    int radix[2][256];         // digit histograms of the radix passes, double-buffered (read by the cluster)
    struct { uint32_t key[kSelectAllCands]; int pos[kSelectAllCands]; } all;   // the cluster's candidates, gathered
  };
  union {
    struct { uint32_t key[kSelectCtaCands]; int pos[kSelectCtaCands]; } cand;  // this CTA's candidates, read by the cluster;
                                                                              // pos: position | kCandUp | kCandDown
    int tot[256];              // radix passes: cluster-wide digit counts
  };
  union {                      // scratch of block-wide reductions, one at a time
    int scan[64];
    uint32_t red[kSelectWarps][6];
    int wtot[kSelectWarps][3];
  };
  uint32_t pub_mm[6], mm[6];   // ranges (as keys) of this CTA, of the cluster
  int n_cand, keep_before;
  int pub_keep, pub_up, pub_down, pub_eq, pub_pos;   // counts of this CTA, read by the cluster
  int cnt_bin[kSelectMaxCtas], cnt_keep[kSelectMaxCtas], cnt_up[kSelectMaxCtas], cnt_down[kSelectMaxCtas];
  int digit, krem;             // (also: the threshold bin and the rank inside it)
  uint32_t T;
  int posT;
};
constexpr int kCandUp = 1 << 31, kCandDown = 1 << 30, kCandPos = kCandDown - 1;

// Range of positions owned by CTA `rank` when N positions are split over `ncta` CTAs.
__device__ __forceinline__ void cta_range(int N, int ncta, int rank, int* begin, int* end) {
  const int span = (N + ncta - 1) / ncta;
  *begin = min(N, rank * span);
  *end = min(N, *begin + span);
}
// Range of a CTA's positions owned by one of its warps.
__device__ __forceinline__ void warp_range(int cnt, int warp, int* lo, int* hi) {
  const int span = ((cnt + kSelectWarps - 1) / kSelectWarps + 31) & ~31;
  *lo = min(cnt, warp * span);
  *hi = min(cnt, *lo + span);
}
__device__ __forceinline__ float key_value(uint32_t key) {   // inverse of rank_key
  return __uint_as_float((key & 0x80000000u) ? (key ^ 0x80000000u) : ~key);
}

// Warp 0 finds the digit whose bin holds the krem-th largest remaining key, given bin counts tot[256].
__device__ __noinline__ void find_digit(const int* tot, int krem, SelectShared* sh) {
  const int tid = threadIdx.x;
  if (tid < 32) {
    int c[8], local = 0;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      c[b] = tot[tid * 8 + b];
      local += c[b];
    }
    int above = local;   // inclusive suffix sum over lanes: keys in this lane's bins and in all higher bins
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_down_sync(0xFFFFFFFFu, above, o);
      if (tid + o < 32) above += y;
    }
    int cum = above - local;
#pragma unroll
    for (int b = 7; b >= 0; --b) {
      if (cum < krem && cum + c[b] >= krem) {
        sh->digit = tid * 8 + b;
        sh->krem = krem - cum;
      }
      cum += c[b];
    }
  }
}

// Digit histogram of the keys that match (mask, prefix).  Keys of one step share their leading bits, so lanes
// of a warp mostly hit the same bin: lanes with equal digits are grouped and one of them adds the group's count.
__device__ __noinline__ void digit_histogram(const uint32_t* keys, int cnt, uint32_t mask, uint32_t prefix,
                                                int shift, int* hist) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  for (int i0 = 0; i0 < cnt; i0 += nthr) {
    const int i = i0 + tid;
    int digit = -1;
    if (i < cnt) {
      const uint32_t key = keys[i];
      if ((key & mask) == prefix) digit = (int)((key >> shift) & 255u);
    }
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, digit);
    if (digit >= 0 && (int)(__ffs(peers) - 1) == (tid & 31)) atomicAdd(&hist[digit], __popc(peers));
  }
}

// Sum over the block, added to *out (shared memory, zeroed by the caller and synchronised around the call).
__device__ __forceinline__ void block_add(int x, int* out) {
  x = __reduce_add_sync(0xFFFFFFFFu, x);
  if ((threadIdx.x & 31) == 0 && x != 0) atomicAdd(out, x);
}

// (T, posT) of the B-th largest of the cluster's keys by radix passes, for any distribution of keys; N > B >= 1.  Returns
// whether more protected rows than B exist (only the first B of them can then stay).  keys[0 .. cnt): this CTA's keys.
template <bool SINGLE>
__device__ __noinline__ bool radix_threshold(const uint32_t* keys, int begin, int cnt, int B, SelectShared* sh) {
  using G = Peers<SINGLE>;
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int ncta = G::count(), rank = G::rank();
  G::sync();                                    // (the histograms below lie over data the cluster may still read)
  uint32_t prefix = 0, mask = 0;
  int krem = B, buf = 0;
#pragma unroll 1
  for (int shift = 24; shift >= 0; shift -= 8, buf ^= 1) {
    int* hist = sh->radix[buf];
    for (int b = tid; b < 256; b += nthr) hist[b] = 0;
    __syncthreads();
    digit_histogram(keys, cnt, mask, prefix, shift, hist);
    G::sync();
    // every CTA folds all histograms and finds the same digit
    if (tid < 256) {
      int v[G::kMax];
#pragma unroll
      for (int r = 0; r < G::kMax; ++r)      // all remote loads in flight before the first add
        v[r] = r < ncta ? G::of(hist, r)[tid] : 0;
      int t = 0;
#pragma unroll
      for (int r = 0; r < G::kMax; ++r) t += v[r];
      sh->tot[tid] = t;
    }
    __syncthreads();
    find_digit(sh->tot, krem, sh);
    __syncthreads();
    prefix |= (uint32_t)sh->digit << shift;
    mask |= 255u << shift;
    krem = sh->krem;
  }
  // the krem-th tie, counted over the CTAs in order: its position
  const int chunk = (cnt + nthr - 1) / nthr;
  const int lo = min(cnt, tid * chunk), hi = min(cnt, lo + chunk);
  int eq = 0, eq_total;
  for (int i = lo; i < hi; ++i) eq += keys[i] == prefix;
  int before = block_excl_scan_int(eq, sh->scan, &eq_total);
  if (tid == 0) {
    sh->pub_eq = eq_total;
    sh->pub_pos = -1;
  }
  G::sync();
  int eq_all = 0;
  for (int r = 0; r < ncta; ++r) {
    const int e = *G::of(&sh->pub_eq, r);
    if (r < rank) before += e;
    eq_all += e;
  }
  if (before < krem && before + eq >= krem)          // one thread of the cluster
    for (int i = lo; i < hi; ++i)
      if (keys[i] == prefix && ++before == krem) sh->pub_pos = begin + i;
  G::sync();
  if (tid == 0) {
    int p = -1;
    for (int r = 0; r < ncta; ++r) p = max(p, *G::of(&sh->pub_pos, r));
    sh->T = prefix;
    sh->posT = p;
  }
  __syncthreads();
  return prefix == kKeyProtected && eq_all > krem;
}

// The bin of the target-th row from the top, of the cluster's histograms hist[0 .. bins), into sh->digit, its rank inside
// the bin into sh->krem and the CTAs' shares of the bin into sh->cnt_bin; what the lower ranks hold in the bins above is
// added to sh->keep_before.  Thread t looks at bin (last - t); every CTA finds the bin for itself.
template <bool SINGLE>
__device__ __forceinline__ void find_bin(int* hist, int bins, int target, SelectShared* sh) {
  using G = Peers<SINGLE>;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, ncta = G::count(), rank = G::rank(), b = bins - 1 - tid;
  int v[G::kMax], tot = 0, before = 0;
#pragma unroll
  for (int r = 0; r < G::kMax; ++r) v[r] = b >= 0 && r < ncta ? G::of(hist, r)[b] : 0;
#pragma unroll
  for (int r = 0; r < G::kMax; ++r) {
    tot += v[r];
    before += r < rank ? v[r] : 0;
  }
  int above = tot;                                     // inclusive over the warp's lanes, then over its lower warps
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xFFFFFFFFu, above, o);
    if (lane >= o) above += y;
  }
  if (lane == 31) sh->wtot[warp][0] = above;
  __syncthreads();
  above += __reduce_add_sync(0xFFFFFFFFu, lane < warp ? sh->wtot[lane][0] : 0) - tot;
  if (above < target && above + tot >= target) {
    sh->digit = b;
    sh->krem = target - above;
#pragma unroll
    for (int r = 0; r < G::kMax; ++r) sh->cnt_bin[r] = v[r];
  }
  __syncthreads();
  block_add(b > sh->digit ? before : 0, &sh->keep_before);
}

// Finer bins of a crowded one: equal steps of the key between its edges (monotone, so a key may be a step off).
struct SubBins {
  uint32_t lo;
  float scale;
  __device__ __forceinline__ int of(uint32_t key) const {
    return key > lo ? (int)fminf((float)(kSelectSubBins - 1), (float)(key - lo) * scale) : 0;
  }
};

// The threshold bin, bf's sh->digit, in finer ones: as find_bin, for the sh->krem-th row of it.  Returns whether the finer
// bin holds one key only, which is then sh->T.  mem: 3 kSelectSubBins words that the cluster may read until the next barrier.
template <bool SINGLE>
__device__ __noinline__ bool refine_bin(const uint32_t* keys, const uint16_t* bf, int cnt, SubBins sub, uint32_t* mem, SelectShared* sh) {
  using G = Peers<SINGLE>;
  const int tid = threadIdx.x, lane = tid & 31, bstar = sh->digit, target = sh->krem;
  int* hist = reinterpret_cast<int*>(mem);
  uint32_t *lo = mem + kSelectSubBins, *hi = lo + kSelectSubBins;
  if (tid < kSelectSubBins) {
    hist[tid] = 0;
    lo[tid] = 0xFFFFFFFFu;
    hi[tid] = 0;
  }
  __syncthreads();
#pragma unroll 1
  for (int i = tid; i < cnt; i += (int)blockDim.x)
    if ((bf[i] & (kSelectBins - 1)) == bstar) {
      const uint32_t key = keys[i];
      const int b = sub.of(key);
      atomicAdd(&hist[b], 1);
      atomicMin(&lo[b], key);
      atomicMax(&hi[b], key);
    }
  G::sync();
  find_bin<SINGLE>(hist, kSelectSubBins, target, sh);
  const int b = sh->digit;
  const uint32_t first = __reduce_min_sync(0xFFFFFFFFu, lane < G::count() ? G::of(lo, lane)[b] : 0xFFFFFFFFu);
  const uint32_t last = __reduce_max_sync(0xFFFFFFFFu, lane < G::count() ? G::of(hi, lane)[b] : 0u);
  if (tid == 0) sh->T = first;
  __syncthreads();
  return first == last;
}

// Where all rows of the threshold bin have the key sh->T: up to which position those of this CTA stay (N: all of its own, -1:
// none).  The lower ranks' ties come first, then the lower positions; the CTA that holds the last one to stay leaves its
// position in sh->pub_pos, the others -1, so that after the next barrier all can judge rows of any CTA.
__device__ __noinline__ int last_tie(const uint32_t* keys, int begin, int cnt, int N, int rank, SelectShared* sh) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  int mine = sh->krem;
  for (int r = 0; r < rank; ++r) mine -= sh->cnt_bin[r];
  const bool holds = mine > 0 && mine <= sh->cnt_bin[rank];
  if (tid == 0) sh->pub_pos = -1;
  if (holds) {
    const int chunk = (cnt + nthr - 1) / nthr, lo = min(cnt, tid * chunk), hi = min(cnt, lo + chunk);
    const uint32_t T = sh->T;
    int eq = 0, all;
    for (int i = lo; i < hi; ++i) eq += keys[i] == T;
    int before = block_excl_scan_int(eq, sh->scan, &all);
    if (before < mine && before + eq >= mine)            // one thread
      for (int i = lo; i < hi; ++i)
        if (keys[i] == T && ++before == mine) sh->pub_pos = begin + i;
  }
  __syncthreads();
  return holds ? sh->pub_pos : (mine > 0 ? N : -1);
}

// Single-CTA pick used for the small top-A choice over the confidence map: marks the A largest of cnt keys
// in keep[], ties to the lower index.
__device__ inline void block_top_mark(const uint32_t* keys, uint8_t* keep, int cnt, int A, SelectShared* sh) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const bool keep_all = cnt <= A;
  uint32_t T = 0;
  int need_eq = 0;
  if (!keep_all && A > 0) {
    uint32_t prefix = 0, mask = 0;
    int krem = A;
#pragma unroll 1
    for (int shift = 24; shift >= 0; shift -= 8) {
      for (int b = tid; b < 256; b += nthr) sh->tot[b] = 0;
      __syncthreads();
      digit_histogram(keys, cnt, mask, prefix, shift, sh->tot);
      __syncthreads();
      find_digit(sh->tot, krem, sh);
      __syncthreads();
      prefix |= (uint32_t)sh->digit << shift;
      mask |= 255u << shift;
      krem = sh->krem;
      __syncthreads();
    }
    T = prefix;
    need_eq = krem;
  }
  const int chunk = (cnt + nthr - 1) / nthr;
  const int lo = min(cnt, tid * chunk), hi = min(cnt, lo + chunk);
  int cnt_eq = 0;
  if (!keep_all && A > 0)
    for (int i = lo; i < hi; ++i) cnt_eq += keys[i] == T;
  int tot;
  int eq_rank = block_excl_scan_int(cnt_eq, sh->scan, &tot);
  for (int i = lo; i < hi; ++i) {
    bool k = keep_all;
    if (!keep_all && A > 0) k = keys[i] > T || (keys[i] == T && eq_rank++ < need_eq);
    keep[i] = k ? 1 : 0;
  }
  __syncthreads();
}

__host__ __device__ inline size_t select_header_bytes() { return (sizeof(SelectShared) + 15) & ~(size_t)15; }

// Shared memory a CTA of the stand-alone selection needs for `span` owned positions: their keys.
__host__ __device__ inline size_t select_smem_bytes(int span) { return select_header_bytes() + (((size_t)span * 4 + 15) & ~(size_t)15); }

// The fused per-step kernel keeps, per position, the value or key (4 bytes), bin and flag (2), id (8), stored score (4)
// and slot (4) on chip.  Behind them lie the frame's m raw residual norms and the np confidence keys and marks, which the
// flags and values are made of, and later, in the same place, a block of sums and a list of rows for the key sums' corrections: a
// CTA lists at most m rows that leave and its share of the m that come.  Largest caches of small frames do without that
// block (room 0: their sums are taken afresh each step) rather than be refused.
constexpr int kDeltaCols = 1024;
static_assert(3 * kSelectSubBins <= kDeltaCols, "the finer bins lie in the block of sums");
__host__ __device__ inline size_t compress_smem_bytes(int span, int ncta, int np, int m, bool room) {
  const size_t s4 = ((size_t)span + 3) & ~(size_t)3, m4 = ((size_t)m + 3) & ~(size_t)3, np4 = ((size_t)np + 3) & ~(size_t)3;
  const size_t early = m4 * 4 + np4 * 4 + ((np4 + 15) & ~(size_t)15);
  const size_t late = room ? (size_t)kDeltaCols * 4 + ((size_t)m + (size_t)sums_share(m, ncta)) * 4 : 0;
  return select_header_bytes() + s4 * (8 + 3 * 4) + ((s4 + 7) & ~(size_t)7) * 2 + (early > late ? early : late);
}

// Per-warp totals of the rows that stay, and of two marked kinds of rows, for the warp's range of positions; then the
// block's exclusive prefix of them.  `row(i, keep, up, down)` classifies a position.  All threads call it.
template <typename F>
__device__ __forceinline__ void warp_totals(int lo, int hi, SelectShared* sh, F row, int* keep0, int* up0, int* down0) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int k = 0, u = 0, d = 0;
  for (int i = lo + lane; i < hi; i += 32) {
    bool keep, up, down;
    row(i, keep, up, down);
    k += keep;
    u += up;
    d += down;
  }
  k = __reduce_add_sync(0xFFFFFFFFu, k);
  u = __reduce_add_sync(0xFFFFFFFFu, u);
  d = __reduce_add_sync(0xFFFFFFFFu, d);
  if (lane == 0) {
    sh->wtot[warp][0] = k;
    sh->wtot[warp][1] = u;
    sh->wtot[warp][2] = d;
  }
  __syncthreads();
  const bool mine = lane < warp;                     // (16 warps: the lanes of one warp cover them)
  *keep0 = __reduce_add_sync(0xFFFFFFFFu, mine ? sh->wtot[lane][0] : 0);
  *up0 = __reduce_add_sync(0xFFFFFFFFu, mine ? sh->wtot[lane][1] : 0);
  *down0 = __reduce_add_sync(0xFFFFFFFFu, mine ? sh->wtot[lane][2] : 0);
}

// ---- standalone selection over given priorities: one cluster per independent problem (blockIdx.y)

template <bool SINGLE>
__global__ void __launch_bounds__(kSelectThreads) k_select(const float* __restrict__ r,
                                                           const uint8_t* __restrict__ flags_in, int N, int B,
                                                           int* __restrict__ survivors, int* status) {
  extern __shared__ __align__(16) unsigned char smem_select[];
  using G = Peers<SINGLE>;
  SelectShared* sh = reinterpret_cast<SelectShared*>(smem_select);
  uint32_t* keys = reinterpret_cast<uint32_t*>(smem_select + select_header_bytes());
  const int ncta = G::count(), rank = G::rank();
  int begin, end;
  cta_range(N, ncta, rank, &begin, &end);
  const int cnt = end - begin;
  const size_t prob = blockIdx.y;
  const float* rr = r + prob * (size_t)N;
  const uint8_t* ff = flags_in + prob * (size_t)N;
  for (int i = threadIdx.x; i < cnt; i += blockDim.x)
    keys[i] = ff[begin + i] != 0 ? kKeyProtected : rank_key(rr[begin + i]);
  __syncthreads();
  uint32_t T = 0;
  int posT = N;
  bool bad = false;
  if (N > B) {
    bad = radix_threshold<SINGLE>(keys, begin, cnt, B, sh);
    T = sh->T;
    posT = sh->posT;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int lo, hi, j, u0, d0;
  warp_range(cnt, warp, &lo, &hi);
  auto kept = [&](int i) { return keys[i] > T || (keys[i] == T && begin + i <= posT); };
  warp_totals(lo, hi, sh, [&](int i, bool& k, bool& u, bool& d) { k = kept(i); u = d = false; }, &j, &u0, &d0);
  if (threadIdx.x == kSelectThreads - 32) sh->pub_keep = j + sh->wtot[warp][0];   // (the last warp knows the total)
  G::sync();
  int all = 0;
  for (int q = 0; q < ncta; ++q) {
    const int c = *G::of(&sh->pub_keep, q);
    if (q < rank) j += c;
    all += c;
  }
  int* out = survivors + prob * (size_t)min(N, B);
  for (int i0 = lo; i0 < hi; i0 += 32) {
    const int i = i0 + lane;
    const bool k = i < hi && kept(i);
    const unsigned m = __ballot_sync(0xFFFFFFFFu, k);
    if (k) out[j + __popc(m & ((1u << lane) - 1))] = begin + i;
    j += __popc(m);
  }
  if ((bad || all != min(N, B)) && threadIdx.x == 0 && status) atomicCAS(status, 0, OVGGT_ERR_DEVICE_STATUS);
  G::leave();
}

// ---- the fused per-step kernel

struct CompressParams {
  int n, M, B;                      // cached rows, new rows, budget
  int n_special, grid_h, grid_w;
  float alpha, w_center, w_edge, w_corner;   // Eq. 6: blend and the normalised 3x3 Gaussian weights
  float beta;
  int mode;                         // OVGGT_SCORE_*
  int protect_new;                  // != 0: give every new row this flag (INIT: first frame; HIST: a camera-cache anchor)
  unsigned long long step_key;      // OVGGT_SCORE_RANDOM: SplitMix64(seed ^ frame id) of this step
  float lone_new;                   // >= 0: normalised score of a new group without a range (Eq. 7's 0/0); < 0: 0
  int register_anchor, A;           // 1: flag the A most confident patches of the new frame HIST
  long long demote_frame;           // >= 0: release the HIST rows of that frame
  const float* s_raw;               // [M] residual norms of the new rows
  const float* d;                   // key diversity (hybrid mode), indexed by the row's physical slot
  const float* conf;                // [grid_h*grid_w]
  const float* override_r;          // [N] or nullptr
  const long long* ids_src; const uint8_t* flags_src; const float* stored_src;   // [N] pre-compaction meta
  long long* ids_dst; uint8_t* flags_dst; float* stored_dst;                     // [<=B] compacted meta
  float* r_out;                     // [N] priorities as computed here
  int* survivors;                   // [min(N, B)]
  int* status;
  int* n_keep_out;
  // Hole-filling layout (fill != 0): the K/V row of logical position g lives in slot slot_src[g] (g < n) or g
  // (new rows); the K/V rows are not gathered.  Survivors whose slot is >= B have to move into the slots < B
  // that evicted rows leave: the i-th such survivor (in logical order) goes to the i-th such slot (in the logical
  // order of the rows that leave).  The kernel writes the pairs, the survivors' slots, and the step's stamp beside every
  // slot that will be filled; the layer's next append copies the rows and patches slot_dst[move_j[i]] = move_dst[i].
  int fill;
  const int* slot_src;              // [n]
  int* slot_dst;                    // [<= B]
  int* move_src; int* move_dst; int* move_j;   // [<= M] each
  int* tail_move;                   // [M]: for slot B + i, the index of the move that empties it, or -1
  int* n_moves_out;
  int* hole_stamp; int stamp;       // [B]
  uint4 *move_k, *move_v;           // not nullptr (a frame of one row, one CTA): the pair is moved here, not by the next append
  const uint4* resid;               // [M, C] or nullptr: compute the residual norms here instead of reading s_raw (small M)
  // Column sums of the keys that stay: ksum_next = ksum (or 0) + admitted keys - evicted keys; ksum_next nullptr: not asked for.
  const uint4* k_cache; int nvec;
  int room;                         // the block of sums and the list have their place in shared memory (needed for ksum_next)
  const float* ksum; float* ksum_next;   // [C]
  // Where the attention beside this kernel takes the sums instead (see KeySums): the list of rows, by CTA of the cluster.
  int* sums_list; int sums_cap;     // [CTAs][sums_cap]: ~slot of a row that leaves, the slot of one that comes, or kSumsNone
  int* sums_out;                    // [CTAs] rows that leave
};

// Eq. 6 for new-frame token j (aux tokens keep their raw score); s_raw: the frame's M residual norms.
__device__ __forceinline__ float smoothed_score(const CompressParams& P, const float* s_raw, int j) {
  float v = s_raw[j];
  if (j >= P.n_special) {
    const int q = j - P.n_special, y = q / P.grid_w, x = q - y * P.grid_w;
    const float* S = s_raw + P.n_special;
    float conv = 0.0f;
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        const int yy = min(max(y + dy, 0), P.grid_h - 1), xx = min(max(x + dx, 0), P.grid_w - 1);
        const float w = (dx == 0 && dy == 0) ? P.w_center : ((dx == 0 || dy == 0) ? P.w_edge : P.w_corner);
        conv = __fmaf_rn(w, S[yy * P.grid_w + xx], conv);
      }
    v = __fmaf_rn(P.alpha, conv, __fmul_rn(1.0f - P.alpha, v));
  }
  return v;
}

// ksum_next = ksum + (keys admitted - keys evicted) by the whole cluster: each CTA adds up the rows of its list, whose first
// n_out entries leave and whose others come (< 0: nothing), then the CTAs are folded in rank order.  A warp owns a line of
// eight vectors of all rows, its four lane groups take every fourth row with eight loads in flight each, so the fold inside
// the CTA is two shuffles; every order is fixed, whatever the timing.
template <int DT, bool SINGLE>
__device__ __noinline__ void fold_key_sums(const CompressParams& P, const int* list, int n_out, int n_list, float* part) {
  constexpr int VEC = VecOf<DT>::n, VB = kDeltaCols / VEC;        // vectors of a block of columns
  using G = Peers<SINGLE>;
  const int ncta = G::count(), rank = G::rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, grp = lane >> 3;
  const int C = P.nvec * VEC, share = kDeltaCols / G::kMax;       // columns of a block that a CTA finishes
  for (int v0 = 0; v0 < P.nvec; v0 += VB) {
    float base[(kDeltaCols + kSelectThreads - 1) / kSelectThreads];
#pragma unroll
    for (int k = 0; k * kSelectThreads < share; ++k) {
      const int x = k * kSelectThreads + tid, c = v0 * VEC + rank * share + x;
      base[k] = P.ksum != nullptr && x < share && c < C ? P.ksum[c] : 0.0f;
    }
#pragma unroll 1
    for (int w = warp; w < VB / 8 && v0 + w * 8 < P.nvec; w += kSelectWarps) {
      const int vec = v0 + w * 8 + (lane & 7);
      const bool in = vec < P.nvec;
      float acc[VEC];
#pragma unroll
      for (int e = 0; e < VEC; ++e) acc[e] = 0.0f;
#pragma unroll 1
      for (int e0 = grp; e0 < n_list; e0 += 32) {
        uint4 u[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int slot = e0 + 4 * k < n_list && in ? list[e0 + 4 * k] : -1;
          u[k] = slot >= 0 ? P.k_cache[(size_t)slot * P.nvec + vec] : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float sign = e0 + 4 * k < n_out ? -1.0f : 1.0f;
          float f[VEC];
          unpack<DT>(u[k], f);
#pragma unroll
          for (int e = 0; e < VEC; ++e) acc[e] = __fmaf_rn(f[e], sign, acc[e]);
        }
      }
#pragma unroll
      for (int e = 0; e < VEC; ++e) {
        acc[e] += __shfl_xor_sync(0xFFFFFFFFu, acc[e], 8);
        acc[e] += __shfl_xor_sync(0xFFFFFFFFu, acc[e], 16);
      }
      if (grp == 0)
#pragma unroll
        for (int e = 0; e < VEC; ++e) part[(w * 8 + lane) * VEC + e] = acc[e];
    }
    G::sync();
#pragma unroll
    for (int k = 0; k * kSelectThreads < share; ++k) {
      const int x = k * kSelectThreads + tid, y = rank * share + x, c = v0 * VEC + y;
      if (x < share && c < C) {
        float v[G::kMax];                             // all remote reads in flight before the first add
#pragma unroll
        for (int q = 0; q < G::kMax; ++q) v[q] = q < ncta ? G::of(part, q)[y] : 0.0f;
#pragma unroll
        for (int q = 0; q < G::kMax; ++q) base[k] += v[q];
        P.ksum_next[c] = base[k];
      }
    }
    if (v0 + VB < P.nvec) G::sync();                  // (part is written again)
  }
}

// ONE: a single CTA and one row more than the budget, as in a cache of one token a frame that is full; two reductions find the row
// that leaves, and the admitted one is moved here where that is asked for.  An instance of its own, since its code slows the
// general one down (steps over 300 rows of 5 / 20 / 69 tokens, bf16: 16.3 / 16.8 / 19.0 us beside it, 15.6 / 16.1 / 18.6 without)
// and the other way round (camera head, 16 heads and 144 rows, fp32: 13.2 and 12.7 us a layer).
template <int DT, bool SINGLE, bool ONE = false>
__device__ __forceinline__ void compress_select_body(const CompressParams& P, unsigned char* smem) {
  using G = Peers<SINGLE>;
  const int ncta = G::count(), rank = G::rank();
  SelectShared* sh = reinterpret_cast<SelectShared*>(smem);
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int n = P.n, M = P.M, N = n + M, Np = P.grid_h * P.grid_w;
  int begin, end;
  cta_range(N, ncta, rank, &begin, &end);
  const int cnt = end - begin, span4 = ((N + ncta - 1) / ncta + 3) & ~3;
  unsigned char* p = smem + select_header_bytes();
  long long* sid = reinterpret_cast<long long*>(p);               // ids of the owned positions
  uint32_t* keys = reinterpret_cast<uint32_t*>(sid + ((span4 + 1) & ~1));   // their values, then the priorities' keys, in place
  float* val = reinterpret_cast<float*>(keys);
  float* sst = reinterpret_cast<float*>(keys + span4);            // their stored scores
  int* ssl = reinterpret_cast<int*>(sst + span4);                 // their physical slots
  uint16_t* bf = reinterpret_cast<uint16_t*>(ssl + span4);        // flag << 14 | bin of the owned positions
  float* sraw = reinterpret_cast<float*>(bf + ((span4 + 7) & ~7));        // [M] the frame's residual norms
  uint32_t* ckeys = reinterpret_cast<uint32_t*>(sraw + ((M + 3) & ~3));   // [Np] confidence keys
  uint8_t* cmark = reinterpret_cast<uint8_t*>(ckeys + ((Np + 3) & ~3));   // [Np] the most confident patches
  float* part = sraw;   // over the last three, which are dead by then: [kDeltaCols] this CTA's corrections of the key sums
  int* list = reinterpret_cast<int*>(part + kDeltaCols);          // [M + its share of M] slots of the rows they are made of
  const bool hybrid = P.mode == OVGGT_SCORE_HYBRID, choose = N > P.B;
  pdl_wait();
  pdl_trigger();   // an attention queued behind this kernel reads nothing of it: it starts as soon as this one runs
  const bool own_rank = P.override_r == nullptr;                  // rank the priorities computed here

  // -- anchor registration (Sec. 3.3): the A most confident patch tokens of the new frame, ties to the lower
  //    index.  Every CTA that owns new rows computes the same marks and uses those of the positions it owns.
  const bool reg = P.register_anchor && P.A > 0 && end > n;
  if (reg) {
    for (int i = tid; i < Np; i += nthr) ckeys[i] = rank_key(P.conf[i]);
    __syncthreads();
    block_top_mark(ckeys, cmark, Np, P.A, sh);
  }

  // -- protection flags and values of the owned positions, and the ranges of the evictable ones (as keys): cached group,
  //    new group (Eq. 7), ranked values.  A CTA that owns new rows first stages the frame's raw norms (Eq. 6 reads each
  //    nine times); all global loads of four positions are issued before any is used.
  sh->hist[tid] = 0;
  if (tid == 0) sh->n_cand = sh->pub_up = sh->pub_down = sh->keep_before = 0;
  if (end > n) {
    if (P.resid != nullptr) {
      // (from the last warp on: the first ones have positions to load)
      for (int j = kSelectWarps - 1 - warp; j < M; j += kSelectWarps) warp_row_norm<DT>(P.resid, j, P.nvec, sraw);
    } else {
      for (int j = tid; j < M; j += nthr) sraw[j] = P.s_raw[j];
    }
  }
  uint32_t mn[3] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu}, mx[3] = {0u, 0u, 0u};
  // (a thread touches its own positions only, so the passes need no barrier among them; all loads of a pass are independent)
#pragma unroll 4
  for (int i = tid; i < cnt; i += nthr) {
    const int g = begin + i;
    int sl = g;
    float st = 0.0f;
    if (g < n) {
      st = P.stored_src[g];
      if (P.fill) {
        sl = P.slot_src[g];
        if (!index_ok(sl, P.B + P.M, P.status)) sl = g;
      }
    }
    bf[i] = (uint16_t)((P.flags_src[g] & 3) << 14);
    sid[i] = P.ids_src[g];
    sst[i] = st;
    ssl[i] = sl;
  }
  if (hybrid)
#pragma unroll 4
    for (int i = tid; i < cnt; i += nthr) val[i] = begin + i < n ? P.d[ssl[i]] : 0.0f;
  __syncthreads();                                     // the staged norms are complete
#pragma unroll 1
  for (int i = tid; i < cnt; i += nthr) {
    const int g = begin + i;
    int f = bf[i] >> 14;
    float x;
    if (g >= n) {
      const int j = g - n;
      if (P.protect_new) f = P.protect_new;
      if (reg && j >= P.n_special && cmark[j - P.n_special]) f = OVGGT_FLAG_HIST;
      x = smoothed_score(P, sraw, j);
      sst[i] = x;                // the score the row keeps
    } else {
      if (P.demote_frame >= 0 && f == OVGGT_FLAG_HIST && sid[i] / M == P.demote_frame) f = OVGGT_FLAG_EVICTABLE;
      x = hybrid ? val[i] : sst[i];
    }
    if (P.mode == OVGGT_SCORE_RANDOM) x = random_priority(P.step_key, sid[i]);   // Supp. A: uniform, fresh per step
    bf[i] = (uint16_t)(f << 14);
    val[i] = x;
    if (f == 0) {
      const uint32_t k = rank_key(x);
      if (x == x) {              // (a NaN takes no part in its group's range)
        const bool cached = g < n;
        mn[0] = cached ? min(mn[0], k) : mn[0];
        mx[0] = cached ? max(mx[0], k) : mx[0];
        mn[1] = cached ? mn[1] : min(mn[1], k);
        mx[1] = cached ? mx[1] : max(mx[1], k);
      }
      const float v = own_rank ? x : P.override_r[g];
      if (fabsf(v) < INFINITY) {
        const uint32_t kv = rank_key(v);
        mn[2] = min(mn[2], kv);
        mx[2] = max(mx[2], kv);
      }
    }
  }
  if (hybrid || choose) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      mn[q] = __reduce_min_sync(0xFFFFFFFFu, mn[q]);
      mx[q] = __reduce_max_sync(0xFFFFFFFFu, mx[q]);
    }
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        sh->red[warp][2 * q] = mn[q];
        sh->red[warp][2 * q + 1] = mx[q];
      }
    __syncthreads();
    if (warp < 6) {                                   // one warp per quantity: lanes are the block's warps
      const bool is_max = warp & 1;
      const uint32_t v = lane < kSelectWarps ? sh->red[lane][warp] : (is_max ? 0u : 0xFFFFFFFFu);
      const uint32_t r = is_max ? __reduce_max_sync(0xFFFFFFFFu, v) : __reduce_min_sync(0xFFFFFFFFu, v);
      if (lane == 0) sh->pub_mm[warp] = r;
    }
    G::sync();
    if (warp < 6) {                                   // lanes are the CTAs of the cluster
      const bool is_max = warp & 1;
      const uint32_t v = lane < ncta ? G::of(sh, lane)->pub_mm[warp] : (is_max ? 0u : 0xFFFFFFFFu);
      const uint32_t r = is_max ? __reduce_max_sync(0xFFFFFFFFu, v) : __reduce_min_sync(0xFFFFFFFFu, v);
      if (lane == 0) sh->mm[warp] = r;
    }
    __syncthreads();
  }

  // -- Eq. 7, and a bin for every priority: equal steps of the priority (hybrid, random), or equal steps of its key, which
  //    is logarithmic (residual norms spread over octaves; given priorities may do anything).  Bins only have to be
  //    monotone; how evenly they fill decides how few candidates the last stage ranks.
  const float lo_h = key_value(sh->mm[0]), hi_h = key_value(sh->mm[1]), lo_n = key_value(sh->mm[2]), hi_n = key_value(sh->mm[3]);
  const bool linear = own_rank && (hybrid || P.mode == OVGGT_SCORE_RANDOM);
  const uint32_t bin_key0 = sh->mm[4];
  const float bin_lo = linear ? (hybrid ? 0.0f : key_value(bin_key0)) : 0.0f;
  const float bin_hi = linear ? (hybrid ? fmaxf(P.beta, 1.0f - P.beta) : key_value(sh->mm[5]))
                              : (float)(sh->mm[5] > bin_key0 ? sh->mm[5] - bin_key0 : 0u);
  const float bin_scale = bin_hi - bin_lo > 0.0f && bin_hi - bin_lo < INFINITY ? (float)(kSelectBins - 1) / (bin_hi - bin_lo) : 0.0f;
#pragma unroll 1
  for (int i = tid; i < ((cnt + 31) & ~31); i += nthr) {
    bool prot = false;
    if (i < cnt) {
      const int g = begin + i;
      const int f = bf[i] >> 14;
      float r;
      uint32_t key;
      int bin;
      prot = f != 0;
      if (prot) {
        r = INFINITY;
        key = kKeyProtected;
        bin = kSelectBins - 1;
      } else {
        if (hybrid) {
          const float lo = g < n ? lo_h : lo_n, hi = g < n ? hi_h : hi_n;
          const float w = g < n ? 1.0f - P.beta : P.beta;
          r = hi > lo ? __fmul_rn(w, __fdiv_rn(val[i] - lo, hi - lo))
                      : ((g >= n && P.lone_new >= 0.0f) ? __fmul_rn(w, P.lone_new) : 0.0f);
        } else {
          r = val[i];
        }
        const float v = own_rank ? r : P.override_r[g];
        key = rank_key(v);
        const float steps = linear ? __fmul_rn(v - bin_lo, bin_scale) : (key > bin_key0 ? __fmul_rn((float)(key - bin_key0), bin_scale) : 0.0f);
        bin = (int)fminf((float)(kSelectBins - 2), fmaxf(0.0f, steps));
        if (choose && !ONE) atomicAdd(&sh->hist[bin], 1);
      }
      // The kernel's own priority, also when an override is ranked instead.  Where it can be told from its key it is
      // written with the survivors: a cluster barrier waits for the global stores before it.
      if (!own_rank || !(prot || fabsf(r) < INFINITY)) P.r_out[g] = r;
      keys[i] = key;
      bf[i] = (uint16_t)(f << 14 | bin);
    }
    const unsigned m = __ballot_sync(0xFFFFFFFFu, prot);
    if (m != 0 && lane == 0) atomicAdd(&sh->hist[kSelectBins - 1], __popc(m));
  }

  // -- Eq. 8: (T, posT), and what the lower ranks of the cluster keep and move
  const bool fill = P.fill != 0;
  auto is_up = [&](int i) { return fill ? ssl[i] >= P.B : begin + i >= n; };
  uint32_t T = 0;
  int posT = N, keep_before = begin, up_before = 0, down_before = 0, keep_all = N, up_all = 0, down_all = 0;
  bool bad = false;
  auto classify = [&](int i, bool& keep, bool& up, bool& down) {
    const uint32_t key = keys[i];
    keep = key > T || (key == T && begin + i <= posT);
    const bool u = choose && is_up(i);
    up = keep && u;
    down = choose && !keep && !u;
  };
  int wlo, whi, kw = 0, uw = 0, dw = 0;                // this warp's positions, and what the block's lower warps hold
  warp_range(cnt, warp, &wlo, &whi);
  if constexpr (ONE) {
    // the row that leaves: the lowest key, of equal ones the last
    uint32_t key = 0xFFFFFFFFu;
    int pos = -1;
    for (int i = tid; i < cnt; i += nthr)
      if (keys[i] <= key) {
        key = keys[i];
        pos = i;
      }
    auto lowest = [&]() {
      const uint32_t k = __reduce_min_sync(0xFFFFFFFFu, key);
      pos = __reduce_max_sync(0xFFFFFFFFu, key == k ? pos : -1);
      key = k;
    };
    lowest();
    if (lane == 0) {
      sh->red[warp][0] = key;
      sh->red[warp][1] = (uint32_t)pos;
    }
    __syncthreads();
    key = lane < kSelectWarps ? sh->red[lane][0] : 0xFFFFFFFFu;
    pos = lane < kSelectWarps ? (int)sh->red[lane][1] : -1;
    lowest();
    __syncthreads();                                   // (warp_totals writes over them)
    T = key;
    posT = pos - 1;
    bad = key == kKeyProtected;
    keep_before = 0;
    keep_all = P.B;
    warp_totals(wlo, whi, sh, classify, &kw, &uw, &dw);
    up_all = __reduce_add_sync(0xFFFFFFFFu, lane < kSelectWarps ? sh->wtot[lane][1] : 0);
    down_all = __reduce_add_sync(0xFFFFFFFFu, lane < kSelectWarps ? sh->wtot[lane][2] : 0);
  } else if (!choose) {
    __syncthreads();
    kw = wlo;                                          // everything stays
  } else {
    G::sync();
    find_bin<SINGLE>(sh->hist, kSelectBins, P.B, sh);
    const int bstar = sh->digit;
    int cands = 0, sstar = -1;
    bool crowded = bstar == kSelectBins - 1;           // (more protected rows than B: an error the slow way reports)
    auto count = [&]() {
      cands = 0;
      for (int r = 0; r < ncta; ++r) {
        cands += sh->cnt_bin[r];
        crowded |= sh->cnt_bin[r] > kSelectCtaCands;
      }
      crowded |= cands > kSelectAllCands;
    };
    count();
    // a crowded bin in finer ones, equal steps of the key between its edges (monotone, so a key may be a step off)
    SubBins sub = {0, 1.0f};
    bool ties = false;
    if (!SINGLE && P.room && crowded && bstar < kSelectBins - 1) {   // (one CTA's radix passes are cheap: no cluster barriers)
      const float step = bin_scale > 0.0f ? 1.0f / bin_scale : 0.0f, e0 = (float)bstar * step, e1 = (float)(bstar + 1) * step;
      sub.lo = linear ? rank_key(bin_lo + e0) : bin_key0 + (uint32_t)e0;
      const uint32_t hi = linear ? rank_key(bin_lo + e1) : bin_key0 + (uint32_t)e1;
      if (hi > sub.lo) sub.scale = (float)kSelectSubBins / (float)(hi - sub.lo);
      ties = refine_bin<SINGLE>(keys, bf, cnt, sub, reinterpret_cast<uint32_t*>(part), sh);   // (the block of sums is not in use yet)
      sstar = sh->digit;
      crowded = false;
      count();
    }
    if (!crowded) {
      int up = 0, down = 0;
#pragma unroll 1
      for (int i = tid; i < cnt; i += nthr) {
        int side = (bf[i] & (kSelectBins - 1)) - bstar;
        if (!SINGLE && side == 0 && sstar >= 0) side = sub.of(keys[i]) - sstar;
        const bool u = is_up(i);
        up += side > 0 && u;
        down += side < 0 && !u;
        if (side == 0) {
          const int c = atomicAdd(&sh->n_cand, 1);     // (in whatever order: they are ranked by key and position)
          if (c < kSelectCtaCands) {
            sh->cand.key[c] = keys[i];
            sh->cand.pos[c] = (begin + i) | (u ? kCandUp : kCandDown);
          }
        }
      }
      block_add(up, &sh->pub_up);
      block_add(down, &sh->pub_down);
      G::sync();
      uint32_t key = 0;
      int pos = 0, owner = 0, idx = tid;
      if (tid < cands) {
        while (idx >= sh->cnt_bin[owner]) idx -= sh->cnt_bin[owner++];
        const SelectShared* o = G::of(sh, owner);
        key = sh->all.key[tid] = o->cand.key[idx];
        pos = sh->all.pos[tid] = o->cand.pos[idx];
      }
      if (tid >= cands && tid < ((cands + 3) & ~3)) {  // (the ranking loop reads four at a time)
        sh->all.key[tid] = 0;
        sh->all.pos[tid] = kCandPos;
      }
      if (tid >= nthr - 32 && lane < ncta) {
        sh->cnt_up[lane] = G::of(sh, lane)->pub_up;
        sh->cnt_down[lane] = G::of(sh, lane)->pub_down;
      }
      __syncthreads();
      const int krem = sh->krem;
      if (tid < cands) {
        int before = 0;
        const int at = pos & kCandPos;
        for (int j = 0; j < cands; j += 4) {
          const uint4 k4 = *reinterpret_cast<const uint4*>(&sh->all.key[j]);
          const int4 p4 = *reinterpret_cast<const int4*>(&sh->all.pos[j]);
          before += (k4.x > key || (k4.x == key && (p4.x & kCandPos) < at)) + (k4.y > key || (k4.y == key && (p4.y & kCandPos) < at)) +
                    (k4.z > key || (k4.z == key && (p4.z & kCandPos) < at)) + (k4.w > key || (k4.w == key && (p4.w & kCandPos) < at));
        }
        if (before == krem - 1) {
          sh->T = key;
          sh->posT = pos & kCandPos;
        }
        const bool in = before < krem;
        if (in && owner < rank) atomicAdd(&sh->keep_before, 1);
        if (in && (pos & kCandUp)) atomicAdd(&sh->cnt_up[owner], 1);
        if (!in && (pos & kCandDown)) atomicAdd(&sh->cnt_down[owner], 1);
      }
      __syncthreads();
      T = sh->T;
      posT = sh->posT;
      keep_before = sh->keep_before;
      keep_all = P.B;
      warp_totals(wlo, whi, sh, classify, &kw, &uw, &dw);
    } else {
      if (!SINGLE && ties) {
        T = sh->T;
        posT = last_tie(keys, begin, cnt, N, rank, sh);
      } else {
        bad = radix_threshold<SINGLE>(keys, begin, cnt, P.B, sh);
        T = sh->T;
        posT = sh->posT;
      }
      warp_totals(wlo, whi, sh, classify, &kw, &uw, &dw);
      if (tid == nthr - 32) {                          // the last warp: its prefix and its own count are the CTA's total
        sh->pub_keep = kw + sh->wtot[kSelectWarps - 1][0];
        sh->pub_up = uw + sh->wtot[kSelectWarps - 1][1];
        sh->pub_down = dw + sh->wtot[kSelectWarps - 1][2];
      }
      G::sync();
      if (warp == 0) {                                 // lanes are the CTAs of the cluster
        const SelectShared* o = G::of(sh, min(lane, ncta - 1));
        if (lane < ncta) {
          sh->cnt_keep[lane] = o->pub_keep;
          sh->cnt_up[lane] = o->pub_up;
          sh->cnt_down[lane] = o->pub_down;
        }
        const int pos = __reduce_max_sync(0xFFFFFFFFu, o->pub_pos);
        if (lane == 0) sh->posT = pos;
      }
      __syncthreads();
      posT = sh->posT;                                 // (of the whole cluster, also where ties were settled by each CTA)
      keep_before = keep_all = 0;
      for (int r = 0; r < ncta; ++r) {
        if (r < rank) keep_before += sh->cnt_keep[r];
        keep_all += sh->cnt_keep[r];
      }
    }
    for (int r = 0; r < ncta; ++r) {
      if (r < rank) {
        up_before += sh->cnt_up[r];
        down_before += sh->cnt_down[r];
      }
      up_all += sh->cnt_up[r];
      down_all += sh->cnt_down[r];
    }
  }

  // -- column sums of the keys that stay, before anything is written (a cluster barrier waits for the global stores before
  //    it).  A CTA takes the rows that leave from its own positions, and of the frame's rows, which the last CTAs own, its
  //    share, by a look at their keys.
  const unsigned below = (1u << lane) - 1;
  if (P.ksum_next != nullptr) {
    int n_out = 0;
    if (choose) {
      int d = dw;
#pragma unroll 1
      for (int i0 = wlo; i0 < whi; i0 += 32) {
        bool keep, up, down = false;
        if (i0 + lane < whi) classify(i0 + lane, keep, up, down);
        const unsigned m = __ballot_sync(0xFFFFFFFFu, down);
        const int at = d + __popc(m & below);
        if (down && at < M) list[at] = ssl[i0 + lane];
        d += __popc(m);
      }
      n_out = min(M, (int)__reduce_add_sync(0xFFFFFFFFu, lane < kSelectWarps ? sh->wtot[lane][2] : 0));
    }
    const int span = (N + ncta - 1) / ncta, per = sums_share(M, ncta), first = min(M, rank * per), n_in = min(M, first + per) - first;
    for (int j = tid; j < n_in; j += nthr) {
      const int g = n + first + j, owner = g / span;
      const uint32_t key = choose ? G::of(keys, owner)[g - owner * span] : 0u;
      list[n_out + j] = !choose || key > T || (key == T && g <= posT) ? g : -1;
    }
    __syncthreads();
    fold_key_sums<DT, SINGLE>(P, list, n_out, n_out + n_in, part);
  }

  // -- survivors, compacted meta (order preserved), and the lists of rows that come and go
  int j0 = keep_before + kw, u0 = up_before + uw, d0 = down_before + dw;
#pragma unroll 1
  for (int i0 = wlo; i0 < whi; i0 += 32) {
    const int i = i0 + lane, g = begin + i;
    bool keep = false, up = false, down = false;
    if (i < whi) classify(i, keep, up, down);
    const unsigned mk = __ballot_sync(0xFFFFFFFFu, keep), mu = __ballot_sync(0xFFFFFFFFu, up),
                   md = __ballot_sync(0xFFFFFFFFu, down);
    const int j = j0 + __popc(mk & below), iu = u0 + __popc(mu & below), id = d0 + __popc(md & below);
    j0 += __popc(mk);
    u0 += __popc(mu);
    d0 += __popc(md);
    if (i < whi) {
      const int slot = ssl[i];
      const float r = keys[i] == kKeyProtected ? INFINITY : key_value(keys[i]);
      if (own_rank && (keys[i] == kKeyProtected || fabsf(r) < INFINITY)) P.r_out[g] = r;
      if (keep && j < P.B) {
        P.survivors[j] = g;
        P.ids_dst[j] = sid[i];
        P.flags_dst[j] = (uint8_t)(bf[i] >> 14);
        P.stored_dst[j] = sst[i];
        if (fill) P.slot_dst[j] = slot;
      }
      if (fill && up && iu < M) {
        P.move_src[iu] = slot;
        P.move_j[iu] = j;
        if (ONE && P.move_k != nullptr) {
          sh->cnt_bin[0] = slot;
          sh->cnt_bin[1] = j;
        }
      }
      if (fill && down && id < M) {
        P.move_dst[id] = slot;
        if (ONE && P.move_k != nullptr) sh->cnt_bin[2] = slot;
        P.hole_stamp[slot] = P.stamp;
        if (P.sums_list != nullptr) P.sums_list[rank * P.sums_cap + min(M - 1, id - down_before)] = ~slot;
      }
      if (P.sums_list != nullptr && g >= n) {
        const int q = (g - n) / sums_share(M, ncta);
        P.sums_list[q * P.sums_cap + (choose ? min(M, sh->cnt_down[q]) : 0) + (g - n - q * sums_share(M, ncta))] = keep ? slot : kSumsNone;
      }
      // which move empties a slot above B: none if its row leaves (or if the list is full: an inconsistency, see below)
      if (fill && slot >= P.B && slot - P.B < M) P.tail_move[slot - P.B] = up && iu < M ? iu : -1;
    }
  }
  if (ONE && P.move_k != nullptr && up_all == 1 && down_all == 1) {
    __syncthreads();
    const int src = sh->cnt_bin[0], dst = sh->cnt_bin[2];
    for (int v = tid; v < P.nvec; v += nthr) {
      const uint4 k = P.move_k[(size_t)src * P.nvec + v], w = P.move_v[(size_t)src * P.nvec + v];
      P.move_k[(size_t)dst * P.nvec + v] = k;
      P.move_v[(size_t)dst * P.nvec + v] = w;
    }
    if (tid == 0) P.slot_dst[sh->cnt_bin[1]] = dst;
  }
  // slots above B that no row occupies yet (the cache has just filled up) hold nothing to move
  if (fill && rank == 0)
    for (int i = max(0, N - P.B) + tid; i < M; i += nthr) P.tail_move[i] = -1;
  if (P.sums_list != nullptr && rank == 0 && tid < ncta) P.sums_out[tid] = choose ? min(M, sh->cnt_down[tid]) : 0;
  if (rank == 0 && tid == 0) {
    *P.n_keep_out = keep_all;
    if (bad || keep_all != min(N, P.B)) atomicCAS(P.status, 0, OVGGT_ERR_DEVICE_STATUS);
    if (fill) {
      // the two counts agree whenever the slots below min(N, B) were all occupied, which the layout guarantees
      const bool consistent = up_all == down_all && up_all <= M;
      *P.n_moves_out = consistent ? up_all : 0;
      if (!consistent) atomicCAS(P.status, 0, OVGGT_ERR_DEVICE_STATUS);
    }
  }
  G::leave();
}

template <int DT, bool SINGLE, bool ONE>
__global__ void __launch_bounds__(kSelectThreads, 2) k_compress_select(const __grid_constant__ CompressParams P) {
  extern __shared__ __align__(16) unsigned char smem_select[];
  compress_select_body<DT, SINGLE, ONE>(P, smem_select);
}

// The same step for several layers in one launch (Sec. 3.2: every layer has its own budget B^(l) and cache): one
// cluster per layer, blockIdx.y = position in the batch.  The parameter blocks travel as kernel arguments.
constexpr int kMaxBatchLayers = 32;
struct CompressBatch {
  CompressParams p[kMaxBatchLayers];
};
template <int DT, bool SINGLE>
__global__ void __launch_bounds__(kSelectThreads, 2) k_compress_select_batched(const __grid_constant__ CompressBatch batch) {
  extern __shared__ __align__(16) unsigned char smem_select[];
  compress_select_body<DT, SINGLE>(batch.p[blockIdx.y], smem_select);
}

}  // namespace ovggt
