// Compaction of the surviving rows (Eq. 8): the order-preserving gather, the hole-filling moves; key-norm bound.
// Rows are 16-byte-vector arrays; one warp moves one K or V row at a time with all of its
// loads issued before its stores, so many independent 16-byte transactions are in flight per SM.
#pragma once

#include "common.cuh"

namespace ovggt {

__device__ __forceinline__ void warp_copy_row(const uint4* src, uint4* dst, int nvec, int lane) {
  for (int v0 = lane; v0 < nvec; v0 += 128) {
    uint4 u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (v0 + 32 * i < nvec) u[i] = ld_nc(src + v0 + 32 * i);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (v0 + 32 * i < nvec) dst[v0 + 32 * i] = u[i];
  }
}

// dst[j, :] = src[survivors[j], :] for K and V.  Work item 2j is K row j, 2j+1 is V row j.
__global__ void __launch_bounds__(256) k_compact(const uint4* __restrict__ k_src, const uint4* __restrict__ v_src,
                                                 const int* __restrict__ survivors, int n_keep, int nvec,
                                                 uint4* __restrict__ k_dst, uint4* __restrict__ v_dst, int n_src,
                                                 int* status) {
  const int lane = threadIdx.x & 31;
  const int warps_total = (int)((gridDim.x * (unsigned)blockDim.x) >> 5);
  for (int item = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5); item < 2 * n_keep;
       item += warps_total) {
    const int j = item >> 1;
    const int src = survivors[j];
    if (!index_ok(src, n_src, status)) continue;
    if (item & 1) warp_copy_row(v_src + (size_t)src * nvec, v_dst + (size_t)j * nvec, nvec, lane);
    else          warp_copy_row(k_src + (size_t)src * nvec, k_dst + (size_t)j * nvec, nvec, lane);
  }
}

// Running upper bound of the squared per-head key norms of a bf16 cache, head_dim 64: kmax2[h] = max(kmax2[h],
// |K[row, 64h .. 64h+63]|^2).  A warp holds the row as 16-byte vectors (lane + 32 i); a head is eight consecutive
// vectors, i.e. eight neighbouring lanes of one i.  Non-negative floats order like their bit patterns, so the maximum
// is an integer atomicMax, which does not depend on the order of arrival.
// top: kmax2 of the lane's heads as read some time before (it only grows).  A key that is not a number has an infinite norm here:
// no bound holds for its scores, and the attention's exponentials may leave their range check out only where one does.
__device__ __forceinline__ void warp_key_norm_max(const uint4* u, int nvec, int lane, float* kmax2, const float* top) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float ss = 0.0f;
    if (lane + 32 * i < nvec) {
      const uint32_t w[4] = {u[i].x, u[i].y, u[i].z, u[i].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xFFFF0000u);
        ss = fmaf(lo, lo, ss);
        ss = fmaf(hi, hi, ss);
      }
    }
    ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 1);
    ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 2);
    ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 4);
    if ((lane & 7) == 0 && lane + 32 * i < nvec) {
      const int head = (lane + 32 * i) >> 3;
      if (!(ss <= top[i])) atomicMax(reinterpret_cast<int*>(kmax2) + head, __float_as_int(ss == ss ? ss : INFINITY));
    }
  }
}

// kmax2 over rows [0, rows) of K (after an import).  bf16, nvec <= 128.
__global__ void __launch_bounds__(256) k_key_norm_max(const uint4* __restrict__ K, int rows, int nvec,
                                                      float* __restrict__ kmax2) {
  const int lane = threadIdx.x & 31;
  const int warps_total = (int)((gridDim.x * (unsigned)blockDim.x) >> 5);
  for (int r = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5); r < rows; r += warps_total) {
    uint4 u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (lane + 32 * i < nvec) u[i] = ld_nc(K + (size_t)r * nvec + lane + 32 * i);
    float top[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) top[i] = lane + 32 * i < nvec ? kmax2[(lane + 32 * i) >> 3] : 0.0f;
    warp_key_norm_max(u, nvec, lane, kmax2, top);
  }
}

// ---- hole-filling compaction (Eq. 8 fixes the survivor set, not where the rows live)
//
// The selection kernel leaves n_moves pairs: the K/V row in slot move_src[i] (a survivor above slot B) goes to
// slot move_dst[i] (a slot below B whose row was evicted), and the survivor's meta entry move_j[i] learns its new
// slot.  Nothing else moves, so a step at steady state copies at most M rows instead of B.  The next append carries
// the moves out; this kernel is for whoever reads the rows before that.
__global__ void __launch_bounds__(256) k_fill_holes(uint4* __restrict__ k_cache, uint4* __restrict__ v_cache,
                                                    const int* __restrict__ move_src, const int* __restrict__ move_dst,
                                                    const int* __restrict__ move_j, const int* __restrict__ n_moves_ptr,
                                                    int max_moves, int nvec, int* __restrict__ slot_meta,
                                                    int rows_cap, int n_meta, int* status) {
  const int lane = threadIdx.x & 31;
  const int warps_total = (int)((gridDim.x * (unsigned)blockDim.x) >> 5);
  const int n_moves = min(*n_moves_ptr, max_moves);
  for (int m = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5); m < n_moves; m += warps_total) {
    const int src = move_src[m], dst = move_dst[m];
    if (!index_ok(src, rows_cap, status) || !index_ok(dst, rows_cap, status) || !index_ok(move_j[m], n_meta, status))
      continue;
    warp_copy_row(k_cache + (size_t)src * nvec, k_cache + (size_t)dst * nvec, nvec, lane);
    warp_copy_row(v_cache + (size_t)src * nvec, v_cache + (size_t)dst * nvec, nvec, lane);
    if (lane == 0) slot_meta[move_j[m]] = dst;
  }
}

}  // namespace ovggt
