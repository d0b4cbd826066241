// The attend half of the camera head's cache (Supp. C: one token a frame) in one launch: the append, the attention of the
// one query over all rows, and the key diversity of the cached rows.
//
// Nothing here is bound by bytes (145 rows of 16 heads: 0.6 MB) but by launches and by trips to memory, so everything that
// can run at once does: the first H CTAs take a head each, all K and V rows of a batch requested before any is used, on the
// FMA pipes; the others score four rows a warp, as k_front does.  The new row is read where the caller has it and written to the cache
// on the way; no move is pending, since the selection of such a cache moves its one row itself.  Before, k_front and then the
// tensor-core attention, 128 query rows for one, were two launches in a row: a frame through four layers of 16 heads and 145
// rows took 81.5 us and takes 70.5, of which the kernels are 48 and the caller's and the launches' host time bounds the rest.
#pragma once

#include "front_kernel.cuh"

namespace ovggt {

struct TokenArgs {
  const uint4 *q, *k_new, *v_new;             // [C]
  uint4 *k_cache, *v_cache;                   // rows [0, n) cached, row n := the new one
  void* out;                                  // [C]
  int n, H;
  long long frame_id;
  long long* ids; uint8_t* flags; float* stored; int* slot;   // as in FrontArgs
  const float* ksum; float* d;
};

constexpr int kTokenThreads = 256, kTokenWarps = kTokenThreads / 32;
constexpr int kTokenBatch = 8;                // K and V rows that a thread has in flight

template <int DT>
__global__ void __launch_bounds__(kTokenThreads) k_token_attend(const __grid_constant__ TokenArgs A, int nvec) {
  constexpr int VEC = VecOf<DT>::n, kLanes = 64 / VEC, kGroups = kTokenThreads / kLanes;   // lanes of a row of a head
  extern __shared__ __align__(16) float sh_ksum[];
  __shared__ float sh_m[kTokenWarps], sh_l[kTokenWarps], sh_o[kTokenWarps][64];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_wait();
  if ((int)blockIdx.x >= A.H) {
    // ------------------------------------------------ key diversity, four rows a warp
    for (int c = tid * 4; c < nvec * VEC; c += kTokenThreads * 4)
      *reinterpret_cast<float4*>(sh_ksum + c) = *reinterpret_cast<const float4*>(A.ksum + c);
    __syncthreads();
    float kn = 0.0f;
    for (int v = lane; v < nvec; v += 32)
#pragma unroll
      for (int e = 0; e < VEC; ++e) kn = __fmaf_rn(sh_ksum[v * VEC + e], sh_ksum[v * VEC + e], kn);
    kn = warp_sum(kn);
    const int warps = ((int)gridDim.x - A.H) * kTokenWarps;
    for (int item = ((int)blockIdx.x - A.H) * kTokenWarps + warp; item < front_score_items(A.n); item += warps) {
      const int row0 = item * kFrontRows;
      float dot[kFrontRows] = {}, nrm[kFrontRows] = {};
      for (int v0 = lane; v0 < nvec; v0 += 128) {
        uint4 u[kFrontRows][4];
#pragma unroll
        for (int r = 0; r < kFrontRows; ++r)
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (v0 + 32 * i < nvec) u[r][i] = A.k_cache[(size_t)min(row0 + r, A.n - 1) * nvec + v0 + 32 * i];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (v0 + 32 * i < nvec)
#pragma unroll
            for (int r = 0; r < kFrontRows; ++r) {
              float f[VEC];
              unpack<DT>(u[r][i], f);
#pragma unroll
              for (int e = 0; e < VEC; ++e) {
                dot[r] = __fmaf_rn(f[e], sh_ksum[(v0 + 32 * i) * VEC + e], dot[r]);
                nrm[r] = __fmaf_rn(f[e], f[e], nrm[r]);
              }
            }
      }
      float dt = 0.0f, nr = 0.0f;
#pragma unroll
      for (int r = 0; r < kFrontRows; ++r) {
        const float a = warp_sum(dot[r]), b = warp_sum(nrm[r]);
        if (lane == r) {
          dt = a;
          nr = b;
        }
      }
      if (lane < kFrontRows && row0 + lane < A.n) A.d[row0 + lane] = key_diversity(dt, nr, kn);
    }
    return;
  }
  // ------------------------------------------------ append and attention of one head
  const int h = blockIdx.x, c = tid % kLanes, group = tid / kLanes, vec = h * kLanes + c;
  const float scale = 1.4426950408889634f * 0.125f;    // log2(e) / sqrt(64)
  float q[VEC], o[VEC], mref = -INFINITY, l = 0.0f;
  const uint4 q4 = A.q[vec];
#pragma unroll
  for (int e = 0; e < VEC; ++e) o[e] = 0.0f;
#pragma unroll 1
  for (int r0 = group; r0 - group <= A.n; r0 += kTokenBatch * kGroups) {
    uint4 k[kTokenBatch], v[kTokenBatch];
#pragma unroll
    for (int i = 0; i < kTokenBatch; ++i) {
      const int r = r0 + i * kGroups;
      k[i] = v[i] = make_uint4(0u, 0u, 0u, 0u);
      if (r < A.n) {
        k[i] = A.k_cache[(size_t)r * nvec + vec];
        v[i] = A.v_cache[(size_t)r * nvec + vec];
      } else if (r == A.n) {
        k[i] = A.k_new[vec];
        v[i] = A.v_new[vec];
      }
    }
    if (r0 == group) unpack<DT>(q4, q);
    float s[kTokenBatch], top = mref;
#pragma unroll
    for (int i = 0; i < kTokenBatch; ++i) {
      float f[VEC];
      unpack<DT>(k[i], f);
      s[i] = 0.0f;
#pragma unroll
      for (int e = 0; e < VEC; ++e) s[i] = fmaf(q[e], f[e], s[i]);
    }
#pragma unroll
    for (int x = 1; x < kLanes; x <<= 1)
#pragma unroll
      for (int i = 0; i < kTokenBatch; ++i) s[i] += __shfl_xor_sync(0xFFFFFFFFu, s[i], x);
#pragma unroll
    for (int i = 0; i < kTokenBatch; ++i) {
      s[i] = r0 + i * kGroups <= A.n ? s[i] * scale : -INFINITY;
      top = fmaxf(top, s[i]);
    }
    const float corr = mref == -INFINITY ? 0.0f : exp2f(mref - top);    // (a score of -inf is a weight of 0, also before any other)
    l *= corr;
#pragma unroll
    for (int e = 0; e < VEC; ++e) o[e] *= corr;
#pragma unroll
    for (int i = 0; i < kTokenBatch; ++i) {
      const int r = r0 + i * kGroups;
      if (r > A.n) continue;
      const float p = s[i] == -INFINITY ? 0.0f : exp2f(s[i] - top);
      float f[VEC];
      unpack<DT>(v[i], f);
      l += p;
#pragma unroll
      for (int e = 0; e < VEC; ++e) o[e] = fmaf(p, f[e], o[e]);
      if (r == A.n) {
        A.k_cache[(size_t)r * nvec + vec] = k[i];
        A.v_cache[(size_t)r * nvec + vec] = v[i];
      }
    }
    mref = top;
  }
  // the warp's groups, then the warps
#pragma unroll
  for (int x = kLanes; x < 32; x <<= 1) {
    const float m2 = __shfl_xor_sync(0xFFFFFFFFu, mref, x), l2 = __shfl_xor_sync(0xFFFFFFFFu, l, x), top = fmaxf(mref, m2);
    const float w1 = mref == -INFINITY ? 0.0f : exp2f(mref - top), w2 = m2 == -INFINITY ? 0.0f : exp2f(m2 - top);
    l = l * w1 + l2 * w2;
#pragma unroll
    for (int e = 0; e < VEC; ++e) o[e] = o[e] * w1 + __shfl_xor_sync(0xFFFFFFFFu, o[e], x) * w2;
    mref = top;
  }
  if (lane < kLanes) {
#pragma unroll
    for (int e = 0; e < VEC; ++e) sh_o[warp][lane * VEC + e] = o[e];
    if (lane == 0) {
      sh_m[warp] = mref;
      sh_l[warp] = l;
    }
  }
  __syncthreads();
  if (tid < 64) {
    float top = -INFINITY, num = 0.0f, den = 0.0f;
#pragma unroll
    for (int w = 0; w < kTokenWarps; ++w) top = fmaxf(top, sh_m[w]);
#pragma unroll
    for (int w = 0; w < kTokenWarps; ++w) {
      const float f = sh_m[w] == -INFINITY ? 0.0f : exp2f(sh_m[w] - top);
      num = fmaf(f, sh_o[w][tid], num);
      den = fmaf(f, sh_l[w], den);
    }
    if constexpr (DT == kBF16) static_cast<__nv_bfloat16*>(A.out)[h * 64 + tid] = __float2bfloat16_rn(num / den);
    else                       static_cast<float*>(A.out)[h * 64 + tid] = num / den;
  }
  if (h == 0 && tid == 0) {
    A.ids[A.n] = A.frame_id;
    A.flags[A.n] = OVGGT_FLAG_EVICTABLE;
    A.stored[A.n] = 0.0f;
    if (A.slot != nullptr) A.slot[A.n] = A.n;
  }
}

}  // namespace ovggt
