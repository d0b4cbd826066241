// The front of a step in one launch: append (Eq. 2) with the moves the previous step left behind, key diversity of the
// cached rows (Sec. 3.2) and the residual norms of the new ones (Eq. 5).
//
// The three jobs are independent passes over rows of [.., C]: 11 + up to 14 MB, 34 MB and 3 MB at 1374 new rows, 16384
// cached rows and C = 1024 in bf16, so they are bound by memory and, at that size, by latency: one launch pays the
// start-up, the fill of the memory pipeline and the drain once.  A warp takes one item at a time, one new row or four
// rows to score, with all 16 loads of a lane in flight; items are dealt round-robin to two CTAs per SM, the first one
// requested before the centroid is staged in shared memory.  As three launches (append with a cluster fold of the sums'
// corrections, then diversity beside the attention, whose CTAs leave it no registers) the same work cost a step about
// 10 + 14 us; this takes 14.
#pragma once

#include "compact_kernels.cuh"
#include "score_kernels.cuh"

namespace ovggt {

struct FrontArgs {
  // append: rows [n, n + M) := the frame's K and V
  const uint4* k_new; const uint4* v_new;
  int M, n;
  long long frame_id;
  uint4* k_cache; uint4* v_cache;
  long long* ids; uint8_t* flags; float* stored; int* slot;   // meta of the layer, logical order (slot: nullptr in the stable layout)
  float* kmax2;                               // running bound of the key norms, or nullptr
  // Moves the previous step left (hole-filling layout).  The rows admitted then sit in slots >= B, exactly where this
  // frame goes, and nothing reads the cache in between: the warp that owns new row j first carries the row in its slot
  // down to its destination, then writes the new row over it; program order inside the warp is all the ordering needed.
  int B;
  const int* tail_move; const int* move_dst; const int* move_j; const int* n_moves_ptr;   // tail_move nullptr: nothing pending
  // diversity of the rows in slots [0, n): d = 1 - cos(K[slot], ksum)
  const float* ksum;                          // [C] column sums of the cached keys, or nullptr: not asked for
  float* d;                                   // [n]
  // Slots a pending move fills: the warp that carries the row there scores it from its registers, and whoever meets the
  // slot in the cache, where old and new bytes may be mixed just then, leaves its score alone.
  const int* hole_stamp; int stamp;
  // residual norms of the new rows
  const uint4* resid; float* s_raw;           // [M, C] -> [M]; resid nullptr: not asked for
  int* status;                                // where the checked build reports a bad move index
};

constexpr int kFrontThreads = 256;
constexpr int kFrontRows = 4;                 // rows of a scoring item

__host__ __device__ inline int front_score_items(int rows) { return (rows + kFrontRows - 1) / kFrontRows; }

// 1 - the cosine of a key with the centroid, which is that with the column sums: their product, the squared norms of both; a
// zero vector has cosine 0.
__device__ __forceinline__ float key_diversity(float dot, float nrm, float kn) {
  float cosv = 0.0f;
  if (nrm > 0.0f && kn > 0.0f) cosv = __fdiv_rn(dot, __fmul_rn(__fsqrt_rn(nrm), __fsqrt_rn(kn)));
  return 1.0f - cosv;
}

// The sums over the warp of four rows' products and squared norms; lane 8 r gets those of row r.  The order of warp_sum, bit for
// bit, but each step hands half of what is left to the other half of the lanes: 10 shuffles instead of 40, which an SM
// executes at one a cycle (a step of 1374 + 16384 rows: 154.7 -> 153.5 us).
__device__ __forceinline__ void warp_sum_rows(const float (&dot)[kFrontRows], const float (&nrm)[kFrontRows], float* dt, float* nr) {
  static_assert(kFrontRows == 4, "two bits of the lane name the row");
  const int lane = threadIdx.x & 31;
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  float d[2], n[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    d[j] = (b4 ? dot[j + 2] : dot[j]) + __shfl_xor_sync(0xFFFFFFFFu, b4 ? dot[j] : dot[j + 2], 16);
    n[j] = (b4 ? nrm[j + 2] : nrm[j]) + __shfl_xor_sync(0xFFFFFFFFu, b4 ? nrm[j] : nrm[j + 2], 16);
  }
  const float d1 = (b3 ? d[1] : d[0]) + __shfl_xor_sync(0xFFFFFFFFu, b3 ? d[0] : d[1], 8);
  const float n1 = (b3 ? n[1] : n[0]) + __shfl_xor_sync(0xFFFFFFFFu, b3 ? n[0] : n[1], 8);
  float x = (b2 ? n1 : d1) + __shfl_xor_sync(0xFFFFFFFFu, b2 ? d1 : n1, 4);
  x += __shfl_xor_sync(0xFFFFFFFFu, x, 2);
  x += __shfl_xor_sync(0xFFFFFFFFu, x, 1);
  *dt = x;
  *nr = __shfl_xor_sync(0xFFFFFFFFu, x, 4);
}

template <int DT>
__global__ void __launch_bounds__(kFrontThreads, 2) k_front(const __grid_constant__ FrontArgs A, int nvec) {
  constexpr int VEC = VecOf<DT>::n;
  extern __shared__ __align__(16) float sh_ksum[];
  const int lane = threadIdx.x & 31;
  // (warp by warp over the CTAs, so that each SM gets its share of the new rows, which take longest: steps of 1374 + 4096 and 69 + 16000
  // rows are 2 and 3 % faster for it)
  const int gw = (int)((threadIdx.x >> 5) * gridDim.x + blockIdx.x), warps_total = (int)((gridDim.x * (unsigned)blockDim.x) >> 5);
  const int n_div = A.ksum != nullptr ? front_score_items(A.n) : 0;
  const int n_norm = A.resid != nullptr ? front_score_items(A.M) : 0;
  const int items = A.M + n_div + n_norm;
  const bool pending = A.tail_move != nullptr;

  // The selection behind this kernel may take its place early; behind a front of a few CTAs, which ends sooner than that is
  // worth, it only gets in the way (camera head: 84 us a pass without, 93 with).
  if (gridDim.x >= 148) pdl_trigger();
  pdl_wait();
  uint4 u[4][4];
  // What a new row's append looks up besides its rows is requested with them.  (But for where its slot's move goes, which is known when
  // the move is: waiting for that before the first item costs small steps 0.1 to 0.4 us and gains none anything.)
  const int n_moves = pending && gw < A.M ? min(*A.n_moves_ptr, A.M) : 0;
  int move = -1;
  float top[4];                               // the bounds of the heads whose keys the lane holds
  // the first 128 vectors of an item's rows: the new K and V row and what sits in their slot, or four rows to score
  auto load = [&](int item) {
    if (item < A.M) {
      const int s = A.n + item;
      const bool tail = pending && s >= A.B && s - A.B < A.M;
      move = tail ? A.tail_move[s - A.B] : -1;
#pragma unroll
      for (int i = 0; i < 4; ++i) top[i] = A.kmax2 != nullptr && lane + 32 * i < nvec ? A.kmax2[(lane + 32 * i) >> 3] : 0.0f;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (lane + 32 * i < nvec) {
          u[0][i] = ld_nc(A.k_new + (size_t)item * nvec + lane + 32 * i);
          u[1][i] = ld_nc(A.v_new + (size_t)item * nvec + lane + 32 * i);
          if (tail) {   // (plain loads: these cache lines are rewritten by this very kernel)
            u[2][i] = A.k_cache[(size_t)s * nvec + lane + 32 * i];
            u[3][i] = A.v_cache[(size_t)s * nvec + lane + 32 * i];
          }
        }
      return;
    }
    const bool norm = item >= A.M + n_div;
    const int row0 = (norm ? item - A.M - n_div : item - A.M) * kFrontRows, rows = norm ? A.M : A.n;
    const uint4* base = norm ? A.resid : A.k_cache;
#pragma unroll
    for (int r = 0; r < kFrontRows; ++r) {
      const uint4* p = base + (size_t)min(row0 + r, rows - 1) * nvec;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (lane + 32 * i < nvec) u[r][i] = p[lane + 32 * i];
    }
  };
  if (gw < items) load(gw);
  float kn = 0.0f;                            // |ksum|^2, folded by every warp in the same order
  if (A.ksum != nullptr) {
    const int C = nvec * VEC;
    for (int c = threadIdx.x * 4; c < C; c += kFrontThreads * 4)
      *reinterpret_cast<float4*>(sh_ksum + c) = *reinterpret_cast<const float4*>(A.ksum + c);
    __syncthreads();
    for (int v = lane; v < nvec; v += 32)
#pragma unroll
      for (int e = 0; e < VEC; e += 4) {
        const float4 k4 = *reinterpret_cast<const float4*>(sh_ksum + v * VEC + e);
        kn = __fmaf_rn(k4.x, k4.x, kn);
        kn = __fmaf_rn(k4.y, k4.y, kn);
        kn = __fmaf_rn(k4.z, k4.z, kn);
        kn = __fmaf_rn(k4.w, k4.w, kn);
      }
    kn = warp_sum(kn);
  }
  auto centroid = [&](int vec, float* ks) {   // 16-byte reads: consecutive lanes are VEC floats apart
#pragma unroll
    for (int e = 0; e < VEC; e += 4)
      *reinterpret_cast<float4*>(ks + e) = *reinterpret_cast<const float4*>(sh_ksum + vec * VEC + e);
  };
  auto accumulate = [&](const uint4& x, const float* ks, float& dot, float& nrm) {
    float f[VEC];
    unpack<DT>(x, f);
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
      dot = __fmaf_rn(f[e], ks[e], dot);
      nrm = __fmaf_rn(f[e], f[e], nrm);
    }
  };

  for (int item = gw; item < items; item += warps_total) {
    if (item != gw) load(item);
    if (item < A.M) {
      // ---- append row j, after carrying down what a pending move left in its slot
      const int j = item, s = A.n + j;
      // (a warp collective, reached by every lane whatever part of the row it holds; rows of up to 128 vectors only,
      //  which is all the bound is kept for)
      if (A.kmax2 != nullptr) warp_key_norm_max(u[0], nvec, lane, A.kmax2, top);
      int m = move < n_moves ? move : -1;
      const int dst = m >= 0 ? A.move_dst[m] : 0, meta = m >= 0 ? A.move_j[m] : 0;
      if (m >= 0 && (!index_ok(dst, A.B, A.status) || !index_ok(meta, A.B, A.status))) m = -1;
      float dot = 0.0f, nrm = 0.0f;
      for (int v0 = lane; v0 < nvec; v0 += 128) {
        if (v0 != lane) {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (v0 + 32 * i < nvec) {
              u[0][i] = ld_nc(A.k_new + (size_t)j * nvec + v0 + 32 * i);
              u[1][i] = ld_nc(A.v_new + (size_t)j * nvec + v0 + 32 * i);
              if (m >= 0) {
                u[2][i] = A.k_cache[(size_t)s * nvec + v0 + 32 * i];
                u[3][i] = A.v_cache[(size_t)s * nvec + v0 + 32 * i];
              }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (v0 + 32 * i < nvec) {
            if (m >= 0) {
              A.k_cache[(size_t)dst * nvec + v0 + 32 * i] = u[2][i];
              A.v_cache[(size_t)dst * nvec + v0 + 32 * i] = u[3][i];
              if (A.ksum != nullptr) {
                float ks[VEC];
                centroid(v0 + 32 * i, ks);
                accumulate(u[2][i], ks, dot, nrm);
              }
            }
            A.k_cache[(size_t)s * nvec + v0 + 32 * i] = u[0][i];
            A.v_cache[(size_t)s * nvec + v0 + 32 * i] = u[1][i];
          }
      }
      if (m >= 0 && A.ksum != nullptr) {      // (m is the same in all lanes)
        dot = warp_sum(dot);
        nrm = warp_sum(nrm);
        if (lane == 0) A.d[dst] = key_diversity(dot, nrm, kn);
      }
      if (lane == 0) {
        if (m >= 0) A.slot[meta] = dst;
        A.ids[s] = A.frame_id * (long long)A.M + j;
        A.flags[s] = OVGGT_FLAG_EVICTABLE;
        A.stored[s] = 0.0f;
        if (A.slot != nullptr) A.slot[s] = s;
      }
    } else {
      // ---- score four rows: residual norms, or diversity
      const bool norm = item >= A.M + n_div;
      const int row0 = (norm ? item - A.M - n_div : item - A.M) * kFrontRows, rows = norm ? A.M : A.n;
      const uint4* base = norm ? A.resid : A.k_cache;
      const int row = row0 + (lane >> 3);
      bool mine = (lane & 7) == 0 && row < rows;             // lane 8 r writes the score of row r
      if (!norm && pending && mine) mine = A.hole_stamp[row] != A.stamp;
      float dot[kFrontRows] = {}, nrm[kFrontRows] = {};
      for (int v0 = lane; v0 < nvec; v0 += 128) {
        if (v0 != lane) {
#pragma unroll
          for (int r = 0; r < kFrontRows; ++r) {
            const uint4* p = base + (size_t)min(row0 + r, rows - 1) * nvec;
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (v0 + 32 * i < nvec) u[r][i] = p[v0 + 32 * i];
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (v0 + 32 * i < nvec) {
            float ks[VEC] = {};
            if (!norm) centroid(v0 + 32 * i, ks);
#pragma unroll
            for (int r = 0; r < kFrontRows; ++r) accumulate(u[r][i], ks, dot[r], nrm[r]);
          }
      }
      float dt, nr;
      warp_sum_rows(dot, nrm, &dt, &nr);
      if (mine) {
        if (norm) A.s_raw[row] = __fsqrt_rn(nr);
        else      A.d[row] = key_diversity(dt, nr, kn);
      }
    }
  }
}

}  // namespace ovggt
