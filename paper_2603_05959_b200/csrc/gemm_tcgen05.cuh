// bf16 GEMM for sm_100a: C [M, N] = A [M, K] x B [K, N], row-major, fp32 accumulation in tensor memory, with what the
// layers around the streaming step do to a product folded into its epilogue: GELU, the residual sum, and the split of a
// QKV product into three matrices.
//
// Not part of the streaming step itself: it is what a model wraps around it (QKV / output projections, MLP), provided
// so that the 24-layer workloads can run their scaffold on hand-written kernels too.
//   CTA tile 128 x 128, K in steps of 64: A tile [128 rows, 64 k] K-major (16 KB), B tile [64 k, 128 n] as two
//   [64 k, 64 n] boxes, N-major as the tensor lies in memory (2 x 8 KB), read by one N = 128 MMA per 16 k whose
//   descriptor names the distance between the boxes; three stages;
//   warp 0 produces (TMA), warp 1 issues the MMAs, accumulators in TMEM columns [0, 128), warps 2-5 read them back (one
//   thread per output row), finish and store.
// At these sizes (1041 or 1374 rows, N and K of 1024 to 4096) a product is 72 to 352 tiles of 2 to 9 us each, so it is
// the number of tiles in flight that matters, not the peak rate of one: 96 KB of stages let two CTAs share an SM (one
// fills or drains while the other multiplies), and a product with fewer tiles than SMs is cut along K over a cluster
// of two CTAs, each of which finishes half of the columns with the other's partial sums, sent through distributed shared
// memory.  The kernel is launched programmatically behind its predecessor, so set-up runs under that one's drain.
// (Before: N = 64 MMAs, four stages and one CTA per SM, no split: 17.9 / 8.9 / 16.6 / 22.7 us for the QKV, output, first
// and second MLP product of 1041 rows, and 45 element-wise launches per layer around them.)
// Requirements: K a multiple of 64, N a multiple of 8 (TMA row pitch of 16 bytes), 16-byte aligned bases.  Every
// barrier wait is bounded (about one second); on expiry the CTA records OVGGT_ERR_TIMEOUT and leaves through the
// common teardown, after the MMAs it issued have drained.
#pragma once

#include <cooperative_groups.h>

#include "attn_tcgen05.cuh"

namespace ovggt {

constexpr int kGemmBM = 128, kGemmBN = 128, kGemmBK = 64, kGemmStages = 3;
constexpr int kGemmThreads = 192;
constexpr int kGemmATile = kGemmBM * kGemmBK * 2;          // 16 KB
constexpr int kGemmBBox = kGemmBK * 64 * 2;                // 8 KB: [64 k, 64 n]
constexpr int kGemmBTile = 2 * kGemmBBox;                  // 16 KB
constexpr int kGemmTmemCols = 128;
constexpr int kGemmExchange = kGemmBM * (kGemmBN / 2) * 4; // 32 KB: half a tile of fp32 partial sums from the other CTA

struct GemmBarriers {
  unsigned long long full[kGemmStages], empty[kGemmStages], acc_full, drain;
  uint32_t tmem_base;
  int abort_flag;
};
__host__ __device__ constexpr size_t gemm_smem_bytes(bool split) {
  return (size_t)kGemmStages * (kGemmATile + kGemmBTile) + (split ? kGemmExchange : 0) + sizeof(GemmBarriers) + 64;
}

struct GemmArgs {
  int M, N, K;
  // t = bf16(product), or bf16(gelu(bf16(product)))
  __nv_bfloat16* out[3];            // t, columns [part * i, part * (i + 1)) to out[i] [M, part]; out[0] nullptr: not stored
  int part;
  int gelu;
  const __nv_bfloat16* residual;    // [M, N] or nullptr
  __nv_bfloat16* sum;               // [M, N]: bf16(residual + t)
  int* status;
};

__device__ __forceinline__ float gelu_exact(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }

// Eight finished columns [n, n + 8) of row m.
__device__ __forceinline__ void gemm_store8(const GemmArgs& P, int m, int n, const float* acc) {
  uint4 t;
  uint32_t* w = reinterpret_cast<uint32_t*>(&t);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    w[e] = pack_bf16(acc[2 * e], acc[2 * e + 1]);
    if (P.gelu)
      w[e] = pack_bf16(gelu_exact(__uint_as_float(w[e] << 16)), gelu_exact(__uint_as_float(w[e] & 0xFFFF0000u)));
  }
  if (P.out[0] != nullptr) {
    const int i = n / P.part;       // (8 columns lie in one part: its width is a multiple of 8)
    __nv_bfloat16* o = i == 0 ? P.out[0] : (i == 1 ? P.out[1] : P.out[2]);
    *reinterpret_cast<uint4*>(o + (size_t)m * P.part + (n - i * P.part)) = t;
  }
  if (P.residual != nullptr) {
    const uint4 r = *reinterpret_cast<const uint4*>(P.residual + (size_t)m * P.N + n);
    const uint32_t* rw = reinterpret_cast<const uint32_t*>(&r);
    uint4 s;
    uint32_t* sw = reinterpret_cast<uint32_t*>(&s);
#pragma unroll
    for (int e = 0; e < 4; ++e)
      sw[e] = pack_bf16(__uint_as_float(rw[e] << 16) + __uint_as_float(w[e] << 16),
                        __uint_as_float(rw[e] & 0xFFFF0000u) + __uint_as_float(w[e] & 0xFFFF0000u));
    *reinterpret_cast<uint4*>(P.sum + (size_t)m * P.N + n) = s;
  }
}

// SPLIT: launched as clusters of two CTAs, neighbours in x, each with half of the K steps of one tile.
template <bool SPLIT>
__global__ void __launch_bounds__(kGemmThreads, SPLIT ? 1 : 2)
k_gemm_bf16_tcgen05(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                    const __grid_constant__ GemmArgs P) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* sA = smem;
  unsigned char* sB = sA + kGemmStages * kGemmATile;
  float* xch = reinterpret_cast<float*>(sB + kGemmStages * kGemmBTile);     // [64 columns][128 rows], SPLIT only
  GemmBarriers* B = reinterpret_cast<GemmBarriers*>(sB + kGemmStages * kGemmBTile + (SPLIT ? kGemmExchange : 0));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * kGemmBM, n0 = (SPLIT ? blockIdx.x >> 1 : blockIdx.x) * kGemmBN;
  const int half = SPLIT ? (int)(blockIdx.x & 1) : 0;
  const int k_all = P.K / kGemmBK;
  const int k_begin = SPLIT && half ? (k_all + 1) / 2 : 0, k_tiles = (SPLIT && !half ? (k_all + 1) / 2 : k_all) - k_begin;
  bool aligned = (smem_u32(smem) & 1023u) == 0;     // the 128-byte swizzle needs 1024-byte aligned tiles
  if (!aligned && threadIdx.x == 0) atomicCAS(P.status, 0, OVGGT_ERR_DEVICE_STATUS);

  if (warp == 0 && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_a) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_b) : "memory");
    for (int s = 0; s < kGemmStages; ++s) {
      mbar_init(&B->full[s], 1);
      mbar_init(&B->empty[s], 1);
    }
    mbar_init(&B->acc_full, 1);
    mbar_init(&B->drain, 1);
    B->abort_flag = aligned ? 0 : 1;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&B->tmem_base)),
                 "r"((uint32_t)kGemmTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *(volatile uint32_t*)&B->tmem_base;
  if constexpr (SPLIT) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  pdl_wait();

  bool ok = aligned;
  if (warp == 0) {
    // ------------------------------------------------ TMA producer
    if (lane == 0) {
      int issued = 0;
      for (int kt = 0; kt < k_tiles && ok; ++kt) {
        const int s = kt % kGemmStages;
        const uint32_t ph = (uint32_t)(kt / kGemmStages) & 1u;
        if (kt >= kGemmStages) ok = mbar_wait(&B->empty[s], ph ^ 1u, B, P.status);
        if (!ok) break;
        const int k0 = (k_begin + kt) * kGemmBK;
        mbar_expect_tx(&B->full[s], kGemmATile + kGemmBTile);
        tma_load_2d(sA + s * kGemmATile, &tm_a, k0, m0, &B->full[s]);
        tma_load_2d(sB + s * kGemmBTile, &tm_b, n0, k0, &B->full[s]);
        tma_load_2d(sB + s * kGemmBTile + kGemmBBox, &tm_b, n0 + 64, k0, &B->full[s]);
        ++issued;
      }
      if (!ok)   // leave no bulk copy in flight into this CTA's shared memory
        for (int i = max(0, issued - kGemmStages); i < issued; ++i)
          mbar_wait(&B->full[i % kGemmStages], (uint32_t)(i / kGemmStages) & 1u, B, P.status);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (whole warp in step, one elected lane issues)
    const bool leader = elect_one();
    const uint32_t tm = __reduce_or_sync(0xFFFFFFFFu, tmem);
    constexpr uint32_t idesc = idesc_bf16(kGemmBN, true);       // A K-major, B N-major
    for (int kt = 0; kt < k_tiles && ok; ++kt) {
      const int s = kt % kGemmStages;
      const uint32_t ph = (uint32_t)(kt / kGemmStages) & 1u;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(&B->full[s], ph, B, P.status)) != 0;
      if (!ok) break;
      tc_fence_after();
      const uint64_t da = smem_desc_sw128(smem_u32(sA + s * kGemmATile));
      const uint64_t db = smem_desc_sw128_mn(smem_u32(sB + s * kGemmBTile), kGemmBBox);
      if (leader) {
#pragma unroll
        for (int kk = 0; kk < kGemmBK / 16; ++kk)   // A: 16 k = 32 bytes inside the swizzled row; B: 16 k-rows = 2048 bytes
          mma_ss(tm, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 128), idesc, (kt > 0 || kk > 0));
        tc_commit(&B->empty[s]);
      }
    }
    if (ok) {
      if (leader) tc_commit(&B->acc_full);
    } else if (aligned) {
      if (leader) tc_commit(&B->drain);             // let every issued MMA finish before TMEM is freed
      __all_sync(0xFFFFFFFFu, mbar_wait(&B->drain, 0, B, P.status));
    }
    __syncwarp();
  } else if (ok) {
    ok = __all_sync(0xFFFFFFFFu, mbar_wait(&B->acc_full, 0, B, P.status)) != 0;
    tc_fence_after();
  }
  // ------------------------------------------------ epilogue: warps 2..5 own the TMEM lane quarters 2, 3, 0, 1
  const int quad = warp & 3;
  const int row = quad * 32 + lane, m = m0 + row;
  const uint32_t t_row = tmem + ((uint32_t)(quad * 32) << 16);
  if (!SPLIT) {
    if (warp >= 2 && ok) {
#pragma unroll
      for (int j = 0; j < kGemmBN / 32; ++j) {
        uint32_t o[32];
        tmem_ld32(t_row + j * 32, o);
        tmem_wait_ld();
        if (m < P.M) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int n = n0 + j * 32 + e * 8;
            if (n < P.N) gemm_store8(P, m, n, reinterpret_cast<const float*>(o) + 8 * e);   // (N is a multiple of 8)
          }
        }
      }
    }
  } else {
    // This CTA finishes the columns [64 half, 64 half + 64) of the tile; the other half's partial sums go to the peer.
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    float* peer = cluster.map_shared_rank(xch, (int)cluster.block_rank() ^ 1);
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");      // the peer has started: its shared memory is there
    if (warp >= 2 && ok) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        uint32_t o[32];
        tmem_ld32(t_row + (half ^ 1) * 64 + j * 32, o);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 32; ++e) peer[(j * 32 + e) * kGemmBM + row] = __uint_as_float(o[e]);
      }
    }
    cluster.sync();
    if (warp >= 2 && ok) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        uint32_t o[32];
        tmem_ld32(t_row + half * 64 + j * 32, o);
        tmem_wait_ld();
        if (m < P.M) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int n = n0 + half * 64 + j * 32 + e * 8;
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(o[8 * e + i]) + xch[(j * 32 + e * 8 + i) * kGemmBM + row];
            if (n < P.N) gemm_store8(P, m, n, v);
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)kGemmTmemCols) : "memory");
  }
}

inline int gemm_tcgen05_launch(const void* A, const void* Bm, const GemmArgs& P, cudaStream_t st) {
  CUtensorMap ta, tb;
  int rc = make_rows_map(&ta, A, P.M, P.K, kGemmBM);       // 64 k-columns x 128 rows per box
  if (rc) return rc;
  rc = make_rows_map(&tb, Bm, P.K, P.N, kGemmBK);          // 64 n-columns x 64 k-rows per box
  if (rc) return rc;
  const int tiles_n = (P.N + kGemmBN - 1) / kGemmBN, tiles_m = (P.M + kGemmBM - 1) / kGemmBM;
  // Half the SMs or fewer busy and a K loop long enough to halve: two CTAs a tile.
  const bool split = tiles_n * tiles_m <= 74 && P.K >= 1024;
  static std::atomic<uint64_t> smem_set[2];
  const auto kernel = split ? k_gemm_bf16_tcgen05<true> : k_gemm_bf16_tcgen05<false>;
  cudaError_t e = allow_smem(kernel, gemm_smem_bytes(split), smem_set[split ? 1 : 0]);
  if (e == cudaSuccess)
    e = launch_dependent(kernel, dim3(split ? 2 * tiles_n : tiles_n, tiles_m), kGemmThreads, split ? 2 : 1, gemm_smem_bytes(split), st, true,
                         ta, tb, P);
  if (e != cudaSuccess) { g_attn_last_error = (int)e; return OVGGT_ERR_CUDA; }
  return OVGGT_OK;
}

}  // namespace ovggt
