// bf16 GEMM for sm_100a: C [M, N] = A [M, K] x B [K, N], row-major, fp32 accumulation in tensor memory, with what the
// layers around the streaming step do to a product folded into its epilogue: GELU, the residual sum, and the split of a
// QKV product into three matrices.
//
// Not part of the streaming step itself: it is what a model wraps around it (QKV / output projections, MLP), provided
// so that the 24-layer workloads can run their scaffold on hand-written kernels too.
//   CTA tile 128 x BN (256, 128 or 64), K in steps of 64: A tile [128 rows, 64 k] K-major (16 KB), B tile [64 k, BN n] as
//   [64 k, 64 n] boxes, N-major as the tensor lies in memory (8 KB each), read by one N = BN MMA per 16 k whose descriptor
//   names the distance between the boxes; 192 KB of stages, one CTA per SM;
//   warp 16 produces (TMA), warp 17 issues the MMAs, accumulators in BN TMEM columns; warps 0-15 read them back, one thread
//   per output row and quarter of the columns, finish, and store whole lines by way of shared memory.
// What bounds it at these sizes (1041 or 1374 rows, N and K of 1024 to 4096): one wave of CTAs whose loads all come from
// L2, each at the 64 bytes a clock that an SM takes in (260 ns for the 32 KB of a 128-wide K step, however many CTAs run);
// hence the widest tile where a product has tiles enough for every SM, the narrowest where it has few, and all of shared
// memory in flight.  The kernel is launched programmatically
// behind its predecessor and prefetches its part of B (weights, as a rule) into L2 while that one drains.
// Measured, QKV / output / first (GELU) / second MLP product of 1041 rows, width 1024: 9.7 / 6.3 / 14.1 / 17.0 us; the
// first and the third took 13.9 and 18.1 us with 128 x 128 tiles of three stages and four epilogue warps that stored row by row.
// A residual is requested while the products run, not after them, in instances of their own (RES): output and second MLP product of
// 1041 rows 7.0 -> 6.5 and 18.5 -> 17.8 us, of 1374 rows 8.7 -> 7.8 and 22.6 -> 21.7; in an instance for both the registers it
// waits in cost the QKV product 10.7 -> 11.5.  A table of GELU in shared memory was slower than the error functions (the third product
// 15.1 -> 17.3 us).
// Requirements: K a multiple of 64, N a multiple of 8 (TMA row pitch of 16 bytes), 16-byte aligned bases.  Every
// barrier wait is bounded (about one second); on expiry the CTA records OVGGT_ERR_TIMEOUT and leaves through the
// common teardown, after the MMAs it issued have drained.
#pragma once

#include "attn_tcgen05.cuh"

namespace ovggt {

constexpr int kGemmBM = 128, kGemmBK = 64;
constexpr int kGemmEpilogueWarps = 16, kGemmThreads = (kGemmEpilogueWarps + 2) * 32;
constexpr int kGemmATile = kGemmBM * kGemmBK * 2;          // 16 KB
constexpr int kGemmBBox = kGemmBK * 64 * 2;                // 8 KB: [64 k, 64 n]
constexpr int kGemmMaxStages = 8;
__host__ __device__ constexpr int gemm_stage_bytes(int bn) { return kGemmATile + bn / 64 * kGemmBBox; }
__host__ __device__ constexpr int gemm_stages(int bn) { return bn == 256 ? 4 : (bn == 128 ? 6 : 8); }

struct GemmBarriers {
  unsigned long long full[kGemmMaxStages], empty[kGemmMaxStages], acc_full, drain;
  uint32_t tmem_base;
  int abort_flag;
};
__host__ __device__ constexpr size_t gemm_smem_bytes(int bn) {
  return (size_t)gemm_stages(bn) * gemm_stage_bytes(bn) + sizeof(GemmBarriers) + 64;
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

// x Phi(x), in the form whose bf16 rounding every bf16 input shares with torch's GELU.
__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }

// The same of a pair of bf16 values from -3 on, rounded to bf16: erf(x / sqrt 2) as x times a polynomial of x^2 (of degree 8, through
// the Chebyshev nodes of [0, 3.25^2], beyond which 1 + erf rounds to 2), 14 packed operations a pair instead of two error functions
// of some 40 instructions each.  Its error, 1.1e-6 and its roundings, is far enough from where any bf16 input's result would round the other way, so the
// bits are gelu's (every input is tested); below -3, where 1 + erf cancels, they would not be.
__device__ __forceinline__ uint32_t gelu_pair(uint32_t w) {
  const float2 x = make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
  const float2 c = make_float2(fminf(x.x, 3.25f), fminf(x.y, 3.25f)), zero = make_float2(0.0f, 0.0f);
  const float2 t = fma2(c, c, zero);
  float2 q = make_float2(5.140512460144464e-10f, 5.140512460144464e-10f);
  const float k[8] = {0.7978842258453369f, -0.13297531008720398f, 0.019932821393013f, -0.0023600568529218435f, 0.00022326379257719964f, -1.659831468714401e-05f, 9.056150247488404e-07f, -3.154504923941204e-08f};
#pragma unroll
  for (int i = 7; i >= 0; --i) q = fma2(q, t, make_float2(k[i], k[i]));
  const float2 one = add2(fma2(q, c, zero), make_float2(1.0f, 1.0f));
  return pack_bf16(0.5f * x.x * one.x, 0.5f * x.y * one.y);
}

// The same of a warp's 16 columns of 32 rows: by the polynomial where none of them is below -3, else by the error functions for
// all.  (A choice by value takes both ways in most warps: the first MLP product of 1041 rows, whose values have a deviation of
// 1.6, 0.96 or 0.64: 17.9, 14.3, 13.7 us; so 14.9, 14.1, 12.9; by the error functions alone 14.9.)
__device__ __forceinline__ void gelu_warp(uint32_t (&w)[8]) {
  __nv_bfloat162 low = reinterpret_cast<const __nv_bfloat162*>(w)[0];
#pragma unroll
  for (int e = 1; e < 8; ++e) low = __hmin2(low, reinterpret_cast<const __nv_bfloat162*>(w)[e]);
  if (__any_sync(0xFFFFFFFFu, fminf(__low2float(low), __high2float(low)) < -3.0f)) {
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = pack_bf16(gelu(__uint_as_float(w[e] << 16)), gelu(__uint_as_float(w[e] & 0xFFFF0000u)));
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = gelu_pair(w[e]);
  }
}

// Finished bf16 columns [n, n + 8) of row m: where the caller wants them.  r: those of the residual.
template <bool RES>
__device__ __forceinline__ void gemm_store8(const GemmArgs& P, int m, int n, const uint4& t, const uint4& r) {
  if (P.out[0] != nullptr) {
    const int i = n / P.part;       // (8 columns lie in one part: its width is a multiple of 8)
    __nv_bfloat16* o = i == 0 ? P.out[0] : (i == 1 ? P.out[1] : P.out[2]);
    *reinterpret_cast<uint4*>(o + (size_t)m * P.part + (n - i * P.part)) = t;
  }
  if constexpr (RES) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(&t);
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

__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(map), "r"(x), "r"(y) : "memory");
}

template <int BN, bool RES>
__global__ void __launch_bounds__(kGemmThreads, 1)
k_gemm_bf16_tcgen05(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                    const __grid_constant__ GemmArgs P) {
  constexpr int kStages = gemm_stages(BN), kStage = gemm_stage_bytes(BN);
  constexpr int kProducer = kGemmEpilogueWarps, kIssuer = kGemmEpilogueWarps + 1;
  extern __shared__ __align__(1024) unsigned char smem[];
  GemmBarriers* B = reinterpret_cast<GemmBarriers*>(smem + kStages * kStage);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * kGemmBM, n0 = (int)blockIdx.x * BN, k_tiles = P.K / kGemmBK;
  const bool aligned = (smem_u32(smem) & 1023u) == 0;     // the 128-byte swizzle needs 1024-byte aligned tiles
  if (!aligned && threadIdx.x == 0) atomicCAS(P.status, 0, OVGGT_ERR_DEVICE_STATUS);
  pdl_trigger();

  if (warp == kProducer && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_a) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_b) : "memory");
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&B->full[s], 1);
      mbar_init(&B->empty[s], 1);
    }
    mbar_init(&B->acc_full, 1);
    mbar_init(&B->drain, 1);
    B->abort_flag = aligned ? 0 : 1;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    // the CTAs of one column of tiles share its part of B out among them
    for (int kt = (int)blockIdx.y; kt < k_tiles; kt += (int)gridDim.y)
      for (int x = 0; x < BN && n0 + x < P.N; x += 64) tma_prefetch_2d(&tm_b, n0 + x, kt * kGemmBK);
  }
  if (warp == kIssuer) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&B->tmem_base)),
                 "r"((uint32_t)BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *(volatile uint32_t*)&B->tmem_base;
  pdl_wait();

  // The epilogue's 16-byte units: a warp finishes a quarter of the columns of 32 rows, whole lines of a row by neighbouring lanes.
  constexpr int kCols = BN / 4, kUnits = kCols / 8;        // columns of a warp, their units
  const int quad = warp & 3, side = warp >> 2;
  auto unit_row = [&](int i) { return m0 + quad * 32 + (lane + 32 * i) / kUnits; };
  auto unit_col = [&](int i) { return n0 + side * kCols + (lane + 32 * i) % kUnits * 8; };
  uint4 residual[RES ? kUnits : 1];                        // requested while the products run

  bool ok = aligned;
  if (warp == kProducer) {
    // ------------------------------------------------ TMA producer
    if (lane == 0) {
      int issued = 0;
      for (int kt = 0; kt < k_tiles && ok; ++kt) {
        const int s = kt % kStages;
        const uint32_t ph = (uint32_t)(kt / kStages) & 1u;
        if (kt >= kStages) ok = mbar_wait(&B->empty[s], ph ^ 1u, B, P.status);
        if (!ok) break;
        const int k0 = kt * kGemmBK;
        unsigned char* st = smem + s * kStage;
        mbar_expect_tx(&B->full[s], kStage);
        tma_load_2d(st, &tm_a, k0, m0, &B->full[s]);
#pragma unroll
        for (int x = 0; x < BN / 64; ++x)
          tma_load_2d(st + kGemmATile + x * kGemmBBox, &tm_b, n0 + x * 64, k0, &B->full[s]);
        ++issued;
      }
      if (!ok)   // leave no bulk copy in flight into this CTA's shared memory
        for (int i = max(0, issued - kStages); i < issued; ++i)
          mbar_wait(&B->full[i % kStages], (uint32_t)(i / kStages) & 1u, B, P.status);
    }
    __syncwarp();
  } else if (warp == kIssuer) {
    // ------------------------------------------------ MMA issuer (whole warp in step, one elected lane issues)
    const bool leader = elect_one();
    const uint32_t tm = __reduce_or_sync(0xFFFFFFFFu, tmem);
    constexpr uint32_t idesc = idesc_bf16(BN, true);            // A K-major, B N-major
    for (int kt = 0; kt < k_tiles && ok; ++kt) {
      const int s = kt % kStages;
      const uint32_t ph = (uint32_t)(kt / kStages) & 1u;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(&B->full[s], ph, B, P.status)) != 0;
      if (!ok) break;
      tc_fence_after();
      const uint64_t da = smem_desc_sw128(smem_u32(smem + s * kStage));
      const uint64_t db = smem_desc_sw128_mn(smem_u32(smem + s * kStage + kGemmATile), kGemmBBox);
      if (leader) {
#pragma unroll
        for (int kk = 0; kk < kGemmBK / 16; ++kk)   // A: 16 k = 32 bytes inside the swizzled row; B: 16 k-rows = 2048 bytes
          mma_ss(tm, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 128), idesc, (kt > 0 || kk > 0));
        tc_commit(&B->empty[s]);
      }
    }
    if (ok) {
      if (leader) tc_commit(&B->acc_full);
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(&B->acc_full, 0, B, P.status)) != 0;
    } else if (aligned) {
      if (leader) tc_commit(&B->drain);             // let every issued MMA finish before TMEM is freed
      __all_sync(0xFFFFFFFFu, mbar_wait(&B->drain, 0, B, P.status));
    }
    __syncwarp();
  } else if (ok) {
    if constexpr (RES)
#pragma unroll
      for (int i = 0; i < kUnits; ++i)
        if (unit_row(i) < P.M && unit_col(i) < P.N)        // (N is a multiple of 8)
          residual[i] = *reinterpret_cast<const uint4*>(P.residual + (size_t)unit_row(i) * P.N + unit_col(i));
    ok = __all_sync(0xFFFFFFFFu, mbar_wait(&B->acc_full, 0, B, P.status)) != 0;
    tc_fence_after();
  }
  // ------------------------------------------------ epilogue: warps 0-15; the stages are free now
  const uint32_t t_row = tmem + ((uint32_t)(quad * 32) << 16);
  if (side < 4 && ok) {                                    // (the producer and the issuer are past the last side)
    uint4* stage = reinterpret_cast<uint4*>(smem) + warp * 32 * kUnits;
#pragma unroll 1
    for (int j = 0; j < kCols; j += 16) {
      uint32_t o[16];
      tmem_ld16(t_row + side * kCols + j, o);
      tmem_wait_ld();
      uint32_t w[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) w[e] = pack_bf16(__uint_as_float(o[2 * e]), __uint_as_float(o[2 * e + 1]));
      if (P.gelu) gelu_warp(w);
#pragma unroll
      for (int u = 0; u < 2; ++u)
        stage[lane * kUnits + ((j / 8 + u) ^ (lane & (kUnits - 1)))] = make_uint4(w[4 * u], w[4 * u + 1], w[4 * u + 2], w[4 * u + 3]);
    }
    __syncwarp();
    constexpr int kAtOnce = RES ? kUnits : 4;              // (a residual's registers have to be named)
#pragma unroll kAtOnce
    for (int i = 0; i < kUnits; ++i) {
      const int r = (lane + 32 * i) / kUnits, u = (lane + 32 * i) % kUnits;
      if (unit_row(i) < P.M && unit_col(i) < P.N)
        gemm_store8<RES>(P, unit_row(i), unit_col(i), stage[r * kUnits + (u ^ (r & (kUnits - 1)))], residual[RES ? i : 0]);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kIssuer) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)BN) : "memory");
  }
}

// Tile width, from a model in nanoseconds fitted to a sweep over twenty shapes (261 to 1374 rows, N 768 to 4096, K 1024 to
// 4096): waves over 148 SMs, one CTA each; 350, 260 and 217 per K step of a 256-, 128- and 64-wide tile (loads: 48, 32 and
// 24 KB); 4,200, 3,100 and 2,400 for set-up and epilogue.  1041 x 1024 x 4096 takes 26.8, 20.5 and 17.0 us.  K is not
// split: that product would gain (14.8 us in clusters of two), but its sums would be grouped otherwise, and 24 layers of
// bf16 turn any such change into one or two per cent of the result.
inline int gemm_tile_width(int M, int N, int K) {
  const long tiles_m = (M + kGemmBM - 1) / kGemmBM, steps = K / kGemmBK;
  auto ns = [&](int bn, long step, long fixed) { return (tiles_m * ((N + bn - 1) / bn) + 147) / 148 * (steps * step + fixed); };
  const long wide = ns(256, 350, 4200), middle = ns(128, 260, 3100), narrow = ns(64, 217, 2400);
  return wide <= middle && wide <= narrow ? 256 : (middle <= narrow ? 128 : 64);
}

static inline int gemm_tcgen05_launch(const void* A, const void* Bm, const GemmArgs& P, cudaStream_t st) {
  CUtensorMap ta, tb;
  int rc = make_rows_map(&ta, A, P.M, P.K, kGemmBM);       // 64 k-columns x 128 rows per box
  if (rc) return rc;
  rc = make_rows_map(&tb, Bm, P.K, P.N, kGemmBK);          // 64 n-columns x 64 k-rows per box
  if (rc) return rc;
  const int bn = gemm_tile_width(P.M, P.N, P.K);
  const bool res = P.residual != nullptr;
  const auto kernel = bn == 256   ? (res ? k_gemm_bf16_tcgen05<256, true> : k_gemm_bf16_tcgen05<256, false>)
                      : bn == 128 ? (res ? k_gemm_bf16_tcgen05<128, true> : k_gemm_bf16_tcgen05<128, false>)
                                  : (res ? k_gemm_bf16_tcgen05<64, true> : k_gemm_bf16_tcgen05<64, false>);
  static std::atomic<uint64_t> smem_set[6];
  const size_t smem = gemm_smem_bytes(bn);
  cudaError_t e = allow_smem(kernel, smem, smem_set[(bn == 256 ? 0 : (bn == 128 ? 2 : 4)) + res]);
  if (e == cudaSuccess)
    e = launch_dependent(kernel, dim3((P.N + bn - 1) / bn, (P.M + kGemmBM - 1) / kGemmBM), kGemmThreads, 1, smem, st, true, ta, tb, P);
  if (e != cudaSuccess) { g_attn_last_error = (int)e; return OVGGT_ERR_CUDA; }
  return OVGGT_OK;
}

}  // namespace ovggt
