// fp32 flash attention for sm_100a on the bf16 tensor pipe: out = softmax(Q K^T / sqrt(64)) V per head, head_dim 64.
//
// The tensor cores take no fp32 operands, so every operand is written as the sum of three bf16 numbers,
// x = h + m + l (each the rounded remainder of the ones before: |m| <= 2^-9 |x|, |l| <= 2^-18 |x|, what is left over is
// below 2^-27 |x|), and a product as six of the nine partial products, hh + hm + mh + hl + mm + lh; the three left out
// are below 2^-26 of it, less than the rounding of an fp32 product.  A bf16 product is exact in fp32, the smallest
// partial products are accumulated first, and no accumulation in tensor memory is longer than one 64-row tile: Q K^T
// sums 64 terms, and the P V product of a tile starts from zero and is added to fp32 registers, because long sums in
// tensor memory are not rounded to nearest.  Measured against fp64 the result is as close as that of plain fp32
// arithmetic.
//
// What bounds it: 48 MMAs of 128 x 64 x 16 per 128 x 64 tile, which take the tensor pipe some 61 cycles each, 5,850 for two
// query tiles; the softmax of a tile is busy for 2,500 of them, the splitting of a K and V tile for 1,900.  A plain fp32 kernel is
// bound by the FMA pipes at 64 x 2 x 2 instructions per score instead, an order of magnitude more.
// A CTA owns one or two (TILES) tiles of 128 query rows of one head and a range of 64-row KV tiles.  With two there is one CTA
// per SM; K and V are split once for both tiles, and their planes have room for two stages (1374 x 5470 x 16: 176 us, with one tile
// 215).  With one there are two per SM, of one stage each, whose MMAs wait for the splitting; but such a CTA is set up 2 us sooner,
// and of them a frame has as many as it has tiles, which fill the SMs better (see attn_f32_plan).  (Four MMAs a K step instead of
// six, those that share a plane of A with B planes side by side, leave no room for a second buffer of scores: 259 us.)
// Warps, for each of the TILES:
//   4 softmax    one thread per query row; running maximum, P split and written to tensor memory over the scores it came from,
//                O accumulated in registers
//   1 issuer     of the MMAs of its tile (the whole warp in step, one elected lane); the first one allocates tensor memory
//   3 splitting  read K and V rows from global memory, split them and write the bf16 planes, 128-byte swizzled, to shared
//                memory (done once per CTA and tile: cheaper than a pass over the cache that writes planes, and it needs no
//                scratch memory)
// A result that is not finite is taken again in plain fp32 arithmetic, which says whether it should be (see plain_row).
// Every wait is bounded; on expiry the CTA records OVGGT_ERR_TIMEOUT and leaves through the common teardown.
#pragma once

#include "attn_tcgen05.cuh"

namespace ovggt {

constexpr int kF32BN = 64;                              // KV rows per tile
__host__ __device__ constexpr int f32_threads(int tiles) { return 256 * tiles; }
constexpr int kF32QPlane = kBM * kHD * 2;               // 16 KB
constexpr int kF32KvPlane = kF32BN * kHD * 2;           // 8 KB
constexpr int kF32RegsSoftmax = 168, kF32RegsOther = 88;
static_assert(128 * kF32RegsSoftmax + 128 * kF32RegsOther <= 256 * kRegsLaunch, "register pool of the CTA exceeded");
// Of each query tile's 256 columns: S_b at columns [96 b, 96 b + 64), the planes of P_b over it at [96 b, 96 b + 96), O of a tile at [192, 256)
constexpr int kF32ColBuf = 96, kF32ColO = 192;

struct F32Barriers {
  unsigned long long k_full[2], k_empty[2], v_full[2], v_empty[2];   // by stage
  unsigned long long s_full[2][2], p_full[2], o_full[2], drain[2];   // by query tile
  uint32_t tmem_base;
  int abort_flag;
  int odd[2];             // a result of the tile is not finite
};
__host__ __device__ constexpr int f32_planes(int tiles) { return tiles * (3 * kF32QPlane + 6 * kF32KvPlane); }
static_assert(kJoinStages * kPartBytes <= f32_planes(1), "the parts do not fit the operand planes");
constexpr size_t f32_smem_bytes(int tiles, bool join) { return (size_t)f32_planes(tiles) + sizeof(F32Barriers) + (join ? sizeof(PartJoin) + kJoinTable * 4 : 0) + 64; }

struct F32Params {
  const float *q, *k, *v;
  int M, N, H;
  int splits, tiles_per_split, tiles_total;
  float* out;             // [M, C]            (splits == 1)
  float* o_part;          // these as in AttnParams
  float2* ml_part;
  float* lse;             // [M, H] or nullptr
  int* status;            // or nullptr
  int wait_first;         // these as in AttnParams
  unsigned* tickets;
};

// A pair of floats as three bf16 pairs.
__device__ __forceinline__ void split3(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = pack_bf16(a, b);
  a -= __uint_as_float(h << 16);
  b -= __uint_as_float(h & 0xFFFF0000u);
  m = pack_bf16(a, b);
  a -= __uint_as_float(m << 16);
  b -= __uint_as_float(m & 0xFFFF0000u);
  l = pack_bf16(a, b);
}
// Eight floats of columns [8 j, 8 j + 8) of row r -> the same place of three swizzled planes.
__device__ __forceinline__ void store_planes(unsigned char* base, int plane_bytes, int r, int j, const float4& x, const float4& y) {
  uint4 h, m, l;
  split3(x.x, x.y, h.x, m.x, l.x);
  split3(x.z, x.w, h.y, m.y, l.y);
  split3(y.x, y.y, h.z, m.z, l.z);
  split3(y.z, y.w, h.w, m.w, l.w);
  unsigned char* p = base + r * 128 + ((j ^ (r & 7)) << 4);
  *reinterpret_cast<uint4*>(p) = h;
  *reinterpret_cast<uint4*>(p + plane_bytes) = m;
  *reinterpret_cast<uint4*>(p + 2 * plane_bytes) = l;
}

// The six partial products, (plane of A, plane of B), smallest first.
__device__ constexpr int kSplitA[6] = {2, 0, 1, 1, 0, 0};
__device__ constexpr int kSplitB[6] = {0, 2, 1, 0, 1, 0};

// Takes the rows of this CTA's query tile whose results are not finite again, a warp each; called by the softmax warps, whose
// register budget covers any function's.  A function, not inline: with its loops in the kernel the softmax loop came out 5
// to 11 % slower (1374 x 5470 x 16: 209 us without any of this, 211 so, 220 to 232 inline); one per cent is what looking for such
// rows costs.
__device__ __noinline__ void redo_rows(const F32Params& P, int qt) {
  const int lane = threadIdx.x & 31, h = blockIdx.y;
  const PlainRows plain = {P.q, P.k, P.v, P.N, P.H};
#pragma unroll 1
  for (int r = (threadIdx.x >> 5) & 3; r < kBM && qt * kBM + r < P.M; r += 4) {
    const int m = qt * kBM + r;
    float2* o = reinterpret_cast<float2*>(P.out + ((size_t)m * P.H + h) * kHD) + lane;
    float2 x = *o;
    if (__any_sync(0xFFFFFFFFu, !(x.x * 0.0f + x.y * 0.0f == 0.0f))) {
      plain_row<32>(plain, m, h, P.lse, &x.x);
      *o = x;
    }
  }
}

// JOIN: the parts of a split KV range are joined here (see join_parts); with two TILES only for frames of one.
template <int TILES, bool JOIN>
__global__ void __launch_bounds__(f32_threads(TILES), 2 / TILES) k_attn_f32(const __grid_constant__ F32Params P) {
  constexpr int kThreads = f32_threads(TILES), kConverters = 96 * TILES, kStages = TILES;
  extern __shared__ __align__(1024) unsigned char smem[];
  if (smem_u32(smem) & 1023u) {                      // the 128-byte swizzle needs 1024-byte aligned tiles
    if (threadIdx.x == 0) report_status(P.status, OVGGT_ERR_DEVICE_STATUS);
    return;
  }
  unsigned char* sQ = smem;                            // [2 tiles][3 planes]
  unsigned char* sK = sQ + TILES * 3 * kF32QPlane;         // [stages][3 planes]
  unsigned char* sV = sK + kStages * 3 * kF32KvPlane;
  F32Barriers* B = reinterpret_cast<F32Barriers*>(smem + f32_planes(TILES));
  PartJoin* J = reinterpret_cast<PartJoin*>(B + 1);    // [2]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.y, split = blockIdx.z;
  const int q_tiles = (P.M + kBM - 1) / kBM, tiles = TILES == 1 ? 1 : min(TILES, q_tiles - TILES * (int)blockIdx.x);   // of this CTA
  const int t_begin = split * P.tiles_per_split;
  const int n_tiles = min(P.tiles_total, t_begin + P.tiles_per_split) - t_begin;   // >= 1 by construction
  const int C = P.H * kHD;

  if (P.wait_first) pdl_wait();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&B->k_full[s], kConverters);
      mbar_init(&B->v_full[s], kConverters);
      mbar_init(&B->k_empty[s], tiles);
      mbar_init(&B->v_empty[s], tiles);
    }
    for (int i = 0; i < TILES; ++i) {
      mbar_init(&B->s_full[i][0], 1);
      mbar_init(&B->s_full[i][1], 1);
      mbar_init(&B->p_full[i], 128);
      mbar_init(&B->o_full[i], 1);
      mbar_init(&B->drain[i], 1);
      B->odd[i] = 0;
      if constexpr (JOIN)
        for (int s = 0; s < kJoinStages; ++s) mbar_init(&J->full[s], 1);
    }
    B->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 4 * TILES) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&B->tmem_base)),
                 "r"((uint32_t)(TILES * kTmemCols))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // (K and V, which the front wrote, are read behind the barrier below)
  if (threadIdx.x == kThreads - 32 && !P.wait_first) drop_stale_lines(reinterpret_cast<const int*>(P.q));
#pragma unroll 1
  for (int tile = 0; tile < tiles; ++tile) {           // a query tile's planes: 128 rows x 8 groups of 8 columns, rows past M zero
    constexpr int kPer = kBM * 8 / kThreads;
    float4 x[kPer], y[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int idx = threadIdx.x + i * kThreads, m = (TILES * (int)blockIdx.x + tile) * kBM + (idx >> 3);
      x[i] = y[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (m < P.M) {
        const float4* p = reinterpret_cast<const float4*>(P.q + (size_t)m * C + (size_t)h * kHD + (idx & 7) * 8);
        x[i] = __ldcg(p);
        y[i] = __ldcg(p + 1);
      }
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int idx = threadIdx.x + i * kThreads;
      store_planes(sQ + tile * 3 * kF32QPlane, kF32QPlane, idx >> 3, idx & 7, x[i], y[i]);
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *(volatile uint32_t*)&B->tmem_base;

  if (warp >= 4 * TILES) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kF32RegsOther));
    if (warp < 5 * TILES) {
      // ------------------------------------------------ MMA issuers, one per query tile: QK(0) | QK(1) PV(0) | QK(2) PV(1) | ...
      // QK(t + 1) goes into the other buffer, whose P(t - 1) the already issued PV(t - 1) reads first (the tensor pipe
      // executes one thread's MMAs in order).
      const int i = warp - 4 * TILES;
      if (i < tiles) {
        const bool leader = elect_one();
        const uint32_t tm = __reduce_or_sync(0xFFFFFFFFu, tmem) + i * kTmemCols;
        constexpr uint32_t idesc_qk = idesc_bf16(kF32BN, false), idesc_pv = idesc_bf16(kHD, true);
        const uint64_t dq = smem_desc_sw128(smem_u32(sQ + i * 3 * kF32QPlane));
        const uint64_t dk0 = smem_desc_sw128(smem_u32(sK)), dv0 = smem_desc_sw128(smem_u32(sV));
        auto wait_all = [&](void* bar, uint32_t parity) {
          return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, B, P.status)) != 0;
        };
        auto issue_qk = [&](int t) {
          const uint64_t dk = dk0 + (uint64_t)(t % kStages * (3 * kF32KvPlane >> 4));
          if (leader) {
#pragma unroll
            for (int g = 0; g < 6; ++g)
#pragma unroll
              for (int kk = 0; kk < kHD / 16; ++kk)
                mma_ss(tm + (t & 1) * kF32ColBuf, dq + (uint64_t)(kSplitA[g] * (kF32QPlane >> 4) + kk * 2),
                       dk + (uint64_t)(kSplitB[g] * (kF32KvPlane >> 4) + kk * 2), idesc_qk, g > 0 || kk > 0);
            tc_commit(&B->s_full[i][t & 1]);
            tc_commit(&B->k_empty[t % kStages]);
          }
        };
        bool ok = wait_all(&B->k_full[0], 0);
        if (ok) {
          tc_fence_after();
          issue_qk(0);
        }
        for (int t = 0; t < n_tiles && ok; ++t) {
          if (t + 1 < n_tiles) {
            ok = wait_all(&B->k_full[(t + 1) % kStages], (uint32_t)((t + 1) / kStages) & 1u);
            if (!ok) break;
            tc_fence_after();
            issue_qk(t + 1);
          }
          ok = wait_all(&B->v_full[t % kStages], (uint32_t)(t / kStages) & 1u);
          if (ok) ok = wait_all(&B->p_full[i], (uint32_t)t & 1u);
          if (!ok) break;
          tc_fence_after();
          if (leader) {
            const uint64_t dv = dv0 + (uint64_t)(t % kStages * (3 * kF32KvPlane >> 4));
#pragma unroll
            for (int g = 0; g < 6; ++g)
#pragma unroll
              for (int kk = 0; kk < kF32BN / 16; ++kk)
                mma_ts(tm + kF32ColO, tm + (t & 1) * kF32ColBuf + kSplitA[g] * 32 + kk * 8,
                       dv + (uint64_t)(kSplitB[g] * (kF32KvPlane >> 4) + kk * 128), idesc_pv, g > 0 || kk > 0);
            tc_commit(&B->v_empty[t % kStages]);
            tc_commit(&B->o_full[i]);
          }
        }
        if (ok) {
          wait_all(&B->o_full[i], (uint32_t)(n_tiles - 1) & 1u);
        } else {
          if (leader) tc_commit(&B->drain[i]);          // let every issued MMA finish before TMEM is freed
          wait_all(&B->drain[i], 0);
        }
      }
      __syncwarp();
    } else {
      // ------------------------------------------------ K / V splitting
      // A tile's rows are requested as soon as the registers are free: with two query tiles a tile ahead of the buffer they go to.
      const int ct = (int)threadIdx.x - 160 * TILES;
      constexpr int kVecs = kF32BN * 8, kPer = (kVecs + kConverters - 1) / kConverters;
      struct Rows { float4 x[kPer], y[kPer]; };
      auto load = [&](const float* src, int t, Rows& w) {
        const int row0 = (t_begin + t) * kF32BN;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          const int idx = ct + i * kConverters, r = row0 + (idx >> 3);
          w.x[i] = w.y[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (idx < kVecs && r < P.N) {
            const float4* p = reinterpret_cast<const float4*>(src + (size_t)r * C + (size_t)h * kHD + (idx & 7) * 8);
            w.x[i] = p[0];
            w.y[i] = p[1];
          }
        }
      };
      auto convert = [&](const Rows& w, unsigned char* planes, int t, unsigned long long* empty, unsigned long long* full) -> bool {
        const int s = t % kStages;
        if (t >= kStages && !mbar_wait(&empty[s], (uint32_t)(t / kStages - 1) & 1u, B, P.status)) return false;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          const int idx = ct + i * kConverters;
          if (idx < kVecs) store_planes(planes + s * 3 * kF32KvPlane, kF32KvPlane, idx >> 3, idx & 7, w.x[i], w.y[i]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(&full[s]);
        return true;
      };
      if constexpr (TILES == 2) {
        Rows k, v;
        load(P.k, 0, k);
        load(P.v, 0, v);
#pragma unroll 1
        for (int t = 0; t < n_tiles; ++t) {
          if (!convert(k, sK, t, B->k_empty, B->k_full)) break;
          if (t + 1 < n_tiles) load(P.k, t + 1, k);
          if (!convert(v, sV, t, B->v_empty, B->v_full)) break;
          if (t + 1 < n_tiles) load(P.v, t + 1, v);
        }
      } else {                                          // (twice the rows a thread: registers for one tile's)
        Rows w;
#pragma unroll 1
        for (int t = 0; t < n_tiles; ++t) {
          load(P.k, t, w);
          if (!convert(w, sK, t, B->k_empty, B->k_full)) break;
          load(P.v, t, w);
          if (!convert(w, sV, t, B->v_empty, B->v_full)) break;
        }
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------ softmax and accumulation of O (128 threads a tile, one query row each)
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kF32RegsSoftmax));
    const int tile = warp >> 2, qt = TILES * (int)blockIdx.x + tile, row = (warp & 3) * 32 + lane;
    if (tile < tiles) {
    const uint32_t t_row = tmem + tile * kTmemCols + ((uint32_t)((warp & 3) * 32) << 16);
    const float c = 1.4426950408889634f * 0.125f;     // log2(e) / sqrt(64)
    float mref = -INFINITY, l = 0.0f;
    float acc[kHD];
#pragma unroll
    for (int i = 0; i < kHD; ++i) acc[i] = 0.0f;
    bool ok = true;
    // acc += O of tile t (both under the reference that held when its P was made)
    auto take_o = [&](int t) -> bool {
      if (__all_sync(0xFFFFFFFFu, mbar_wait(&B->o_full[tile], (uint32_t)t & 1u, B, P.status)) == 0) return false;
      tc_fence_after();
#pragma unroll
      for (int j = 0; j < kHD; j += 16) {
        uint32_t o[16];
        tmem_ld16(t_row + kF32ColO + j, o);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[j + e] += __uint_as_float(o[e]);
      }
      return true;
    };
    for (int t = 0; t < n_tiles; ++t) {
      const uint32_t buf = t_row + (t & 1) * kF32ColBuf;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(&B->s_full[tile][t & 1], (uint32_t)(t >> 1) & 1u, B, P.status)) != 0;
      if (!ok) break;
      tc_fence_after();
      uint32_t s[kF32BN];
      tmem_ld32(buf, s);
      tmem_ld32(buf + 32, s + 32);
      tmem_wait_ld();
      const int left = P.N - (t_begin + t) * kF32BN;
      if (left < kF32BN) {
#pragma unroll
        for (int j = 0; j < kF32BN; ++j)
          if (j >= left) s[j] = 0xFF800000u;           // -inf on columns past the last row
      }
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int j = 0; j < kF32BN; j += 2)
        m4[(j >> 1) & 3] = max3(m4[(j >> 1) & 3], __uint_as_float(s[j]), __uint_as_float(s[j + 1]));
      const float mnew = fmaxf(mref, fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * c);
      const float corr = ex2(mref - mnew);             // 0 on the first tile, 1 when the maximum stands
      float sum4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int j = 0; j < kF32BN; j += 16) {
        uint32_t ph[8], pm[8], pl[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float p0 = ex2(fmaf(__uint_as_float(s[j + 2 * e]), c, -mnew));
          const float p1 = ex2(fmaf(__uint_as_float(s[j + 2 * e + 1]), c, -mnew));
          sum4[e & 3] += p0 + p1;
          split3(p0, p1, ph[e], pm[e], pl[e]);
        }
        tmem_st8(buf + j / 2, ph);
        tmem_st8(buf + 32 + j / 2, pm);
        tmem_st8(buf + 64 + j / 2, pl);
      }
      l = fmaf(l, corr, (sum4[0] + sum4[1]) + (sum4[2] + sum4[3]));
      if (t > 0) {
        ok = take_o(t - 1);
        if (!ok) break;
        if (__any_sync(0xFFFFFFFFu, corr != 1.0f)) {
#pragma unroll
          for (int i = 0; i < kHD; ++i) acc[i] *= corr;
        }
      }
      mref = mnew;
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&B->p_full[tile]);
    }
    if (ok) ok = take_o(n_tiles - 1);
    const int m = qt * kBM + row;
    if (ok && m < P.M) {
      const bool whole = P.splits == 1;
      const float f = whole ? 1.0f / l : 1.0f;
      const size_t part_row = JOIN ? join_row0(P.M, qt, h, P.splits) + (size_t)split * min(kBM, P.M - qt * kBM) + row
                                   : (size_t)split * P.M + m;
      float* part = JOIN ? P.o_part + part_row * kHD : P.o_part + part_row * C + (size_t)h * kHD;
      float4* dst = reinterpret_cast<float4*>(whole ? P.out + (size_t)m * C + (size_t)h * kHD : part);
#pragma unroll
      for (int i = 0; i < kHD; i += 4) {
        const float4 x = make_float4(acc[i] * f, acc[i + 1] * f, acc[i + 2] * f, acc[i + 3] * f);
        dst[i / 4] = x;
        if (!JOIN && whole && !all_finite(x)) B->odd[tile] = 1;
      }
      if (!whole) P.ml_part[JOIN ? part_row : part_row * P.H + h] = make_float2(mref, l);
      if (whole && P.lse != nullptr) P.lse[(size_t)m * P.H + h] = mref + log2f(l);
    }
    if constexpr (JOIN) {
      if (join_arrive(J, P.tickets + h * q_tiles + qt, P.splits, ok, tile)) {
        const int m0 = qt * kBM;
        const size_t row0 = join_row0(P.M, qt, h, P.splits);
        join_parts(J, B, smem, reinterpret_cast<float*>(J + 1), P.o_part + row0 * kHD, P.ml_part + row0, min(kBM, P.M - m0),
                   P.splits, P.out + (size_t)m0 * C + h * kHD, C, P.lse != nullptr ? P.lse + (size_t)m0 * P.H + h : nullptr, P.H,
                   P.status, &B->odd[tile], tile);
      }
    }
    softmax_warps_sync(tile);
    if (*(volatile int*)&B->odd[tile]) redo_rows(P, qt);
    }
  }

  // ------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (warp == 4 * TILES) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(TILES * kTmemCols)) : "memory");
  }
  if (!P.wait_first) pdl_wait();
}

// ---------------------------------------------------------------- host side

// Query tiles a CTA and parts of the KV range, by the time that they take in units of 0.05 us, in a step and alone.
// CTAs of one tile: the set-up, and waves over two places an SM, each as long as its KV tiles, less where no two share an SM.
// CTAs of two tiles: a longer set-up, which a step hides under the start of its selection, and waves over an SM each; beside the
// selection that leaves 140, and a CTA more has to wait for its end.  A CTA with a tile missing is over somewhat sooner.  Parts cost a
// merge, which writes and reads them, or joining.  Frames of one tile take the CTA of two: twice the warps to split K and V, 1.1 to
// 1.5 times as fast.  The number of parts decides how sums are grouped, so a step's halves take that of a step; the kind of CTA does
// not, and is their own.  (In a step the constants stand for more than their names: a wave also waits for the selection.)
// Fitted to 20,000 timings (steps: 5 to 1374 rows over 300 to 16,000, alone: 1 to 1374 over 64 to 12,000; 1 to 16 heads, either
// CTA, 1 to 16 parts).  Against CTAs of one tile throughout (two places an SM, a merge as long as three KV tiles) steps take 0.88 and
// the attention alone 0.94 of the time, against CTAs of two throughout 0.99 and 0.88; against the better of both 0.998 (worst 1.13:
// 518 + 4000 x 4) and 0.979 (1.05).  A step of 1041 + 2500 x 16: 118 us, with two tiles a CTA 153; 329 + 6000 x 12: 65 and 71.
struct F32Times {
  int set_up1, wave1, shared, alone, slots1;           // CTAs of one tile; a KV tile of two that share an SM, of one alone
  int set_up2, wave2, pair, single, slots2, odd;       // CTAs of two; a KV tile of such a frame, of a frame of one; a lone tile's share of 20
  int merge, merge_rows, joined, joined_part;          // merge and rows of parts a unit, joining and each part joined
};
constexpr int kF32JoinTiles = 5, kF32JoinTilesOne = 2;  // KV tiles a part up to which parts are joined: CTAs of one tile, frames of one tile
constexpr F32Times kF32Step = {50, 128, 67, 59, 296, 167, 44, 50, 19, 140, 19, 5, 287, 42, 20};
constexpr F32Times kF32Alone = {86, 18, 68, 48, 296, 140, 11, 51, 26, 148, 18, 30, 371, 0, 0};

inline bool attn_f32_join(int tiles, int q_tiles, int H, int splits, long per) {
  return splits > 1 && (long)(q_tiles + tiles - 1) / tiles * H * splits * tiles <= 2 * 148 &&
         (tiles == 1 ? per <= kF32JoinTiles : q_tiles == 1 && per <= kF32JoinTilesOne);
}
inline long attn_f32_time(const F32Times& T, int tiles, int q_tiles, int M, int H, int s, long per) {
  const long heads = (long)H * s, n = q_tiles * heads;
  long t;
  if (tiles == 1) {
    const long rest = n % T.slots1, shared = n / T.slots1 + (rest > T.slots1 / 2), alone = rest > 0 && rest <= T.slots1 / 2;
    t = T.set_up1 + (shared + alone) * T.wave1 + per * (shared * T.shared + alone * T.alone);
    if (T.joined && attn_f32_join(1, q_tiles, H, s, per)) return t + T.joined + T.joined_part * s;
  } else if (q_tiles == 1) {
    t = T.set_up2 + (n + T.slots2 - 1) / T.slots2 * (T.wave2 + T.single * per);
  } else {
    const long n20 = (q_tiles / 2 * 20 + q_tiles % 2 * T.odd) * heads;
    t = T.set_up2 + (n20 + 20 * T.slots2 - 1) / (20 * T.slots2) * (T.wave2 + T.pair * per);
  }
  return s > 1 ? t + T.merge + heads * M / T.merge_rows : t;
}

enum class F32Call { kAlone, kHalf, kStep };           // an attention by itself, the attend half of a step, a step
struct F32Plan { int tiles, splits; };
inline F32Plan attn_f32_plan(int M, int N, int H, int max_splits, F32Call call) {
  const int q_tiles = (M + kBM - 1) / kBM, kv_tiles = (N + kF32BN - 1) / kF32BN;
  auto faster = [&](const F32Times& T, int s, long per, long* time) {   // tiles a CTA
    const long t2 = attn_f32_time(T, 2, q_tiles, M, H, s, per), t1 = q_tiles > 1 ? attn_f32_time(T, 1, q_tiles, M, H, s, per) : t2 + 1;
    *time = std::min(t1, t2);
    return t1 <= t2 ? 1 : 2;
  };
  F32Plan best = {};
  long best_time = -1, time;
  for (int s = 1; s <= max_splits && s <= kv_tiles; ++s) {
    const int per = (kv_tiles + s - 1) / s;
    if ((kv_tiles + per - 1) / per != s) continue;
    const int tiles = faster(call == F32Call::kAlone ? kF32Alone : kF32Step, s, per, &time);
    if (best_time < 0 || time < best_time) {
      best_time = time;
      best = {tiles, s};
    }
  }
  if (call == F32Call::kHalf) best.tiles = faster(kF32Alone, best.splits, (kv_tiles + best.splits - 1) / best.splits, &time);
  return best;
}

// scratch: attn_tcgen05_scratch_bytes, or nullptr (the KV range is then not split).  in_step: a selection runs beside this.
static inline int attn_f32_launch(const void* q, const void* k, const void* v, int M, int N, int H, void* out, void* scratch,
                                  int* status, cudaStream_t st, float* lse, bool beside_previous, unsigned* tickets, int* launches,
                                  bool in_step) {
  const int C = H * kHD;
  F32Params P;
  P.q = static_cast<const float*>(q);
  P.k = static_cast<const float*>(k);
  P.v = static_cast<const float*>(v);
  P.M = M; P.N = N; P.H = H;
  P.tiles_total = (N + kF32BN - 1) / kF32BN;
  const F32Plan plan = attn_f32_plan(M, N, H, scratch ? kMaxSplits : 1, in_step ? F32Call::kStep : tickets ? F32Call::kHalf : F32Call::kAlone);
  P.splits = plan.splits;
  P.tiles_per_split = (P.tiles_total + P.splits - 1) / P.splits;
  P.splits = (P.tiles_total + P.tiles_per_split - 1) / P.tiles_per_split;     // no empty split
  P.out = static_cast<float*>(out);
  P.o_part = static_cast<float*>(scratch);
  P.ml_part = reinterpret_cast<float2*>(static_cast<char*>(scratch) + (size_t)kMaxSplits * M * C * 4);
  P.tickets = tickets;
  P.lse = lse;
  P.status = status;
  P.wait_first = beside_previous ? 0 : 1;
  const int q_tiles = (M + kBM - 1) / kBM;
  const dim3 grid((q_tiles + plan.tiles - 1) / plan.tiles, H, P.splits);
  // (joined where that is no slower in a step: CTAs of one tile 0.93 to 0.98 of the time with a merge up to four KV tiles a part, 1.01 to
  // 1.09 with five, 1.05 to 1.15 from six on; frames of one tile 0.97 up to two, from three on 0.97 to 1.01 but up to 1.18 for some)
  const bool join = tickets && attn_f32_join(plan.tiles, q_tiles, H, P.splits, P.tiles_per_split);
  const auto kernel = plan.tiles == 1 ? (join ? k_attn_f32<1, true> : k_attn_f32<1, false>)
                                      : (join ? k_attn_f32<2, true> : k_attn_f32<2, false>);
  static std::atomic<uint64_t> smem_set[4];
  const size_t smem = f32_smem_bytes(plan.tiles, join);
  cudaError_t e = allow_smem(kernel, smem, smem_set[2 * (plan.tiles - 1) + join]);
  if (e != cudaSuccess) { g_attn_last_error = (int)e; return OVGGT_ERR_CUDA; }
  e = launch_dependent(kernel, grid, f32_threads(plan.tiles), 1, smem, st, true, P);
  if (e != cudaSuccess) { g_attn_last_error = (int)e; return OVGGT_ERR_CUDA; }
  const bool merge = P.splits > 1 && !join;
  *launches = merge ? 2 : 1;
  return merge ? attn_merge_launch<float>(P.o_part, P.ml_part, M, H, P.splits, P.out, lse, st, {P.q, P.k, P.v, N, H}) : OVGGT_OK;
}

}  // namespace ovggt
