// Shared device helpers of the OVGGT step kernels: element access, block primitives.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/ovggt.h"

namespace ovggt {

constexpr int kF32 = OVGGT_DTYPE_F32;
constexpr int kBF16 = OVGGT_DTYPE_BF16;

// Elements per 16-byte vector of a stored row.
template <int DT> struct VecOf { static constexpr int n = (DT == kBF16) ? 8 : 4; };

__host__ __device__ inline int elem_bytes(int dtype) { return dtype == kBF16 ? 2 : 4; }

// Expand one 16-byte vector of stored elements to floats (exact).
template <int DT>
__device__ __forceinline__ void unpack(const uint4& u, float* f) {
  if constexpr (DT == kBF16) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
  } else {
    f[0] = __uint_as_float(u.x);
    f[1] = __uint_as_float(u.y);
    f[2] = __uint_as_float(u.z);
    f[3] = __uint_as_float(u.w);
  }
}

__device__ __forceinline__ uint4 ld_nc(const uint4* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// Sum over the warp in a fixed butterfly order; every lane gets the result.
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
  return x;
}

// Priority -> unsigned key whose integer order is the ranking order:
// NaN ranks with -inf, -0 equals +0, larger float = larger key.
__device__ __forceinline__ uint32_t rank_key(float x) {
  if (x != x) x = -INFINITY;
  if (x == 0.0f) x = 0.0f;
  uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// One output step of the SplitMix64 generator from state x (Steele, Lea, Flood 2014), and the uniform priority in
// [0, 1) that the random-eviction mode gives token `token_id` in the step of frame `frame_id`: the top 24 bits of
// SplitMix64(SplitMix64(seed ^ frame_id) + token_id), exact in fp32.
__host__ __device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
  unsigned long long z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__host__ __device__ __forceinline__ float random_priority(unsigned long long step_key, long long token_id) {
  return (float)(splitmix64(step_key + (unsigned long long)token_id) >> 40) * (1.0f / 16777216.0f);
}

// Range check of an index that a kernel has read from device memory (survivor lists, slots, move lists).  In the
// ordinary build it costs nothing.  Built with -DOVGGT_BOUNDS_CHECK, an index outside [0, n) is not used: the access
// is skipped and OVGGT_ERR_DEVICE_STATUS goes to the status word, which the next ovggt_cache_stats reports - no trap,
// the kernel runs to its end.
#ifdef OVGGT_BOUNDS_CHECK
__device__ __forceinline__ bool index_ok(long long i, long long n, int* status) {
  if (i >= 0 && i < n) return true;
  if (status != nullptr) atomicCAS(status, 0, OVGGT_ERR_DEVICE_STATUS);
  return false;
}
#else
__device__ __forceinline__ bool index_ok(long long, long long, int*) { return true; }
#endif

// Programmatic dependent launch.  A kernel launched with it may start while the one before it in the stream drains;
// pdl_wait returns once that one has completed and its writes are visible (at once when the kernel was launched plainly).
// pdl_trigger lets the kernel after this one start as soon as every CTA of this one has come here or ended.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// A kernel that starts at its predecessor's trigger and does not wait for its end may read what kernels BEFORE that one wrote:
// those are complete (the predecessor waited for them before it triggered) and their writes are in L2, but this SM's first-level
// cache may still hold lines from before.  So such data is read by bulk copies or __ldcg, which go to L2, or by plain loads
// behind a CTA barrier ahead of which one thread has called this: an acquire, which drops the first-level lines.  `word` is
// any word of global memory.  (Loads of the read-only path, __ldg, are not covered.)
__device__ __forceinline__ void drop_stale_lines(const int* word) {
  int x;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(x) : "l"(word) : "memory");
}

// The column sums of the cached keys after a step: those before it, plus the rows that come, less the rows that leave.  The
// selection takes them itself, or leaves the rows in a list per CTA of its cluster for the attention beside it to take (see
// take_key_sums); either way the rows of a list are added in the same order, so the sums are the same bits.
constexpr int kSumsLists = 8;                 // CTAs of the selection's cluster
constexpr int kSumsNone = 0x7FFFFFFF;         // an entry without a row
struct KeySums {
  const uint2* k_cache;                       // [.., C] bf16
  const float* ksum; float* ksum_next;        // [C] before (nullptr: zero) and after the step; ksum_next nullptr: not asked for
  const int* list; const int* out;            // as CompressParams::sums_list, sums_out
  int cap, M, C, rows;                        // rows: of k_cache
};
// New rows that a list names, of a frame of M.
__host__ __device__ constexpr int sums_share(int M, int lists) { return (M + lists - 1) / lists; }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, int threads, int cluster, size_t smem, cudaStream_t st,
                                    bool pdl, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  if (pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Opt a kernel in to `bytes` of dynamic shared memory, and its SMs to the largest shared-memory carve-out: an SM whose
// carve-out was set up for a kernel with little shared memory has to drain before a CTA of the attention (115 KB) can join
// it, so a selection running beside the attention would keep its SMs to itself.  Once per kernel and device (the calls
// are safe to repeat, so threads may race here).  `done` belongs to this copy of the library: a function that keeps one is static
// or in an anonymous namespace, since the statics of an inline function would be shared by all copies a process has loaded.
template <typename K>
inline cudaError_t allow_smem(K kernel, size_t bytes, std::atomic<uint64_t>& done, bool carveout = true) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = 1ull << (dev & 63);
  if (dev < 64 && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && carveout) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess && dev < 64) done.fetch_or(bit);
  return e;
}

// ---- block-wide primitive for a block of up to 1024 threads; `sh` holds >= 32 words.

// Exclusive prefix sum of x over the threads of the block in thread order; *total = block sum.
__device__ __noinline__ int block_excl_scan_int(int x, int* sh, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = (blockDim.x + 31) >> 5;
  int incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += y;
  }
  __syncthreads();
  if (lane == 31) sh[warp] = incl;
  __syncthreads();
  int base = 0, tot = 0;
  for (int w = 0; w < nwarp; ++w) {
    if (w < warp) base += sh[w];
    tot += sh[w];
  }
  *total = tot;
  return base + incl - x;
}

}  // namespace ovggt
