// Reductions shared by the tiled kernels: block sums, the fixed-order sum of the blocks'
// partials, and the last-block-to-arrive finish.  Everything is in a fixed order, so the
// results are deterministic.
#pragma once

#include "excmg_internal.cuh"

namespace excmg {
namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Sums over the block of NV values per thread; sum v is valid in warp v's first thread.  Every
// thread must call.  float64 instructions are scarce on this GPU (2 per clock per SM,
// 64-clock latency), so one warp adds per value, the values side by side: every thread parks
// its values in shared memory, then each lane of warp v sums blockDim/32 of value v in a fixed
// order and the warp reduces by shuffles.  The order is fixed, so the result is deterministic.
template <int NV>
__device__ __forceinline__ double block_sums(const double (&v)[NV]) {
  static_assert(NV <= kThreads / 32, "a warp per value");
  __shared__ double s_v[NV][kThreads];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) s_v[k][threadIdx.x] = v[k];
  __syncthreads();
  double t = 0.0;
  if (warp < NV) {
    // kThreads / 32 values per lane as a pairwise tree (a short dependence chain)
    double w[kThreads / 32];
#pragma unroll
    for (int u = 0; u < kThreads / 32; ++u) w[u] = s_v[warp][lane + 32 * u];
#pragma unroll
    for (int d = 1; d < kThreads / 32; d *= 2)
#pragma unroll
      for (int u = 0; u + d < kThreads / 32; u += 2 * d) w[u] += w[u + d];
    t = warp_sum(w[0]);
  }
  return t;
}

// Sum over the block; the result is valid in thread 0.  Every thread must call.
__device__ double block_sum(double v) {
  const double vs[1] = {v};
  return block_sums(vs);
}

// One warp's sum of src[0 .. n) from global memory (through L2) in a fixed order: each lane
// takes the values lane, lane + 32, ... in chunks of kSumChunk loads in flight, sums a
// chunk as a pairwise tree, then the lanes reduce by shuffles.  Valid in lane 0.
constexpr int kSumChunk = 8;
__device__ __forceinline__ double warp_sum_global(const double* src, int n) {
  const int lane = threadIdx.x & 31;
  double acc = 0.0;
  for (int i0 = 0; i0 < n; i0 += 32 * kSumChunk) {
    double w[kSumChunk];
#pragma unroll
    for (int u = 0; u < kSumChunk; ++u) {
      const int i = i0 + lane + 32 * u;
      w[u] = i < n ? __ldcg(src + i) : 0.0;
    }
#pragma unroll
    for (int d = 1; d < kSumChunk; d *= 2)
#pragma unroll
      for (int u = 0; u + d < kSumChunk; u += 2 * d) w[u] += w[u + d];
    acc += w[0];
  }
  return warp_sum(acc);
}

template <typename D>
__device__ __forceinline__ int find_problem(const D* descs, int nprob, long long t, int p) {
  while (p + 1 < nprob && t >= descs[p + 1].tile_begin) ++p;
  return p;
}

// Publish this block's per-problem partial sums (NV values per problem) and let the
// last block to arrive for problem p reduce the gridDim.x partials of p in index order
// and call fin(p, sums).  The slot of problem p's state is descs[p].slot.
template <int NV, typename Fin>
__device__ void publish_and_finish(int nprob, const int* s_active, const double* s_part,
                                   double* partials, unsigned* counters, const Fin& fin) {
  __shared__ int s_last[kMaxProb];
  __shared__ double s_sums[NV];
  const int G = gridDim.x;
  for (int p = threadIdx.x; p < nprob; p += blockDim.x) {
    s_last[p] = 0;
    if (s_active[p]) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
        partials[((long long)p * NV + v) * G + blockIdx.x] = s_part[p * NV + v];
      __threadfence();
      const unsigned t = atomicAdd(&counters[p], 1u);
      s_last[p] = (t == (unsigned)G - 1u);
    }
  }
  __syncthreads();
  for (int p = 0; p < nprob; ++p) {
    if (!s_last[p]) continue;  // shared value: uniform across the block
    __threadfence();
    const int v = threadIdx.x >> 5;  // a warp per value
    if (v < NV) {
      const double t = warp_sum_global(partials + ((long long)p * NV + v) * G, G);
      if ((threadIdx.x & 31) == 0) s_sums[v] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      fin(p, s_sums);
      counters[p] = 0u;
    }
    __syncthreads();
  }
}

}  // namespace
}  // namespace excmg
