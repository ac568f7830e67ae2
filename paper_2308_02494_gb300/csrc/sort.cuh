// Morton order of batches: the sampler's bin scan and the sorted copies of batches in memory.
#pragma once
#include "common.cuh"

namespace srn {

__device__ __forceinline__ int brick_of_point(const Bricks& br, int64_t g) {
  int lo = 0, hi = br.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (br.off[mid] <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Exclusive scan of one brick's kSortBins counters by a block of 1024 threads: each warp scans
// 1024 consecutive counters, 128 at a time (a lane reads four, so every load of a warp is one
// line), with shuffles, and one warp scans the 32 warp totals.
// (With 32 consecutive counters per thread every load touched 32 lines: 11 us.)
__device__ __forceinline__ void scan_bins(uint32_t* hist) {
  constexpr int rounds = kSortBins / 32 / 128;
  static_assert(rounds * 32 * 128 == kSortBins, "a warp's counters are whole rounds of 128");
  __shared__ uint32_t wsum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint4* h = reinterpret_cast<uint4*>(hist) + warp * (rounds * 32) + lane;
  uint4 v[rounds];
  uint32_t incl[rounds];
#pragma unroll
  for (int k = 0; k < rounds; ++k) v[k] = h[32 * k];
#pragma unroll
  for (int k = 0; k < rounds; ++k) incl[k] = v[k].x + v[k].y + v[k].z + v[k].w;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {   // inclusive scans of the rounds' lane totals, side by side
#pragma unroll
    for (int k = 0; k < rounds; ++k) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl[k], o);
      if (lane >= o) incl[k] += y;
    }
  }
  uint32_t total = 0;
#pragma unroll
  for (int k = 0; k < rounds; ++k) {
    const uint32_t t = __shfl_sync(0xffffffffu, incl[k], 31);
    incl[k] += total - (v[k].x + v[k].y + v[k].z + v[k].w);   // exclusive within the warp
    total += t;
  }
  if (lane == 0) wsum[warp] = total;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = wsum[lane];
    uint32_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += y;
    }
    wsum[lane] = wi - w;   // exclusive
  }
  __syncthreads();
  const uint32_t base = wsum[warp];
#pragma unroll
  for (int k = 0; k < rounds; ++k) {
    const uint32_t s = base + incl[k];
    h[32 * k] = make_uint4(s, s + v[k].x, s + v[k].x + v[k].y, s + v[k].x + v[k].y + v[k].z);
  }
}
// The bins' counts, cleared by the whole grid.
__device__ __forceinline__ void sort_clear(const Bricks& br, const SortedBatch& s) {
  uint4* h4 = reinterpret_cast<uint4*>(s.hist);
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < (int64_t)br.n * kSortBins / 4;
       q += (int64_t)gridDim.x * blockDim.x)
    h4[q] = make_uint4(0u, 0u, 0u, 0u);
}
// Ranks and bin counts.
__device__ __forceinline__ void sort_count(const Bricks& br, const float* __restrict__ xyz, const SortedBatch& s) {
  const int64_t total = br.off[br.n], first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  for (int64_t gi = first; gi - lane < total; gi += step) {
    const bool in = gi < total;
    uint32_t key = 0xffffffffu;
    if (in) {
      const int b = brick_of_point(br, gi);
      const uint32_t c = morton_bin(xyz[3 * gi], xyz[3 * gi + 1], xyz[3 * gi + 2]);
      key = (uint32_t)b * kSortBins + c;
    }
    // one atomic per distinct bin of the warp
    const unsigned grp = __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(grp) - 1;
    uint32_t r = 0;
    if (in && lane == leader) r = atomicAdd(s.hist + key, (uint32_t)__popc(grp));
    r = __shfl_sync(0xffffffffu, r, leader);
    if (in) s.rank[gi] = r + __popc(grp & ((1u << lane) - 1u));
  }
}
// The sorted copy (after the scan).  (Points that another stream is writing meanwhile may have
// another bin than they were counted in: their places stay within their brick.)
__device__ __forceinline__ void sort_scatter(const Bricks& br, const float* __restrict__ xyz,
                                             const float* __restrict__ target, const SortedBatch& s) {
  const int64_t total = br.off[br.n];
  for (int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; gi < total; gi += (int64_t)gridDim.x * blockDim.x) {
    const int b = brick_of_point(br, gi);
    const float x = xyz[3 * gi], y = xyz[3 * gi + 1], z = xyz[3 * gi + 2];
    const int64_t dst = min(br.off[b] + (int64_t)s.hist[(int64_t)b * kSortBins + morton_bin(x, y, z)] + s.rank[gi],
                            br.off[b + 1] - 1);
    s.xyz[3 * dst] = x; s.xyz[3 * dst + 1] = y; s.xyz[3 * dst + 2] = z;
    if (s.target) s.target[dst] = target[gi];
    if (s.index) s.index[dst] = (uint32_t)gi;
  }
}

}  // namespace srn
