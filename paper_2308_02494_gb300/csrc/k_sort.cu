// Sorted copies of batches in memory, and the tile list of the training pass.
//
// Neighbouring points of a batch in no order share nothing: each corner read of a warp
// touches 32 lines, a tile's node boxes cover the grid, and the scatter takes one global
// atomic per corner.  The counting sort of the sampler on points in memory reads and writes
// about 48 bytes per point after the count, with one atomic per distinct bin of a warp (about
// 0.05 ns per point), and makes such a batch what the sampler's is.
// Each sort is one cooperative launch: as launches of their own its phases take 4 to 10 us
// longer in a query, and in a training batch that is in order already (the usual one) the
// launches that find nothing to do held up the 2^18-point gradient by 15 us of 340.
#include <algorithm>
#include <climits>
#include <cooperative_groups.h>

#include "kernels.h"
#include "sort.cuh"

namespace srn {
namespace {

constexpr int kSortNT = 1024;

// The points of this thread, first, first + step, ..., with their predecessors, four points'
// loads in flight: f(point, bin code, predecessor's code, brick, first point of its brick).
template <typename F>
__device__ __forceinline__ void with_predecessors(const Bricks& br, const float* __restrict__ xyz, F f) {
  const int64_t total = br.off[br.n], first = (int64_t)blockIdx.x * kSortNT + threadIdx.x;
  const int64_t step = (int64_t)gridDim.x * kSortNT;
  for (int64_t g0 = first; g0 < total; g0 += 4 * step) {
    float q[4][6];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t gi = g0 + k * step;
#pragma unroll
      for (int j = 0; j < 6; ++j) q[k][j] = gi < total && (gi > 0 || j > 2) ? xyz[3 * gi - 3 + j] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t gi = g0 + k * step;
      if (gi >= total) break;
      const int b = brick_of_point(br, gi);
      f(gi, morton_bin(q[k][3], q[k][4], q[k][5]), morton_bin(q[k][0], q[k][1], q[k][2]), b, gi == br.off[b]);
    }
  }
}

// How many points come before their predecessor, first: a batch in order pays only for that
// (6 us, in which the counters, 128 KB per brick, are cleared too).
__global__ void __launch_bounds__(kSortNT) k_sort_query(Bricks br, const float* __restrict__ xyz, SortedBatch s) {
  cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  const int64_t first = (int64_t)blockIdx.x * kSortNT + threadIdx.x;
  uint32_t back = 0;
  if (first == 0) *s.next = 0u;
  with_predecessors(br, xyz, [&](int64_t, uint32_t c, uint32_t before, int, bool head) { back += !head && before > c; });
  back = __reduce_add_sync(0xffffffffu, back);
  if ((threadIdx.x & 31) == 0 && back) atomicAdd(s.moved, back);   // (cleared by the call before)
  sort_clear(br, s);   // (here, so that a copy has one barrier less)
  grid.sync();
  if (*(volatile uint32_t*)s.moved <= s.limit) return;
  sort_count(br, xyz, s);
  grid.sync();
  for (int b = blockIdx.x; b < br.n; b += gridDim.x) {
    scan_bins(s.hist + (int64_t)b * kSortBins);
    __syncthreads();
  }
  grid.sync();
  sort_scatter(br, xyz, nullptr, s);
}

// The tiles of brick b, by a block of 1024 threads.  The brick's largest tile level lmax is the largest L <= lcap whose
// block, mapped through any of the brick's grids, has a node box of at most capn nodes:
// per grid axis, the image's extent in cells plus the box margin, one partial cell at
// each end and the node past the last cell bound tile_box's count (0 when even one unit
// is too large; such grids add their corners directly).  Units without a recorded start
// take the next recorded one (a suffix minimum; for a sorted batch this is exact, for any
// batch the starts become non-decreasing from 0 to n, so the tiles below always partition
// the brick's points).  Every unit then belongs to the largest aligned range of 2^L units
// (L <= lmax) holding at most tp (<= ST) points; each such range becomes ceil(points / tp)
// tiles of consecutive points.
__device__ __forceinline__ void tile_list(const Bricks& br, int b, const TrainWs& ws, const Model& md, int capn,
                                          int lcap, int tp) {
  constexpr int UPT = kUnits / 1024;
  __shared__ int32_t st[kUnits + 1];
  __shared__ int32_t wred[32];
  __shared__ int32_t gbase;
  __shared__ int32_t s_lv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_lv = lcap;
  __syncthreads();
  if (tid < md.M) {
    const float* g = md.G + (int64_t)b * md.sG + 12 * tid;
    const float hs = 0.5f * (float)(md.R - 1) * (2.f / (float)(1 << kUnitBits));   // cells per unit
    int lv = 0;
    for (int L = lcap; L > 0; --L) {
      const float ext[3] = {(float)(1 << ((L + 2) / 3)), (float)(1 << ((L + 1) / 3)), (float)(1 << (L / 3))};
      int nodes = 1;
      for (int d = 0; d < 3; ++d) {
        const float e = (fabsf(g[4 * d]) * ext[0] + fabsf(g[4 * d + 1]) * ext[1] + fabsf(g[4 * d + 2]) * ext[2]) * hs;
        nodes *= min((int)ceilf(e + 0.01f) + 2, md.R);
      }
      if (nodes <= capn) { lv = L; break; }
    }
    atomicMin(&s_lv, lv);
  }
  __syncthreads();
  const int lmax = s_lv;
  const int64_t o = br.off[b];
  const int32_t n = (int32_t)(br.off[b + 1] - o);
  const int32_t* us = ws.ustart + (int64_t)b * (kUnits + 1);
  const uint32_t* bins = ws.bin_start ? ws.bin_start : ws.sorted.use() ? ws.sorted.hist : nullptr;
  int32_t loc[UPT];
  {
    int32_t m = INT_MAX;
#pragma unroll
    for (int k = UPT - 1; k >= 0; --k) {
      // a batch from the sampler or a sorted copy: unit u starts where its first bin starts
      const int32_t v = bins ? (int32_t)bins[(int64_t)b * kSortBins + ((tid * UPT + k) << 3)] : us[tid * UPT + k] - 1;
      if (v >= 0) m = min(m, v);
      loc[k] = m;
    }
    int32_t incl = loc[0];   // suffix minimum over lanes >= lane
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t y = __shfl_down_sync(0xffffffffu, incl, d);
      if (lane + d < 32) incl = min(incl, y);
    }
    if (lane == 0) wred[warp] = incl;
    __syncthreads();
    const int32_t after = min(n, __reduce_min_sync(0xffffffffu, lane > warp ? wred[lane] : n));
    const int32_t next = __shfl_down_sync(0xffffffffu, incl, 1);
    const int32_t excl = lane < 31 ? min(next, after) : after;
#pragma unroll
    for (int k = 0; k < UPT; ++k) st[tid * UPT + k] = min(loc[k], excl);
    // the first point always opens a tile: in a batch that is not sorted, later points
    // of its unit may have overwritten its recorded start
    if (tid == 0) { st[0] = 0; st[kUnits] = n; }
  }
  __syncthreads();
  int nt[UPT], lv[UPT];
  int tot = 0;
#pragma unroll
  for (int k = 0; k < UPT; ++k) {
    const int u = tid * UPT + k;
    int L = 0;
    for (int l = lmax; l > 0; --l) {
      const int a = u & ~((1 << l) - 1);
      if (st[a + (1 << l)] - st[a] <= tp) { L = l; break; }
    }
    lv[k] = L;
    nt[k] = 0;
    if ((u & ((1 << L) - 1)) == 0) nt[k] = (st[u + (1 << L)] - st[u] + tp - 1) / tp;
    tot += nt[k];
  }
  int incl = tot;   // block-wide exclusive scan of the tile counts
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += y;
  }
  __syncthreads();
  if (lane == 31) wred[warp] = incl;
  __syncthreads();
  const int wt = wred[lane];
  const int base = incl - tot + __reduce_add_sync(0xffffffffu, lane < warp ? wt : 0);
  const int all = __reduce_add_sync(0xffffffffu, wt);
  if (tid == 0) gbase = atomicAdd(ws.tile_ctr, all);
  __syncthreads();
  int idx = gbase + base;
#pragma unroll
  for (int k = 0; k < UPT; ++k) {
    const int u = tid * UPT + k;
    const int c = nt[k] ? st[u + (1 << lv[k])] - st[u] : 0;
    for (int t = 0; t < nt[k]; ++t, ++idx) {
      ScatTile T;
      T.start = o + st[u] + (int64_t)t * c / nt[k];
      T.count = (int32_t)((int64_t)(t + 1) * c / nt[k] - (int64_t)t * c / nt[k]);
      T.code = (uint32_t)b << 20 | (uint32_t)lv[k] << 16 | (uint32_t)u;
      ws.tiles[idx] = T;
    }
  }
}

// The tiles of brick b of a batch in no order, by a block: runs of at most `run` points.
__device__ __forceinline__ void run_list(const Bricks& br, int b, const TrainWs& ws, int run) {
  __shared__ int32_t s_first;
  const int64_t o = br.off[b], n = br.off[b + 1] - o;
  const int32_t nt = (int32_t)((n + run - 1) / run);
  if (threadIdx.x == 0) s_first = atomicAdd(ws.tile_ctr, nt);
  __syncthreads();
  for (int t = threadIdx.x; t < nt; t += blockDim.x) {
    const int64_t from = t * n / nt;
    ScatTile T;
    T.start = o + from;
    T.count = (int32_t)((t + 1) * n / nt - from);
    T.code = (uint32_t)b << 20 | kNoBlock << 16;
    ws.tiles[s_first + t] = T;
  }
}

// The sampler's batch: its histogram gives the unit starts.
__global__ void __launch_bounds__(kSortNT) k_tile_list(Bricks brp, TrainWs ws, Model md, int capn, int lcap, int tp) {
  __shared__ Bricks br;
  load_bricks(brp, br);
  tile_list(br, blockIdx.x, ws, md, capn, lcap, tp);
}

// A caller's batch: the first point of every Morton unit (2 x 2 x 2 bins) that starts a run of
// that unit in its brick (plus one; 0, as cleared with the accumulators, for the others) and
// the number of points whose unit comes before their predecessor's; the sorted copy if the
// batch needs one and has room for it; the tiles.
__global__ void __launch_bounds__(kSortNT)
k_sort_tiles(Bricks br, TrainWs ws, Model md, const float* __restrict__ xyz, const float* __restrict__ target,
             int capn, int capw, int lcap, int tp, int run) {
  cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  const SortedBatch& s = ws.sorted;
  uint32_t back = 0;
  with_predecessors(br, xyz, [&](int64_t gi, uint32_t c, uint32_t before, int b, bool head) {
    const uint32_t u = c >> 3, v = before >> 3;
    if (head || v != u) ws.ustart[(int64_t)b * (kUnits + 1) + u] = (int32_t)(gi - br.off[b]) + 1;
    back += !head && v > u;
  });
  back = __reduce_add_sync(0xffffffffu, back);
  if ((threadIdx.x & 31) == 0 && back) atomicAdd(s.moved, back);
  grid.sync();
  const bool none = *(volatile uint32_t*)s.moved > s.limit;   // in no order
  if (none && s.xyz) {
    sort_clear(br, s);
    grid.sync();
    sort_count(br, xyz, s);
    grid.sync();
    for (int b = blockIdx.x; b < br.n; b += gridDim.x) {
      scan_bins(s.hist + (int64_t)b * kSortBins);
      __syncthreads();
    }
    grid.sync();
    sort_scatter(br, xyz, target, s);
  }
  for (int b = blockIdx.x; b < br.n; b += gridDim.x) {
    __syncthreads();
    if (none && !s.xyz) run_list(br, b, ws, run);
    else tile_list(br, b, ws, md, none ? capw : capn, lcap, tp);
  }
}

// CTAs of a cooperative launch over n points: at most one per SM, so that all are resident,
// as the grid's barriers need.
int sort_blocks(int64_t n, const Launch& L) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + kSortNT - 1) / kSortNT, L.num_sms));
}

}  // namespace

cudaError_t launch_sort_query(const Launch& L, const Bricks& br, const float* xyz, const SortedBatch& s) {
  if (br.off[br.n] == 0) return cudaSuccess;
  void* args[] = {(void*)&br, (void*)&xyz, (void*)&s};
  return cudaLaunchCooperativeKernel((const void*)k_sort_query, dim3(sort_blocks(br.off[br.n], L)), dim3(kSortNT), args,
                                     0, L.stream);
}

cudaError_t launch_tiles(const Launch& L, const Model& md, const Bricks& br, const TrainWs& ws, const float* xyz,
                         const float* target, int capn, int capw, int lcap, int tp, int run) {
  if (ws.bin_start) {
    k_tile_list<<<br.n, kSortNT, 0, L.stream>>>(br, ws, md, capn, lcap, tp);
    return cudaGetLastError();
  }
  void* args[] = {(void*)&br,   (void*)&ws,   (void*)&md,   (void*)&xyz, (void*)&target,
                  (void*)&capn, (void*)&capw, (void*)&lcap, (void*)&tp,  (void*)&run};
  return cudaLaunchCooperativeKernel((const void*)k_sort_tiles, dim3(sort_blocks(br.off[br.n], L)), dim3(kSortNT), args,
                                     0, L.stream);
}

}  // namespace srn
