// Shared memory of the forward query (k_fwd.cuh): its layout, and the node boxes of the grids.
#pragma once
#include "enc_ops.cuh"
#include "render.h"

namespace srn {

// CTAs per SM and samples per thread.  With staged boxes a thread's samples share the reads of
// a grid's map and box (a warp-uniform 16-byte read takes two passes of the shared-memory
// pipe, 65% busy at two samples per thread), which for K >= 64 pays for 128 registers and
// the two CTAs that the feature tile and the boxes leave room for (frame of the paper-scale
// model: 157 ms at two samples, 153 at four); the small models take three CTAs of one sample
// per thread instead (progressive pass at K = 32: 318 and 292 us).  Without boxes what is left
// of shared memory is L1, the corners' latency asks for warps, and three CTAs of one sample
// per thread, of two at K = 128, are best (BF16 queries at two CTAs of four samples, three of
// two, three of one: K = 128, 500000 points in order 198, 189 and 197 us; K = 64, 60000 points
// in no order 46.5, 40.7 and 40.5).  Points far apart in K = 128's grids, whose corners come from
// far, want four samples' reads in flight instead (`far`: point_source).  Float32 has the
// registers for two (K = 128, 20000 points in no order: 63.5 us at two samples per thread, 57.0
// at one).
constexpr int fwd_ctas(int K, bool F32, bool four) { return F32 || (four && K >= 64) ? 2 : 3; }

// One grid's staged box as the encoder sees it.  With t the cell's float bits of
// axis_cell (cell + kMagicBits) per axis, the byte address of the cell's first corner is
// at + tz oz + ty oy + tx (node bytes), all modulo 2^32.
struct __align__(16) FwdBox {
  uint32_t at, oy, oz, pad;
};
// What staging needs: lo | nodes per axis as in block_box, and the pool offset in nodes.
struct FwdStage {
  uint32_t lo, n, at;
};

template <int K, int C, bool F32, bool BOXES>
struct FwdLay {
  static constexpr int M = K / C;
  static constexpr int T = F32 ? 64 : 128;           // samples per feature tile
  static constexpr int GROUP = fwd_group(F32, BOXES);   // samples per group, at most
  static constexpr int YP = K + 4, HP = 64 + 4;      // row pitches of the float32 tiles (floats)
  static constexpr int W1 = 0;                       // [64][K] bf16 swizzled, or [64][YP] f32
  static constexpr int W2 = W1 + (F32 ? 64 * YP * 4 : 64 * K * 2);   // [64][64] bf16, or [64][HP] f32
  static constexpr int Y = W2 + (F32 ? 64 * HP * 4 : 64 * 64 * 2);   // [T][K] bf16, or [T][YP] f32 and over it,
  static constexpr int YB = F32 ? T * (YP > HP ? YP : HP) * 4 : T * K * 2;   // once read, the hidden layer [T][HP]
  static constexpr int X = Y + YB;                   // [GROUP] float4: x, y, z, bits of brick | slot << 8 (-1: no sample)
  static constexpr int W3 = X + GROUP * 16;          // [64] f32
  static constexpr int P = W3 + 64 * 4;              // [4][T] f32 partial outputs (float32)
  static constexpr int G = P + (F32 ? 4 * T * 4 : 0);   // [M][12] f32: column pairs of the x and y rows, then the z row
  static constexpr int BOX = G + M * 48;             // [M] FwdBox
  static constexpr int STG = BOX + M * 16;           // [M] FwdStage
  static constexpr int POOL = (STG + M * 12 + 15) / 16 * 16;   // staged nodes, C float32 each
  // (without boxes the layout ends at BOX)
};

// The box of the nodes blo | bn (as sample_box gives them) whose staged nodes start at byte
// `base` of shared memory.  A sample outside the grid reads, and drops, a cell at the start of
// the pool with these strides: less than the box's size on, and for a grid without staged
// nodes (bn = 0) the pool's first two nodes.
template <int C>
__host__ __device__ inline FwdBox fwd_box(uint32_t blo, uint32_t bn, uint32_t base) {
  constexpr uint32_t nb = 4 * C, mb = (uint32_t)kMagicBits;
  FwdBox q;
  q.oy = (bn & 0xffu) * nb;
  q.oz = (bn & 0xffu) * (bn >> 8 & 0xffu) * nb;
  q.at = base - ((blo >> 16 & 0xffu) + mb) * q.oz - ((blo >> 8 & 0xffu) + mb) * q.oy - ((blo & 0xffu) + mb) * nb;
  q.pad = 0u;
  return q;
}

// Node box of grid g over the block [lo, hi]: block_box with a margin that covers the
// rounding of the per-sample map for any transform, so that every sample of the block
// inside the grid has its cell in the box (no per-sample test is needed).  False, and no
// nodes (also on the axes that the block does reach), if it misses the grid.
// gp: the grid's map as load order keeps it, the column pairs of its x and y rows, then
// its z row.
__host__ __device__ inline bool sample_box(const float (&lo)[3], const float (&hi)[3], const float* gp, int R,
                                           uint32_t& blo, uint32_t& bn) {
  const float h = 0.5f * (float)(R - 1), top = (float)(R - 1);
  uint32_t first = 0, count = 0;
  blo = bn = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    auto g = [&](int k) { return d < 2 ? gp[2 * k + d] : gp[8 + k]; };
    float umin = g(3), umax = umin, mag = fabsf(umin);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float a = g(k), p = a * lo[k], q = a * hi[k];
      umin += fminf(p, q);
      umax += fmaxf(p, q);
      mag += fmaxf(fabsf(p), fabsf(q));
    }
    // per sample and here: at most 5 roundings of sums of at most mag, each 2^-24 of them
    const float pu = mag * 1e-6f, ps = fmaf(h, pu, 1e-3f);
    if (umax + pu < -1.f || umin - pu > 1.f) return false;
    const float a = fmaf(umin, h, h) - ps, b = fmaf(umax, h, h) + ps;
    const float s0 = a >= 0.f ? fminf(a, top) : 0.f;     // (a NaN bound takes the whole axis)
    const float s1 = b <= top ? fmaxf(b, 0.f) : top;
    const int c0 = min((int)s0, R - 2), c1 = min((int)s1, R - 2);
    first |= (uint32_t)c0 << (8 * d);
    count |= (uint32_t)(c1 - c0 + 2) << (8 * d);
  }
  blo = first;
  bn = count;
  return true;
}

// The dynamic shared memory of a CTA with boxes: its share of the SM's (1 KB of it reserved), less the static part.
inline int fwd_smem(int smem_sm, int K, bool F32) {
  constexpr int kStatic = 1536;
  return (smem_sm / fwd_ctas(K, F32, true) - 1024 - kStatic) / 128 * 128;
}

}  // namespace srn
