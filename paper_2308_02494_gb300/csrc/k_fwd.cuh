// Forward query f(x) = d(e(x)) (Eq. 1-3 and Sec. 4.1.2), BF16 or float32, for srn_forward, the
// renderer and the full-volume decode.  Included by one translation unit per feature count
// and precision, which sets kK and kF32 first.
//
// A CTA takes groups of up to 512 neighbouring samples: consecutive points of a brick, a
// bundle of ray samples, or a block of voxels, whose coordinates it forms itself, so the
// renderer and the decode keep no coordinates in memory.  Dense views (boxes_pay) stage nodes
// in shared memory: per group and brick the samples' bounding box, mapped through each grid's
// Eq. 1, bounds the nodes that the grid can read, and boxes that are worth it and fit are
// kept as the float32 values of their nodes.  All others read the corners from global memory.
// Then 128 samples (float32: 64) at a time: a thread evaluates Eq. 1-2 for one to four samples
// and the grids of eight features (float32 at K = 16: four) before it stores them.  BF16: warp w
// runs the two hidden layers for rows 16w..16w+15 on the tensor cores (m16n8k16, FP32
// accumulate) and the 64 -> 1 output layer in FP32; float32: packed FMAs, 32 rows x 16 columns
// a warp.
//
// What bounds it: with boxes, instruction issue and the shared-memory pipe (55% and 65% busy
// in a decode); without, the L1 pipe (82% in a query of 1.0 M sorted points, IPC 2.3).  Reading
// the corners from global memory takes 103 warp instructions per 32 (sample, grid) pairs, of
// which unpacking the BF16 nodes and eight addresses; staged float32 nodes need no unpacking
// and one address for eight reads: 88.  A sample outside a grid reads nothing, by predicated loads: reading, and
// dropping, some cell took 110.9 us where it takes 102.0 (200003 points in no order, K = 64).
// Boxes of points in memory did not pay at any density: 1500000 points in order of the
// paper-scale model took 568 us with them and 470 without, 60000 59 and 46.
// The blend is rounded as the global read's was, so the features are the same bits.
#include <algorithm>

#include "fwd_box.cuh"
#include "kernels.h"

namespace srn {
namespace {

constexpr int NT = 256;

// One grid node in global memory: C bf16 or C float32 values.
template <int C, bool F32>
using FwdNode = std::conditional_t<F32, EncSNode<C>, EncNode<C>>;
template <int C, bool F32>
__device__ __forceinline__ EncSNode<C> widen(FwdNode<C, F32> v) {   // as C float32
  if constexpr (F32) return v;
  else if constexpr (C == 2) return bf2_bits(v);
  else return __uint_as_float((uint32_t)v << 16);
}

// The node at a, or 0.
__device__ __forceinline__ uint16_t load_if(bool p, const uint16_t* a) {
  uint16_t v;
  asm("{.reg .pred q;\n setp.ne.s32 q, %2, 0;\n mov.b16 %0, 0;\n @q ld.global.nc.u16 %0, [%1];}" : "=h"(v) : "l"(a), "r"((int)p));
  return v;
}
__device__ __forceinline__ uint32_t load_if(bool p, const uint32_t* a) {
  uint32_t v;
  asm("{.reg .pred q;\n setp.ne.s32 q, %2, 0;\n mov.b32 %0, 0;\n @q ld.global.nc.u32 %0, [%1];}" : "=r"(v) : "l"(a), "r"((int)p));
  return v;
}
__device__ __forceinline__ float load_if(bool p, const float* a) {
  float v;
  asm("{.reg .pred q;\n setp.ne.s32 q, %2, 0;\n mov.b32 %0, 0;\n @q ld.global.nc.f32 %0, [%1];}" : "=f"(v) : "l"(a), "r"((int)p));
  return v;
}
__device__ __forceinline__ unsigned long long load_if(bool p, const unsigned long long* a) {
  unsigned long long v;
  asm("{.reg .pred q;\n setp.ne.s32 q, %2, 0;\n mov.b64 %0, 0;\n @q ld.global.nc.u64 %0, [%1];}" : "=l"(v) : "l"(a), "r"((int)p));
  return v;
}

// Float order as unsigned integer order (for min/max reductions).
__device__ __forceinline__ uint32_t ord(float v) {
  const uint32_t b = __float_as_uint(v);
  return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
}
__device__ __forceinline__ float unord(uint32_t o) {
  return __uint_as_float(o ^ ((o & 0x80000000u) ? 0x80000000u : 0xffffffffu));
}

// VIEW: ray samples or voxels, else points in memory.  BOXES: with staged boxes.  FAR: points far
// apart.
template <int K, int C, bool EVEN, bool F32, bool VIEW, bool BOXES, bool FAR>
__global__ void __launch_bounds__(NT, fwd_ctas(K, F32, BOXES || FAR))
k_fwd(Model md, Bricks brp, std::conditional_t<VIEW, FwdSource, FwdPointSource> src, float* __restrict__ out,
      uint32_t pool_nodes) {
  using L = FwdLay<K, C, F32, BOXES>;
  using Node = FwdNode<C, F32>;
  constexpr int M = K / C, T = L::T;
  constexpr int CW = F32 && K == 16 ? 4 : 8;   // features per chunk
  constexpr int GPC = CW / C;                // grids per chunk
  constexpr int NCH = K / CW;                // chunks of a feature row
  constexpr int PP = K < 64 || (!BOXES && (F32 || K < 128)) ? 1 : F32 || !(BOXES || FAR) ? 2 : 4;   // samples per thread
  constexpr int NQ = 8 / (T / (32 * PP));    // warps sharing the same samples, each its own chunks
  constexpr uint32_t kNB = 4 * C;            // bytes of a staged node
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ TileMap tm;
  __shared__ Bricks br;
  __shared__ uint32_t s_lo[3], s_hi[3], s_mask[2], s_np;
  __shared__ float s_range[2];            // the brick's minimum and span
  __shared__ int s_run[2];                // the next run of groups
  __shared__ FwdBlock blk;                // the group's voxels (kFwdDecode)
  __shared__ uint16_t s_cnt[L::GROUP / 32];   // a mixed group's samples of a brick in each 32 slots,
  __shared__ uint16_t s_first[SRN_MAX_BRICKS], s_end;   // where its bricks' samples start, and the last one's end
  __shared__ uint32_t s_slow[kMaxGrids / 32];   // bit i: grid i's corners come from global memory
  load_bricks(brp, br);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g8 = lane >> 2, t4 = lane & 3;
  const int R = md.R;
  const int GS = src.group;
  if constexpr (!VIEW) {
    if (tid == 0) build_tile_map_log2(br, __ffs(GS) - 1, tm);   // (a power of two: 64-bit divisions took 0.1 us a brick)
    __syncthreads();
  }
  const int total = VIEW ? src.groups : tm.first[br.n];
  const bool render = VIEW && src.kind == kFwdRender;
  const bool copied = !VIEW && src.sorted.use();
  const float* xyz = copied ? src.sorted.xyz : src.xyz;
  float4* xs = reinterpret_cast<float4*>(sm + L::X);
  float* w3s = reinterpret_cast<float*>(sm + L::W3);
  float* gs = reinterpret_cast<float*>(sm + L::G);
  FwdBox* boxes = reinterpret_cast<FwdBox*>(sm + L::BOX);
  FwdStage* stg = reinterpret_cast<FwdStage*>(sm + L::STG);
  const uint32_t sW1 = su32(sm + L::W1), sW2 = su32(sm + L::W2), sY = su32(sm + L::Y);
  const uint32_t spool = su32(sm + L::POOL);
  const int64_t gsz = (int64_t)R * R * R;   // nodes of a grid
  const float hs = 0.5f * (float)(R - 1);
  const float ct = hs - 0.5f + kMagic;   // an integer when R is even (axis_cell)

  int cur = -1, hint = -1;
  // Runs of src.run consecutive groups (they share a brick and its weights): one for every CTA,
  // and then in turn, or, of rays in many rounds, as CTAs are done (src.next; the next run is
  // taken one ahead).  Dealt in turn, the rows of a view's groups could divide the CTAs evenly,
  // and some had the volume's middle in every round and others its empty sides (a progressive
  // pass with a third of its rays on the volume: 473 us, and 293 taken as they come).
  for (int r = blockIdx.x, k = 0; r * src.run < total; ++k) {
  int after = 0;
  if (VIEW && src.next && tid == 0) after = (int)gridDim.x + atomicAdd(src.next, 1);
  const int r0 = r * src.run, r1 = min(total, r0 + src.run);
  for (int grp = r0; grp < r1; ++grp) {
    // ---- the group's samples: coordinates and brick (-1: no sample)
    if (tid < 2) s_mask[tid] = 0u;
    if constexpr (VIEW)
      if (tid == 2 && !render) blk = decode_block(src.dec, grp);
    __syncthreads();   // also: the previous group is done with xs, the boxes and Y
    // slots of the group that can hold samples, and the first one's point or slot (formed again
    // where it is needed: a 64-bit value kept through the tiles costs registers they lack)
    int ns = GS;
    if (!VIEW) {
      hint = brick_of_tile(tm, br.n, grp, hint);
      ns = (int)min((int64_t)GS, br.off[hint + 1] - br.off[hint] - (int64_t)(grp - tm.first[hint]) * GS);
    } else if (!render) {
      ns = blk.n[0] * blk.n[1] * blk.n[2];
    }
    auto base = [&]() {
      return VIEW ? (int64_t)grp * GS : br.off[hint] + (int64_t)(grp - tm.first[hint]) * GS;
    };
    {
      Ray ray;
      int last = -1;
      uint32_t m0 = 0u, m1 = 0u;
      for (int s = tid; s < GS; s += NT) {
        float4 v = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
        if (s < ns) {
          int b;
          if constexpr (!VIEW) {
            const float* q = xyz + 3 * (base() + s);
            v.x = q[0]; v.y = q[1]; v.z = q[2];
            b = hint;
          } else if (render) {
            const RaySlot rs = ray_slot(src.rp, grp * GS + s);
            if (rs.ray != last) {   // slots NT apart share the ray when rg divides NT
              last = rs.ray;
              ray.hit = false;
              if (rs.ray < src.npix) ray = make_ray(src.rp, pixel_of(src.rp, src.pix0 + rs.ray));
            }
            b = ray.hit && rs.j < src.rp.samples ? ray_sample(src.rp, ray, rs.j, v.x, v.y, v.z) : -1;
          } else {
            b = blk.brick;
            decode_point(src, blk, s, v.x, v.y, v.z);
          }
          v.w = __int_as_float(b < 0 ? -1 : b | s << 8);
          if (render && b >= 0) {
            if (b < 32) m0 |= 1u << b; else m1 |= 1u << (b - 32);
          }
        }
        xs[s] = v;
      }
      if (render) {
        m0 = __reduce_or_sync(0xffffffffu, m0);
        m1 = __reduce_or_sync(0xffffffffu, m1);
        if (lane == 0) {
          if (m0) atomicOr(&s_mask[0], m0);
          if (m1) atomicOr(&s_mask[1], m1);
        }
      }
    }
    unsigned long long mask = render || ns <= 0 ? 0ull : 1ull << (VIEW ? blk.brick : hint);
    // (a decode's block that is empty, at the end of a shorter brick, comes to no other barrier
    // before `blk` is written again)
    if constexpr (VIEW) {
      if (tid == 0) s_run[k & 1] = after;   // (here, so that the samples hide the counter's latency)
      __syncthreads();
    }
    if (render) mask = (unsigned long long)s_mask[0] | ((unsigned long long)s_mask[1] << 32);
    const bool mixed = VIEW && (mask & (mask - 1)) != 0;
    if (mixed) {   // the bricks' samples one brick after the other, in order within each
      constexpr int SPT = L::GROUP / NT;
      float4 v[SPT];
      int at[SPT], first = 0;
#pragma unroll
      for (int k = 0; k < SPT; ++k) {
        at[k] = -1;
        if (tid + k * NT < GS) v[k] = xs[tid + k * NT];
      }
      for (unsigned long long m = mask; m; m &= m - 1) {
        const int b = __ffsll((long long)m) - 1;
        __syncthreads();
        uint32_t bal[SPT];
#pragma unroll
        for (int k = 0; k < SPT; ++k) {
          const int s = tid + k * NT;
          if (s >= GS) continue;   // (whole warps: GS is a multiple of 32)
          const int w = __float_as_int(v[k].w);
          bal[k] = __ballot_sync(0xffffffffu, w >= 0 && (w & 0xff) == b);
          if (lane == 0) s_cnt[s / 32] = (uint16_t)__popc(bal[k]);
        }
        if (tid == 0) s_first[b] = (uint16_t)first;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < SPT; ++k) {
          const int s = tid + k * NT;
          if (s >= GS || !(bal[k] >> lane & 1u)) continue;
          at[k] = first + __popc(bal[k] & ((1u << lane) - 1u));
          for (int q = 0; q < s / 32; ++q) at[k] += s_cnt[q];
        }
        for (int q = 0; q < GS / 32; ++q) first += s_cnt[q];
      }
#pragma unroll
      for (int k = 0; k < SPT; ++k)
        if (at[k] >= 0) xs[at[k]] = v[k];
      // (the other slots keep what they held: the bricks' ranges bound what is read)
      if (tid == 0) s_end = (uint16_t)first;
      __syncthreads();
    }
    while (mask) {   // the bricks of the group (more than one only where rays cross a brick face)
      const int b = __ffsll((long long)mask) - 1;
      mask &= mask - 1;
      // its samples: slots [i0, i1)
      const int i0 = mixed ? s_first[b] : 0;
      const int i1 = !mixed ? ns : mask ? s_first[__ffsll((long long)mask) - 1] : s_end;
      if (tid < 3) { s_lo[tid] = 0xffffffffu; s_hi[tid] = 0u; }
      if (tid == 3) s_np = 0u;
      // (a mixed group's few samples of a brick are not worth the boxes' three barriers)
      const bool stage = BOXES && (!mixed || i1 - i0 > T);
      if (!stage && tid < kMaxGrids / 32) s_slow[tid] = 0xffffffffu;
      if (b != cur) {
        cur = b;
        const void* w1p = F32 ? (const void*)(md.W1f + (int64_t)b * md.sW1) : (const void*)(md.W1h + (int64_t)b * md.sW1);
        const void* w2p = F32 ? (const void*)(md.W2f + (int64_t)b * md.sW2) : (const void*)(md.W2h + (int64_t)b * md.sW2);
        const uint4* w1 = static_cast<const uint4*>(w1p);
        const uint4* w2 = static_cast<const uint4*>(w2p);
        if constexpr (F32) {
          for (int c = tid; c < 64 * K / 4; c += NT)
            *reinterpret_cast<uint4*>(sm + L::W1 + ((c / (K / 4)) * L::YP + (c % (K / 4)) * 4) * 4) = w1[c];
          for (int c = tid; c < 64 * 16; c += NT)
            *reinterpret_cast<uint4*>(sm + L::W2 + ((c / 16) * L::HP + (c % 16) * 4) * 4) = w2[c];
        } else {
          for (int c = tid; c < 64 * K / 8; c += NT)
            *reinterpret_cast<uint4*>(sm + L::W1 + swz<K>(c / (K / 8), (c % (K / 8)) * 8)) = w1[c];
          for (int c = tid; c < 64 * 8; c += NT)
            *reinterpret_cast<uint4*>(sm + L::W2 + swz<64>(c / 8, (c % 8) * 8)) = w2[c];
        }
        if (tid < 64) w3s[tid] = md.w3[(int64_t)b * md.sw3 + tid];
        // each grid's map as the column pairs of its x and y rows, then its z row
        const float* G = md.G + (int64_t)b * md.sG;
        for (int c = tid; c < M * 12; c += NT) {
          const int i = c / 12, j = c - 12 * i;
          gs[c] = G[12 * i + (j < 8 ? (j >> 1) + 4 * (j & 1) : j)];
        }
        if (tid < 2) s_range[tid] = tid ? md.range[2 * b + 1] - md.range[2 * b] : md.range[2 * b];
      }
      __syncthreads();
      const Node* Fb = F32 ? reinterpret_cast<const Node*>(md.F32 + (int64_t)b * md.sF)
                           : reinterpret_cast<const Node*>(md.F16 + (int64_t)b * md.sF);
      if (stage) {
        {  // bounding box of the brick's samples (non-finite ones are inside no grid)
          uint32_t lo[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, hi[3] = {0u, 0u, 0u};
          int n = 0;
          for (int s = i0 + tid; s < i1; s += NT) {
            const float4 v = xs[s];
            if (__float_as_int(v.w) >= 0 && v.x - v.x == 0.f && v.y - v.y == 0.f && v.z - v.z == 0.f) {
              ++n;
              lo[0] = min(lo[0], ord(v.x)); hi[0] = max(hi[0], ord(v.x));
              lo[1] = min(lo[1], ord(v.y)); hi[1] = max(hi[1], ord(v.y));
              lo[2] = min(lo[2], ord(v.z)); hi[2] = max(hi[2], ord(v.z));
            }
          }
          n = __reduce_add_sync(0xffffffffu, n);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            lo[d] = __reduce_min_sync(0xffffffffu, lo[d]);
            hi[d] = __reduce_max_sync(0xffffffffu, hi[d]);
          }
          if (lane == 0 && n) {
            atomicAdd(&s_np, (uint32_t)n);
#pragma unroll
            for (int d = 0; d < 3; ++d) { atomicMin(&s_lo[d], lo[d]); atomicMax(&s_hi[d], hi[d]); }
          }
        }
        __syncthreads();
        if (warp == 0) {   // the grids' boxes, packed into the pool in grid order
          const uint32_t np = s_np;
          const float lo[3] = {unord(s_lo[0]), unord(s_lo[1]), unord(s_lo[2])};
          const float hi[3] = {unord(s_hi[0]), unord(s_hi[1]), unord(s_hi[2])};
          uint32_t used = 0u;
          for (int i0 = 0; i0 < M; i0 += 32) {
            const int i = i0 + lane;
            uint32_t blo = 0u, bn = 0u, nodes = 0u;
            bool any = false;
            if (i < M && np) any = sample_box(lo, hi, gs + 12 * i, R, blo, bn);
            const uint32_t nx = bn & 0xffu, ny = (bn >> 8) & 0xffu, nz = (bn >> 16) & 0xffu;
            // staging a node costs about half of what it saves on one sample
            if (any && nx * ny * nz <= np) nodes = nx * ny * nz;
            uint32_t incl = nodes;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
              if (lane >= o) incl += y;
            }
            const uint32_t at = used + incl - nodes;
            const bool fits = nodes && at + nodes <= pool_nodes;
            if (i < M) {
              boxes[i] = fwd_box<C>(blo, fits ? bn : 0u, spool + at * kNB);
              stg[i] = FwdStage{blo, fits ? bn : 0u, at};
            }
            const uint32_t slow = __ballot_sync(0xffffffffu, any && !fits);
            if (lane == 0) s_slow[i0 / 32] = slow;
            used += __shfl_sync(0xffffffffu, incl, 31);
          }
        }
        __syncthreads();
        // ---- staging: a warp per grid, a lane per node
        for (int i = warp; i < M; i += NT / 32) {
          const FwdStage q = stg[i];
          if (!q.n) continue;
          const uint32_t nx = q.n & 0xffu, ny = (q.n >> 8) & 0xffu, nxy = nx * ny, n = nxy * (q.n >> 16 & 0xffu);
          const float ixy = 1.f / (float)nxy, ix = 1.f / (float)nx;
          const Node* Fg = Fb + i * gsz + (((q.lo >> 16 & 0xffu) * R + (q.lo >> 8 & 0xffu)) * R + (q.lo & 0xffu));
          EncSNode<C>* dst = reinterpret_cast<EncSNode<C>*>(sm + L::POOL) + q.at;
#pragma unroll 2
          for (uint32_t k = lane; k < n; k += 32) {   // n <= 512: the float quotients are exact
            const uint32_t z = (uint32_t)(((float)k + 0.5f) * ixy), r = k - z * nxy;
            const uint32_t y = (uint32_t)(((float)r + 0.5f) * ix), x = r - y * nx;
            dst[k] = widen<C, F32>(__ldg(Fg + ((z * R + y) * R + x)));
          }
        }
        __syncthreads();
      }
      for (int t0 = i0; t0 < i1; t0 += T) {
        {  // ---- encode
          const int pr = (warp / NQ) * 32 * PP + lane;   // this thread's rows: pr, pr + 32, ...
          f2_t xx[PP], yy[PP], zz[PP];
          bool valid[PP];
#pragma unroll
          for (int p = 0; p < PP; ++p) {
            const int s = t0 + pr + 32 * p;
            const float4 v = xs[min(s, GS - 1)];
            xx[p] = f2_pack(v.x, v.x); yy[p] = f2_pack(v.y, v.y); zz[p] = f2_pack(v.z, v.z);
            valid[p] = s < i1 && __float_as_int(v.w) >= 0;
          }
          // Eq. 1 and the cell of Eq. 2 of sample p in grid i
          struct Place {
            uint32_t tx, ty, tz;
            float wx, wy, wz;
            bool in;
          };
          auto place = [&](int i, Place (&c)[PP]) {
            const ulonglong2 ab = *reinterpret_cast<const ulonglong2*>(gs + 12 * i);
            const ulonglong2 cd = *reinterpret_cast<const ulonglong2*>(gs + 12 * i + 4);
            const float4 gz = *reinterpret_cast<const float4*>(gs + 12 * i + 8);
#pragma unroll
            for (int p = 0; p < PP; ++p) {
              const f2_t uxy = f2_fma(ab.x, xx[p], f2_fma(ab.y, yy[p], f2_fma(cd.x, zz[p], cd.y)));
              const float uz = fmaf(gz.x, f2_lo(xx[p]), fmaf(gz.y, f2_lo(yy[p]), fmaf(gz.z, f2_lo(zz[p]), gz.w)));
              c[p].in = valid[p] & (fabsf(f2_lo(uxy)) <= 1.f) & (fabsf(f2_hi(uxy)) <= 1.f) & (fabsf(uz) <= 1.f);
              if constexpr (EVEN) {
                int32_t tx, ty;
                axis_cell2(uxy, f2_pack(hs, hs), f2_pack(ct, ct), f2_pack(kMagic, kMagic), tx, ty, c[p].wx, c[p].wy);
                c[p].tx = (uint32_t)tx;
                c[p].ty = (uint32_t)ty;
                c[p].tz = (uint32_t)axis_cell(uz, hs, ct, c[p].wz);
              } else {   // (s - 1/2) + kMagic: the cell floor(s) or, on a node, an even neighbour; at most R - 2
                const float top = kMagic + (float)(R - 2);
                auto axis = [&](float u, uint32_t& t, float& w) {
                  const float sv = fmaf(u, hs, hs), cv = fminf(__fadd_rn(sv - 0.5f, kMagic), top);
                  w = sv - (cv - kMagic);
                  t = __float_as_uint(cv);
                };
                axis(f2_lo(uxy), c[p].tx, c[p].wx);
                axis(f2_hi(uxy), c[p].ty, c[p].wy);
                axis(uz, c[p].tz, c[p].wz);
              }
            }
          };
          // Eq. 2's blend of the eight corners (x fastest)
          auto blend = [&](const EncSNode<C> (&v)[8], const Place& c) -> EncSNode<C> {
            const float vx = 1.f - c.wx, vy = 1.f - c.wy, vz = 1.f - c.wz;
            if constexpr (C == 2) {
              const f2_t px = f2_pack(c.wx, c.wx), qx = f2_pack(vx, vx), py = f2_pack(c.wy, c.wy), qy = f2_pack(vy, vy);
              const f2_t e0 = blend2(v[0], v[1], px, qx), e1 = blend2(v[2], v[3], px, qx);
              const f2_t e2 = blend2(v[4], v[5], px, qx), e3 = blend2(v[6], v[7], px, qx);
              return blend2(blend2(e0, e1, py, qy), blend2(e2, e3, py, qy), f2_pack(c.wz, c.wz), f2_pack(vz, vz));
            } else {
              const float e0 = blend1(v[0], v[1], c.wx, vx), e1 = blend1(v[2], v[3], c.wx, vx);
              const float e2 = blend1(v[4], v[5], c.wx, vx), e3 = blend1(v[6], v[7], c.wx, vx);
              return blend1(blend1(e0, e1, c.wy, vy), blend1(e2, e3, c.wy, vy), c.wz, vz);
            }
          };
          // from a staged box (a sample outside the grid reads, and drops, nodes at the pool's
          // start, see fwd_box)
          auto from_box = [&](const FwdBox& q, const Place& c) -> EncSNode<C> {
            const uint32_t a = q.at + c.tz * q.oz + c.ty * q.oy + c.tx * kNB, a0 = c.in ? a : spool;
            const uint32_t a1 = a0 + q.oy, a2 = a0 + q.oz, a3 = a2 + q.oy;
            const EncSNode<C> v[8] = {enc_node<C, 0>(a0), enc_node<C, kNB>(a0), enc_node<C, 0>(a1), enc_node<C, kNB>(a1),
                                      enc_node<C, 0>(a2), enc_node<C, kNB>(a2), enc_node<C, 0>(a3), enc_node<C, kNB>(a3)};
            const EncSNode<C> f = blend(v, c);
            return c.in ? f : EncSNode<C>(0);
          };
          auto from_grid = [&](int i, const Place& c) -> EncSNode<C> {
            // (predicated loads and no branch, so that the reads of several samples and grids are
            // in flight together; a sample outside the grid reads nothing)
            constexpr uint32_t mb = (uint32_t)kMagicBits;
            const Node* F0 = Fb + i * gsz + ((c.tz - mb) * R + (c.ty - mb)) * R + (c.tx - mb);
            const Node* F2 = F0 + (uint32_t)(R * R);
            const Node n[8] = {load_if(c.in, F0), load_if(c.in, F0 + 1), load_if(c.in, F0 + R), load_if(c.in, F0 + R + 1),
                               load_if(c.in, F2), load_if(c.in, F2 + 1), load_if(c.in, F2 + R), load_if(c.in, F2 + R + 1)};
            EncSNode<C> v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = widen<C, F32>(n[k]);
            const EncSNode<C> f = blend(v, c);
            return c.in ? f : EncSNode<C>(0);
          };
          // the features of the chunk's grid j: packed pairs of bf16, or float32
          uint32_t o[PP][F32 ? CW : CW / 2];
          auto put = [&](int p, int j, EncSNode<C> f) {
            if constexpr (F32 && C == 2) {
              o[p][2 * j] = (uint32_t)f;
              o[p][2 * j + 1] = (uint32_t)(f >> 32);
            } else if constexpr (F32) {
              o[p][j] = __float_as_uint(f);
            } else if constexpr (C == 2) {
              o[p][j] = pack_bf16(f2_lo(f), f2_hi(f));
            } else {
              const uint32_t h = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(f));
              o[p][j / 2] = j % 2 ? o[p][j / 2] | h << 16 : h;
            }
          };
#pragma unroll 1
          for (int ch = warp % NQ; ch < NCH; ch += NQ) {
            const uint32_t unstaged = !BOXES ? (1u << GPC) - 1u : (s_slow[ch * GPC / 32] >> (ch * GPC % 32)) & ((1u << GPC) - 1u);
            if (unstaged == 0u) {   // straight-line code over the chunk's grids
#pragma unroll
              for (int j = 0; j < GPC; ++j) {
                Place c[PP];
                place(ch * GPC + j, c);
                const FwdBox q = boxes[ch * GPC + j];
#pragma unroll
                for (int p = 0; p < PP; ++p) put(p, j, from_box(q, c[p]));
              }
            } else if (PP == 1 && unstaged == (1u << GPC) - 1u) {
#pragma unroll
              for (int j = 0; j < GPC; ++j) {
                Place c[PP];
                place(ch * GPC + j, c);
#pragma unroll
                for (int p = 0; p < PP; ++p) put(p, j, from_grid(ch * GPC + j, c[p]));
              }
            } else {
#pragma unroll
              for (int j = 0; j < GPC; ++j) {
                Place c[PP];
                place(ch * GPC + j, c);
                EncSNode<C> f[PP];
                if (unstaged >> j & 1u) {
#pragma unroll
                  for (int p = 0; p < PP; ++p) f[p] = from_grid(ch * GPC + j, c[p]);
                } else {
                  const FwdBox q = boxes[ch * GPC + j];
#pragma unroll
                  for (int p = 0; p < PP; ++p) f[p] = from_box(q, c[p]);
                }
#pragma unroll
                for (int p = 0; p < PP; ++p) put(p, j, f[p]);
              }
            }
#pragma unroll
            for (int p = 0; p < PP; ++p) {
              if constexpr (F32) {
                uint4* y = reinterpret_cast<uint4*>(sm + L::Y + ((pr + 32 * p) * L::YP + CW * ch) * 4);
#pragma unroll
                for (int q = 0; q < CW / 4; ++q) y[q] = make_uint4(o[p][4 * q], o[p][4 * q + 1], o[p][4 * q + 2], o[p][4 * q + 3]);
              } else {
                unsigned char* y = sm + L::Y + swz<K>(pr + 32 * p, CW * ch);
                if constexpr (CW == 8) *reinterpret_cast<uint4*>(y) = make_uint4(o[p][0], o[p][1], o[p][2], o[p][3]);
                else *reinterpret_cast<uint2*>(y) = make_uint2(o[p][0], o[p][1]);
              }
            }
          }
        }
        __syncthreads();
        auto write = [&](int r, float f) {   // the sample at r of the group, if there is one
          if (r >= i1) return;
          const int w = __float_as_int(xs[r].w), s = w >> 8;
          if (w < 0) return;
          f = fmaf(f, s_range[1], s_range[0]);
          if constexpr (VIEW) out[render ? base() + s : decode_index(src, blk, s)] = f;
          else if (!copied) out[base() + s] = f;
          else if (const int64_t at = src.sorted.index[base() + s]; at < br.off[br.n]) out[at] = f;   // (sort_scatter)
        };
        if constexpr (F32) {
          // ---- decoder in float32: warp w takes 32 rows x 16 columns of a hidden layer, lane
          // (ty, tx) rows ty + 8 r and columns tx + 4 c: eight 16-byte reads feed 64 products
          // (packed over even and odd k), each read one or two passes of the pipe
          const int ty = lane >> 2, tx = lane & 3, row0 = (warp & 1) * 32 + ty, col0 = (warp >> 1) * 16 + tx;
          auto layer = [&](const unsigned char* a, int ap, const unsigned char* w, int wp, int n, float (&z)[4][4]) {
            f2_t acc[4][4];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
              for (int c = 0; c < 4; ++c) acc[r][c] = 0ull;
#pragma unroll 2
            for (int k = 0; k < n; k += 4) {
              ulonglong2 y[4], q[4];
#pragma unroll
              for (int r = 0; r < 4; ++r) y[r] = *reinterpret_cast<const ulonglong2*>(a + ((row0 + 8 * r) * ap + k) * 4);
#pragma unroll
              for (int c = 0; c < 4; ++c) q[c] = *reinterpret_cast<const ulonglong2*>(w + ((col0 + 4 * c) * wp + k) * 4);
#pragma unroll
              for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = f2_fma(y[r].y, q[c].y, f2_fma(y[r].x, q[c].x, acc[r][c]));
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
              for (int c = 0; c < 4; ++c) z[r][c] = fmaxf(f2_lo(acc[r][c]) + f2_hi(acc[r][c]), 0.f);
          };
          float z[4][4];
          layer(sm + L::Y, L::YP, sm + L::W1, L::YP, K, z);
          __syncthreads();   // every warp has read Y: the hidden layer goes over it
          float* h1 = reinterpret_cast<float*>(sm + L::Y);
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) h1[(row0 + 8 * r) * L::HP + col0 + 4 * c] = z[r][c];
          __syncthreads();
          layer(sm + L::Y, L::HP, sm + L::W2, L::HP, 64, z);
          float* part = reinterpret_cast<float*>(sm + L::P);
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) s = fmaf(z[r][c], w3s[col0 + 4 * c], s);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (tx == 0) part[(warp >> 1) * T + row0 + 8 * r] = s;
          }
          __syncthreads();
          if (tid < T) write(t0 + tid, (part[tid] + part[T + tid]) + (part[2 * T + tid] + part[3 * T + tid]));
        } else {  // ---- decoder on the tensor cores
          const int r0w = warp * 16;
          float acc[8][4];
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll
          for (int ks = 0; ks < K / 16; ++ks) {
            uint32_t a[4];
            ldsm4(a, sY + swz<K>(r0w + (lane & 15), ks * 16 + (lane >> 4) * 8));
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t bb[4];
              ldsm4(bb, sW1 + swz<K>(q * 16 + (lane & 7) + ((lane >> 4) << 3), ks * 16 + ((lane >> 3) & 1) * 8));
              mma(acc[2 * q], a, bb[0], bb[1]);
              mma(acc[2 * q + 1], a, bb[2], bb[3]);
            }
          }
          uint32_t h1a[4][4];
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            h1a[kk][0] = pack_bf16(fmaxf(acc[2 * kk][0], 0.f), fmaxf(acc[2 * kk][1], 0.f));
            h1a[kk][1] = pack_bf16(fmaxf(acc[2 * kk][2], 0.f), fmaxf(acc[2 * kk][3], 0.f));
            h1a[kk][2] = pack_bf16(fmaxf(acc[2 * kk + 1][0], 0.f), fmaxf(acc[2 * kk + 1][1], 0.f));
            h1a[kk][3] = pack_bf16(fmaxf(acc[2 * kk + 1][2], 0.f), fmaxf(acc[2 * kk + 1][3], 0.f));
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t bb[4];
              ldsm4(bb, sW2 + swz<64>(q * 16 + (lane & 7) + ((lane >> 4) << 3), kk * 16 + ((lane >> 3) & 1) * 8));
              mma(acc[2 * q], h1a[kk], bb[0], bb[1]);
              mma(acc[2 * q + 1], h1a[kk], bb[2], bb[3]);
            }
          }
          float mlo = 0.f, mhi = 0.f;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float w = w3s[j * 8 + 2 * t4 + e];
              mlo = fmaf(fmaxf(acc[j][e], 0.f), w, mlo);
              mhi = fmaf(fmaxf(acc[j][2 + e], 0.f), w, mhi);
            }
          }
          mlo += __shfl_xor_sync(0xffffffffu, mlo, 1);
          mlo += __shfl_xor_sync(0xffffffffu, mlo, 2);
          mhi += __shfl_xor_sync(0xffffffffu, mhi, 1);
          mhi += __shfl_xor_sync(0xffffffffu, mhi, 2);
          // lane t4 = 0 writes row g8, lane 1 row g8 + 8
          if (t4 < 2) write(t0 + r0w + g8 + 8 * t4, t4 ? mhi : mlo);
        }
        __syncthreads();
      }
    }
  }
  // (the next run's barriers come before s_run[k & 1] is written again)
  r = VIEW && src.next ? s_run[k & 1] : r + (int)gridDim.x;
  }
}

template <int K, int C, bool EVEN, bool F32, bool VIEW, bool BOXES, bool FAR = false>
cudaError_t launch_k(const Launch& L, const Model& md, const Bricks& br, const FwdSource& src, float* out) {
  using Lay = FwdLay<K, C, F32, BOXES>;
  auto kern = k_fwd<K, C, EVEN, F32, VIEW, BOXES, FAR>;
  const int smem = BOXES ? fwd_smem(L.smem_sm, K, F32) : Lay::BOX;   // (what is left is L1)
  if (BOXES && smem < Lay::POOL + 64) return cudaErrorInvalidConfiguration;   // room for dropped reads (fwd_box)
  const int pool = BOXES ? (smem - Lay::POOL) / (4 * C) : 0;
  cudaError_t e;
  if (smem > (48 << 10) &&
      (e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess)
    return e;
  int total = src.groups;
  if (!VIEW) {
    total = 0;
    for (int b = 0; b < br.n; ++b) total += (int)((br.off[b + 1] - br.off[b] + src.group - 1) / src.group);
  }
  if (total == 0) return cudaSuccess;
  FwdSource s = src;
  const int ctas = fwd_ctas(K, F32, BOXES || FAR) * L.num_sms;
  s.run = std::max(1, std::min(4, total / (8 * ctas)));
  // (taken one ahead, the last runs of a few rounds go to whichever CTAs began first, three of an
  // SM: batches of 512 groups 45 us each, dealt in turn 36)
  if (total < 8 * ctas) s.next = nullptr;
  const int grid = std::min((total + s.run - 1) / s.run, ctas);
  kern<<<grid, NT, smem, L.stream>>>(md, br, s, out, (uint32_t)pool);
  return cudaGetLastError();
}

template <int K, int C, bool EVEN>
cudaError_t launch_e(const Launch& L, const Model& md, const Bricks& br, const FwdSource& src, float* out) {
  if (src.kind == kFwdPoints) {
    if constexpr (K == 128 && !kF32)
      if (src.far) return launch_k<K, C, EVEN, kF32, false, false, true>(L, md, br, src, out);
    return launch_k<K, C, EVEN, kF32, false, false>(L, md, br, src, out);
  }
  return src.boxes ? launch_k<K, C, EVEN, kF32, true, true>(L, md, br, src, out)
                   : launch_k<K, C, EVEN, kF32, true, false>(L, md, br, src, out);
}
template <int K, int C>
cudaError_t launch_c(const Launch& L, const Model& md, const Bricks& br, const FwdSource& src, float* out) {
  return md.R % 2 ? launch_e<K, C, false>(L, md, br, src, out) : launch_e<K, C, true>(L, md, br, src, out);
}

}  // namespace

template <>
cudaError_t launch_forward_k<kK, kF32>(const Launch& L, const Model& md, const Bricks& br, const FwdSource& src,
                                       float* out) {
  return md.C == 2 ? launch_c<kK, 2>(L, md, br, src, out) : launch_c<kK, 1>(L, md, br, src, out);
}

}  // namespace srn
