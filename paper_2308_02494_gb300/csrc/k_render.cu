// Headless neural volume renderer (Sec. 6) over a domain decomposition (Sec. 5.3).
//
// Per batch of rays the forward query forms its samples itself, bundle by bundle (render.h),
// and leaves their values in slot order; then each ray reads its values in sample order and
// is composited front to back.  Sampling and opacity: midpoints t_j = t0 + (j + 1/2) dt of the ray's
// segment inside [-1,1]^3, alpha = 1 - exp(-a dt / (2/512)), the 256-entry RGBA
// transfer function read with linear interpolation.
#include <algorithm>
#include <climits>
#include <cmath>

#include "common.cuh"
#include "kernels.h"
#include "render.h"

namespace srn {
namespace {

// Position of pixel (x, y) in the progressive order (the inverse of pixel_of).
__device__ __forceinline__ int order_of(const RenderParams& rp, int x, int y) {
  if ((x | y) == 0) return 0;
  const int l = __ffs(x | y) - 1;   // the finest level holding the pixel; < L since x, y < 2^L
  const int a = x >> l, b = y >> l, wa = level_cols(rp, l), half = wa >> 1;
  return level_pixels(rp, l + 1) + (b >> 1) * (half + wa) + ((b & 1) ? half + a : a >> 1);
}

// Front-to-back compositing of 32 rays per block of 256 threads: thread (ray, segment)
// composites one eighth of the ray's samples, then the segments are joined in order (the
// compositing operator is associative).  One thread per ray left a batch of 8192 rays
// with 54 threads per SM, each a chain of 512 dependent reads.
constexpr int kSegs = 8;
__global__ void __launch_bounds__(32 * kSegs)
k_render_composite(RenderParams rp, int pix0, int npix, const float* __restrict__ val,
                   const float* __restrict__ lut, float* __restrict__ rgba, int32_t* __restrict__ next) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *next = 0;   // for the next batch's groups
  __shared__ float4 part[kSegs][32];
  const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
  const int ray = blockIdx.x * 32 + lane;
  const int pix = ray < npix ? pixel_of(rp, pix0 + ray) : 0;
  float cr = 0.f, cg = 0.f, cb = 0.f, T = 1.f;
  if (ray < npix) {
    const Ray r = make_ray(rp, pix);
    if (r.hit) {
      const float k = r.dt / (2.f / 512.f);
      const float inv_span = 1.f / (rp.vmax - rp.vmin);
      const int j0 = (int)((int64_t)rp.samples * seg / kSegs), j1 = (int)((int64_t)rp.samples * (seg + 1) / kSegs);
      const int s0 = render_slot(rp, ray, 0);
#pragma unroll 8
      for (int j = j0; j < j1; ++j) {
        const float f = val[s0 + j * rp.rg];
        const float s = fminf(fmaxf((f - rp.vmin) * inv_span, 0.f), 1.f) * 255.f;
        const int i0 = min((int)s, 254);
        const float fr = s - (float)i0;
        const float4 a = reinterpret_cast<const float4*>(lut)[i0];
        const float4 c = reinterpret_cast<const float4*>(lut)[i0 + 1];
        const float red = a.x + (c.x - a.x) * fr, grn = a.y + (c.y - a.y) * fr, blu = a.z + (c.z - a.z) * fr;
        const float op = a.w + (c.w - a.w) * fr;
        const float alpha = 1.f - expf(-op * k);
        const float w = T * alpha;
        cr = fmaf(w, red, cr); cg = fmaf(w, grn, cg); cb = fmaf(w, blu, cb);
        T *= 1.f - alpha;
      }
    }
  }
  part[seg][lane] = make_float4(cr, cg, cb, T);
  __syncthreads();
  if (seg == 0 && ray < npix) {
#pragma unroll
    for (int q = 1; q < kSegs; ++q) {
      const float4 p = part[q][lane];
      cr = fmaf(T, p.x, cr); cg = fmaf(T, p.y, cg); cb = fmaf(T, p.z, cb);
      T *= p.w;
    }
    reinterpret_cast<float4*>(rgba)[pix] = make_float4(cr, cg, cb, 1.f - T);
  }
}

// In-progress image of progressive rendering: evaluated pixels as they are, the others
// bilinear between the four samples of the finest complete level around (x, y) / 2^l.
__global__ void k_render_preview(RenderParams rp, int done, int level, const float4* __restrict__ rgba,
                                 float4* __restrict__ out) {
  const int pix = blockIdx.x * blockDim.x + threadIdx.x;
  if (pix >= rp.width * rp.height) return;
  const int x = pix % rp.width, y = pix / rp.width;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (order_of(rp, x, y) < done) {
    v = rgba[pix];
  } else if (done > 0) {
    const int nx = level_cols(rp, level), ny = (rp.height + (1 << level) - 1) >> level;
    const float s = 1.f / (float)(1 << level);
    const float fx = (float)x * s, fy = (float)y * s;   // exact: a power-of-two scale
    const int a0 = min(x >> level, nx - 1), b0 = min(y >> level, ny - 1);
    const int a1 = min(a0 + 1, nx - 1), b1 = min(b0 + 1, ny - 1);
    const float tx = a1 == a0 ? 0.f : fx - (float)a0, ty = b1 == b0 ? 0.f : fy - (float)b0;
    const float4 p00 = rgba[(b0 << level) * rp.width + (a0 << level)];
    const float4 p10 = rgba[(b0 << level) * rp.width + (a1 << level)];
    const float4 p01 = rgba[(b1 << level) * rp.width + (a0 << level)];
    const float4 p11 = rgba[(b1 << level) * rp.width + (a1 << level)];
    const float ux = 1.f - tx, uy = 1.f - ty;
    v.x = uy * (ux * p00.x + tx * p10.x) + ty * (ux * p01.x + tx * p11.x);
    v.y = uy * (ux * p00.y + tx * p10.y) + ty * (ux * p01.y + tx * p11.y);
    v.z = uy * (ux * p00.z + tx * p10.z) + ty * (ux * p01.z + tx * p11.z);
    v.w = uy * (ux * p00.w + tx * p10.w) + ty * (ux * p01.w + tx * p11.w);
  }
  out[pix] = v;
}

}  // namespace

bool boxes_pay(const Model& md, int group, float each, float x, float y, float z) {
  const float cells = 0.5f * (float)(md.R - 1) * 1.15f, e = cbrtf((float)group);
  const float nodes = (e * x * cells + 2.f) * (e * y * cells + 2.f) * (e * z * cells + 2.f);
  return nodes * each <= (float)group;
}

cudaError_t launch_render_batch(const Launch& L, const RenderParams& rp, float* val, int32_t* next, int pix0, int npix,
                                const Model& md, const float* lut, float* rgba) {
  Bricks br{};
  br.n = rp.grid[0] * rp.grid[1] * rp.grid[2];
  FwdSource src{};
  src.kind = kFwdRender;
  // Groups as large as they go while there are two for every SM; a group is about a cube.
  const int64_t slots = render_slots(rp, npix);
  const int least = md.F16 ? 128 : 64;
  const float edge = cbrtf(rp.cell);
  src.group = fwd_group(!md.F16, true);
  while (src.group > least && slots < (int64_t)src.group * 2 * L.num_sms) src.group /= 2;
  src.boxes = boxes_pay(md, src.group, ray_samples_per_node(!md.F16), edge, edge, edge);
  if (!src.boxes) src.group = std::min(src.group, fwd_group(!md.F16, false));
  src.groups = (int)((slots + src.group - 1) / src.group);
  src.next = next;
  src.pix0 = pix0;
  src.npix = npix;
  src.rp = rp;
  const cudaError_t e = launch_forward(L, md, br, src, val);
  if (e != cudaSuccess) return e;
  k_render_composite<<<(npix + 31) / 32, 32 * kSegs, 0, L.stream>>>(rp, pix0, npix, val, lut, rgba, next);
  return cudaGetLastError();
}

cudaError_t launch_render_preview(const Launch& L, const RenderParams& rp, int done, int level,
                                  const float* rgba, float* preview) {
  const int n = rp.width * rp.height;
  k_render_preview<<<(n + 255) / 256, 256, 0, L.stream>>>(rp, done, level, reinterpret_cast<const float4*>(rgba),
                                                         reinterpret_cast<float4*>(preview));
  return cudaGetLastError();
}

cudaError_t launch_decode(const Launch& L, const RenderParams& rp, const Model& md, float* out) {
  FwdSource src{};
  src.kind = kFwdDecode;
  src.rp = rp;
  src.dec.vox = rp.vox;
  int n[3], nb = 1;
  int64_t voxels = 1;
  for (int a = 0; a < 3; ++a) {
    src.dec.grid[a] = rp.grid[a];
    nb *= rp.grid[a];
    voxels *= rp.vox;
    n[a] = 0;   // the longest brick along the axis
    for (int c = 0; c < rp.grid[a]; ++c)
      n[a] = std::max(n[a], (int)(decode_first(rp.vox, c + 1, rp.grid[a]) - decode_first(rp.vox, c, rp.grid[a])));
    if (n[a] == 0) return cudaSuccess;
  }
  // Blocks of at most `cap` voxels: as large as they go while there are a few for every CTA,
  // and of the shape with the fewest tiles of samples over the bricks, compact ones first.
  const int tile = md.F16 ? 128 : 64;   // (the kernel's)
  int cap = fwd_group(!md.F16, true);
  while (cap > tile && voxels / cap < 8 * (int64_t)L.num_sms) cap /= 2;
  // A block of voxels is a cube along the bricks' axes, so full ones of BF16 pay sooner than rays
  // (boxes and without, in us, at voxels per node: 64 grids, 3.0 1389 and 1362, 4.1 612 and 638, 4.5
  // 2344 and 2600; 32 grids, 2.5 155 and 158, 4.4 337 and 387; 16 grids of 16^3, 3.9 101 and 109).
  const float full = md.K == 128 ? 4.f : 2.5f;
  const float each = md.F16 && cap == fwd_group(false, true) ? full : ray_samples_per_node(!md.F16);
  src.boxes = boxes_pay(md, cap, each, 2.f / (float)n[0], 2.f / (float)n[1], 2.f / (float)n[2]);
  if (!src.boxes) cap = std::min(cap, fwd_group(!md.F16, false));
  double best = 0.0;
  for (int x = 1; x <= std::min(16, n[0]); ++x)
    for (int y = 1; y <= std::min(16, n[1]); ++y)
      for (int z = 1; z <= std::min(16, n[2]) && x * y * z <= cap; ++z) {
        const int64_t blocks = (int64_t)((n[0] + x - 1) / x) * ((n[1] + y - 1) / y) * ((n[2] + z - 1) / z);
        const double cost = (double)blocks * ((x * y * z + tile - 1) / tile + 0.25) * (1.0 + 0.01 * (x + y + z));
        if (best == 0.0 || cost < best) {
          best = cost;
          src.dec.blk[0] = x; src.dec.blk[1] = y; src.dec.blk[2] = z;
        }
      }
  int64_t groups = nb;
  for (int a = 0; a < 3; ++a) {
    src.dec.nblk[a] = (n[a] + src.dec.blk[a] - 1) / src.dec.blk[a];
    groups *= src.dec.nblk[a];
  }
  if (groups > INT32_MAX) return cudaErrorInvalidValue;
  src.group = (src.dec.blk[0] * src.dec.blk[1] * src.dec.blk[2] + tile - 1) / tile * tile;
  src.groups = (int)groups;
  Bricks br{};
  br.n = nb;
  return launch_forward(L, md, br, src, out);
}

}  // namespace srn
