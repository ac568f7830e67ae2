// Sample sources of the forward query: points in memory, the renderer's ray samples and
// the decode's voxels (internal to libsrn).
#pragma once
#include "common.cuh"
#include "kernels.h"

namespace srn {

struct RenderParams {
  srn_camera cam;
  int32_t width, height, samples;
  int32_t order;    // 0: raster order, in 8 x 8 pixel blocks; 1: the progressive (image-hierarchy) order
  int32_t levels;   // L: the coarsest hierarchy level, 2^L >= max(width, height)
  // Sample slots of a batch: groups of rg consecutive rays, each group's samples one after
  // the other (spr per ray, the last ones empty), its rays fastest.  Consecutive slots are
  // then a compact bundle of ray segments, and a sample's slots are read coalesced over rays.
  int32_t rg, spr;
  float cell;       // volume per sample in a brick's coordinates (about)
  int32_t grid[3];
  int64_t vox;
  float vmin, vmax;
  int32_t lo[SRN_MAX_BRICKS][3];
  int32_t hi[SRN_MAX_BRICKS][3];
};

// Slot of sample j of ray `ray` of a batch (batches hold fewer than 2^31 slots).
__host__ __device__ inline int32_t render_slot(const RenderParams& rp, int ray, int j) {
  return ((ray / rp.rg) * rp.spr + j) * rp.rg + ray % rp.rg;
}
__host__ __device__ inline int64_t render_slots(const RenderParams& rp, int64_t npix) {
  return (npix + rp.rg - 1) / rp.rg * rp.rg * rp.spr;
}
struct RaySlot {
  int ray, j;
};
__device__ __forceinline__ RaySlot ray_slot(const RenderParams& rp, int slot) {   // the inverse
  const int q = slot / rp.rg, g = q / rp.spr;
  return RaySlot{g * rp.rg + slot % rp.rg, q - g * rp.spr};
}

struct Ray {
  float ox, oy, oz, dx, dy, dz, t0, dt;
  bool hit;
};

__device__ __forceinline__ Ray make_ray(const RenderParams& rp, int pix) {
  const int px = pix % rp.width, py = pix / rp.width;
  const float aspect = (float)rp.width / (float)rp.height;
  const float nx = (2.f * ((float)px + 0.5f) / (float)rp.width - 1.f) * rp.cam.scale * aspect;
  const float ny = (1.f - 2.f * ((float)py + 0.5f) / (float)rp.height) * rp.cam.scale;
  Ray r;
  const float* e = rp.cam.eye;
  const float* f = rp.cam.forward;
  const float* ri = rp.cam.right;
  const float* u = rp.cam.up;
  if (rp.cam.ortho) {
    r.ox = e[0] + nx * ri[0] + ny * u[0];
    r.oy = e[1] + nx * ri[1] + ny * u[1];
    r.oz = e[2] + nx * ri[2] + ny * u[2];
    r.dx = f[0]; r.dy = f[1]; r.dz = f[2];
  } else {
    r.ox = e[0]; r.oy = e[1]; r.oz = e[2];
    float dx = f[0] + nx * ri[0] + ny * u[0];
    float dy = f[1] + nx * ri[1] + ny * u[1];
    float dz = f[2] + nx * ri[2] + ny * u[2];
    const float inv = rsqrtf(dx * dx + dy * dy + dz * dz);
    r.dx = dx * inv; r.dy = dy * inv; r.dz = dz * inv;
  }
  // slab test against [-1, 1]^3
  float tmin = -INFINITY, tmax = INFINITY;
  const float o[3] = {r.ox, r.oy, r.oz}, d[3] = {r.dx, r.dy, r.dz};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float inv = 1.f / d[a];
    const float ta = (-1.f - o[a]) * inv, tb = (1.f - o[a]) * inv;
    tmin = fmaxf(tmin, fminf(ta, tb));
    tmax = fminf(tmax, fmaxf(ta, tb));
  }
  tmin = fmaxf(tmin, 0.f);
  r.hit = tmax > tmin;
  r.t0 = tmin;
  r.dt = r.hit ? (tmax - tmin) / (float)rp.samples : 0.f;
  return r;
}

// Sample j of a ray that hits: its brick, and its coordinates in the brick's [-1, 1]^3.
__device__ __forceinline__ int ray_sample(const RenderParams& rp, const Ray& r, int j, float& x, float& y, float& z) {
  const float t = r.t0 + ((float)j + 0.5f) * r.dt;
  const float p[3] = {r.ox + t * r.dx, r.oy + t * r.dy, r.oz + t * r.dz};
  int cell[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {   // Sec. 5.3 hash, clamped to the brick grid
    const int n = rp.grid[a];
    cell[a] = min(max((int)floorf((float)n * (p[a] + 1.f) * 0.5f), 0), n - 1);
  }
  const int b = cell[0] + rp.grid[0] * (cell[1] + rp.grid[1] * cell[2]);
  const float half = 0.5f * (float)(rp.vox - 1);
  float q[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {   // global -> brick-local [-1, 1]
    const float sc = (p[a] + 1.f) * half;
    const float lo = (float)rp.lo[b][a], hi = (float)rp.hi[b][a];
    q[a] = (sc - lo) / (hi - lo) * 2.f - 1.f;
  }
  x = q[0]; y = q[1]; z = q[2];
  return b;
}

// Pixels of level l of the image hierarchy: its grid (a 2^l, b 2^l), ceil(W / 2^l) by
// ceil(H / 2^l).  Together, the levels coarser than l hold exactly level l+1's grid.
__device__ __forceinline__ int level_cols(const RenderParams& rp, int l) { return (rp.width + (1 << l) - 1) >> l; }
__device__ __forceinline__ int level_pixels(const RenderParams& rp, int l) {
  return level_cols(rp, l) * ((rp.height + (1 << l) - 1) >> l);
}

// Flat pixel of the k-th pixel of the render order.  Raster order: bands of 8 rows, in each
// band blocks of 8 columns one after the other (the last band and block may be smaller), so
// that 64 consecutive rays are neighbours in both directions.  Progressive order (Sec. 6):
// the coarsest level's pixel (0, 0), then each finer level l's pixels not on level l+1's
// grid, row by row: an even row b of the level has its odd columns, an odd row all.  (Taking
// a level's rows in blocks of 8 x 8 as well, within a pass, was slower: 284 -> 308 us for the
// 14400 pixels of a VGA view.)
__device__ __forceinline__ int pixel_of(const RenderParams& rp, int k) {
  if (!rp.order) {
    const int band = k / (8 * rp.width), q = k - band * 8 * rp.width, hb = min(8, rp.height - 8 * band);
    const int blk = q / (8 * hb), r = q - blk * 8 * hb, wb = min(8, rp.width - 8 * blk);
    const int y = r / wb;
    return (8 * band + y) * rp.width + 8 * blk + r - y * wb;
  }
  if (k == 0) return k;
  int l = rp.levels - 1;
  while (level_pixels(rp, l) <= k) --l;   // level_pixels(0) = W H > k
  const int q = k - level_pixels(rp, l + 1);
  const int wa = level_cols(rp, l), half = wa >> 1, pair = q / (half + wa), r = q - pair * (half + wa);
  const int a = r < half ? 2 * r + 1 : r - half, b = r < half ? 2 * pair : 2 * pair + 1;
  return (b << l) * rp.width + (a << l);
}

// The voxels of a decode: per brick (x fastest) the same number of blocks per axis, each of
// at most blk[] voxels; a brick's voxels along an axis are [first(c), first(c + 1)).
struct DecodeParams {
  int64_t vox;
  int32_t grid[3];
  int32_t blk[3], nblk[3];
};
struct FwdBlock {
  int brick;
  int v0[3], n[3];   // first voxel and voxels per axis (0: nothing)
};
// First voxel of brick c of n along an axis of `vox` voxels: voxel i belongs to brick
// min(floor(n i / (vox - 1)), n - 1).
__host__ __device__ inline int64_t decode_first(int64_t vox, int c, int n) {
  return c >= n ? vox : (c * (vox - 1) + n - 1) / n;
}
__device__ __forceinline__ FwdBlock decode_block(const DecodeParams& d, int g) {
  FwdBlock k;
  const int per = d.nblk[0] * d.nblk[1] * d.nblk[2];
  k.brick = g / per;
  int r = g - k.brick * per, c = k.brick;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int ia = r % d.nblk[a], ca = c % d.grid[a];
    r /= d.nblk[a];
    c /= d.grid[a];
    const int end = (int)decode_first(d.vox, ca + 1, d.grid[a]);
    k.v0[a] = (int)decode_first(d.vox, ca, d.grid[a]) + ia * d.blk[a];
    k.n[a] = max(0, min(d.blk[a], end - k.v0[a]));
  }
  return k;
}
// Voxel s of a block (x fastest).
__device__ __forceinline__ void decode_voxel(const FwdBlock& k, int s, int (&v)[3]) {
  const int q = s / k.n[0], z = q / k.n[1];
  v[0] = k.v0[0] + s - q * k.n[0];
  v[1] = k.v0[1] + q - z * k.n[1];
  v[2] = k.v0[2] + z;
}

// Where the forward query takes its samples from, in groups of `group` (a multiple of the
// kernel's tile, 128 or, in float32, 64, at most fwd_group()) neighbouring ones.
enum FwdKind { kFwdPoints = 0, kFwdRender = 1, kFwdDecode = 2 };
constexpr int fwd_group(bool f32, bool boxes) { return f32 || !boxes ? 256 : 512; }
struct FwdPointSource {   // what a kernel over points in memory gets (the rest is 2 KB of arguments)
  int32_t kind;
  int32_t group, groups;   // (kFwdPoints counts its groups per brick itself)
  int32_t run;             // consecutive groups of a CTA (set by the launch)
  int32_t* next;           // kFwdRender: zero; runs of groups taken beyond the CTAs' first (NULL: in turn)
  int32_t boxes;           // 0 (always for points in memory): read every corner from global memory
  int32_t far;             // kFwdPoints: the points of a group are far apart
  const float* xyz;        // kFwdPoints, and their sorted copy, if one was made
  SortedBatch sorted;
};
struct FwdSource : FwdPointSource {
  int32_t pix0, npix;      // kFwdRender: rays pix0 .. pix0 + npix - 1 of rp's order
  DecodeParams dec;        // kFwdDecode; the bricks' boxes are rp.lo, rp.hi
  RenderParams rp;
};
// The points of br in memory, in groups that leave a few for every CTA.
inline FwdSource point_source(const Launch& L, const Bricks& br, const float* xyz, bool f32) {
  FwdSource s{};
  s.kind = kFwdPoints;
  s.group = 256;
  while (s.group > (f32 ? 64 : 128) && br.off[br.n] < (int64_t)s.group * 4 * L.num_sms) s.group /= 2;
  // (BF16, 64 grids of 32^3, far and not, in us: in no order, 3905 points through 8 bricks 35 and
  // 53, 20000 47 and 51, 60000 through 64 bricks 127 and 182; in order, 60000 46 and 46, 500000
  // 202 and 192, 8 bricks of 25000 157 and 157)
  s.far = br.off[br.n] < (int64_t)60000 * br.n;
  s.xyz = xyz;
  return s;
}
__device__ __forceinline__ void decode_point(const FwdSource& src, const FwdBlock& k, int s, float& x, float& y,
                                             float& z) {
  int v[3];
  float q[3];
  decode_voxel(k, s, v);
#pragma unroll
  for (int a = 0; a < 3; ++a) {   // voxel index = (p + 1)/2 (vox - 1): global -> brick-local [-1, 1]
    const int lo = src.rp.lo[k.brick][a], hi = src.rp.hi[k.brick][a];
    q[a] = ((float)v[a] - (float)lo) / (float)(hi - lo) * 2.f - 1.f;
  }
  x = q[0]; y = q[1]; z = q[2];
}
__device__ __forceinline__ int64_t decode_index(const FwdSource& src, const FwdBlock& k, int s) {
  int v[3];
  decode_voxel(k, s, v);
  return ((int64_t)v[2] * src.dec.vox + v[1]) * src.dec.vox + v[0];
}

// f of every sample of the source: out[point], out[slot] (slots without a sample are left
// alone) or out[voxel].
// (One translation unit per feature count K and precision.)
template <int K, bool F32>
cudaError_t launch_forward_k(const Launch& L, const Model& md, const Bricks& br, const FwdSource& src, float* out);
#define SRN_FWD(K, F32)                                                                            \
  template <>                                                                                      \
  cudaError_t launch_forward_k<K, F32>(const Launch&, const Model&, const Bricks&, const FwdSource&, float*);
SRN_FWD(16, false) SRN_FWD(32, false) SRN_FWD(64, false) SRN_FWD(128, false)
SRN_FWD(16, true) SRN_FWD(32, true) SRN_FWD(64, true) SRN_FWD(128, true)
#undef SRN_FWD
inline cudaError_t launch_forward(const Launch& L, const Model& md, const Bricks& br, const FwdSource& src, float* out) {
  const bool f32 = !md.F16;
  switch (md.K) {
    case 16: return f32 ? launch_forward_k<16, true>(L, md, br, src, out) : launch_forward_k<16, false>(L, md, br, src, out);
    case 32: return f32 ? launch_forward_k<32, true>(L, md, br, src, out) : launch_forward_k<32, false>(L, md, br, src, out);
    case 64: return f32 ? launch_forward_k<64, true>(L, md, br, src, out) : launch_forward_k<64, false>(L, md, br, src, out);
    case 128: return f32 ? launch_forward_k<128, true>(L, md, br, src, out) : launch_forward_k<128, false>(L, md, br, src, out);
    default: return cudaErrorInvalidValue;
  }
}

// Whether staged boxes pay for groups of `group` of a brick's samples, x, y and z apart in its
// coordinates: a cube's nodes in a grid are those of its extent in cells (the maps are on the
// device: they are taken to zoom by 15%), a partial cell and a node at either end, and a node
// should serve `each` samples or more.  Rays: eight, sixteen in float32.  With boxes and without, in us, at
// samples per node by this count: BF16, 64 grids, 11 (frame of 512^2 x 256 rays through 8 bricks)
// 20300 and 23600, 6.6 (progressive pass of 9000 x 256) 967 and 925, 2.9 (the same, 4 bricks)
// 1475 and 1059; 32 grids, 13 460 and 459; 16 grids, 14 (14400 x 256) 258 and 283.  Float32, 64
// grids, 7 (frame of 160^2 x 320) 7036 and 7548, 2.6 (8 bricks) 10780 and 8910; 16 grids of 9^3,
// 20 2805 and 2600.
bool boxes_pay(const Model& md, int group, float each, float x, float y, float z);
inline float ray_samples_per_node(bool f32) { return f32 ? 16.f : 8.f; }
// Rays pix0 .. pix0 + npix - 1 of rp's order; val: [max_points] scratch for their samples'
// values, next: a counter that is zero, and again after a batch whose launches succeed.
cudaError_t launch_render_batch(const Launch& L, const RenderParams& rp, float* val, int32_t* next, int pix0, int npix,
                                const Model& md, const float* lut, float* rgba);
// In-progress image after `done` pixels of the progressive order; `level` is the finest
// complete hierarchy level (ignored when done = 0).
cudaError_t launch_render_preview(const Launch& L, const RenderParams& rp, int done, int level,
                                  const float* rgba, float* preview);

// The whole decode: rp holds the bricks' grid, boxes and vox.
cudaError_t launch_decode(const Launch& L, const RenderParams& rp, const Model& md, float* out);

}  // namespace srn
