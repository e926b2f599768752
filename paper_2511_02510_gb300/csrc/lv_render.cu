// lv_render.cu -- forward / backward passes of the sparse-voxel tile
// rasterizer (LiteVoxel Sec. III, Eq. 1-5) for sm_103a.
//
// Pipeline of lv_rasterize_forward (one stream, no host synchronisation):
//   k_bin       per (voxel, view): FP32 cull / near-plane clipping / corner
//               projection / tile rect / depth key with a fixed operation
//               order; depth statistics; each block's pair and slot totals.
//   k_block_offsets  the blocks' first pairs and slots (item order), with the
//               slot and pair totals.
//   k_emit      per (voxel, view): the item's (tile, slot) pairs, written in
//               item order by whole warps; per visible item the 64-byte render
//               record (centre relative to the camera, half-size, 8 corner
//               densities, SH colour, 1 / (2 h)), its pixel box, voxel id and
//               depth key.
//   radix sort  the pairs by tile id (stable: each tile's list stays in
//               voxel-id order); its last pass also notes every tile's range.
//   k_tile_sort_warp, k_tile_sort  per tile: its slots sorted by depth key in
//               shared memory (stable), front to back with ties by voxel id, and
//               written with the pixel strips they meet; of very long lists only
//               the front.  The depth keys are sorted per tile, where they fit
//               in shared memory, instead of by global passes over all slots.
//   k_fwd       per tile, one thread per pixel: each warp stages the records
//               that meet its pixel strip through shared memory and marches
//               front to back (Eq. 2-4); w_max (Eq. 5) is reduced over the
//               warp before one global atomicMax; a warp stops when all its
//               pixels have T < t_stop.
//   k_tile_rest, k_fwd  the rest of the very long lists whose pixels are still
//               open, and their march from there on.
// lv_rasterize_backward walks the same lists back to front (k_bwd) and
// reduces the SH colour gradient per voxel (k_sh_bwd).
#include <math.h>
#include <stdio.h>

#include "lv_prims.cuh"

namespace lv {

// ------------------------------------------------------------------ views
struct DevView {
  float R[9];  // w2c rotation, row-major
  float t[3];
  float o[3];  // camera centre in world coordinates
  float fx, fy, cx, cy, z_near;
  int W, H, tiles_x, tiles_y;
  int tile_off;       // first global tile of the view
  long long pix_off;  // first global pixel of the view
  // k_bin's early-out planes: the frustum of the tile grid widened by 2 pixels has side planes
  // f u - m z = 0 (u the camera x or y coordinate) with m = cx + 2, cx - tiles_x ts - 2,
  // cy + 2, cy - tiles_y ts - 2 (cull_m), and |(f, m)| rounded up (cull_n)
  float cull_m[4], cull_n[4];
};
struct ViewSet {
  int n;
  int ts;
  long long id_base;  // global id of the call's first pixel (w_max argmax ids)
  DevView v[LV_MAX_VIEWS];
};

static void make_views(const lv_camera* cams, int nv, int ts, ViewSet* vs, int64_t* tiles, int64_t* pixels) {
  vs->n = nv;
  vs->ts = ts;
  vs->id_base = 0;
  int64_t to = 0, po = 0;
  for (int i = 0; i < nv; ++i) {
    const lv_camera& c = cams[i];
    DevView& d = vs->v[i];
    for (int r = 0; r < 3; ++r) {
      for (int k = 0; k < 3; ++k) d.R[r * 3 + k] = c.w2c[r * 4 + k];
      d.t[r] = c.w2c[r * 4 + 3];
    }
    for (int k = 0; k < 3; ++k) {
      double s = 0;
      for (int r = 0; r < 3; ++r) s += (double)c.w2c[r * 4 + k] * (double)c.w2c[r * 4 + 3];
      d.o[k] = (float)(-s);
    }
    d.fx = c.fx; d.fy = c.fy; d.cx = c.cx; d.cy = c.cy; d.z_near = c.z_near;
    d.W = c.width; d.H = c.height;
    d.tiles_x = (c.width + ts - 1) / ts;
    d.tiles_y = (c.height + ts - 1) / ts;
    d.tile_off = (int)to;
    d.pix_off = po;
    d.cull_m[0] = d.cx + 2.f;
    d.cull_m[1] = d.cx - (float)(d.tiles_x * ts) - 2.f;
    d.cull_m[2] = d.cy + 2.f;
    d.cull_m[3] = d.cy - (float)(d.tiles_y * ts) - 2.f;
    for (int k = 0; k < 4; ++k) {
      const double f = k < 2 ? (double)d.fx : (double)d.fy, m = (double)d.cull_m[k];
      d.cull_n[k] = nextafterf((float)sqrt(f * f + m * m), INFINITY);  // at least the exact norm
    }
    to += (int64_t)d.tiles_x * d.tiles_y;
    po += (int64_t)c.width * c.height;
  }
  *tiles = to;
  *pixels = po;
}

// ------------------------------------------------------------------ workspace
// Tiles by list length, longest first: class 0 above 4096 pairs (long), 1 to 4 above 2048, 1024, 512 and
// 256 (medium), 5 to 7 above 128, 64 and the rest (short).  The depth sort and the composites take them
// in this order: a long list begun last would keep its warps marching after all others have ended.
constexpr int TILE_CLASSES = 8, TILE_CLASS_SHORT = 5;
struct TileOrder {
  uint32_t* tiles;      // [TILE_CLASSES][stride]
  unsigned int* count;  // [TILE_CLASSES], 16-byte aligned
  uint32_t stride;
  static __device__ __forceinline__ int cls(uint32_t length) {
    // 12 bits and more: 0 and 1, each bit less a class on, at most 64: 7
    return length > 4096u ? 0 : (length <= 64u ? 7 : __clz(length - 1u) - 19);
  }
  // the i-th tile, and (nullable) its class
  __device__ __forceinline__ uint32_t tile(uint32_t i, int* c_out = nullptr) const {
    const uint4 a = *(const uint4*)count, b = *(const uint4*)(count + 4);
    const uint32_t n[TILE_CLASSES] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    int c = 0;
    uint32_t at = i;
#pragma unroll
    for (int k = 0; k + 1 < TILE_CLASSES; ++k) {
      if (c == k && at >= n[k]) {
        at -= n[k];
        c = k + 1;
      }
    }
    if (c_out) *c_out = c;
    return tiles[(size_t)c * stride + at];
  }
};
// progress of a long tile's depth order
struct TileProg {
  uint32_t done;  // entries sorted
  uint32_t next;  // smallest order key not sorted yet
  uint32_t kmax;  // largest order key of the list
  uint32_t open;  // 1: listed in open_tiles
  uint32_t front; // where the resumed composite starts (list entry)
};
// items are (view, voxel) pairs in view-major order: item = view * n + voxel
struct FwdWs {
  unsigned long long* counters;  // [0] pairs, [1] slots
  uint32_t* cnt;                 // [items] tiles covered (visible: not 0)
  uint2* rect;                   // [items] of visible items: (tx0 | tx1 << 16, ty0 | ty1 << 16)
  uint2* pbox;                   // [items] of visible items: conservative pixel box (x0 | x1 << 16,
                                 // y0 | y1 << 16), [x0, x1)
  uint32_t* dkey;                // [items] of visible items: order key of z_centre
  uint32_t* slot;                // [items] of visible items: render slot
  unsigned long long* blk_pairs; // [blocks of 256 voxels x views, view-major] pairs, then the block's first
                                 // within its group
  uint32_t* blk_slots;           // the same for slots
  unsigned long long* grp_pairs; // totals of groups of BO_GROUP blocks
  uint32_t* grp_slots;
  uint2* rec_bb;                 // [slots] pixel box of the render record
  uint32_t* slot_vox;            // [slots] voxel id of the render record
  uint32_t* s_dkey;              // [slots] order key
  unsigned int* work;            // [32] work-item counters: [0..1] the persistent composites, [2] the
                                 // resumed composite, [3] k_tile_rest, [5] k_tile_sort, [7] count of the
                                 // open tiles; [8..10] block arrivals of the persistent forward, backward
                                 // and resumed composites (sm_leave); [16..23] tiles per length class
  uint32_t* class_tiles;         // [TILE_CLASSES][tiles] the tiles of each length class
  uint32_t* open_tiles;          // [tiles] long tiles with pixels open at the end of the sorted part
  uint32_t* ready;               // [tiles] end of the list's depth-sorted part
  TileProg* prog;                // [tiles] progress of the long tiles' depth order
  float* dep;                    // [pixels] depth and sample count of the pixels of open tiles
  uint32_t* nsamp;
  float4* rec;                   // [slots][4]
  float4* d_rgb;                 // [slots] colour gradient (xyz) scratch of the backward; w = clamp mask
  uint32_t* ranges;              // [tiles][2]
  float* tau;                    // [pixels] final optical depth
  void* sort_tmp;                // scratch of the sort by tile
  int32_t* status;               // fallback status word
  uint32_t *k0, *v0, *k1, *v1;   // [pair capacity] (tile, slot) pairs and the sort's other buffer
  // once the pairs are sorted by tile, their slots in one of v0 and v1 (item order within a tile), the
  // sort's other buffer and the sorted tile ids, which the ranges replace, serve the depth order:
  uint32_t* tile_slots;          // the sorted slots
  uint2* plist;                  // [pair capacity] (slot, strip mask) of every tile's list in depth order
  uint32_t* long_keys;           // [pair capacity] the long lists' order keys
  size_t bytes;
};

constexpr int BIN_THREADS = 256;  // voxels per block of k_bin and k_emit
constexpr int BO_THREADS = 1024, BO_ITEMS = 4, BO_GROUP = BO_THREADS * BO_ITEMS;  // blocks per group of their offsets
static int64_t bin_blocks(int64_t n) { return (n + BIN_THREADS - 1) / BIN_THREADS; }

static int tile_bits(int64_t tiles) {
  int b = 0;
  while (b < 32 && ((int64_t)1 << b) < tiles) ++b;
  return b;
}

static FwdWs carve_fwd(void* base, int64_t n, int nv, int64_t tiles, int64_t pixels, int64_t pair_cap) {
  FwdWs w;
  Carve c(base);
  int64_t items = n * nv;
  w.counters = c.take<unsigned long long>(8);
  w.status = c.take<int32_t>(4);
  w.work = c.take<unsigned int>(32);
  w.cnt = c.take<uint32_t>(items);
  w.rect = c.take<uint2>(items);
  w.pbox = c.take<uint2>(items);
  w.dkey = c.take<uint32_t>(items);
  w.slot = c.take<uint32_t>(items);
  w.blk_pairs = c.take<unsigned long long>(bin_blocks(n) * nv);
  w.blk_slots = c.take<uint32_t>(bin_blocks(n) * nv);
  w.grp_pairs = c.take<unsigned long long>(bin_blocks(n) * nv / BO_GROUP + 1);
  w.grp_slots = c.take<uint32_t>(bin_blocks(n) * nv / BO_GROUP + 1);
  w.rec_bb = c.take<uint2>(items);
  w.slot_vox = c.take<uint32_t>(items);
  w.s_dkey = c.take<uint32_t>(items);
  w.rec = c.take<float4>(items * 4);
  w.d_rgb = c.take<float4>(items);
  w.ranges = c.take<uint32_t>(tiles * 2);
  w.class_tiles = c.take<uint32_t>(TILE_CLASSES * tiles);
  w.open_tiles = c.take<uint32_t>(tiles);
  w.ready = c.take<uint32_t>(tiles);
  w.prog = c.take<TileProg>(tiles);
  w.dep = c.take<float>(pixels);
  w.nsamp = c.take<uint32_t>(pixels);
  w.tau = c.take<float>(pixels);
  w.sort_tmp = c.take<char>(sort_tmp_bytes(pair_cap));
  // keys and values of a buffer side by side, so that the unused buffer holds 8-byte words
  const size_t half = align_up((size_t)pair_cap, 64);
  w.k0 = c.take<uint32_t>(2 * half);
  w.k1 = c.take<uint32_t>(2 * half);
  w.v0 = w.k0 ? w.k0 + half : nullptr;
  w.v1 = w.k1 ? w.k1 + half : nullptr;
  const bool odd = sort_passes(tile_bits(tiles)) & 1;  // the sorted pairs are in (k1, v1)
  w.tile_slots = odd ? w.v1 : w.v0;
  w.long_keys = odd ? w.k1 : w.k0;
  w.plist = (uint2*)(odd ? w.k0 : w.k1);
  w.bytes = c.off + 256;
  return w;
}



__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// ------------------------------------------------------------------ binning (FP32, fixed op order)
__device__ __forceinline__ void cam_point32(const DevView& c, float X, float Y, float Z, float* q) {
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    float a = __fmul_rn(c.R[r * 3 + 0], X);
    float b = __fmul_rn(c.R[r * 3 + 1], Y);
    float e = __fmul_rn(c.R[r * 3 + 2], Z);
    float s = __fadd_rn(a, b);
    s = __fadd_rn(s, e);
    q[r] = __fadd_rn(s, c.t[r]);
  }
}

// one (voxel, view) item: its number of tiles, and the outputs of a visible one
__device__ __forceinline__ uint32_t bin_item(const DevView& c, int ts, const float4* __restrict__ geom, int64_t vox,
                                             int64_t i, uint2* __restrict__ rect, uint2* __restrict__ pbox,
                                             uint32_t* __restrict__ dkey, float* z_min, float* delta_min,
                                             uint8_t* seen) {
  float4 g = geom[vox];
  float qc[3];
  cam_point32(c, g.x, g.y, g.z, qc);
  {
    // Early out for voxels far outside the view: the circumscribed sphere lies behind the near
    // plane or beyond a side plane of the frustum of the tile grid (which may reach past the image
    // edge) widened by 2 pixels, with a relative slack far above FP32 rounding.  Such a voxel's
    // exact tile rectangle below (1-pixel margin, clamped to the tile grid) is empty, so skipping it
    // changes no output.
    const float r = g.w * 1.7320508f;
    const float rs = r + 1e-4f * (fabsf(qc[0]) + fabsf(qc[1]) + fabsf(qc[2]) + r) + 1e-6f;
    // (the planes and their norms are per view, set up on the host)
    const bool out = qc[2] + rs < c.z_near ||
                     c.fx * qc[0] + c.cull_m[0] * qc[2] < -rs * c.cull_n[0] ||
                     c.fx * qc[0] + c.cull_m[1] * qc[2] > rs * c.cull_n[1] ||
                     c.fy * qc[1] + c.cull_m[2] * qc[2] < -rs * c.cull_n[2] ||
                     c.fy * qc[1] + c.cull_m[3] * qc[2] > rs * c.cull_n[3];
    if (out) return 0u;
  }
  float umin = 0.f, umax = 0.f, vmin = 0.f, vmax = 0.f;
  float px[8], py[8], pz[8];
  int n_front = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    float X = (k & 1) ? __fadd_rn(g.x, g.w) : __fsub_rn(g.x, g.w);
    float Y = (k & 2) ? __fadd_rn(g.y, g.w) : __fsub_rn(g.y, g.w);
    float Z = (k & 4) ? __fadd_rn(g.z, g.w) : __fsub_rn(g.z, g.w);
    float p[3];
    cam_point32(c, X, Y, Z, p);
    px[k] = p[0]; py[k] = p[1]; pz[k] = p[2];
    n_front += p[2] >= c.z_near ? 1 : 0;
  }
  auto project = [&](int k, float* u, float* v) {
    const float iz = __frcp_rn(pz[k]);  // one correctly rounded reciprocal per corner
    *u = __fadd_rn(__fmul_rn(c.fx, __fmul_rn(px[k], iz)), c.cx);
    *v = __fadd_rn(__fmul_rn(c.fy, __fmul_rn(py[k], iz)), c.cy);
  };
  if (n_front == 8) {
    // the usual case, with no test per corner: 3-input minima and maxima of all eight (the order of
    // minima and maxima changes nothing)
    float u[8], v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) project(k, &u[k], &v[k]);
    umin = fminf(min3(u[0], u[1], u[2]), fminf(min3(u[3], u[4], u[5]), fminf(u[6], u[7])));
    umax = fmaxf(max3(u[0], u[1], u[2]), fmaxf(max3(u[3], u[4], u[5]), fmaxf(u[6], u[7])));
    vmin = fminf(min3(v[0], v[1], v[2]), fminf(min3(v[3], v[4], v[5]), fminf(v[6], v[7])));
    vmax = fmaxf(max3(v[0], v[1], v[2]), fmaxf(max3(v[3], v[4], v[5]), fmaxf(v[6], v[7])));
  } else {
    bool first = true;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (pz[k] >= c.z_near) {
        float u, v;
        project(k, &u, &v);
        if (first) { umin = umax = u; vmin = vmax = v; first = false; }
        else { umin = fminf(umin, u); umax = fmaxf(umax, u); vmin = fminf(vmin, v); vmax = fmaxf(vmax, v); }
      }
    }
  }
  int tx0 = 0, tx1 = 0, ty0 = 0, ty1 = 0;
  int px0 = 0, px1 = 0, py0 = 0, py1 = 0;  // pixels x in [px0, px1) may be hit (their centres lie in the box)
  if (n_front > 0) {
    if (n_front < 8) {
      // near-plane clipping: crossing points of the box edges (k, k|bit) with z = z_near
#pragma unroll
      for (int k = 0; k < 8; ++k) {
#pragma unroll
        for (int bit = 1; bit < 8; bit <<= 1) {
          if (k & bit) continue;
          const int j = k | bit;
          if ((pz[k] >= c.z_near) == (pz[j] >= c.z_near)) continue;
          const float f = __fdiv_rn(__fsub_rn(c.z_near, pz[k]), __fsub_rn(pz[j], pz[k]));
          const float x = __fadd_rn(px[k], __fmul_rn(f, __fsub_rn(px[j], px[k])));
          const float y = __fadd_rn(py[k], __fmul_rn(f, __fsub_rn(py[j], py[k])));
          const float u = __fadd_rn(__fmul_rn(c.fx, __fdiv_rn(x, c.z_near)), c.cx);
          const float v = __fadd_rn(__fmul_rn(c.fy, __fdiv_rn(y, c.z_near)), c.cy);
          umin = fminf(umin, u); umax = fmaxf(umax, u); vmin = fminf(vmin, v); vmax = fmaxf(vmax, v);
        }
      }
    }
    // ts is a power of two, so multiplying by 1/ts rounds exactly as dividing by ts
    const float its = 1.0f / (float)ts;
    const float a0 = floorf(__fmul_rn(__fsub_rn(umin, 1.0f), its));
    const float a1 = ceilf(__fmul_rn(__fadd_rn(umax, 1.0f), its));
    const float b0 = floorf(__fmul_rn(__fsub_rn(vmin, 1.0f), its));
    const float b1 = ceilf(__fmul_rn(__fadd_rn(vmax, 1.0f), its));
    tx0 = (int)fminf(fmaxf(a0, 0.0f), (float)c.tiles_x);
    tx1 = (int)fminf(fmaxf(a1, 0.0f), (float)c.tiles_x);
    ty0 = (int)fminf(fmaxf(b0, 0.0f), (float)c.tiles_y);
    ty1 = (int)fminf(fmaxf(b1, 0.0f), (float)c.tiles_y);
    // The composites only cull with the pixel box: a ray through the centre (x + 1/2, y + 1/2) of
    // pixel (x, y) meets the box only if that centre lies in the footprint's bounding box
    // [umin, umax] x [vmin, vmax].  The FP32 projection and the FP32 ray of the chord test are
    // each within about 1e-3 pixel of exact, so widening the box by 1/16 pixel plus 2^-14 of the
    // coordinate keeps every pixel an FP32 chord test can hit; the tile rectangle above keeps its
    // 1-pixel margin.
    const float eu = fmaf(6.1035156e-5f, fmaxf(fabsf(umin), fabsf(umax)), 0.0625f);
    const float ev = fmaf(6.1035156e-5f, fmaxf(fabsf(vmin), fabsf(vmax)), 0.0625f);
    px0 = (int)fminf(fmaxf(ceilf(umin - eu - 0.5f), 0.0f), (float)c.W);
    px1 = (int)fminf(fmaxf(floorf(umax + eu - 0.5f) + 1.0f, (float)px0), (float)c.W);
    py0 = (int)fminf(fmaxf(ceilf(vmin - ev - 0.5f), 0.0f), (float)c.H);
    py1 = (int)fminf(fmaxf(floorf(vmax + ev - 0.5f) + 1.0f, (float)py0), (float)c.H);
  }
  uint32_t count = (tx1 > tx0 && ty1 > ty0) ? (uint32_t)(tx1 - tx0) * (uint32_t)(ty1 - ty0) : 0u;
  if (!count) return 0u;
  dkey[i] = order_key(qc[2]);
  rect[i] = make_uint2((uint32_t)tx0 | ((uint32_t)tx1 << 16), (uint32_t)ty0 | ((uint32_t)ty1 << 16));
  pbox[i] = make_uint2((uint32_t)px0 | ((uint32_t)px1 << 16), (uint32_t)py0 | ((uint32_t)py1 << 16));
  float zs = fmaxf(qc[2], c.z_near);
  float dl = __fdiv_rn(zs, c.fx);
  if (z_min) atomicMin((unsigned int*)&z_min[vox], __float_as_uint(zs));
  if (delta_min) atomicMin((unsigned int*)&delta_min[vox], __float_as_uint(dl));
  if (seen) seen[vox] = 1;
  return count;
}

// Block b covers 256 consecutive voxels of view b % views, as in k_emit: the
// views' blocks of one voxel range run side by side, so its geometry comes from
// HBM once; a warp's lanes share one view (warp-uniform camera loads; the
// statistics' atomics hit distinct voxels).  The block leaves its pair and slot
// totals, from which k_block_offsets and k_emit place the items: per-item
// offsets, scanned by three more launches, cost 28 bytes of traffic an item
// (48M items: 290 us), and only visible items write anything but their count
// (48M items: 854 -> 607 us with that, the geometry read once, the usual case's
// projections without a test per corner and six blocks an SM, for which 56 bytes a
// thread are spilled; 2M items: 39 -> 31 us).
__global__ void __launch_bounds__(BIN_THREADS, 6)
    k_bin(const float4* __restrict__ geom, int64_t n, int64_t blocks, const __grid_constant__ ViewSet vs,
          uint32_t* __restrict__ cnt, uint2* __restrict__ rect, uint2* __restrict__ pbox, uint32_t* __restrict__ dkey,
          unsigned long long* __restrict__ blk_pairs, uint32_t* __restrict__ blk_slots, float* z_min,
          float* delta_min, uint8_t* seen, const ZeroRanges zr) {
  grid_begin();
  __shared__ unsigned long long s_pairs[BIN_THREADS / 32];
  __shared__ uint32_t s_slots[BIN_THREADS / 32];
  // the later kernels' counters are cleared by the first blocks, not by a launch of their own (about
  // 2100 32-bit words)
  constexpr unsigned ZERO_BLOCKS = 8;
  if (blockIdx.x < ZERO_BLOCKS) {
    const size_t stride = (size_t)min(gridDim.x, ZERO_BLOCKS) * BIN_THREADS;
    for (int k = 0; k < 4; ++k)
      for (size_t x = blockIdx.x * (size_t)BIN_THREADS + threadIdx.x; x < zr.bytes[k] / 4; x += stride)
        ((uint32_t*)zr.p[k])[x] = 0u;
  }
  const int view = (int)(blockIdx.x % (unsigned)vs.n);
  const int64_t vb = blockIdx.x / (unsigned)vs.n, vox = vb * BIN_THREADS + threadIdx.x;
  const int64_t i = (int64_t)view * n + vox;  // items are view-major
  uint32_t count = 0;
  if (vox < n) {
    count = bin_item(vs.v[view], vs.ts, geom, vox, i, rect, pbox, dkey, z_min, delta_min, seen);
    cnt[i] = count;
  }
  // (32 counts can exceed 32 bits: halves are summed)
  const uint32_t lo = __reduce_add_sync(FULL, count & 0xffffu), hi = __reduce_add_sync(FULL, count >> 16);
  const uint32_t vis = __popc(__ballot_sync(FULL, count != 0u));
  if ((threadIdx.x & 31) == 0) {
    s_pairs[threadIdx.x >> 5] = ((unsigned long long)hi << 16) + lo;
    s_slots[threadIdx.x >> 5] = vis;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long p = 0;
    uint32_t q = 0;
#pragma unroll
    for (int w = 0; w < BIN_THREADS / 32; ++w) {
      p += s_pairs[w];
      q += s_slots[w];
    }
    blk_pairs[view * blocks + vb] = p;
    blk_slots[view * blocks + vb] = q;
  }
}

// Offsets of the binning blocks' pairs and slots within groups of BO_GROUP
// blocks, in place, the groups' totals, and the grand totals added to
// counters[0] and [1] (zero before).  k_emit sums the groups before its own: up
// to 1M items there is one group, at 48M items 46.  (One block over all entries
// took 196 us for 48M items, 4 us a round of 4096.)
__global__ void __launch_bounds__(BO_THREADS) k_block_offsets(unsigned long long* pairs,
                                                              uint32_t* slots, int64_t m,
                                                              unsigned long long* grp_pairs,
                                                              uint32_t* grp_slots,
                                                              unsigned long long* counters) {
  grid_begin();
  __shared__ unsigned long long s_a[BO_THREADS / 32];
  __shared__ uint32_t s_b[BO_THREADS / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t i0 = blockIdx.x * (int64_t)BO_GROUP + BO_ITEMS * t;
  unsigned long long a[BO_ITEMS], xa = 0;
  uint32_t b[BO_ITEMS], xb = 0;
#pragma unroll
  for (int k = 0; k < BO_ITEMS; ++k) {
    a[k] = i0 + k < m ? pairs[i0 + k] : 0ull;
    b[k] = i0 + k < m ? slots[i0 + k] : 0u;
  }
#pragma unroll
  for (int k = 0; k < BO_ITEMS; ++k) {
    xa += a[k];
    xb += b[k];
  }
  const unsigned long long own_a = xa;
  const uint32_t own_b = xb;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long ya = __shfl_up_sync(FULL, xa, o);
    const uint32_t yb = __shfl_up_sync(FULL, xb, o);
    if (lane >= o) {
      xa += ya;
      xb += yb;
    }
  }
  if (lane == 31) {
    s_a[warp] = xa;
    s_b[warp] = xb;
  }
  __syncthreads();
  unsigned long long wa = s_a[lane];
  uint32_t wb = s_b[lane];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long ya = __shfl_up_sync(FULL, wa, o);
    const uint32_t yb = __shfl_up_sync(FULL, wb, o);
    if (lane >= o) {
      wa += ya;
      wb += yb;
    }
  }
  const unsigned long long pa = __shfl_sync(FULL, wa, (warp + 31) & 31);
  const uint32_t pb = __shfl_sync(FULL, wb, (warp + 31) & 31);
  unsigned long long ra = (warp ? pa : 0ull) + xa - own_a;
  uint32_t rb = (warp ? pb : 0u) + xb - own_b;
#pragma unroll
  for (int k = 0; k < BO_ITEMS; ++k) {
    if (i0 + k < m) {
      pairs[i0 + k] = ra;
      slots[i0 + k] = rb;
    }
    ra += a[k];
    rb += b[k];
  }
  if (t == BO_THREADS - 1) {
    grp_pairs[blockIdx.x] = wa;  // lane 31: the whole group
    grp_slots[blockIdx.x] = wb;
    atomicAdd(&counters[0], wa);
    atomicAdd(&counters[1], (unsigned long long)wb);
  }
}

// ------------------------------------------------------------------ SH (real, degree <= 3)
// Orthonormal real spherical harmonics written from the associated Legendre
// functions: Y0 = 1/(2 sqrt(pi)); l=1 sqrt(3/4pi) {y, z, x}; l=2 sqrt(15/4pi)
// {xy, yz, xz}, sqrt(5/16pi)(3z^2-1), sqrt(15/16pi)(x^2-y^2); l=3
// sqrt(35/32pi) y(3x^2-y^2), sqrt(105/4pi) xyz, sqrt(21/32pi) y(5z^2-1),
// sqrt(7/16pi) z(5z^2-3), sqrt(21/32pi) x(5z^2-1), sqrt(105/16pi) z(x^2-y^2),
// sqrt(35/32pi) x(x^2-3y^2).
__device__ __forceinline__ void sh_basis(float x, float y, float z, float* Y) {
  const float C0 = 0.28209479177387814f;
  const float C1 = 0.48860251190291992f;
  const float C2a = 1.0925484305920792f, C2b = 0.31539156525252005f, C2c = 0.54627421529603959f;
  const float C3a = 0.59004358992664352f, C3b = 2.8906114426405538f, C3c = 0.45704579946446572f;
  const float C3d = 0.37317633259011540f, C3e = 1.4453057213202769f;
  float xx = x * x, yy = y * y, zz = z * z;
  Y[0] = C0;
  Y[1] = C1 * y;
  Y[2] = C1 * z;
  Y[3] = C1 * x;
  Y[4] = C2a * x * y;
  Y[5] = C2a * y * z;
  Y[6] = C2b * (3.f * zz - 1.f);
  Y[7] = C2a * x * z;
  Y[8] = C2c * (xx - yy);
  Y[9] = C3a * y * (3.f * xx - yy);
  Y[10] = C3b * x * y * z;
  Y[11] = C3c * y * (5.f * zz - 1.f);
  Y[12] = C3d * z * (5.f * zz - 3.f);
  Y[13] = C3c * x * (5.f * zz - 1.f);
  Y[14] = C3e * z * (xx - yy);
  Y[15] = C3a * x * (xx - 3.f * yy);
}

// A lane's own row in 32-byte loads, whole sectors, where the row is aligned for
// them: with 16-byte loads every sector of a row is asked for twice, and by the
// second time the other lanes' rows may have pushed it out of L1.
__device__ __forceinline__ void ld_row32(const void* p, uint32_t* w) {
  asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
      : "l"(p));
}
__device__ __forceinline__ void st_row32(void* p, float4 a, float4 b) {  // p: 32-byte aligned
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z),
               "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
               : "memory");
}
__device__ __forceinline__ bool aligned32(const void* p) { return ((uintptr_t)p & 31) == 0; }
__device__ __forceinline__ void bf16_pair(uint32_t w, float* c) {
  c[0] = __uint_as_float(w << 16);
  c[1] = __uint_as_float(w & 0xffff0000u);
}

// c = max(0, raw) with raw = sum_j coef[j] Y_j + 0.5 per channel, from a voxel's row of 48 coefficients
// ([j][rgb], 16-byte aligned).  The row is read 32 bytes at a time, each word used before the next is
// asked for, and only as far as the degree needs, to keep k_emit's registers few: it is bound by the
// latency of its scattered reads and writes, so warps in flight count for more than loads in flight per
// warp.  Eight views of 6M voxels, FP16 and BF16: 1474 us at 5 blocks an SM, 1362 at 6, 1271 at 8 (32
// registers and 16 bytes spilled), 1100 with the records stored in whole sectors; one view of 2M, FP32: 97, 91, 97 us, and 86.
template <int PER, typename F>
__device__ __forceinline__ void sh_add(int k, const F (&c)[PER], int nb, const float* Y, float* raw) {
#pragma unroll
  for (int h = 0; h < PER; ++h) {
    const int i = PER * k + h, j = i / 3;
    if (j < nb) raw[i % 3] = fmaf(c[h], Y[j], raw[i % 3]);
  }
}
__device__ __forceinline__ void sh_raw_row(const float* __restrict__ row, int nb, const float* dir, float* raw) {
  float Y[16];
  sh_basis(dir[0], dir[1], dir[2], Y);
  raw[0] = raw[1] = raw[2] = 0.f;
  const bool wide = aligned32(row);
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    if (8 * k < 3 * nb) {  // grid-uniform
      float c[8];
      if (wide) {
        uint32_t w[8];
        ld_row32(row + 8 * k, w);
#pragma unroll
        for (int h = 0; h < 8; ++h) c[h] = __uint_as_float(w[h]);
      } else {
        const float4 a = __ldg((const float4*)row + 2 * k), b = __ldg((const float4*)row + 2 * k + 1);
        c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w;
        c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
      }
      sh_add<8>(k, c, nb, Y, raw);
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) raw[k] += 0.5f;
}
__device__ __forceinline__ void sh_raw_row(const __nv_bfloat16* __restrict__ row, int nb, const float* dir,
                                           float* raw) {
  float Y[16];
  sh_basis(dir[0], dir[1], dir[2], Y);
  raw[0] = raw[1] = raw[2] = 0.f;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    if (8 * k < 3 * nb) {  // grid-uniform
      const uint4 q = __ldg((const uint4*)row + k);
      float c[8];
      bf16_pair(q.x, c);
      bf16_pair(q.y, c + 2);
      bf16_pair(q.z, c + 4);
      bf16_pair(q.w, c + 6);
      sh_add<8>(k, c, nb, Y, raw);
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) raw[k] += 0.5f;
}

// one voxel's 8 corner densities (any alignment)
__device__ __forceinline__ void load_corners(const float* __restrict__ row, float* d) {
  if (aligned32(row)) {
    uint32_t w[8];
    ld_row32(row, w);
#pragma unroll
    for (int k = 0; k < 8; ++k) d[k] = __uint_as_float(w[k]);
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) d[k] = row[k];
  }
}
__device__ __forceinline__ void load_corners(const __half* __restrict__ row, float* d) {
  if (((uintptr_t)row & 15) == 0) {
    const uint4 q = __ldg((const uint4*)row);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 f = __half22float2(*(const __half2*)&w[k]);
      d[2 * k] = f.x;
      d[2 * k + 1] = f.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) d[k] = to_f32(row[k]);
  }
}

__device__ __forceinline__ void unit_dir(float rx, float ry, float rz, float* d) {
  float nn = rx * rx + ry * ry + rz * rz;
  if (nn > 0.f) {
    float inv = rsqrtf(nn);
    d[0] = rx * inv; d[1] = ry * inv; d[2] = rz * inv;
  } else {
    d[0] = 0.f; d[1] = 0.f; d[2] = 1.f;
  }
}

// ------------------------------------------------------------------ emit
// One thread per (voxel, view) item, blocks as in k_bin: an item's slot and first
// pair are its block's plus a scan inside the block.  First the warp writes the (tile, slot)
// pairs of its 32 items: items are consecutive, so their pairs form one
// contiguous range in item order (view-major, voxel id within a view), which
// the warp fills 32 pairs per step, each lane finding the item of its pair by
// a 5-step search over the lanes' first pairs.  More pairs than capacity:
// none are written and the status word says LV_ERR_CAPACITY.  Then each
// visible item writes the render record of its slot (camera-relative centre
// and h | 8 corner densities | clamped SH colour and 1/(2h)), the slot's order
// key, and the colour-gradient scratch (cleared; w = clamp mask).
template <typename DT, typename ST>
__global__ void __launch_bounds__(BIN_THREADS, sizeof(ST) == 4 ? 6 : 8)
    k_emit(const float4* __restrict__ geom, const DT* __restrict__ dens, const ST* __restrict__ sh, int sh_nb,
           int64_t n, const __grid_constant__ ViewSet vs, const uint32_t* cnt, const uint2* rect, const uint2* pbox,
           uint2* rec_bb, uint32_t* slot_vox, const uint32_t* dkey, uint32_t* slot, int64_t blocks,
           const unsigned long long* blk_pairs, const uint32_t* blk_slots, const unsigned long long* grp_pairs,
           const uint32_t* grp_slots, const unsigned long long* counters, int64_t pair_cap, uint32_t* pair_tile,
           uint32_t* pair_slot, int32_t* status, uint2* ranges, int64_t tiles, const SortCountTargets sc, int passes,
           float4* rec, float4* d_rgb, uint32_t* s_dkey, const uint32_t* __restrict__ vidx) {
  grid_begin();
  // Block b covers 256 consecutive voxels of view b % views, so the blocks of
  // all views of one voxel range run side by side: a voxel's SH row comes
  // from HBM once and from L2 for its other views.  Items are view-major
  // (i = view * n + voxel), so each block still writes consecutive slots.
  const int view = (int)(blockIdx.x % (unsigned)vs.n);
  const int64_t vox = (int64_t)(blockIdx.x / (unsigned)vs.n) * 256 + threadIdx.x;
  const int64_t i = (int64_t)view * n + vox;
  const bool in = vox < n;
  // the sort by tile's last pass reduces every tile's [first, end) into ranges
  for (int64_t x = blockIdx.x * 256ll + threadIdx.x; x < tiles; x += (int64_t)gridDim.x * 256)
    ranges[x] = make_uint2(~0u, 0u);
  const uint32_t cn = in ? cnt[i] : 0u;  // nonzero exactly for the visible items
  const unsigned long long total = counters[0];
  // the sort by tile's digit counts (every pass) are counted here, and its first look-back words cleared
  __shared__ uint32_t s_cnt[4 * 256];
  for (int x = threadIdx.x; x < passes * 256; x += 256) s_cnt[x] = 0u;
  if (total <= (unsigned long long)pair_cap) {
    const int64_t words = (int64_t)((total + sc.tile - 1) / sc.tile) * 256;
    for (int64_t x = blockIdx.x * 256ll + threadIdx.x; x < words; x += (int64_t)gridDim.x * 256) sc.look0[x] = 0ull;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t blk = view * blocks + blockIdx.x / (unsigned)vs.n;
  // items of the warp before this one: visible, and their pairs (32 bits do: nothing is written when
  // the pairs exceed the capacity, and that is below 2^32)
  const uint32_t vism = __ballot_sync(FULL, cn != 0u);
  uint32_t pre = cn;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(FULL, pre, o);
    if (lane >= o) pre += y;
  }
  __shared__ uint32_t s_wp[8], s_wv[8];
  if (lane == 31) {
    s_wp[warp] = pre;
    s_wv[warp] = __popc(vism);
  }
  uint32_t sl = blk_slots[blk];
  unsigned long long p_block = blk_pairs[blk];
  // the groups before this block's: summed by the first warp (none up to 1M items)
  __shared__ unsigned long long s_gp;
  __shared__ uint32_t s_gs;
  const int64_t grp = blk / BO_GROUP;
  if (warp == 0) {
    unsigned long long a = 0;
    uint32_t b = 0;
    for (int64_t g = lane; g < grp; g += 32) {
      a += grp_pairs[g];
      b += grp_slots[g];
    }
    if (grp) {  // block-uniform
#pragma unroll
      for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(FULL, a, o);
      b = __reduce_add_sync(FULL, b);
    }
    if (lane == 0) {
      s_gp = a;
      s_gs = b;
    }
  }
  __syncthreads();
  p_block += s_gp;
  sl += s_gs;
  uint32_t wp = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    wp += w < warp ? s_wp[w] : 0u;
    sl += w < warp ? s_wv[w] : 0u;
  }
  sl += __popc(vism & ((1u << lane) - 1u));
  if (total > (unsigned long long)pair_cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) report(status, LV_ERR_CAPACITY);
  } else {
    const uint32_t wn = __shfl_sync(FULL, pre, 31);  // the warp's pairs
    if (wn) {                                        // warp-uniform
      const uint32_t po = pre - cn;  // first pair of the item within the warp's
      uint32_t rx = 0u, ry = 0u;
      if (cn) {
        const uint2 rc = rect[i];
        rx = rc.x;
        ry = rc.y;
      }
      const unsigned long long p_begin = p_block + wp;
      const DevView& c = vs.v[view];
      const uint32_t toff = (uint32_t)c.tile_off, tiles_x = (uint32_t)c.tiles_x;
      for (uint32_t e0 = 0; e0 < wn; e0 += 32) {  // warp-uniform
        const uint32_t e = e0 + lane;
        int j = 0;  // the largest lane whose first pair is <= e (lane 0's is 0)
#pragma unroll
        for (int step = 16; step; step >>= 1) {
          const uint32_t x = __shfl_sync(FULL, po, (j + step) & 31);
          if (j + step < 32 && x <= e) j += step;
        }
        const uint32_t pj = __shfl_sync(FULL, po, j);
        const uint32_t jx = __shfl_sync(FULL, rx, j), jy = __shfl_sync(FULL, ry, j);
        const uint32_t js = __shfl_sync(FULL, sl, j);
        if (e < wn) {
          const uint32_t q = e - pj;
          const uint32_t tx0 = jx & 0xffffu, wx = (jx >> 16) - tx0, ty0 = jy & 0xffffu;
          const uint32_t key = toff + (ty0 + q / wx) * tiles_x + tx0 + q % wx;
          pair_tile[p_begin + e] = key;
          pair_slot[p_begin + e] = js;
          for (int p = 0; p < passes; ++p) atomicAdd(&s_cnt[p * 256 + ((key >> (8 * p)) & 255u)], 1u);
        }
      }
    }
  }
  __syncthreads();
  for (int x = threadIdx.x; x < passes * 256; x += 256)
    if (s_cnt[x]) atomicAdd(&sc.counts[x], s_cnt[x]);
  if (!cn) return;
  const DevView& c = vs.v[view];
  const uint32_t s = sl;
  slot[i] = s;
  const float4 g = geom[vox];
  const float rx = g.x - c.o[0], ry = g.y - c.o[1], rz = g.z - c.o[2];
  float dir[3];
  unit_dir(rx, ry, rz, dir);
  float raw[3];
  sh_raw_row(sh + 48 * vox, sh_nb, dir, raw);
  float d[8];
  if (vidx) {  // shared grid-vertex densities
    const uint4 i0 = *(const uint4*)(vidx + 8 * vox), i1 = *(const uint4*)(vidx + 8 * vox + 4);
    d[0] = to_f32(dens[i0.x]); d[1] = to_f32(dens[i0.y]); d[2] = to_f32(dens[i0.z]); d[3] = to_f32(dens[i0.w]);
    d[4] = to_f32(dens[i1.x]); d[5] = to_f32(dens[i1.y]); d[6] = to_f32(dens[i1.z]); d[7] = to_f32(dens[i1.w]);
  } else {
    load_corners(dens + 8 * vox, d);
  }
  float4* r = rec + 4 * (int64_t)s;
  // whole sectors: a lane's rows are 64 bytes apart, and 16-byte stores would write each sector twice
  st_row32(r, make_float4(rx, ry, rz, g.w), make_float4(d[0], d[1], d[2], d[3]));
  st_row32(r + 2, make_float4(d[4], d[5], d[6], d[7]),
           make_float4(fmaxf(raw[0], 0.f), fmaxf(raw[1], 0.f), fmaxf(raw[2], 0.f), __fdiv_rn(0.5f, g.w)));
  const uint2 box = pbox[i];
  const uint32_t key = dkey[i];
  slot_vox[s] = (uint32_t)vox;
  // colour-gradient scratch: xyz cleared, w = which channels passed the clamp
  // (bit c set when raw_c > 0) as a small exact float, read by the SH backward
  d_rgb[s] = make_float4(0.f, 0.f, 0.f,
                         (float)((raw[0] > 0.f ? 1 : 0) | (raw[1] > 0.f ? 2 : 0) | (raw[2] > 0.f ? 4 : 0)));
  rec_bb[s] = box;
  s_dkey[s] = key;
}

// pairs usable by the later stages: all of them, or none after an overflow
__device__ __forceinline__ int64_t usable_pairs(const unsigned long long* d_count, int64_t cap) {
  unsigned long long c = *d_count;
  return c <= (unsigned long long)cap ? (int64_t)c : 0;
}

// ------------------------------------------------------------------ per-tile depth order
// After the stable sort by tile id, each tile's pairs are in item order (voxel
// id within a view), and the sort's last pass has left every tile's range in
// ranges (empty tiles: (0xffffffff, 0)).  Each tile's slots are then put in
// order of their keys, ties in item order, and written with their strip masks
// to plist: the order one stable sort of (tile, order key) pairs in voxel-id
// order gives.  A list is sorted in shared memory, by an LSD radix sort of
// 9-bit digits of the key minus the smallest key (3 passes for spans below
// 2^27).  Each pass ranks stably (warp-private digit counts; the lanes holding
// a digit found by bit ballots or by __match_any_sync).  The tiles are shared
// out by list length:
//   k_tile_sort_warp  one warp per tile: lists of up to TW_MAX pairs; it also
//                     writes every tile's range in final form (empty: (0, 0))
//                     and lists the longer tiles;
//   k_tile_sort       persistent blocks of 512 threads: lists of up to TS_CHUNK
//                     pairs in one go, longer ones range of keys by range of
//                     keys (as many whole bins of a histogram of the keys as
//                     hold TS_CHUNK pairs), and of those above TS_LAZY only
//                     the front, the nearest ranges up to TS_FRONT pairs: one
//                     range, unless a crowded bin cut it short;
//   k_tile_rest       the rest of those whose pixels are still open after the
//                     composite of the sorted parts.
// Opaque scenes seldom read a long list past its front: of eight 980 x 545
// views of 6M voxels with tile 32 (lists of up to 68,000 pairs, 38M in all) hardly
// a tile does (with fronts of 2048 pairs 2 to 5 % of them, and 480 us for the rest
// and the resumed composite).  Sorting every list whole, in chunks merged
// afterwards, took 4.7 ms of those views' 8.2 ms; their fronts take 0.41 ms.  Lists
// of a few chunks are sorted whole: where their pixels stay open, the composite in two launches costs more than the sort
// saves (one 1237 x 822 view of 2M voxels, lists of up to 7,800 pairs: 217 + 151 us
// against 297 us).  Scenes of up to TS_LAZY_VOXELS seldom have longer lists, and go
// without the two launches that the rest takes (6 us when there is none).
constexpr int TS_BITS = 9, TS_BINS = 1 << TS_BITS;
constexpr int TS_THREADS = 512, TS_WARPS = TS_THREADS / 32, TS_ITEMS = 8, TS_CHUNK = TS_THREADS * TS_ITEMS;
constexpr uint32_t TS_LAZY = 4 * TS_CHUNK;          // lists up to here are sorted whole at once
constexpr uint32_t TS_FRONT = TS_CHUNK / 2;         // at least this many entries of the others are
constexpr int64_t TS_LAZY_VOXELS = 1 << 19;         // and all lists of scenes up to here
constexpr int TL_BITS = 11, TL_BINS = 1 << TL_BITS;  // key histogram of a long list
constexpr int TW_MAX = 256, TW_ITEMS = TW_MAX / 32, TW_WARPS = 16;
static_assert(TS_THREADS == TS_BINS, "a thread for each digit");

struct TileSortSmem {
  uint32_t k[TS_CHUNK];                // keys
  uint32_t v[TS_CHUNK];                // slots
  uint16_t wc[TS_WARPS][TS_BINS + 2];  // warp digit counts -> warp prefixes (bin TS_BINS: padding)
  uint32_t base[TS_BINS];              // start of each digit
  uint32_t w[TS_WARPS];
  uint32_t item, kmin, kmax;
};
struct WarpSortSmem {
  uint32_t k[2][TW_MAX];     // keys, ping-pong
  uint32_t v[2][TW_MAX];     // slots, ping-pong
  uint16_t wc[TS_BINS + 2];  // digit counts (bin TS_BINS: padding)
  uint16_t base[TS_BINS];    // start of each digit
};
struct TileSortWarpSmem {
  WarpSortSmem w[TW_WARPS];
};
struct TileLongSmem {
  TileSortSmem s;
  uint32_t inc[TL_BINS];  // keys of a bin or an earlier one
  uint32_t b0, b1;
};

// exclusive scan of one value per thread over a block of WARPS warps
template <int WARPS>
__device__ __forceinline__ uint32_t ts_block_excl(uint32_t c, uint32_t* s_w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  uint32_t pre = 0;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) pre += w < warp ? s_w[w] : 0u;
  return pre + x - c;
}

// Stable ranks of R rounds held warp-striped (round j of a warp holds item
// 32 j + lane of the warp's items).  dr[j] holds the digit (TS_BINS for
// padding) on entry; on exit also the item's rank among the warp's items of
// its digit, from bit 10 up.  The warp's counts per digit accumulate in wc.
template <int ITEMS>
__device__ __forceinline__ void ts_rank(uint32_t (&dr)[ITEMS], int R, uint16_t* wc, bool use_match, int lane) {
  const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    if (j >= R) break;  // warp-uniform
    const uint32_t d = dr[j];
    uint32_t peers;
    if (use_match) {  // warp-uniform
      peers = __match_any_sync(FULL, d);
    } else {
      const uint32_t valid = __ballot_sync(FULL, d < TS_BINS);
      peers = d < TS_BINS ? valid : ~valid;
#pragma unroll
      for (int b = 0; b < TS_BITS; ++b) {
        const uint32_t m = __ballot_sync(FULL, (d >> b) & 1u);
        peers &= ((d >> b) & 1u) ? m : ~m;
      }
    }
    const bool leader = (peers & lt_mask) == 0;
    use_match = __popc(__ballot_sync(FULL, leader)) <= 16;
    const uint32_t cur = wc[d];
    dr[j] = d | ((cur + __popc(peers & lt_mask)) << 10);
    __syncwarp();
    if (leader) wc[d] = (uint16_t)(cur + __popc(peers));
    __syncwarp();
  }
}

// smallest and largest of the per-thread values into *kmin / *kmax (set to ~0u / 0 before a barrier)
__device__ __forceinline__ void ts_min_max(uint32_t mn, uint32_t mx, uint32_t* kmin, uint32_t* kmax) {
  mn = __reduce_min_sync(FULL, mn);
  mx = __reduce_max_sync(FULL, mx);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(kmin, mn);
    atomicMax(kmax, mx);
  }
}

// the tile's pair range: from the sort's last pass, or the whole list when no pass ran (one tile)
__device__ __forceinline__ void ts_range(const uint32_t* ranges, uint32_t tile, int64_t n, bool ranges_ready,
                                         uint32_t* lo, uint32_t* hi) {
  *lo = *hi = 0u;
  if (n <= 0) return;
  if (!ranges_ready) {
    *hi = (uint32_t)n;
    return;
  }
  const uint2 r = reinterpret_cast<const uint2*>(ranges)[tile];
  if (r.x < r.y) {
    *lo = r.x;
    *hi = r.y;
  }
}

__device__ __forceinline__ int ts_passes(uint32_t span) {
  return span ? (32 - __clz(span) + TS_BITS - 1) / TS_BITS : 0;
}

// The strips (4 x 8 pixel blocks, one warp of a composite each) of a tile that a
// pixel box meets, as a bit mask: bit s for strip s, ts / 8 strips across.  The
// sorted list carries it beside the slot, so a composite's warp finds its
// records from one coalesced 8-byte word per entry.  Before, every one of a
// tile's 2, 8 or 32 warps gathered the pixel box of every entry by slot; the
// gather is now done once per pair, where the sorted list is written.
struct TileBox {
  int x0, y0;   // the tile's first pixel
  int cshift;   // log2 of the strips across: ts = 8 << cshift
  __device__ __forceinline__ TileBox(const ViewSet& vs, uint32_t gtile) {
    int v = 0;
    while (v + 1 < vs.n && (int)gtile >= vs.v[v + 1].tile_off) ++v;
    const int lt = (int)gtile - vs.v[v].tile_off, tx = vs.v[v].tiles_x;
    x0 = (lt % tx) * vs.ts;
    y0 = (lt / tx) * vs.ts;
    cshift = vs.ts == 8 ? 0 : (vs.ts == 16 ? 1 : 2);
  }
  // box: (bx0 | bx1 << 16, by0 | by1 << 16), [bx0, bx1) x [by0, by1)
  __device__ __forceinline__ uint32_t mask(uint2 box) const {
    const int ts = 8 << cshift;
    const int bx0 = max((int)(box.x & 0xffffu) - x0, 0), bx1 = min((int)(box.x >> 16) - x0, ts);
    const int by0 = max((int)(box.y & 0xffffu) - y0, 0), by1 = min((int)(box.y >> 16) - y0, ts);
    if (bx1 <= bx0 || by1 <= by0) return 0u;
    const uint32_t cols = (1u << ((bx1 + 7) >> 3)) - (1u << (bx0 >> 3));
    const int r0 = (by0 >> 2) << cshift, r1 = ((by1 + 3) >> 2) << cshift;  // bit range [r0, r1) of the rows
    const uint32_t rows = ((r1 < 32 ? 1u << r1 : 0u) - (1u << r0)) &
                          (cshift == 0 ? 0xffffffffu : (cshift == 1 ? 0x55555555u : 0x11111111u));
    return rows * cols;  // the column bits at every row: no carries, cols < 2^(strips across)
  }
};

// ---- short lists: one warp each, TW_WARPS tiles per block
__global__ void __launch_bounds__(TW_WARPS * 32, 2)
    k_tile_sort_warp(const uint32_t* tvals, const uint32_t* s_dkey, const unsigned long long* d_count, int64_t cap,
                     bool ranges_ready, int64_t tiles, uint32_t* ranges, const TileOrder order, uint32_t* ready,
                     TileProg* prog, const __grid_constant__ ViewSet vs, const uint2* rec_bb, uint2* plist) {
  grid_begin();
  extern __shared__ __align__(16) unsigned char tw_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  WarpSortSmem& W = reinterpret_cast<TileSortWarpSmem*>(tw_raw)->w[warp];
  __shared__ uint32_t s_cnt[TILE_CLASSES], s_at[TILE_CLASSES];
  const int64_t tile64 = (int64_t)blockIdx.x * TW_WARPS + warp;
  const uint32_t tile = (uint32_t)tile64;
  uint32_t lo = 0, hi = 0, at = 0;
  int cls = 0;
  if (threadIdx.x < TILE_CLASSES) s_cnt[threadIdx.x] = 0u;
  __syncthreads();
  if (lane == 0 && tile64 < tiles) {
    ts_range(ranges, tile, usable_pairs(d_count, cap), ranges_ready, &lo, &hi);
    reinterpret_cast<uint2*>(ranges)[tile] = make_uint2(lo, hi);
    const uint32_t L = hi - lo;
    ready[tile] = hi;
    cls = TileOrder::cls(L);
    if (cls == 0) prog[tile].open = 0u;
    at = atomicAdd(&s_cnt[cls], 1u);
  }
  __syncthreads();
  if (threadIdx.x < TILE_CLASSES)
    s_at[threadIdx.x] = s_cnt[threadIdx.x] ? atomicAdd(&order.count[threadIdx.x], s_cnt[threadIdx.x]) : 0u;
  __syncthreads();
  if (tile64 >= tiles) return;  // warp-uniform; no block-wide barrier below
  if (lane == 0) order.tiles[(size_t)cls * order.stride + s_at[cls] + at] = tile;
  lo = __shfl_sync(FULL, lo, 0);
  const int L = (int)(__shfl_sync(FULL, hi, 0) - lo);
  if (L < 1 || L > TW_MAX) return;  // warp-uniform
  const TileBox tb(vs, tile);
  const int R = (L + 31) / 32;
  uint32_t mn = ~0u, mx = 0u;
  {
    uint32_t kk[TW_ITEMS], vv[TW_ITEMS];
#pragma unroll
    for (int j = 0; j < TW_ITEMS; ++j) {
      if (j >= R) break;
      vv[j] = j * 32 + lane < L ? tvals[lo + j * 32 + lane] : 0u;
    }
#pragma unroll
    for (int j = 0; j < TW_ITEMS; ++j) {
      if (j >= R) break;
      kk[j] = j * 32 + lane < L ? s_dkey[vv[j]] : 0u;
    }
#pragma unroll
    for (int j = 0; j < TW_ITEMS; ++j) {
      if (j >= R) break;
      const int q = j * 32 + lane;
      if (q < L) {
        W.k[0][q] = kk[j];
        W.v[0][q] = vv[j];
        mn = min(mn, kk[j]);
        mx = max(mx, kk[j]);
      }
    }
  }
  const uint32_t kmin = __reduce_min_sync(FULL, mn);
  const int npass = ts_passes(__reduce_max_sync(FULL, mx) - kmin);
  __syncwarp();  // no pass (one pair, or all keys equal): item order is the order
  int cur = 0;
  for (int pass = 0; pass < npass; ++pass) {
    const int shift = TS_BITS * pass;
    uint32_t dr[TW_ITEMS];
#pragma unroll
    for (int j = 0; j < TW_ITEMS; ++j) {
      if (j >= R) break;
      const int q = j * 32 + lane;
      dr[j] = q < L ? ((W.k[cur][q] - kmin) >> shift) & (TS_BINS - 1) : (uint32_t)TS_BINS;
    }
    uint32_t* wcw = reinterpret_cast<uint32_t*>(W.wc);
    for (int x = lane; x < (TS_BINS + 2) / 2; x += 32) wcw[x] = 0u;
    __syncwarp();
    ts_rank<TW_ITEMS>(dr, R, W.wc, pass > 0, lane);
    __syncwarp();
    // digit starts: lane l takes digits 16 l .. 16 l + 15 (8 words of two counts), the lanes'
    // totals are scanned, then each lane writes its digits' starts
    const uint32_t* wc2 = reinterpret_cast<const uint32_t*>(W.wc) + 8 * lane;
    uint32_t tot = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t c2 = wc2[i];
      tot += (c2 & 0xffffu) + (c2 >> 16);
    }
    uint32_t x = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL, x, o);
      if (lane >= o) x += y;
    }
    uint32_t run = x - tot;
    uint32_t* base2 = reinterpret_cast<uint32_t*>(W.base) + 8 * lane;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t c2 = wc2[i];
      const uint32_t b0 = run, b1 = run + (c2 & 0xffffu);
      base2[i] = b0 | (b1 << 16);
      run = b1 + (c2 >> 16);
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < TW_ITEMS; ++j) {
      if (j >= R) break;
      const uint32_t d = dr[j] & 1023u;
      if (d < TS_BINS) {
        const int q = j * 32 + lane;
        const uint32_t pos = W.base[d] + (dr[j] >> 10);
        W.k[cur ^ 1][pos] = W.k[cur][q];
        W.v[cur ^ 1][pos] = W.v[cur][q];
      }
    }
    __syncwarp();
    cur ^= 1;
  }
#pragma unroll
  for (int j = 0; j < TW_ITEMS; ++j) {
    if (j >= R) break;
    const int q = j * 32 + lane;
    if (q < L) {
      const uint32_t v = W.v[cur][q];
      plist[lo + q] = make_uint2(v, tb.mask(rec_bb[v]));
    }
  }
}

// the blocks' shared memory, named in each function (not handed down as a
// pointer) so that calls keep its address space
__device__ __forceinline__ TileLongSmem& ts_smem() {
  extern __shared__ __align__(16) unsigned char ts_raw[];
  return *reinterpret_cast<TileLongSmem*>(ts_raw);
}

// Sorts the m <= TS_CHUNK (key, slot) pairs of S by key, stably, with the whole
// block (all of it past a barrier since they were written, and S.kmin and S.kmax
// their extremes); ends with a barrier where it moved anything.
__device__ __forceinline__ void ts_sort_pairs(int m) {
  TileSortSmem& S = ts_smem().s;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int R = (m + TS_THREADS - 1) / TS_THREADS;  // items per thread, and rounds per warp
  const uint32_t kmin = S.kmin;
  const int npass = ts_passes(S.kmax - kmin);
  for (int pass = 0; pass < npass; ++pass) {
    const int shift = TS_BITS * pass;
    uint32_t kk[TS_ITEMS], vv[TS_ITEMS], dr[TS_ITEMS];
#pragma unroll
    for (int j = 0; j < TS_ITEMS; ++j) {
      if (j >= R) break;
      const int q = warp * 32 * R + j * 32 + lane;
      const bool ok = q < m;
      kk[j] = ok ? S.k[q] : 0u;
      vv[j] = ok ? S.v[q] : 0u;
      dr[j] = ok ? ((kk[j] - kmin) >> shift) & (TS_BINS - 1) : (uint32_t)TS_BINS;
    }
    {
      uint32_t* p = reinterpret_cast<uint32_t*>(&S.wc[0][0]);
      for (int x = t; x < TS_WARPS * (TS_BINS + 2) / 2; x += TS_THREADS) p[x] = 0u;
    }
    __syncthreads();
    ts_rank<TS_ITEMS>(dr, R, S.wc[warp], pass > 0, lane);
    __syncthreads();
    uint32_t c = 0;  // digit t: warp counts -> warp prefixes
#pragma unroll
    for (int w = 0; w < TS_WARPS; ++w) {
      const uint32_t x = S.wc[w][t];
      S.wc[w][t] = (uint16_t)c;
      c += x;
    }
    S.base[t] = ts_block_excl<TS_WARPS>(c, S.w);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < TS_ITEMS; ++j) {
      if (j >= R) break;
      const uint32_t d = dr[j] & 1023u;
      if (d < TS_BINS) {
        const uint32_t pos = S.base[d] + S.wc[warp][d] + (dr[j] >> 10);
        S.k[pos] = kk[j];
        S.v[pos] = vv[j];
      }
    }
    __syncthreads();
  }
}

// the sorted pairs of S as (slot, strip mask) to plist[0, m)
__device__ __forceinline__ void ts_write(int m, const TileBox& tb, const uint2* rec_bb,
                                         uint2* plist) {
  const TileSortSmem& S = ts_smem().s;
  for (int q = threadIdx.x; q < m; q += TS_THREADS) {
    const uint32_t v = S.v[q];
    plist[q] = make_uint2(v, tb.mask(rec_bb[v]));
  }
}

__device__ __noinline__ void ts_sort_smem(int m) { ts_sort_pairs(m); }
// sort and write in one function: the depth order of one view of 2M voxels takes 71 us so, 76 in two
__device__ __noinline__ void ts_sort_write(int m, const TileBox& tb, const uint2* rec_bb, uint2* plist) {
  ts_sort_pairs(m);
  ts_write(m, tb, rec_bb, plist);
}

// a whole list of m <= TS_CHUNK slots
__device__ __noinline__ void ts_sort_list(const uint32_t* src, const uint32_t* s_dkey,
                                          int m, const TileBox& tb, const uint2* rec_bb,
                                          uint2* plist) {
  TileSortSmem& S = ts_smem().s;
  const int t = threadIdx.x;
  if (t == 0) {
    S.kmin = ~0u;
    S.kmax = 0u;
  }
  __syncthreads();
  const int R = (m + TS_THREADS - 1) / TS_THREADS;
  // every slot load, then every key load, in flight at once
  uint32_t kk[TS_ITEMS], vv[TS_ITEMS];
#pragma unroll
  for (int j = 0; j < TS_ITEMS; ++j) {
    if (j >= R) break;
    const int q = t + j * TS_THREADS;
    vv[j] = q < m ? src[q] : 0u;
  }
#pragma unroll
  for (int j = 0; j < TS_ITEMS; ++j) {
    if (j >= R) break;
    const int q = t + j * TS_THREADS;
    kk[j] = q < m ? s_dkey[vv[j]] : 0u;
  }
  uint32_t mn = ~0u, mx = 0u;
#pragma unroll
  for (int j = 0; j < TS_ITEMS; ++j) {
    if (j >= R) break;
    const int q = t + j * TS_THREADS;
    if (q < m) {
      S.k[q] = kk[j];
      S.v[q] = vv[j];
      mn = min(mn, kk[j]);
      mx = max(mx, kk[j]);
    }
  }
  ts_min_max(mn, mx, &S.kmin, &S.kmax);
  __syncthreads();
  ts_sort_write(m, tb, rec_bb, plist);
}

// The entries of a long list with keys in [k0, k1], in item order, to S as (key,
// slot).  Without ONE_KEY there are at most TS_CHUNK of them, and their extremes go
// to S too.  With ONE_KEY (k0 == k1: item order is the order) there may be any
// number: flush(m) gets each round's, at most TS_CHUNK, at S's start.
template <bool ONE_KEY, typename Flush>
__device__ __forceinline__ void tl_collect(TileSortSmem& S, const uint32_t* sv, const uint32_t* xk, uint32_t L,
                                           uint32_t k0, uint32_t k1, Flush&& flush) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (t == 0) {
    S.kmin = ~0u;
    S.kmax = 0u;
  }
  uint32_t at = 0, mn = ~0u, mx = 0u;
  for (uint32_t base = 0; base < L; base += TS_CHUNK) {  // block-uniform
    // warp w takes entries [base + 256 w, + 256), 32 at a time
    uint32_t k[TS_ITEMS], in[TS_ITEMS], c = 0;
    const uint32_t e0 = base + warp * 32 * TS_ITEMS + lane;
#pragma unroll
    for (int j = 0; j < TS_ITEMS; ++j) k[j] = e0 + 32 * j < L ? xk[e0 + 32 * j] : 0u;
#pragma unroll
    for (int j = 0; j < TS_ITEMS; ++j) {
      in[j] = __ballot_sync(FULL, e0 + 32 * j < L && k[j] >= k0 && k[j] <= k1);
      c += __popc(in[j]);
    }
    __syncthreads();  // the last round's counts are read, and its entries flushed
    if (lane == 0) S.w[warp] = c;
    __syncthreads();
    if (ONE_KEY) at = 0;
    uint32_t pos = at;
#pragma unroll
    for (int w = 0; w < TS_WARPS; ++w) {
      const uint32_t x = S.w[w];
      pos += w < warp ? x : 0u;
      at += x;
    }
#pragma unroll
    for (int j = 0; j < TS_ITEMS; ++j) {
      if ((in[j] >> lane) & 1u) {
        const uint32_t q = pos + __popc(in[j] & ((1u << lane) - 1u));
        S.k[q] = k[j];
        S.v[q] = sv[e0 + 32 * j];
        mn = min(mn, k[j]);
        mx = max(mx, k[j]);
      }
      pos += __popc(in[j]);
    }
    if (ONE_KEY && at) {  // block-uniform
      __syncthreads();
      flush(at);
    }
  }
  if (!ONE_KEY) ts_min_max(mn, mx, &S.kmin, &S.kmax);
  __syncthreads();
}

// Depth order of a long list's entries with keys from cur up (`done` of its L
// entries have smaller ones), nearest first: a histogram of the keys not sorted yet
// cuts them into ranges of at most TS_CHUNK entries, and each range is collected in
// item order and sorted in shared memory.  A bin of more than TS_CHUNK entries is
// cut by a finer histogram of its own keys; once a bin is one key, item order is the
// order.  sink(at, m, sorted) gets the pieces in order: the m (key, slot) pairs at S's
// start are the list's entries from `at` on, which it sorts first unless they are;
// once it returns true (to the whole block) the work stops after that key.
struct TlAt {
  uint32_t done;  // entries handed out
  uint32_t next;  // smallest key not handed out yet
};
template <typename Sink>
__device__ __forceinline__ TlAt tl_ranges(uint32_t L, const uint32_t* sv, const uint32_t* xk, uint32_t done,
                                          uint32_t cur, uint32_t kmax, Sink&& sink) {
  TileLongSmem& M = ts_smem();
  TileSortSmem& S = M.s;
  const int t = threadIdx.x;
  uint32_t top = kmax;  // keys [cur, top] are cut by one histogram
  while (done < L) {    // block-uniform
    const uint32_t span = top - cur;
    const int shift = span < (uint32_t)TL_BINS ? 0 : 32 - __clz(span) - TL_BITS;
    for (int x = t; x < TL_BINS; x += TS_THREADS) M.inc[x] = 0u;
    __syncthreads();
    for (uint32_t base = t; base < L; base += TS_CHUNK) {
      uint32_t k[TS_ITEMS];
#pragma unroll
      for (int j = 0; j < TS_ITEMS; ++j) k[j] = base + j * TS_THREADS < L ? xk[base + j * TS_THREADS] : 0u;
#pragma unroll
      for (int j = 0; j < TS_ITEMS; ++j)
        if (base + j * TS_THREADS < L && k[j] >= cur && k[j] <= top) atomicAdd(&M.inc[(k[j] - cur) >> shift], 1u);
    }
    __syncthreads();
    {
      constexpr int PER = TL_BINS / TS_THREADS;
      uint32_t c[PER], sum = 0;
#pragma unroll
      for (int i = 0; i < PER; ++i) sum += c[i] = M.inc[PER * t + i];
      uint32_t run = ts_block_excl<TS_WARPS>(sum, S.w);
#pragma unroll
      for (int i = 0; i < PER; ++i) M.inc[PER * t + i] = run += c[i];
    }
    __syncthreads();
    const uint32_t total = M.inc[TL_BINS - 1];
    uint32_t b0 = 0, cum = 0;
    bool finer = false;
    while (cum < total) {  // block-uniform
      if (t == 0) {
        // bins [b0, b1): as many as fit (b1 == b0: bin b0 alone does not)
        auto count_upto = [&](uint32_t limit) {  // bins with inc <= limit
          uint32_t n = 0;
          for (uint32_t step = TL_BINS; step; step >>= 1)
            if (n + step <= (uint32_t)TL_BINS && M.inc[n + step - 1] <= limit) n += step;
          return n;
        };
        M.b0 = count_upto(cum);  // past empty bins, so that an oversized bin is met as b0
        M.b1 = count_upto(cum + TS_CHUNK);
      }
      __syncthreads();
      b0 = M.b0;
      const uint32_t b1 = M.b1;
      __syncthreads();
      bool stop = false;
      uint32_t k1;
      if (b1 > b0) {
        const uint32_t k0 = cur + (b0 << shift);
        k1 = b1 < (uint32_t)TL_BINS && top - cur >= b1 << shift ? cur + ((b1 << shift) - 1u) : top;
        const uint32_t m = M.inc[b1 - 1] - cum;
        tl_collect<false>(S, sv, xk, L, k0, k1, [](uint32_t) {});
        stop = sink(done, m, false);
        __syncthreads();  // S is reused
        done += m;
        cum += m;
        b0 = b1;
      } else if (shift == 0) {  // one key with more entries than TS_CHUNK
        k1 = cur + b0;
        cum = M.inc[b0];
        tl_collect<true>(S, sv, xk, L, k1, k1, [&](uint32_t m) {
          stop |= sink(done, m, true);
          done += m;
        });
        ++b0;
      } else {  // the bin's own keys, finer
        cur += b0 << shift;
        if (top - cur >= 1u << shift) top = cur + ((1u << shift) - 1u);
        finer = true;
        break;
      }
      if (stop) return {done, k1 + 1u};
    }
    if (!finer) {  // everything up to top is sorted
      cur = top + 1u;
      top = kmax;
    }
  }
  return {done, kmax};
}

// A long list's depth order to plist.  START: the keys are gathered first (to xk), and
// above `lazy` entries the work stops at the first range's end past TS_FRONT entries; else
// it goes on from the progress of such a start.
template <bool START>
__device__ __noinline__ void tl_order(uint32_t lo, uint32_t L, uint32_t lazy, const uint32_t* sv_all,
                         uint32_t* xk_all, const uint32_t* s_dkey, TileProg* prog,
                         uint32_t* ready, const TileBox& tb, const uint2* rec_bb,
                         uint2* plist_all) {
  TileSortSmem& S = ts_smem().s;
  const int t = threadIdx.x;
  const uint32_t* sv = sv_all + lo;
  uint32_t* xk = xk_all + lo;
  uint2* plist = plist_all + lo;
  uint32_t done, cur, kmax;
  const bool front = START && L > lazy;
  if (START) {
    if (t == 0) {
      S.kmin = ~0u;
      S.kmax = 0u;
    }
    __syncthreads();
    uint32_t mn = ~0u, mx = 0u;
    for (uint32_t base = t; base < L; base += TS_CHUNK) {
      uint32_t v[TS_ITEMS], k[TS_ITEMS];
#pragma unroll
      for (int j = 0; j < TS_ITEMS; ++j) v[j] = base + j * TS_THREADS < L ? sv[base + j * TS_THREADS] : 0u;
#pragma unroll
      for (int j = 0; j < TS_ITEMS; ++j) k[j] = base + j * TS_THREADS < L ? s_dkey[v[j]] : 0u;
#pragma unroll
      for (int j = 0; j < TS_ITEMS; ++j)
        if (base + j * TS_THREADS < L) {
          xk[base + j * TS_THREADS] = k[j];
          mn = min(mn, k[j]);
          mx = max(mx, k[j]);
        }
    }
    ts_min_max(mn, mx, &S.kmin, &S.kmax);
    __syncthreads();  // also orders the block's writes of xk before its reads below
    done = 0u;
    cur = S.kmin;
    kmax = S.kmax;
  } else {
    done = prog->done;
    cur = prog->next;
    kmax = prog->kmax;
  }
  const TlAt end = tl_ranges(L, sv, xk, done, cur, kmax, [&](uint32_t at, uint32_t m, bool sorted) {
    if (sorted) ts_write((int)m, tb, rec_bb, plist + at);
    else ts_sort_write((int)m, tb, rec_bb, plist + at);
    return front && at + m >= TS_FRONT;
  });
  if (t == 0) {
    prog->done = end.done;
    prog->next = end.next;
    prog->kmax = kmax;
    *ready = lo + end.done;
  }
}

// Persistent blocks over the long tiles, then over the medium ones.
__global__ void __launch_bounds__(TS_THREADS, 2)
    k_tile_sort(const uint32_t* tvals, uint32_t* xk, const uint32_t* s_dkey, const uint32_t* ranges,
                const TileOrder order, unsigned int* work, uint32_t* ready, TileProg* prog, uint32_t lazy,
                const __grid_constant__ ViewSet vs, const uint2* rec_bb, uint2* plist) {
  grid_begin();
  TileLongSmem& M = ts_smem();
  static_assert(TILE_CLASS_SHORT == 5 && TS_CHUNK == 4096 && TW_MAX == 256, "the length classes");
  unsigned int total = 0;
#pragma unroll
  for (int c = 0; c < TILE_CLASS_SHORT; ++c) total += order.count[c];
  while (true) {
    if (threadIdx.x == 0) M.s.item = atomicAdd(work, 1u);
    __syncthreads();
    const unsigned int item = M.s.item;
    __syncthreads();  // everyone has read the item before it is overwritten
    if (item >= total) return;  // block-uniform
    int cls;
    const uint32_t tile = order.tile(item, &cls);
    const uint2 r = reinterpret_cast<const uint2*>(ranges)[tile];
    const TileBox tb(vs, tile);
    if (cls == 0)
      tl_order<true>(r.x, r.y - r.x, lazy, tvals, xk, s_dkey, prog + tile, ready + tile, tb, rec_bb, plist);
    else
      ts_sort_list(tvals + r.x, s_dkey, (int)(r.y - r.x), tb, rec_bb, plist + r.x);
    __syncthreads();
  }
}

// Persistent blocks over the listed long tiles: what k_tile_sort left unsorted.
__global__ void __launch_bounds__(TS_THREADS, 2)
    k_tile_rest(const uint32_t* tvals, uint32_t* xk, const uint32_t* ranges, const uint32_t* list,
                const unsigned int* n_list, unsigned int* work, uint32_t* ready, TileProg* prog,
                const __grid_constant__ ViewSet vs, const uint2* rec_bb, uint2* plist) {
  grid_begin();
  TileLongSmem& M = ts_smem();
  const unsigned int total = *n_list;
  if (total == 0u) return;
  while (true) {
    if (threadIdx.x == 0) M.s.item = atomicAdd(work, 1u);
    __syncthreads();
    const unsigned int item = M.s.item;
    __syncthreads();
    if (item >= total) return;  // block-uniform
    const uint32_t tile = list[item];
    const uint2 r = reinterpret_cast<const uint2*>(ranges)[tile];
    tl_order<false>(r.x, r.y - r.x, 0u, tvals, xk, nullptr, prog + tile, ready + tile, TileBox(vs, tile), rec_bb,
                    plist);
    __syncthreads();
  }
}

// ------------------------------------------------------------------ per-pixel ray
struct Ray {
  float dx, dy, dz;     // unit direction
  float ix, iy, iz;     // 1 / direction (1e30 for a zero component)
  float ax, ay, az;     // |1 / direction|
  float tnear;          // ray parameter of the near plane (camera depth z_near)
};

__device__ __forceinline__ Ray make_ray(const DevView& c, int px, int py) {
  float dcx = __fdiv_rn((float)px + 0.5f - c.cx, c.fx);
  float dcy = __fdiv_rn((float)py + 0.5f - c.cy, c.fy);
  float wx = c.R[0] * dcx + c.R[3] * dcy + c.R[6];
  float wy = c.R[1] * dcx + c.R[4] * dcy + c.R[7];
  float wz = c.R[2] * dcx + c.R[5] * dcy + c.R[8];
  float inv = rsqrtf(wx * wx + wy * wy + wz * wz);
  Ray r;
  r.dx = wx * inv; r.dy = wy * inv; r.dz = wz * inv;
  r.ix = r.dx != 0.f ? __frcp_rn(r.dx) : 1e30f;
  r.iy = r.dy != 0.f ? __frcp_rn(r.dy) : 1e30f;
  r.iz = r.dz != 0.f ? __frcp_rn(r.dz) : 1e30f;
  r.ax = fabsf(r.ix); r.ay = fabsf(r.iy); r.az = fabsf(r.iz);
  r.tnear = c.z_near * (wx * wx + wy * wy + wz * wz) * inv;  // z_near * |(dcx, dcy, 1)|
  return r;
}

// Chord of the ray (origin at the camera) through the box centred at rc
// (relative to the camera) with half-size h, clipped to start at the near
// plane: slab a enters at (rc_a - h sign) / d_a and leaves at (rc_a + h sign) / d_a.
// Identical code in the forward and backward kernels, so both take the same
// hit decisions.
__device__ __forceinline__ bool chord(const Ray& r, float4 g, float& t_in, float& t_out) {
  const float qx = g.x * r.ix, qy = g.y * r.iy, qz = g.z * r.iz;
  t_in = fmaxf(max3(fmaf(-g.w, r.ax, qx), fmaf(-g.w, r.ay, qy), fmaf(-g.w, r.az, qz)), r.tnear);
  t_out = min3(fmaf(g.w, r.ax, qx), fmaf(g.w, r.ay, qy), fmaf(g.w, r.az, qz));
  return t_out > t_in;
}

// local coordinates u = (p - (c - h)) / (2h) = (t d - rc) / (2h) + 1/2 of the
// ray point at t, clamped to [0,1]^3, and the trilinear density there
__device__ __forceinline__ float trilin(const Ray& r, float4 g, float4 d0, float4 d1, float i2h, float t, float* u) {
  u[0] = __saturatef(fmaf(fmaf(t, r.dx, -g.x), i2h, 0.5f));
  u[1] = __saturatef(fmaf(fmaf(t, r.dy, -g.y), i2h, 0.5f));
  u[2] = __saturatef(fmaf(fmaf(t, r.dz, -g.z), i2h, 0.5f));
  float c00 = fmaf(u[0], d0.y - d0.x, d0.x);
  float c10 = fmaf(u[0], d0.w - d0.z, d0.z);
  float c01 = fmaf(u[0], d1.y - d1.x, d1.x);
  float c11 = fmaf(u[0], d1.w - d1.z, d1.z);
  float c0 = fmaf(u[1], c10 - c00, c00);
  float c1 = fmaf(u[1], c11 - c01, c01);
  return fmaf(u[2], c1 - c0, c0);
}

// Raw density of a sample: the trilinear field at the chord midpoint (u[0..2]),
// or, for the exact-segment variant (SEG), its mean over the chord: along a
// line the field is a cubic in t, so Simpson's rule (f_in + 4 f_mid + f_out) / 6
// is exact (u[3..5] at t_in, u[6..8] at t_out).
template <bool SEG>
__device__ __forceinline__ float sample_density(const Ray& r, float4 g, float4 d0, float4 d1, float i2h, float t_in,
                                                float tm, float t_out, float* u) {
  const float fm = trilin(r, g, d0, d1, i2h, tm, u);
  if constexpr (!SEG) {
    return fm;
  } else {
    const float fa = trilin(r, g, d0, d1, i2h, t_in, u + 3);
    const float fb = trilin(r, g, d0, d1, i2h, t_out, u + 6);
    return (fa + 4.f * fm + fb) * (1.f / 6.f);
  }
}

// v[c] = s * (trilinear weight of corner c at u), or += with ADD
template <bool ADD>
__device__ __forceinline__ void corner_weights(float* v, float s, const float* u) {
  const float ux = u[0], uy = u[1], uz = u[2];
  const float mx = 1.f - ux, my = 1.f - uy, mz = 1.f - uz;
  const float a00 = s * my * mz, a10 = s * uy * mz, a01 = s * my * uz, a11 = s * uy * uz;
  const float w[8] = {mx * a00, ux * a00, mx * a10, ux * a10, mx * a01, ux * a01, mx * a11, ux * a11};
#pragma unroll
  for (int c = 0; c < 8; ++c) v[c] = ADD ? v[c] + w[c] : w[c];
}

// 1 - exp(-x) given e = exp(-x): a 5-term series below 1/8 (relative error
// < 5e-8 there), 1 - e above; branch-free
__device__ __forceinline__ float one_minus_exp(float x, float e) {
  float p = fmaf(x, -1.f / 120.f, 1.f / 24.f);
  p = fmaf(x, p, -1.f / 6.f);
  p = fmaf(x, p, 0.5f);
  p = fmaf(x, -p, 1.f);
  p *= x;
  return x < 0.125f ? p : 1.f - e;
}

__device__ __forceinline__ int find_view(const ViewSet& vs, int gtile) {
  int v = 0;
  while (v + 1 < vs.n && gtile >= vs.v[v + 1].tile_off) ++v;
  return v;
}

// The pixels of a warp form a 4 x 8 block of its tile (rows x columns; the
// warps of a TS x TS tile are laid out TS/8 across and TS/4 down, lanes
// row-major inside the block, so pixel ids grow with the lane).  Compared with
// a 2 x 16 strip, a small voxel's footprint meets fewer warps and more lanes
// of each.  A record whose conservative pixel box misses the block cannot be
// hit by any lane, so the whole warp skips it (a warp-uniform branch); the hit
// decisions are exactly those of the per-lane chord test.
template <int TS>
struct Strip {
  uint32_t x0, x1, y0, y1;  // [x0, x1) x [y0, y1) in image pixels
  __device__ __forceinline__ Strip(int tile_x, int tile_y, int warp) {
    x0 = (uint32_t)(tile_x * TS + (warp % (TS / 8)) * 8);
    x1 = x0 + 8;
    y0 = (uint32_t)(tile_y * TS + (warp / (TS / 8)) * 4);
    y1 = y0 + 4;
  }
  __device__ __forceinline__ int px(int lane) const { return (int)x0 + (lane & 7); }
  __device__ __forceinline__ int py(int lane) const { return (int)y0 + (lane >> 3); }
};

// Work items are (tile, warp strip) pairs, item = position in the tile order * (TS*TS/32) + strip.
// Without PERSIST every warp takes the item of its own block and warp index;
// with PERSIST a grid sized to the resident warps loops, each warp taking the
// next item from a global counter (one atomicAdd per item, no waiting), so a
// warp that finishes a cheap strip moves on without waiting for its block.
__device__ __forceinline__ uint32_t next_item(unsigned int* work, int lane) {
  uint32_t it = 0;
  if (lane == 0) it = atomicAdd(work, 1u);
  return __shfl_sync(FULL, it, 0);
}
// the same for a block of CW warps, which take CW items together (every thread calls)
template <int CW>
__device__ __forceinline__ uint32_t next_items(unsigned int* work) {
  __shared__ uint32_t s_at;
  __syncthreads();  // the last items' number is read
  if (threadIdx.x == 0) s_at = atomicAdd(work, 1u);
  __syncthreads();
  return s_at * CW + (threadIdx.x >> 5);
}

// A persistent grid limited to sm_cut of the n_sms SMs (0: all) is launched at
// full size; a block that lands on an SM outside the first sm_cut (by SM id,
// scaled to the id range) returns at once, so the kept SMs hold their full
// share of blocks and the others stay free for concurrent streams.  The work
// counter hands every item to the blocks that stay.
__device__ __forceinline__ bool sm_excluded(int sm_cut, int n_sms) {
  if (sm_cut <= 0) return false;
  uint32_t smid, nsmid;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
  asm volatile("mov.u32 %0, %%nsmid;" : "=r"(nsmid));
  return (unsigned long long)smid * (unsigned)n_sms >= (unsigned long long)sm_cut * nsmid;
}

// Whether this block of a grid cut to sm_cut SMs leaves at once.  Some block must
// stay, or the work counter's items would be taken by nobody (every block could
// land on an excluded SM while streams of higher priority hold the kept ones), so
// each block counts its arrival in *arrivals (zero before the launch; a block on
// a kept SM adds 1 << 16 as well), and the grid's last block to arrive stays,
// wherever it runs, when no block before it stayed.  Called by every thread of
// the block (block barrier); grids of up to 65535 blocks.
__device__ __forceinline__ bool sm_leave(int sm_cut, int n_sms, unsigned int* arrivals) {
  if (sm_cut <= 0) return false;  // grid-uniform
  __shared__ int s_leave;
  if (threadIdx.x == 0) {
    const bool excl = sm_excluded(sm_cut, n_sms);
    const unsigned int old = atomicAdd(arrivals, excl ? 1u : 0x10001u);
    const bool last_alone = (old & 0xffffu) == gridDim.x - 1 && (old >> 16) == 0;
    s_leave = excl && !last_alone;
  }
  __syncthreads();
  return s_leave != 0;
}

// ------------------------------------------------------------------ forward composite
// Each warp walks its strip's list on its own, with no block-wide barrier, and
// stops as soon as all its pixels have.  The list entries carry the strips they
// meet, so a warp reads a round of them at a time (coalesced 8-byte words,
// three or four per lane) and queues the few that meet its strip; the records of a
// batch of queued entries are then copied to shared memory and every lane marches
// its pixel through them.  A pixel that stays open walks thousands of entries, and
// the walk is then one serial chain per warp, so its memory latency is taken out
// of the chain: the entries of the next round are loaded before they are needed,
// and the records of the next batch are copied (cp.async) while the current ones are
// marched.  The rounds and batches are the same for every lv_raster_opts.batch.
//
// Where strips fill the SMs the composites are bound by instruction issue, and in an
// opaque scene most strips stop within some 20 records, so what is read, copied and
// computed ahead is wasted: the first batch takes 16 records and more only if the round
// holds them, the forward copies nothing ahead before that is marched, a march ends
// where its last pixel does, and a record's chord is computed when its turn comes.  One
// 1237 x 822 view of 2M opaque voxels, tile 16, forward (with statistics) + backward:
// 62M + 99M warp instructions, 75 + 109 us, against 84M + 111M and 91 + 123 us with
// batches of 32 copied ahead from the start and every chord a record ahead.
// With LOOK they look ahead like that: where few strips are in flight the latency of one
// march counts, and the next record's chord does not wait for a sample (256 x 256 view of
// an open scene, 2048 strips: 1.57 ms against 1.76).
//
// per-warp slice of shared memory: two buffers of 32 records (64 B), voxel ids and
// (slot, list entry), and the queue: at most 31 entries left over and one round of new ones
template <bool LOOK>
struct WalkShape {
  static constexpr int ENTRIES = LOOK ? 128 : 96;
  static constexpr uint32_t FIRST = LOOK ? 32 : 16;
  static constexpr int QUEUE = LOOK ? 256 : 128;
  static constexpr size_t SLICE = 2 * 32 * (64 + 4 + 8) + (size_t)QUEUE * 8;
  static_assert(31 + ENTRIES <= QUEUE, "the queue holds every waiting entry");
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The records of one strip in list order (REV: from the last entry to the
// first), a batch of up to 32 at a time.  All members are called by the whole warp.
template <bool REV, bool LOOK>
struct StripWalk {
  using Shape = WalkShape<LOOK>;
  static constexpr int K = Shape::ENTRIES / 32;
  static constexpr uint32_t QM = Shape::QUEUE - 1;
  const uint2* plist;
  const float4* rec;
  const uint32_t* slot_vox;
  float4* s_rec;     // [2][32][4]
  uint32_t* s_vox;   // [2][32]
  uint2* s_ent;      // [2][32] (slot, entry)
  uint2* s_q;        // (slot, entry)
  uint32_t lo, hi;   // entries [lo, hi) not scanned yet, those in `ahead` not counted
  uint32_t base;     // first entry of `ahead`
  uint2 ahead[K];
  uint32_t head, tail;  // queue positions: next to copy, next to fill
  uint32_t want;        // records that a batch waits for
  uint32_t bit;
  bool live;            // `ahead` holds entries not queued yet
  int lane;

  __device__ __forceinline__ StripWalk(const uint2* plist_, const float4* rec_, const uint32_t* slot_vox_,
                                       char* smem, int warp, int lane_)
      : plist(plist_), rec(rec_), slot_vox(slot_vox_), lane(lane_) {
    s_rec = (float4*)(smem + Shape::SLICE * warp);
    s_vox = (uint32_t*)(s_rec + 2 * 32 * 4);
    s_ent = (uint2*)(s_vox + 2 * 32);
    s_q = s_ent + 2 * 32;
  }
  __device__ __forceinline__ void load_ahead() {
    const uint32_t r = min((uint32_t)Shape::ENTRIES, hi - lo);
    base = REV ? hi - r : lo;
    const uint2* p = plist + (base + lane);
#pragma unroll
    for (int k = 0; k < K; ++k) ahead[k] = 32 * k + lane < r ? p[32 * k] : make_uint2(0u, 0u);
    if (REV) hi = base;
    else lo += r;
  }
  __device__ __forceinline__ void begin(uint32_t start, uint32_t end, int strip) {
    lo = start;
    hi = end;
    head = tail = 0u;
    want = Shape::FIRST;
    bit = 1u << strip;
    live = start < end;
    load_ahead();
  }
  // queue entries until a batch of them waits or the list ends
  __device__ __forceinline__ void fill() {
    while (tail - head < want && live) {
      const uint32_t b = base;
      uint2 cur[K];
#pragma unroll
      for (int k = 0; k < K; ++k) cur[k] = ahead[k];
      live = lo < hi;
      if (live) load_ahead();
#pragma unroll
      for (int kk = 0; kk < K; ++kk) {
        const int k = REV ? K - 1 - kk : kk;
        const bool in = (cur[k].y & bit) != 0u;
        const uint32_t m = __ballot_sync(FULL, in);
        if (in) {
          const uint32_t before = REV ? m & (0xfffffffeu << lane) : m & ((1u << lane) - 1u);
          s_q[(tail + __popc(before)) & QM] = make_uint2(cur[k].x, b + 32 * k + lane);
        }
        tail += __popc(m);
      }
    }
    __syncwarp();
  }
  // start copying the next batch's records into buffer b; returns their number
  __device__ __forceinline__ int copy(int b) {
    const int m = (int)min(32u, tail - head);
    want = 32u;
    if (m) {
      // four lanes per record: a record's 64 bytes in one request
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int r = 8 * k + (lane >> 2);
        if (r < m) {
          const uint32_t sl = s_q[(head + r) & QM].x;
          cp_async16(s_rec + 128 * b + 4 * r + (lane & 3), rec + 4 * (size_t)sl + (lane & 3));
        }
      }
      if (lane < m) {
        const uint2 e = s_q[(head + lane) & QM];
        cp_async4(s_vox + 32 * b + lane, slot_vox + e.x);
        s_ent[32 * b + lane] = e;
      }
      __syncwarp();  // the queue's words are read before they are filled again
    }
    cp_async_commit();
    head += m;
    return m;
  }
};

// The LF-weighted loss fused into the backward composite (Sec. IV-B, Eq. 8 and
// 18): per pixel dL/drgb = 2 / (3 |P_v|) * (w / <w>) * (rgb - gt), in the
// operation order lv_lf_loss_from_weights uses, and the view's summed
// weighted squared error (FP32 per warp item, FP64 per warp in shared memory,
// summed per block, one global FP64 atomic per block and view into one of
// LF_SLOTS sums; a block is 1 to 8 warps, and with one sum a view and each view's
// constants computed in every block 16 views took 1708 us instead of 1608).
// w == nullptr: not fused.
struct LfFuse {
  const float* rgb;    // [P][3] the forward's image
  const float* gt;     // [P][3]
  const float* w;      // [P] unnormalised weights (lv_lf_weights)
  const double* wsum;  // [views] their sums
  const float2* view_k;  // [views] mean weight, gradient scale
  double* lsum;        // [LF_SLOTS][LV_MAX_VIEWS] loss sums
  float* dL;           // [P][3] dL/drgb, also written out (nullable)
};

// The composite of a list's sorted part and, for the tiles whose pixels were
// still open at its end, of the rest in a second launch (resume): the pixels'
// sums are read back from the outputs (the depth and the sample count, which a
// caller may not want, from dep and nsamp) and the march goes on where it
// stopped, so the results are those of one march.
struct Front {
  uint32_t* ready;
  TileProg* prog;
  uint32_t* open_tiles;
  unsigned int* n_open;
  float* dep;
  uint32_t* nsamp;
};

// A strip's march needs no other warp, so a block is a few warps whatever the
// tile size, few where each warp has one item (a block's place is free once its
// last warp ends).  Blocks of 4 share their tile's list entries and records in L1, so the
// persistent forward takes 4 items at a time as well, with a barrier (an item per warp
// and atomic, 8 warps a block: 97 us against 88 on an opaque view, 578 against 559 on an
// open one, tile 32); the persistent backward, whose strips differ more, takes single items.
// As many blocks share an SM as leave a thread 64 (forward) and 72 (backward)
// registers: with fewer the march spills (at these the exact-segment forward of
// tile 8, 28 bytes), with more too few warps hide the memory's latency.  1237 x 822 views of 2M voxels, opaque and open, tile 16, forward:
// 78 and 494 us at 72 registers, 74 and 490 at 64, 77 and 499 at 56; backward 115 and 714 us
// at 80, 109 and 684 at 72, 115 and 715 at 64.  Looking ahead takes 8 more of them.
template <int TS, bool PERSIST, bool LOOK>
__host__ __device__ constexpr int fwd_warps() { return PERSIST ? (LOOK ? 8 : 4) : (TS == 8 ? 1 : 4); }
template <int TS, bool PERSIST, bool LOOK>
__host__ __device__ constexpr int fwd_blocks() { return (LOOK ? 28 : 32) / fwd_warps<TS, PERSIST, LOOK>(); }
template <int TS, bool PERSIST>
__host__ __device__ constexpr int bwd_warps() { return PERSIST ? 8 : (TS == 8 ? 1 : 4); }
template <int TS, bool PERSIST, bool LOOK>
__host__ __device__ constexpr int bwd_blocks() { return (PERSIST || LOOK ? 24 : 28) / bwd_warps<TS, PERSIST>(); }

template <int TS, bool SEG, bool PERSIST, bool LOOK>
__global__ void __launch_bounds__(fwd_warps<TS, PERSIST, LOOK>() * 32, fwd_blocks<TS, PERSIST, LOOK>())
    k_fwd(const __grid_constant__ ViewSet vs, const uint32_t* ranges, const uint2* plist, const float4* rec,
          const uint32_t* slot_vox, float t_stop, float* rgb, float* depth, float* T_out, uint32_t* n_contrib,
          uint32_t* n_samples, float* tau_out, unsigned long long* wmax, unsigned int* work, uint32_t n_items,
          int sm_cut, int n_sms, unsigned int* arrivals, const TileOrder order, const Front fr) {
  grid_wait();
  constexpr int NW = TS * TS / 32, CW = fwd_warps<TS, PERSIST, LOOK>();
  constexpr bool RESUME = PERSIST && LOOK;  // the second launch, over the open tiles
  extern __shared__ float4 smem_f4[];
  if (PERSIST && sm_leave(sm_cut, n_sms, arrivals)) return;  // block-uniform
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (RESUME) {
    n_items = *fr.n_open * NW;
    if (n_items == 0u) return;
  }
  StripWalk<false, LOOK> walk(plist, rec, slot_vox, (char*)smem_f4, warp, lane);
  constexpr bool BY_BLOCK = PERSIST && !RESUME;  // items taken CW at a time
  auto next = [&]() {
    return BY_BLOCK ? next_items<CW>(work) : (PERSIST ? next_item(work, lane) : n_items);
  };
  for (uint32_t item = PERSIST ? next() : blockIdx.x * CW + warp; item - (BY_BLOCK ? warp : 0) < n_items;
       item = next()) {  // warp-uniform
    if (BY_BLOCK && item >= n_items) continue;
    const int gtile = RESUME ? (int)fr.open_tiles[item / NW] : (int)order.tile(item / NW);
    const int view = find_view(vs, gtile);
    const DevView& c = vs.v[view];
    const uint32_t start = ranges[2 * gtile], end = fr.ready[gtile];
    walk.begin(RESUME ? fr.prog[gtile].front : start, end, (int)(item % NW));
    const int lt = gtile - c.tile_off;
    const int tile_x = lt % c.tiles_x, tile_y = lt / c.tiles_x;
    const Strip<TS> strip(tile_x, tile_y, (int)(item % NW));
    const int px = strip.px(lane), py = strip.py(lane);
    const bool inside = px < c.W && py < c.H;
    const Ray r = make_ray(c, px, py);
    const unsigned long long gid = (unsigned long long)(c.pix_off + (long long)py * c.W + px);
    const unsigned long long gid_key = 0xffffffffull - ((gid + (unsigned long long)vs.id_base) & 0xffffffffull);
    float T = 1.f, tau = 0.f, cr = 0.f, cg = 0.f, cb = 0.f, dep = 0.f;
    uint32_t last = 0, nsamp = 0;
    bool done = !inside;
    if (RESUME) {
      if (inside) {
        const size_t p = (size_t)gid;
        T = T_out[p];
        done = T < t_stop;
      }
      if (__all_sync(FULL, done)) continue;  // the strip stopped within the front
      if (inside) {
        const size_t p = (size_t)gid;
        cr = rgb[3 * p + 0];
        cg = rgb[3 * p + 1];
        cb = rgb[3 * p + 2];
        dep = fr.dep[p];
        tau = tau_out[p];
        last = n_contrib[p];
        nsamp = fr.nsamp[p];
      }
    }
    walk.fill();
    int m = walk.copy(0);
    bool ahead = LOOK;  // batches are copied ahead from the second one on
    for (int b = 0; m; b ^= 1) {  // warp-uniform
      int m_next = 0;
      if (ahead) {
        walk.fill();
        m_next = walk.copy(b ^ 1);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncwarp();
      const float4* wr = walk.s_rec + 128 * b;
      const uint32_t* w_vox = walk.s_vox + 32 * b;
      int last_j = -1;  // the lane's last sample of this batch (its list entry is read once, below)
      float4 g_n;
      float in_n, out_n;
      bool h_n = false;
      if (LOOK) {
        g_n = wr[0];
        h_n = chord(r, g_n, in_n, out_n);
      }
      for (int j = 0; j < m; ++j) {
        float4 g;
        float t_in, t_out;
        bool hit;
        if (LOOK) {
          hit = h_n && !done;
          g = g_n;
          t_in = in_n;
          t_out = out_n;
          // (past the last record: whatever follows in the slice, and the result is not used)
          g_n = wr[4 * (j + 1)];
          h_n = chord(r, g_n, in_n, out_n);
        } else {
          g = wr[4 * j];
          hit = chord(r, g, t_in, t_out) && !done;
        }
        if (!__any_sync(FULL, hit)) {
          if (!LOOK && __all_sync(FULL, done)) break;
          continue;
        }
        float w = 0.f;
        if (hit) {
          const float4 d0 = wr[4 * j + 1], d1 = wr[4 * j + 2], col = wr[4 * j + 3];
          const float l = t_out - t_in, tm = 0.5f * (t_in + t_out);
          float u[SEG ? 9 : 3];
          const float sigma = fmaxf(sample_density<SEG>(r, g, d0, d1, col.w, t_in, tm, t_out, u), 0.f);
          const float x = sigma * l;
          const float ex = __expf(-x);
          const float alpha = one_minus_exp(x, ex);
          w = T * alpha;
          cr = fmaf(w, col.x, cr);
          cg = fmaf(w, col.y, cg);
          cb = fmaf(w, col.z, cb);
          dep = fmaf(w, tm, dep);
          tau += x;
          T *= ex;
          last_j = j;
          ++nsamp;
          done = T < t_stop;
        }
        if (wmax) {  // grid-uniform
          // the warp's largest w (ties to the lowest lane = smallest pixel id), one global atomic
          const uint32_t v = hit ? __float_as_uint(w) + 1u : 0u;
          const uint32_t mx = __reduce_max_sync(FULL, v);
          const uint32_t who = __ballot_sync(FULL, v == mx);
          if (lane == __ffs(who) - 1)
            atomicMax(&wmax[w_vox[j]], ((unsigned long long)(mx - 1u) << 32) | gid_key);
        }
      }
      if (last_j >= 0) last = walk.s_ent[32 * b + last_j].y - start + 1;
      if (__all_sync(FULL, done)) break;
      __syncwarp();  // the buffer is copied into next
      if (!ahead) {
        ahead = true;
        walk.fill();
        m_next = walk.copy(b ^ 1);
      }
      m = m_next;
    }
    cp_async_wait<0>();  // a batch copied ahead of the stop
    // a long list sorted only so far, and pixels that go on: listed for k_tile_rest and the second launch
    const bool open = end < ranges[2 * gtile + 1] && !__all_sync(FULL, done);
    if (open && lane == 0 && atomicExch(&fr.prog[gtile].open, 1u) == 0u) {
      fr.prog[gtile].front = end;
      fr.open_tiles[atomicAdd(fr.n_open, 1u)] = (uint32_t)gtile;
    }
    if (inside) {
      if (open) {
        fr.dep[gid] = dep;
        fr.nsamp[gid] = nsamp;
      }
      const size_t p = (size_t)gid;
      rgb[3 * p + 0] = cr;
      rgb[3 * p + 1] = cg;
      rgb[3 * p + 2] = cb;
      if (depth) depth[p] = dep;
      T_out[p] = T;
      n_contrib[p] = last;
      if (n_samples) n_samples[p] = nsamp;
      tau_out[p] = tau;
    }
    __syncwarp();  // the slice is reused by the next item
  }
}

// ------------------------------------------------------------------ backward composite
// Transposed butterfly: after 16 shuffles even lane l holds the warp sum of
// value (l >> 1) of the 16 inputs (instead of 16 * 5 shuffles).
__device__ __forceinline__ float warp_reduce16(float* v, int lane) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const bool up = lane & 16;
    float send = up ? v[i] : v[i + 8];
    float keep = up ? v[i + 8] : v[i];
    v[i] = keep + __shfl_xor_sync(FULL, send, 16);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool up = lane & 8;
    float send = up ? v[i] : v[i + 4];
    float keep = up ? v[i + 4] : v[i];
    v[i] = keep + __shfl_xor_sync(FULL, send, 8);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const bool up = lane & 4;
    float send = up ? v[i] : v[i + 2];
    float keep = up ? v[i + 2] : v[i];
    v[i] = keep + __shfl_xor_sync(FULL, send, 4);
  }
  {
    const bool up = lane & 2;
    float send = up ? v[0] : v[1];
    float keep = up ? v[1] : v[0];
    v[0] = keep + __shfl_xor_sync(FULL, send, 2);
  }
  return v[0] + __shfl_xor_sync(FULL, v[0], 1);
}

// Backward: each warp walks its strip's list back to front from the last entry
// any of its pixels used, through the same queue and copies as the forward; the
// per-record gradients (8 corners + colour) are
// reduced over the warp and sent with three 16-byte global reductions.
template <int TS, bool SEG, bool PERSIST, bool LOOK>
__global__ void __launch_bounds__(bwd_warps<TS, PERSIST>() * 32, bwd_blocks<TS, PERSIST, LOOK>())
    k_bwd(const __grid_constant__ ViewSet vs, const uint32_t* __restrict__ ranges, const uint2* __restrict__ plist,
          const float4* __restrict__ rec, const uint32_t* __restrict__ slot_vox, const float* __restrict__ T_fwd,
          const float* __restrict__ tau_in, const uint32_t* __restrict__ n_contrib, const float* __restrict__ dL_drgb,
          const float* __restrict__ dL_ddepth, const float* __restrict__ dL_dT, float* __restrict__ d_density,
          float4* __restrict__ d_rgb, unsigned int* work, uint32_t n_items, int sm_cut, int n_sms,
          unsigned int* arrivals, const TileOrder order, const LfFuse lf) {
  grid_wait();
  constexpr int NW = TS * TS / 32, CW = bwd_warps<TS, PERSIST>();
  extern __shared__ float4 smem_f4[];
  __shared__ double s_lf[CW][LV_MAX_VIEWS];  // each warp's loss sums (fused LF loss; no atomics)
  // view_k, computed by a block of many items (reading it there: +1.5 % with 16 views)
  __shared__ float2 s_vk[PERSIST ? LV_MAX_VIEWS : 1];
  if (PERSIST && sm_leave(sm_cut, n_sms, arrivals)) return;  // block-uniform
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (lf.w) {  // grid-uniform; a warp clears and then adds to its own row only
    for (int v = lane; v < vs.n; v += 32) s_lf[warp][v] = 0.0;
    if (PERSIST) {
      for (int v = tid; v < vs.n; v += CW * 32) {
        const double np = (double)vs.v[v].W * (double)vs.v[v].H;
        s_vk[v] = make_float2((float)(lf.wsum[v] / np), (float)(2.0 / (3.0 * np)));
      }
      __syncthreads();
    } else {
      __syncwarp();
    }
  }
  StripWalk<true, LOOK> walk(plist, rec, slot_vox, (char*)smem_f4, warp, lane);
  for (uint32_t item = PERSIST ? next_item(work, lane) : blockIdx.x * CW + warp; item < n_items;
       item = PERSIST ? next_item(work, lane) : n_items) {  // warp-uniform
    const int gtile = (int)order.tile(item / NW);
    const int view = find_view(vs, gtile);
    const DevView& c = vs.v[view];
    const int lt = gtile - c.tile_off;
    const int tile_x = lt % c.tiles_x, tile_y = lt / c.tiles_x;
    const Strip<TS> strip(tile_x, tile_y, (int)(item % NW));
    const int px = strip.px(lane), py = strip.py(lane);
    const bool inside = px < c.W && py < c.H;
    const Ray r = make_ray(c, px, py);
    const uint32_t start = ranges[2 * gtile];
    const size_t p = (size_t)(c.pix_off + (long long)py * c.W + px);
    uint32_t nc = 0;
    float tau = 0.f, Tf = 1.f, gr = 0.f, gg = 0.f, gb = 0.f, gD = 0.f, gT = 0.f;
    if (inside) {
      nc = n_contrib[p];
      tau = tau_in[p];
      Tf = T_fwd[p];
      if (!lf.w) {
        gr = dL_drgb[3 * p + 0];
        gg = dL_drgb[3 * p + 1];
        gb = dL_drgb[3 * p + 2];
      }
      if (dL_ddepth) gD = dL_ddepth[p];
      if (dL_dT) gT = dL_dT[p];
    }
    if (lf.w) {  // grid-uniform: dL/drgb of the LF-weighted loss from the forward's image
      const float2 vk = PERSIST ? s_vk[view] : lf.view_k[view];
      const float mean = vk.x, gscale = vk.y;
      float part = 0.f;
      if (inside) {
        const float wt = lf.w[p] / mean;
        const float r0 = lf.rgb[3 * p] - lf.gt[3 * p], r1 = lf.rgb[3 * p + 1] - lf.gt[3 * p + 1],
                    r2 = lf.rgb[3 * p + 2] - lf.gt[3 * p + 2];
        part = wt * (r0 * r0 + r1 * r1 + r2 * r2);
        const float cf = gscale * wt;
        gr = cf * r0;
        gg = cf * r1;
        gb = cf * r2;
        if (lf.dL) {
          lf.dL[3 * p + 0] = gr;
          lf.dL[3 * p + 1] = gg;
          lf.dL[3 * p + 2] = gb;
        }
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
      if (lane == 0) s_lf[warp][view] += (double)part;
    }
    const uint32_t my_hi = start + nc;  // entries [start, my_hi) were used by this pixel
    const uint32_t warp_hi = start + __reduce_max_sync(FULL, nc);
    const float tgT = Tf * gT;
    float S = 0.f;
    float Tcur = __expf(-tau);  // T after the last sample, from the stored optical depth
    walk.begin(start, warp_hi, (int)(item % NW));
    walk.fill();
    int m = walk.copy(0);
    for (int b = 0; m; b ^= 1) {  // warp-uniform
      walk.fill();
      const int m_next = walk.copy(b ^ 1);
      cp_async_wait<1>();
      __syncwarp();
      const float4* wr = walk.s_rec + 128 * b;
      const uint32_t* w_vox = walk.s_vox + 32 * b;
      const uint2* w_ent = walk.s_ent + 32 * b;
      float4 g_n;
      uint2 ent_n;
      float in_n, out_n;
      bool h_n = false;
      if (LOOK) {
        g_n = wr[0];
        ent_n = w_ent[0];
        h_n = chord(r, g_n, in_n, out_n) && ent_n.y < my_hi;
      }
      for (int j = 0; j < m; ++j) {
        float4 g;
        uint2 ent;
        float t_in, t_out;
        bool hit;
        if (LOOK) {
          hit = h_n;
          g = g_n;
          ent = ent_n;
          t_in = in_n;
          t_out = out_n;
          // (past the last record: whatever follows in the slice, and the result is not used)
          g_n = wr[4 * (j + 1)];
          ent_n = w_ent[j + 1];
          h_n = chord(r, g_n, in_n, out_n) && ent_n.y < my_hi;
        } else {
          g = wr[4 * j];
          ent = w_ent[j];
          hit = chord(r, g, t_in, t_out) && ent.y < my_hi;
        }
        const uint32_t slot = ent.x;
        const unsigned hb = __ballot_sync(FULL, hit);
        if (!hb) continue;
        float v[16];
  #pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = 0.f;
        if (hit) {
          const float4 d0 = wr[4 * j + 1], d1 = wr[4 * j + 2], col = wr[4 * j + 3];
          const float l = t_out - t_in, tm = 0.5f * (t_in + t_out);
          float u[SEG ? 9 : 3];
          const float sraw = sample_density<SEG>(r, g, d0, d1, col.w, t_in, tm, t_out, u);
          const float sigma = fmaxf(sraw, 0.f);
          const float x = sigma * l;
          const float Tk = Tcur;  // transmittance after this sample: the previous step's T_prev
          const float tau_prev = fmaxf(tau - x, 0.f);
          const float T_prev = __expf(-tau_prev);
          Tcur = T_prev;
          const float alpha = one_minus_exp(x, __expf(-x));
          const float w = T_prev * alpha;
          const float a = fmaf(gr, col.x, fmaf(gg, col.y, fmaf(gb, col.z, gD * tm)));
          const float ds = l * (Tk * a - S - tgT);
          S = fmaf(w, a, S);
          tau = tau_prev;
          const float dr = sraw > 0.f ? ds : 0.f;
          corner_weights<false>(v, SEG ? dr * (4.f / 6.f) : dr, u);
          if constexpr (SEG) {
            corner_weights<true>(v, dr * (1.f / 6.f), u + 3);
            corner_weights<true>(v, dr * (1.f / 6.f), u + 6);
          }
          v[8] = w * gr;
          v[9] = w * gg;
          v[10] = w * gb;
        }
        float* dd = d_density + 8 * (size_t)w_vox[j];
        float* dc = (float*)(d_rgb + slot);
        if (__popc(hb) <= 8) {
          // up to eight lanes: each sends its own values, cheaper than the butterfly (measured: 8 lanes
          // 2 % faster than 2; every lane, 12x slower, the reductions to one address serialise)
          if (hit) {
            red_add_v4(dd, v[0], v[1], v[2], v[3]);
            red_add_v4(dd + 4, v[4], v[5], v[6], v[7]);
            red_add_v4(dc, v[8], v[9], v[10], 0.f);
          }
        } else {
          const float sum = warp_reduce16(v, lane);  // value (l >> 1) on even lane l
          // gather four values each into lanes 0 (corners 0-3), 1 (corners 4-7) and 2 (colour)
          const int src0 = lane == 0 ? 0 : (lane == 1 ? 8 : 16);
          const float q0 = __shfl_sync(FULL, sum, src0 + 0);
          const float q1 = __shfl_sync(FULL, sum, src0 + 2);
          const float q2 = __shfl_sync(FULL, sum, src0 + 4);
          const float q3 = __shfl_sync(FULL, sum, src0 + 6);
          if (lane == 0) red_add_v4(dd, q0, q1, q2, q3);
          else if (lane == 1) red_add_v4(dd + 4, q0, q1, q2, q3);
          else if (lane == 2) red_add_v4(dc, q0, q1, q2, 0.f);
        }
      }
      m = m_next;
      __syncwarp();  // the buffer is copied into next
    }
    cp_async_wait<0>();
    __syncwarp();  // the slice is reused by the next item
  }
  if (lf.w) {
    __syncthreads();
    for (int v = tid; v < vs.n; v += CW * 32) {
      double t = 0.0;
      for (int w = 0; w < CW; ++w) t += s_lf[w][v];
      if (t != 0.0) atomicAdd(&lf.lsum[(blockIdx.x % LF_SLOTS) * LV_MAX_VIEWS + v], t);
    }
  }
}

// ------------------------------------------------------------------ SH backward
// A warp handles 32 consecutive voxels, one per lane.  d c / d SH_j = Y_j(dir)
// where the clamp c = max(0, SH + 0.5) passed; the forward left that per-channel
// mask in the w component of the slot's colour-gradient scratch, so the SH rows
// themselves are not read again.  Each lane sums its voxel's gradients over the
// views; the 32 rows leave through shared memory as coalesced 16-byte stores
// (row stride 49 floats: conflict-free per lane).  With `accumulate`, warps
// without any visible voxel touch nothing.
__global__ void __launch_bounds__(128)
    k_sh_bwd(const float4* __restrict__ rec, int sh_nb, int64_t n, const __grid_constant__ ViewSet vs,
             const uint32_t* __restrict__ cnt, const uint32_t* __restrict__ slot, float4* d_rgb, float* d_sh,
             int accumulate) {
  grid_wait();
  constexpr int RS = 49;
  __shared__ float s_rows[4][32 * RS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t v0 = (blockIdx.x * 4 + warp) * (int64_t)32;
  if (v0 >= n) return;  // warp-uniform
  const int nrows = (int)min((int64_t)32, n - v0);
  float* buf = s_rows[warp];
  float acc[48];
#pragma unroll
  for (int k = 0; k < 48; ++k) acc[k] = 0.f;
  bool any_vis = false;
  if (lane < nrows) {
    const int64_t vox = v0 + lane;
    for (int view = 0; view < vs.n; ++view) {
      const int64_t i = (int64_t)view * n + vox;  // view-major items
      if (!cnt[i]) continue;
      any_vis = true;
      const uint32_t s = slot[i];
      // the record holds the centre relative to this view's camera, as k_emit computed it, so the
      // voxel arrays are not read (a topology change may rewrite them meanwhile)
      const float4 g = rec[4 * (int64_t)s];
      float dir[3];
      unit_dir(g.x, g.y, g.z, dir);
      float Y[16];
      sh_basis(dir[0], dir[1], dir[2], Y);
      const float4 dc = d_rgb[s];
      const int m = (int)dc.w;
      const float dr = (m & 1) ? dc.x : 0.f;
      const float dg = (m & 2) ? dc.y : 0.f;
      const float db = (m & 4) ? dc.z : 0.f;
      d_rgb[s] = make_float4(0.f, 0.f, 0.f, dc.w);  // cleared for the next backward call; mask kept
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (j < sh_nb) {
          acc[3 * j + 0] = fmaf(Y[j], dr, acc[3 * j + 0]);
          acc[3 * j + 1] = fmaf(Y[j], dg, acc[3 * j + 1]);
          acc[3 * j + 2] = fmaf(Y[j], db, acc[3 * j + 2]);
        }
      }
    }
  }
  if (accumulate && !__any_sync(FULL, any_vis)) return;  // nothing to add for these 32 voxels
  if (lane < nrows) {
#pragma unroll
    for (int k = 0; k < 48; ++k) buf[lane * RS + k] = acc[k];
  }
  __syncwarp();
  float4* dst = (float4*)(d_sh + 48 * v0);
  for (int w = lane; w < nrows * 12; w += 32) {
    const float* a = buf + (w / 12) * RS + (w % 12) * 4;
    float4 o = make_float4(a[0], a[1], a[2], a[3]);
    if (accumulate) {
      const float4 p = dst[w];
      o.x += p.x; o.y += p.y; o.z += p.z; o.w += p.w;
    }
    dst[w] = o;
  }
}

__global__ void k_unpack_wmax(const unsigned long long* __restrict__ packed, int64_t n, float* __restrict__ w,
                              int64_t* __restrict__ arg) {
  grid_begin();
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  unsigned long long v = packed[i];
  if (v == 0ull) {
    w[i] = 0.f;
    if (arg) arg[i] = -1;
  } else {
    w[i] = __uint_as_float((uint32_t)(v >> 32));
    if (arg) arg[i] = (int64_t)(0xffffffffull - (v & 0xffffffffull));
  }
}

__global__ void k_gather_edge(const int64_t* __restrict__ argmax, int64_t n, const float* __restrict__ edge_map,
                              int64_t n_pix, float* __restrict__ edge) {
  grid_begin();
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t a = argmax[i];
  edge[i] = (a >= 0 && a < n_pix) ? edge_map[a] : 0.f;
}

// The lists of a forward workspace, for the calls that read them whole.  A list the
// forward left partly sorted is put in order in shared memory, by the cuts k_tile_rest
// makes, so these calls only read the workspace and any number may share one.
struct ListView {
  const uint2* ranges;
  const uint32_t* ready;
  const uint2* plist;
  const uint32_t* tile_slots;
  const uint32_t* long_keys;
  const TileProg* prog;
  const uint32_t* slot_vox;
};
// sink as in tl_ranges (`at` counts from the list's start); the whole block calls
template <typename Sink>
__device__ __forceinline__ void list_rest(const ListView& lv, uint32_t tile, uint2 r, Sink&& sink) {
  const TileProg p = lv.prog[tile];
  tl_ranges(r.y - r.x, lv.tile_slots + r.x, lv.long_keys + r.x, p.done, p.next, p.kmax, sink);
}

// a block per tile, in turn
__global__ void __launch_bounds__(TS_THREADS) k_debug_pairs(const ListView lv, int64_t tiles,
                                                           const uint32_t* __restrict__ s_dkey, uint64_t* ko,
                                                           uint32_t* vo) {
  grid_begin();
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const uint2 r = lv.ranges[tile];
    auto put = [&](uint32_t i, uint32_t s) {
      if (ko) ko[i] = ((uint64_t)tile << 32) | s_dkey[s];
      if (vo) vo[i] = lv.slot_vox[s];
    };
    const uint32_t sorted = lv.ready[tile];
    for (uint32_t i = r.x + threadIdx.x; i < sorted; i += TS_THREADS) put(i, lv.plist[i].x);
    if (sorted < r.y)  // block-uniform
      list_rest(lv, (uint32_t)tile, r, [&](uint32_t at, uint32_t m, bool ordered) {
        const TileSortSmem& S = ts_smem().s;
        if (!ordered) {
          ts_sort_smem((int)m);
          __syncthreads();
        }
        for (uint32_t q = threadIdx.x; q < m; q += TS_THREADS) put(r.x + at + q, S.v[q]);
        return false;
      });
  }
}

// ------------------------------------------------------------------ FP64 re-render (gradient checks)
// Each listed pixel's tile list (from a forward workspace) is walked front to
// back in FP64 from the original voxel arrays (geometry, corner densities and SH
// converted exactly to double): the FP64 counterpart of k_fwd, used only to take
// finite differences of the loss.
__device__ __forceinline__ void sh_basis64(double x, double y, double z, double* Y) {
  const double pi = 3.14159265358979323846;
  Y[0] = 0.5 / sqrt(pi);
  const double c1 = sqrt(3.0 / (4.0 * pi));
  Y[1] = c1 * y; Y[2] = c1 * z; Y[3] = c1 * x;
  const double c2a = sqrt(15.0 / (4.0 * pi)), c2b = sqrt(5.0 / (16.0 * pi)), c2c = sqrt(15.0 / (16.0 * pi));
  Y[4] = c2a * x * y; Y[5] = c2a * y * z; Y[6] = c2b * (3.0 * z * z - 1.0); Y[7] = c2a * x * z;
  Y[8] = c2c * (x * x - y * y);
  const double c3a = sqrt(35.0 / (32.0 * pi)), c3b = sqrt(105.0 / (4.0 * pi)), c3c = sqrt(21.0 / (32.0 * pi));
  const double c3d = sqrt(7.0 / (16.0 * pi)), c3e = sqrt(105.0 / (16.0 * pi));
  Y[9] = c3a * y * (3.0 * x * x - y * y); Y[10] = c3b * x * y * z; Y[11] = c3c * y * (5.0 * z * z - 1.0);
  Y[12] = c3d * z * (5.0 * z * z - 3.0); Y[13] = c3c * x * (5.0 * z * z - 1.0); Y[14] = c3e * z * (x * x - y * y);
  Y[15] = c3a * x * (x * x - 3.0 * y * y);
}

// the voxel arrays and options of an FP64 march
template <typename DT, typename ST>
struct Scene64 {
  const float4* geom;
  const DT* dens;
  const ST* sh;
  const uint32_t* vidx;
  int sh_nb, segment;
  double t_stop;
};

// one pixel's FP64 march
struct March64 {
  int gtile;
  double o[3], d[3], t_near;
  double T, cr, cg, cb;

  __device__ March64(const ViewSet& vs, long long gp) {
    int view = 0;
    while (view + 1 < vs.n && gp >= vs.v[view + 1].pix_off) ++view;
    const DevView& c = vs.v[view];
    const long long loc = gp - c.pix_off;
    const int px = (int)(loc % c.W), py = (int)(loc / c.W);
    const int ts = vs.ts;
    gtile = c.tile_off + (py / ts) * c.tiles_x + px / ts;
    for (int k = 0; k < 3; ++k)
      o[k] = -((double)c.R[k] * c.t[0] + (double)c.R[3 + k] * c.t[1] + (double)c.R[6 + k] * c.t[2]);
    const double dcx = ((double)px + 0.5 - (double)c.cx) / (double)c.fx;
    const double dcy = ((double)py + 0.5 - (double)c.cy) / (double)c.fy;
    double nn = 0.0;
    for (int k = 0; k < 3; ++k) {
      d[k] = (double)c.R[k] * dcx + (double)c.R[3 + k] * dcy + (double)c.R[6 + k];
      nn += d[k] * d[k];
    }
    nn = sqrt(nn);
    for (int k = 0; k < 3; ++k) d[k] /= nn;
    t_near = (double)c.z_near * nn;  // camera depth z_near along this ray
    T = 1.0;
    cr = cg = cb = 0.0;
  }
  __device__ bool chord(float4 g, double* lo_out, double* hi_out) const {
    const double h = (double)g.w, cc[3] = {(double)g.x, (double)g.y, (double)g.z};
    double lo_t = t_near, hi_t = 1e300;
    bool miss = false;
    for (int a = 0; a < 3; ++a) {
      const double lo = cc[a] - h, hi = cc[a] + h;
      if (d[a] == 0.0) {
        if (o[a] < lo || o[a] > hi) miss = true;
        continue;
      }
      const double t1 = (lo - o[a]) / d[a], t2 = (hi - o[a]) / d[a];
      lo_t = fmax(lo_t, fmin(t1, t2));
      hi_t = fmin(hi_t, fmax(t1, t2));
    }
    *lo_out = lo_t;
    *hi_out = hi_t;
    return !(miss || !(hi_t - lo_t > 0.0));
  }
  // the list's next voxel; true once the ray stops
  template <typename DT, typename ST>
  __device__ bool add(const Scene64<DT, ST>& sc, uint32_t vox) {
    const float4 g = sc.geom[vox];
    const double h = (double)g.w, cc[3] = {(double)g.x, (double)g.y, (double)g.z};
    double lo_t, hi_t;
    if (!chord(g, &lo_t, &hi_t)) return false;
    const double l = hi_t - lo_t, tm = 0.5 * (lo_t + hi_t);
    // the trilinear field at the midpoint, or its mean over the chord (Simpson, exact for the cubic)
    const double ts3[3] = {tm, lo_t, hi_t}, ws3[3] = {sc.segment ? 4.0 / 6.0 : 1.0, 1.0 / 6.0, 1.0 / 6.0};
    double sr = 0.0;
    for (int q3 = 0; q3 < (sc.segment ? 3 : 1); ++q3) {
      double u[3];
      for (int a = 0; a < 3; ++a)
        u[a] = fmin(fmax((o[a] + ts3[q3] * d[a] - (cc[a] - h)) / (2.0 * h), 0.0), 1.0);
      for (int i = 0; i < 8; ++i) {
        const double w =
            ((i & 1) ? u[0] : 1.0 - u[0]) * ((i & 2) ? u[1] : 1.0 - u[1]) * ((i & 4) ? u[2] : 1.0 - u[2]);
        const size_t di = sc.vidx ? (size_t)sc.vidx[8 * (size_t)vox + i] : 8 * (size_t)vox + i;
        sr += ws3[q3] * w * (double)to_f32(sc.dens[di]);
      }
    }
    const double sigma = fmax(sr, 0.0);
    const double alpha = -expm1(-sigma * l);
    double dir[3] = {cc[0] - o[0], cc[1] - o[1], cc[2] - o[2]};
    const double dn = sqrt(dir[0] * dir[0] + dir[1] * dir[1] + dir[2] * dir[2]);
    for (int k = 0; k < 3; ++k) dir[k] = dn > 0.0 ? dir[k] / dn : (k == 2 ? 1.0 : 0.0);
    double Y[16];
    sh_basis64(dir[0], dir[1], dir[2], Y);
    double col[3] = {0.5, 0.5, 0.5};
    for (int j = 0; j < sc.sh_nb; ++j)
      for (int ch = 0; ch < 3; ++ch) col[ch] += (double)to_f32(sc.sh[48 * (size_t)vox + 3 * j + ch]) * Y[j];
    const double w = T * alpha;
    cr += w * fmax(col[0], 0.0);
    cg += w * fmax(col[1], 0.0);
    cb += w * fmax(col[2], 0.0);
    T *= exp(-sigma * l);
    return T < sc.t_stop;
  }
  __device__ void store(double* rgb_out, double* T_out, int64_t q) const {
    rgb_out[3 * q + 0] = cr;
    rgb_out[3 * q + 1] = cg;
    rgb_out[3 * q + 2] = cb;
    if (T_out) T_out[q] = T;
  }
};

// a thread per pixel; those whose list is not sorted to its end are k_render_f64_rest's
template <typename DT, typename ST>
__global__ void k_render_f64(const __grid_constant__ ViewSet vs, const ListView lv, const Scene64<DT, ST> sc,
                             const int64_t* __restrict__ pixels, int64_t n_px, double* __restrict__ rgb_out,
                             double* __restrict__ T_out) {
  grid_begin();
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q >= n_px) return;
  March64 m(vs, pixels[q]);
  const uint2 r = lv.ranges[m.gtile];
  if (lv.ready[m.gtile] < r.y) return;
  for (uint32_t e = r.x; e < r.y; ++e)
    if (m.add(sc, lv.slot_vox[lv.plist[e].x])) break;
  m.store(rgb_out, T_out, q);
}

// a block per pixel, in turn: it tests 512 of the list's entries at a time, and its first thread
// marches through those the ray meets
template <typename DT, typename ST>
__global__ void __launch_bounds__(TS_THREADS) k_render_f64_rest(const __grid_constant__ ViewSet vs, const ListView lv,
                                                               const Scene64<DT, ST> sc,
                                                               const int64_t* __restrict__ pixels, int64_t n_px,
                                                               double* __restrict__ rgb_out,
                                                               double* __restrict__ T_out) {
  grid_begin();
  __shared__ uint32_t s_hit[TS_WARPS];
  __shared__ int s_done;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int64_t q = blockIdx.x; q < n_px; q += gridDim.x) {  // block-uniform
    March64 m(vs, pixels[q]);
    const uint2 r = lv.ranges[m.gtile];
    const uint32_t sorted = lv.ready[m.gtile];
    if (sorted >= r.y) continue;
    __syncthreads();  // the last pixel's s_done is read
    if (t == 0) s_done = 0;
    __syncthreads();
    // entries [0, n) with the voxel of entry e given by vox_at(e); true once the ray stops
    auto march = [&](uint32_t n, auto&& vox_at) {
      for (uint32_t e0 = 0; e0 < n && !s_done; e0 += TS_THREADS) {  // block-uniform
        double lo_t, hi_t;
        const bool hit = e0 + t < n && m.chord(sc.geom[vox_at(e0 + t)], &lo_t, &hi_t);
        const uint32_t who = __ballot_sync(FULL, hit);
        if (lane == 0) s_hit[warp] = who;
        __syncthreads();
        if (t == 0) {
          bool done = false;
          for (int w = 0; w < TS_WARPS && !done; ++w)
            for (uint32_t h = s_hit[w]; h && !done; h &= h - 1)
              done = m.add(sc, vox_at(e0 + 32 * w + __ffs(h) - 1));
          if (done) s_done = 1;
        }
        __syncthreads();
      }
      return s_done != 0;
    };
    if (!march(sorted - r.x, [&](uint32_t e) { return lv.slot_vox[lv.plist[r.x + e].x]; }))
      list_rest(lv, (uint32_t)m.gtile, r, [&](uint32_t, uint32_t n, bool ordered) {
        const TileSortSmem& S = ts_smem().s;
        if (!ordered) {
          ts_sort_smem((int)n);
          __syncthreads();
        }
        return march(n, [&](uint32_t e) { return lv.slot_vox[S.v[e]]; });
      });
    if (t == 0) m.store(rgb_out, T_out, q);
  }
}

// ------------------------------------------------------------------ host side
static lv_status check_common(const lv_voxels* vox, const lv_camera* cams, int nv, const lv_raster_opts* o) {
  if (!vox || !cams || !o) { set_error("null argument"); return LV_ERR_INVALID_ARG; }
  if (nv < 1 || nv > LV_MAX_VIEWS) { set_error("n_views %d outside [1, %d]", nv, LV_MAX_VIEWS); return LV_ERR_INVALID_ARG; }
  if (vox->n < 0 || vox->n > 0x7fffffffLL) { set_error("voxel count %lld out of range", (long long)vox->n); return LV_ERR_INVALID_ARG; }
  if (vox->n > 0 && (!vox->geom || !vox->density || !vox->sh)) { set_error("null voxel array"); return LV_ERR_INVALID_ARG; }
  if (vox->density_dtype != LV_F32 && vox->density_dtype != LV_F16) { set_error("density dtype must be F32 or F16"); return LV_ERR_INVALID_ARG; }
  if (vox->sh_dtype != LV_F32 && vox->sh_dtype != LV_BF16) { set_error("sh dtype must be F32 or BF16"); return LV_ERR_INVALID_ARG; }
  if (vox->sh_degree < 0 || vox->sh_degree > 3) { set_error("sh_degree must be 0..3"); return LV_ERR_INVALID_ARG; }
  if (vox->vidx && ((uintptr_t)vox->vidx & 15)) { set_error("vidx must be 16-byte aligned"); return LV_ERR_INVALID_ARG; }
  if (o->tile != 8 && o->tile != 16 && o->tile != 32) { set_error("tile must be 8, 16 or 32"); return LV_ERR_INVALID_ARG; }
  if (o->batch != 32 && o->batch != 64 && o->batch != 128) { set_error("batch must be 32, 64 or 128"); return LV_ERR_INVALID_ARG; }
  if (o->tile == 32 && o->batch == 128) {
    set_error("tile 32 takes batch 32 or 64 (as it always has; the batch changes no launch)");
    return LV_ERR_UNSUPPORTED;
  }
  if (!(o->t_stop >= 0.f && o->t_stop < 1.f)) { set_error("t_stop must be in [0, 1)"); return LV_ERR_INVALID_ARG; }
  if (o->persistent_sms < 0) { set_error("persistent_sms must be >= 0"); return LV_ERR_INVALID_ARG; }
  int64_t tiles = 0, pixels = 0;
  for (int i = 0; i < nv; ++i) {
    const lv_camera& c = cams[i];
    if (c.width < 1 || c.height < 1 || c.width > 32768 || c.height > 32768) { set_error("view %d: bad size", i); return LV_ERR_INVALID_ARG; }
    if (!(c.fx > 0.f && c.fy > 0.f && c.z_near > 0.f)) { set_error("view %d: fx, fy, z_near must be > 0", i); return LV_ERR_INVALID_ARG; }
    tiles += (int64_t)((c.width + o->tile - 1) / o->tile) * ((c.height + o->tile - 1) / o->tile);
    pixels += (int64_t)c.width * c.height;
  }
  if (tiles > 0x7fffffffLL || pixels > 0xfffffffeLL) { set_error("too many tiles or pixels"); return LV_ERR_INVALID_ARG; }
  if (o->pixel_id_base < 0 || o->pixel_id_base + pixels > 0xfffffffeLL) {
    set_error("pixel_id_base %lld: the pixel ids must stay in [0, 2^32 - 1)", (long long)o->pixel_id_base);
    return LV_ERR_INVALID_ARG;
  }
  if (vox->n * nv > 0x7fffffffLL) { set_error("voxels x views exceeds 2^31"); return LV_ERR_INVALID_ARG; }
  return LV_OK;
}

static lv_status finish(lv_status st, uint32_t flags, int32_t* d_status, cudaStream_t s, const char* what) {
  if (st != LV_OK) return st;
  lv_status e = cuda_check(cudaGetLastError(), what);
  if (e != LV_OK) return e;
  if (flags & LV_FLAG_SYNC_CHECK) {
    e = cuda_check(cudaStreamSynchronize(s), what);
    if (e != LV_OK) return e;
    int32_t h = 0;
    e = cuda_check(cudaMemcpy(&h, d_status, sizeof(h), cudaMemcpyDeviceToHost), "status readback");
    if (e != LV_OK) return e;
    if (h != 0) { set_error("%s: device reported status %d", what, h); return (lv_status)h; }
  }
  return LV_OK;
}

// resident blocks of a persistent composite (once per kernel)
template <typename K>
static int persistent_blocks(K kernel, int threads, size_t smem) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  return (sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
}

// a persistent grid of pb blocks over all SMs, cut to sm_limit SMs (0: all)
// the SM count, and the cut for a persistent grid limited to sm_limit SMs (0: no limit)
static void sm_limits(int sm_limit, int dev, int* sms, int* sm_cut) {
  cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  *sm_cut = (sm_limit > 0 && *sms > 0 && sm_limit < *sms) ? sm_limit : 0;
}


static uint32_t strip_items(int ts, int64_t tiles) { return (uint32_t)tiles * (uint32_t)(ts * ts / 32); }

static TileOrder tile_order(const FwdWs& w, int64_t tiles) {
  return {w.class_tiles, w.work + 16, (uint32_t)tiles};
}

template <int TS, bool SEG, bool PERSIST, bool LOOK>
static void launch_fwd_t(int64_t tiles, cudaStream_t s, const ViewSet& vs, const FwdWs& w, float t_stop,
                         const lv_fwd_out* out, int sm_limit) {
  constexpr int CW = fwd_warps<TS, PERSIST, LOOK>();
  constexpr bool RESUME = PERSIST && LOOK;
  const auto kernel = k_fwd<TS, SEG, PERSIST, LOOK>;
  const size_t smem = WalkShape<LOOK>::SLICE * CW;
  static int pblocks[64];  // per device
  static std::atomic<unsigned long long> done{0};
  const int dev = current_device();
  once_per_device(done, [&] {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (PERSIST && dev < 64) pblocks[dev] = persistent_blocks(kernel, CW * 32, smem);
  });
  const int pb = dev < 64 ? pblocks[dev] : persistent_blocks(kernel, CW * 32, smem);
  int sms = 0, sm_cut = 0;
  sm_limits(sm_limit, dev, &sms, &sm_cut);
  const uint32_t n_items = strip_items(TS, tiles);
  unsigned grid = (n_items + CW - 1) / CW;
  if (PERSIST) grid = std::min(grid, (unsigned)pb);  // the work counters were cleared at the start of the forward
  const Front fr = {w.ready, w.prog, w.open_tiles, w.work + 7, w.dep, w.nsamp};
  auto k = out->composite_event && !RESUME ? launch(kernel, grid, CW * 32, smem, s)
                                           : chain(kernel, grid, CW * 32, smem, s);
  k(vs, w.ranges, w.plist, w.rec, w.slot_vox, t_stop, out->rgb, out->depth, out->T, out->n_contrib, out->n_samples,
    w.tau, out->wmax_packed, w.work + (RESUME ? 2 : 0), n_items, sm_cut, sms, w.work + (RESUME ? 10 : 8),
    tile_order(w, tiles), fr);
}

template <int TS, bool SEG, bool PERSIST, bool LOOK>
static void launch_bwd_t(int64_t tiles, cudaStream_t s, const ViewSet& vs, const FwdWs& w, const lv_fwd_out* fwd,
                         const float* gC, const float* gD, const float* gT, float* dd,
                         int sm_limit, const LfFuse& lf) {
  constexpr int CW = bwd_warps<TS, PERSIST>();
  const auto kernel = k_bwd<TS, SEG, PERSIST, LOOK>;
  const size_t smem = WalkShape<LOOK>::SLICE * CW;
  static int pblocks[64];  // per device
  static std::atomic<unsigned long long> done{0};
  const int dev = current_device();
  once_per_device(done, [&] {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (PERSIST && dev < 64) pblocks[dev] = persistent_blocks(kernel, CW * 32, smem);
  });
  const int pb = dev < 64 ? pblocks[dev] : persistent_blocks(kernel, CW * 32, smem);
  int sms = 0, sm_cut = 0;
  sm_limits(sm_limit, dev, &sms, &sm_cut);
  const uint32_t n_items = strip_items(TS, tiles);
  unsigned grid = (n_items + CW - 1) / CW;
  if (PERSIST) {
    zero_async(s, w.work + 1, sizeof(unsigned int), w.work + 9, sizeof(unsigned int));
    grid = std::min(grid, (unsigned)pb);
  }
  launch(kernel, grid, CW * 32, smem, s)(vs, w.ranges, w.plist, w.rec, w.slot_vox, fwd->T, w.tau, fwd->n_contrib, gC,
                                         gD, gT, dd, w.d_rgb, w.work + 1, n_items, sm_cut, sms, w.work + 9,
                                         tile_order(w, tiles), lf);
}

// One warp per tile first (short lists, ranges, the lists of longer tiles), then persistent blocks over
// the long tiles' fronts and the medium tiles.
static int tile_sort_blocks() {
  static std::atomic<unsigned long long> attr_done{0};
  static int blocks[64];
  const int dev = current_device();
  once_per_device(attr_done, [dev] {
    cudaFuncSetAttribute(k_tile_sort_warp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TileSortWarpSmem));
    cudaFuncSetAttribute(k_tile_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TileLongSmem));
    cudaFuncSetAttribute(k_tile_rest, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TileLongSmem));
    if (dev < 64) blocks[dev] = persistent_blocks(k_tile_sort, TS_THREADS, sizeof(TileLongSmem));
  });
  return dev < 64 ? blocks[dev] : persistent_blocks(k_tile_sort, TS_THREADS, sizeof(TileLongSmem));
}
static void launch_tile_sort(const FwdWs& w, const ViewSet& vs, int64_t n, int64_t tiles, int64_t pair_cap,
                             cudaStream_t s) {
  const int64_t nb = std::min<int64_t>(tile_sort_blocks(), tiles);
  const bool ready = sort_passes(tile_bits(tiles)) > 0;
  const uint32_t* sv = w.tile_slots;
  const unsigned wblocks = (unsigned)((tiles + TW_WARPS - 1) / TW_WARPS);
  chain(k_tile_sort_warp, wblocks, TW_WARPS * 32, sizeof(TileSortWarpSmem), s)(
      sv, w.s_dkey, w.counters, pair_cap, ready, tiles, w.ranges, tile_order(w, tiles), w.ready, w.prog, vs, w.rec_bb,
      w.plist);
  count_launch(1);
  if (n <= TW_MAX) return;  // a tile lists a voxel once: every list is short
  chain(k_tile_sort, (unsigned)nb, TS_THREADS, sizeof(TileLongSmem), s)(
      sv, w.long_keys, w.s_dkey, w.ranges, tile_order(w, tiles), w.work + 5,
      w.ready, w.prog, n > TS_LAZY_VOXELS ? TS_LAZY : ~0u, vs, w.rec_bb, w.plist);
  count_launch(1);
}
// the rest of the open tiles' lists
static void launch_tile_rest(const FwdWs& w, const ViewSet& vs, int64_t tiles, cudaStream_t s) {
  const int64_t nb = std::min<int64_t>(tile_sort_blocks(), tiles);
  chain(k_tile_rest, (unsigned)nb, TS_THREADS, sizeof(TileLongSmem), s)(
      w.tile_slots, w.long_keys, w.ranges, w.open_tiles, w.work + 7, w.work + 3, w.ready, w.prog, vs, w.rec_bb,
      w.plist);
  count_launch(1);
}

static ListView list_view(const FwdWs& w) {
  return {(const uint2*)w.ranges, w.ready, w.plist, w.tile_slots, w.long_keys, w.prog, w.slot_vox};
}

// dynamic shared memory for the kernels that put a list's rest in order (once per kernel and device)
template <typename K>
static void allow_long_smem(K kernel, std::atomic<unsigned long long>& done) {
  once_per_device(done, [&] {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TileLongSmem));
  });
}

template <typename DT, typename ST>
static void launch_render_f64(const lv_voxels* vox, const lv_raster_opts* o, const ViewSet& vs, const FwdWs& w,
                              const int64_t* pixels, int64_t n_px, double* rgb, double* T, cudaStream_t s) {
  const Scene64<DT, ST> sc = {(const float4*)vox->geom, (const DT*)vox->density, (const ST*)vox->sh, vox->vidx,
                              (vox->sh_degree + 1) * (vox->sh_degree + 1),
                              (o->flags & LV_FLAG_EXACT_SEGMENT) ? 1 : 0, (double)o->t_stop};
  const ListView lv = list_view(w);
  launch(k_render_f64<DT, ST>, (unsigned)((n_px + 127) / 128), 128, 0, s)(vs, lv, sc, pixels, n_px, rgb, T);
  count_launch(1);
  if (vox->n > TS_LAZY_VOXELS) {  // else every list is sorted whole
    static std::atomic<unsigned long long> done{0};
    allow_long_smem(k_render_f64_rest<DT, ST>, done);
    const unsigned grid = (unsigned)std::min<int64_t>(n_px, 1216);
    chain(k_render_f64_rest<DT, ST>, grid, TS_THREADS, sizeof(TileLongSmem), s)(vs, lv, sc, pixels, n_px, rgb, T);
    count_launch(1);
  }
}

// The looking-ahead composites, with either schedule, where few strips are in flight on an SM (see WalkShape):
// up to `waves` times 28 an SM, in the forward 5 with tile 8 and 3 with the others, in the backward 1.  Forward
// and backward in us, open 2M-voxel scene, looking ahead against not: tile 8, 2,048 strips 1611 + 714 against
// 1759 + 755; 9,600 strips 511 + 487 against 559 + 489; 17,000 strips 348 + 459 against 379 + 426 (opaque 57 + 74
// against 51 + 68), 32,400 strips 480 + 735 against 479 + 681; tile 16, 9,600 strips 503 + 524 against 536 + 504,
// 17,000 strips 363 + 485 against 363 + 440 (opaque 57 + 74 against 49 + 68).
static bool look_ahead(const lv_raster_opts* o, int64_t tiles, uint32_t waves) {
  int sms = 0, cut = 0;
  sm_limits((o->flags & LV_FLAG_PERSISTENT) ? o->persistent_sms : 0, current_device(), &sms, &cut);
  return cut == 0 && strip_items(o->tile, tiles) <= waves * 28u * (uint32_t)sms;
}

// resume: the second launch, over the open tiles (its grid is persistent whatever the schedule: only the
// device knows their number)
static void launch_fwd(const lv_raster_opts* o, int64_t tiles, cudaStream_t s, const ViewSet& vs, const FwdWs& w,
                       const lv_fwd_out* out, bool resume) {
  const bool seg = (o->flags & LV_FLAG_EXACT_SEGMENT) != 0, per = (o->flags & LV_FLAG_PERSISTENT) != 0;
  const int sml = per ? o->persistent_sms : 0;
  const bool look = look_ahead(o, tiles, o->tile == 8 ? 5 : 3);
#define LV_FWD_S(TS, SEG)                                                                        \
  if (resume) launch_fwd_t<TS, SEG, true, true>(tiles, s, vs, w, o->t_stop, out, sml);           \
  else if (look) launch_fwd_t<TS, SEG, false, true>(tiles, s, vs, w, o->t_stop, out, 0);         \
  else if (per) launch_fwd_t<TS, SEG, true, false>(tiles, s, vs, w, o->t_stop, out, sml);        \
  else launch_fwd_t<TS, SEG, false, false>(tiles, s, vs, w, o->t_stop, out, 0)
#define LV_FWD(TS)                 \
  if (seg) { LV_FWD_S(TS, true); } \
  else { LV_FWD_S(TS, false); }
  if (o->tile == 8) { LV_FWD(8); }
  else if (o->tile == 16) { LV_FWD(16); }
  else { LV_FWD(32); }
#undef LV_FWD
#undef LV_FWD_S
}

static void launch_bwd(const lv_raster_opts* o, int64_t tiles, cudaStream_t s, const ViewSet& vs, const FwdWs& w,
                       const lv_fwd_out* fwd, const float* gC, const float* gD, const float* gT,
                       float* dd, const LfFuse& lf) {
  const bool seg = (o->flags & LV_FLAG_EXACT_SEGMENT) != 0, per = (o->flags & LV_FLAG_PERSISTENT) != 0;
  const int sml = per ? o->persistent_sms : 0;
  const bool look = look_ahead(o, tiles, 1);
#define LV_BWD_S(TS, SEG)                                                                              \
  if (look) launch_bwd_t<TS, SEG, false, true>(tiles, s, vs, w, fwd, gC, gD, gT, dd, 0, lf);           \
  else if (per) launch_bwd_t<TS, SEG, true, false>(tiles, s, vs, w, fwd, gC, gD, gT, dd, sml, lf);     \
  else launch_bwd_t<TS, SEG, false, false>(tiles, s, vs, w, fwd, gC, gD, gT, dd, 0, lf)
#define LV_BWD(TS)                 \
  if (seg) { LV_BWD_S(TS, true); } \
  else { LV_BWD_S(TS, false); }
  if (o->tile == 8) { LV_BWD(8); }
  else if (o->tile == 16) { LV_BWD(16); }
  else { LV_BWD(32); }
#undef LV_BWD_S
#undef LV_BWD
}

}  // namespace lv

using namespace lv;

extern "C" size_t lv_forward_workspace_size(int64_t n, const lv_camera* cams, int n_views, const lv_raster_opts* opts,
                                            int64_t pair_capacity) {
  if (!cams || !opts || n_views < 1 || n_views > LV_MAX_VIEWS || n < 0 || pair_capacity < 0 ||
      pair_capacity > 0xffffffffLL)
    return 0;
  if (opts->tile != 8 && opts->tile != 16 && opts->tile != 32) return 0;
  ViewSet vs;
  int64_t tiles, pixels;
  make_views(cams, n_views, opts->tile, &vs, &tiles, &pixels);
  return carve_fwd(nullptr, n, n_views, tiles, pixels, pair_capacity).bytes;
}

extern "C" lv_status lv_rasterize_forward(const lv_voxels* vox, const lv_camera* cams, int n_views,
                                          const lv_raster_opts* opts, const lv_fwd_out* out, void* workspace,
                                          size_t ws_bytes, int64_t pair_capacity, int32_t* d_status, void* stream) {
  lv_status st = check_common(vox, cams, n_views, opts);
  if (st != LV_OK) return st;
  if (!out || !out->rgb || !out->T || !out->n_contrib) { set_error("rgb, T and n_contrib outputs are required"); return LV_ERR_INVALID_ARG; }
  if (!workspace || ((uintptr_t)workspace & 255)) { set_error("workspace must be non-null and 256-byte aligned"); return LV_ERR_INVALID_ARG; }
  if (pair_capacity < 0 || pair_capacity > 0xffffffffLL) { set_error("pair_capacity out of range"); return LV_ERR_INVALID_ARG; }
  cudaStream_t s = (cudaStream_t)stream;
  ViewSet vs;
  int64_t tiles, pixels;
  make_views(cams, n_views, opts->tile, &vs, &tiles, &pixels);
  vs.id_base = opts->pixel_id_base;
  FwdWs w = carve_fwd(workspace, vox->n, n_views, tiles, pixels, pair_capacity);
  if (ws_bytes < w.bytes) { set_error("workspace %zu bytes < required %zu", ws_bytes, w.bytes); return LV_ERR_WORKSPACE; }
  if (!d_status) d_status = w.status;
  const int64_t n = vox->n, items = n * n_views;
  // counters, the fallback status word, the work counters of the persistent kernels and the
  // sort by tile's digit counts, which k_emit accumulates (k_tile_sort_warp writes every tile's range)
  const SortCountTargets sc = sort_count_targets(w.sort_tmp, pair_capacity);
  const int passes = std::min(sort_passes(tile_bits(tiles)), 4);
  const bool own_status = d_status == w.status;
  const ZeroRanges zr = {{w.counters, w.status, w.work, sc.counts},
                         {8 * sizeof(unsigned long long), own_status ? sizeof(int32_t) : 0, 32 * sizeof(unsigned int),
                          sc.zero_bytes}};
  if (items == 0)
    zero_async(s, zr.p[0], zr.bytes[0], zr.p[1], zr.bytes[1], zr.p[2], zr.bytes[2], zr.p[3], zr.bytes[3]);
  if (items > 0) {
    const int64_t blocks = bin_blocks(n);
    const unsigned item_blocks = (unsigned)(blocks * n_views);  // (voxel range, view) blocks
    const unsigned bo_blocks = (unsigned)((blocks * n_views + BO_GROUP - 1) / BO_GROUP);
    launch(k_bin, item_blocks, BIN_THREADS, 0, s)(
        (const float4*)vox->geom, n, blocks, vs, w.cnt, w.rect, w.pbox, w.dkey, w.blk_pairs, w.blk_slots, out->z_min,
        out->delta_min, out->seen, zr);
    if (out->stats_event) cudaEventRecord((cudaEvent_t)out->stats_event, s);  // statistics final
    auto offsets = out->stats_event ? launch(k_block_offsets, bo_blocks, BO_THREADS, 0, s)
                                    : chain(k_block_offsets, bo_blocks, BO_THREADS, 0, s);
    offsets(w.blk_pairs, w.blk_slots, blocks * n_views, w.grp_pairs, w.grp_slots, w.counters);
    const int nb = (vox->sh_degree + 1) * (vox->sh_degree + 1);
#define LV_EMIT(DT, ST)                                                                                              \
  chain(k_emit<DT, ST>, item_blocks, BIN_THREADS, 0, s)(                                                             \
      (const float4*)vox->geom, (const DT*)vox->density, (const ST*)vox->sh, nb, n, vs, w.cnt, w.rect, w.pbox,       \
      w.rec_bb, w.slot_vox, w.dkey, w.slot, blocks, w.blk_pairs, w.blk_slots, w.grp_pairs, w.grp_slots, w.counters,  \
      pair_capacity, w.k0, w.v0, d_status, (uint2*)w.ranges, tiles, sc, passes, w.rec, w.d_rgb, w.s_dkey, vox->vidx)
    if (vox->density_dtype == LV_F32 && vox->sh_dtype == LV_F32) LV_EMIT(float, float);
    else if (vox->density_dtype == LV_F16 && vox->sh_dtype == LV_F32) LV_EMIT(__half, float);
    else if (vox->density_dtype == LV_F32 && vox->sh_dtype == LV_BF16) LV_EMIT(float, __nv_bfloat16);
    else LV_EMIT(__half, __nv_bfloat16);
#undef LV_EMIT
    count_launch(3);
  } else if (out->stats_event) {
    cudaEventRecord((cudaEvent_t)out->stats_event, s);  // no voxel: nothing to bin
  }
  // stable sort by tile: each tile's list stays in item order; the last pass notes every tile's range
  radix_sort_pairs(w.k0, w.v0, w.k0, w.v0, w.k1, w.v1, w.sort_tmp, w.counters, pair_capacity, tile_bits(tiles),
                   d_status, s, w.ranges, items > 0);
  // each tile's range, and its list front to back
  launch_tile_sort(w, vs, n, tiles, pair_capacity, s);
  if (out->composite_event) {
    // a timing mark: inside a stream capture it becomes an event record node of the graph
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(s, &cs);
    if (cs == cudaStreamCaptureStatusActive)
      cudaEventRecordWithFlags((cudaEvent_t)out->composite_event, s, cudaEventRecordExternal);
    else
      cudaEventRecord((cudaEvent_t)out->composite_event, s);
  }
  launch_fwd(opts, tiles, s, vs, w, out, false);
  count_launch(2);
  if (n > TS_LAZY_VOXELS) {
    launch_tile_rest(w, vs, tiles, s);
    launch_fwd(opts, tiles, s, vs, w, out, true);
    count_launch(1);
  }
  return finish(LV_OK, opts->flags, d_status, s, "lv_rasterize_forward");
}

namespace lv {
namespace {
// four voxels per thread: one 32-byte store of w_max, 16-byte stores of the
// depths, one 4-byte store of seen (scalar at a ragged end or misaligned arrays)
__global__ void k_reset_stats(int64_t n, unsigned long long* wmax, float* z_min, float* delta_min, uint8_t* seen) {
  grid_begin();
  const float inf = __int_as_float(0x7f800000);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x * 4;
  const bool vec = (((uintptr_t)wmax | (uintptr_t)z_min | (uintptr_t)delta_min) & 15) == 0 &&
                   ((uintptr_t)seen & 3) == 0;
  for (int64_t i0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * 4; i0 < n; i0 += stride) {
    if (vec && i0 + 3 < n) {
      if (wmax) {
        ((uint4*)(wmax + i0))[0] = make_uint4(0u, 0u, 0u, 0u);
        ((uint4*)(wmax + i0))[1] = make_uint4(0u, 0u, 0u, 0u);
      }
      if (z_min) *(float4*)(z_min + i0) = make_float4(inf, inf, inf, inf);
      if (delta_min) *(float4*)(delta_min + i0) = make_float4(inf, inf, inf, inf);
      if (seen) *(uint32_t*)(seen + i0) = 0u;
    } else {
      for (int64_t i = i0; i < n && i < i0 + 4; ++i) {
        if (wmax) wmax[i] = 0ull;
        if (z_min) z_min[i] = inf;
        if (delta_min) delta_min[i] = inf;
        if (seen) seen[i] = 0;
      }
    }
  }
}
}  // namespace
}  // namespace lv

extern "C" lv_status lv_reset_stats(int64_t n, unsigned long long* wmax_packed, float* z_min, float* delta_min,
                                    uint8_t* seen, void* stream) {
  if (n < 0) { set_error("bad voxel count"); return LV_ERR_INVALID_ARG; }
  if (n == 0) return LV_OK;
  int64_t blocks = (n / 4 + 255) / 256;
  if (blocks < 1) blocks = 1;
  if (blocks > 4 * 1216) blocks = 4 * 1216;
  launch(k_reset_stats, (unsigned)blocks, 256, 0, (cudaStream_t)stream)(n, wmax_packed, z_min, delta_min, seen);
  count_launch(1);
  return cuda_check(cudaGetLastError(), "lv_reset_stats");
}

extern "C" lv_status lv_workspace_counters(const void* workspace, size_t ws_bytes, int64_t* out2, void* stream) {
  if (!workspace || !out2 || ws_bytes < 64) { set_error("bad arguments"); return LV_ERR_INVALID_ARG; }
  unsigned long long h[2];
  cudaStream_t s = (cudaStream_t)stream;
  lv_status e = cuda_check(cudaMemcpyAsync(h, workspace, sizeof(h), cudaMemcpyDeviceToHost, s), "counters");
  if (e != LV_OK) return e;
  e = cuda_check(cudaStreamSynchronize(s), "counters");
  if (e != LV_OK) return e;
  out2[0] = (int64_t)h[0];
  out2[1] = (int64_t)h[1];
  return LV_OK;
}

static lv_status launch_sh_bwd(const lv_voxels* vox, const ViewSet& vs, const FwdWs& w, float* d_sh, int accumulate,
                               cudaStream_t s, bool chained) {
  const int64_t n = vox->n;
  if (n == 0) return LV_OK;
  const int nb = (vox->sh_degree + 1) * (vox->sh_degree + 1);
  const int blocks = (int)((n + 127) / 128);  // 4 warps x 32 voxels
  auto k = chained ? chain(k_sh_bwd, blocks, 128, 0, s) : launch(k_sh_bwd, blocks, 128, 0, s);
  k(w.rec, nb, n, vs, w.cnt, w.slot, w.d_rgb, d_sh, accumulate);
  count_launch(1);
  return LV_OK;
}

extern "C" lv_status lv_rasterize_backward(const lv_voxels* vox, const lv_camera* cams, int n_views,
                                           const lv_raster_opts* opts, const lv_fwd_out* fwd, void* workspace,
                                           size_t ws_bytes, int64_t pair_capacity, const float* dL_drgb,
                                           const float* dL_ddepth, const float* dL_dT, float* d_density, float* d_sh,
                                           int accumulate, int32_t* d_status, void* stream) {
  lv_status st = check_common(vox, cams, n_views, opts);
  if (st != LV_OK) return st;
  if (!fwd || !fwd->T || !fwd->n_contrib || !d_density || (!dL_drgb && !fwd->lf_workspace)) { set_error("null argument"); return LV_ERR_INVALID_ARG; }
  if (!workspace || ((uintptr_t)workspace & 255)) { set_error("workspace must be non-null and 256-byte aligned"); return LV_ERR_INVALID_ARG; }
  if (pair_capacity < 0 || pair_capacity > 0xffffffffLL) { set_error("pair_capacity out of range"); return LV_ERR_INVALID_ARG; }
  cudaStream_t s = (cudaStream_t)stream;
  ViewSet vs;
  int64_t tiles, pixels;
  make_views(cams, n_views, opts->tile, &vs, &tiles, &pixels);
  FwdWs w = carve_fwd(workspace, vox->n, n_views, tiles, pixels, pair_capacity);
  if (ws_bytes < w.bytes) { set_error("workspace %zu bytes < required %zu", ws_bytes, w.bytes); return LV_ERR_WORKSPACE; }
  if (!d_status) d_status = w.status;
  // the LF-weighted loss fused in: dL/drgb from the forward's image, the ground truth and the weights
  LfFuse lf = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  if (!dL_drgb) {
    if (!fwd->lf_gt || !fwd->rgb) { set_error("the fused LF loss needs lf_gt and the forward's rgb"); return LV_ERR_INVALID_ARG; }
    int32_t wd[LV_MAX_VIEWS], ht[LV_MAX_VIEWS];
    for (int v = 0; v < n_views; ++v) {
      wd[v] = cams[v].width;
      ht[v] = cams[v].height;
    }
    lv_status e = lf_fused_buffers(wd, ht, n_views, fwd->lf_workspace, fwd->lf_ws_bytes, &lf.w, &lf.wsum, &lf.view_k, &lf.lsum);
    if (e != LV_OK) return e;
    lf.rgb = fwd->rgb;
    lf.gt = fwd->lf_gt;
    lf.dL = fwd->lf_dL;
    if (fwd->lf_wait_event) cudaStreamWaitEvent(s, (cudaEvent_t)fwd->lf_wait_event, 0);  // the weights
  }
  const int64_t n = vox->n;
  if (!accumulate && n > 0) cudaMemsetAsync(d_density, 0, sizeof(float) * 8 * n, s);
  launch_bwd(opts, tiles, s, vs, w, fwd, dL_drgb, dL_ddepth, dL_dT, d_density, lf);
  count_launch(1);
  if (d_sh) launch_sh_bwd(vox, vs, w, d_sh, accumulate, s, true);
  return finish(LV_OK, opts->flags, d_status, s, "lv_rasterize_backward");
}

extern "C" lv_status lv_sh_backward(const lv_voxels* vox, const lv_camera* cams, int n_views,
                                    const lv_raster_opts* opts, void* workspace, size_t ws_bytes,
                                    int64_t pair_capacity, float* d_sh, int accumulate, void* stream) {
  lv_status st = check_common(vox, cams, n_views, opts);
  if (st != LV_OK) return st;
  if (!d_sh || !workspace || ((uintptr_t)workspace & 255)) { set_error("bad arguments"); return LV_ERR_INVALID_ARG; }
  cudaStream_t s = (cudaStream_t)stream;
  ViewSet vs;
  int64_t tiles, pixels;
  make_views(cams, n_views, opts->tile, &vs, &tiles, &pixels);
  FwdWs w = carve_fwd(workspace, vox->n, n_views, tiles, pixels, pair_capacity);
  if (ws_bytes < w.bytes) { set_error("workspace %zu bytes < required %zu", ws_bytes, w.bytes); return LV_ERR_WORKSPACE; }
  launch_sh_bwd(vox, vs, w, d_sh, accumulate, s, false);
  return cuda_check(cudaGetLastError(), "lv_sh_backward");
}

extern "C" lv_status lv_unpack_wmax(const unsigned long long* packed, int64_t n, float* w_max, int64_t* argmax,
                                    void* stream) {
  if (n < 0 || (n > 0 && (!packed || !w_max))) { set_error("bad arguments"); return LV_ERR_INVALID_ARG; }
  if (n == 0) return LV_OK;
  launch(k_unpack_wmax, (unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream)(packed, n, w_max, argmax);
  count_launch(1);
  return cuda_check(cudaGetLastError(), "lv_unpack_wmax");
}

extern "C" lv_status lv_gather_edge(const int64_t* argmax, int64_t n, const float* edge_map, int64_t n_pix,
                                    float* edge, void* stream) {
  if (n < 0 || n_pix < 0 || (n > 0 && (!argmax || !edge || (n_pix > 0 && !edge_map)))) {
    set_error("bad arguments");
    return LV_ERR_INVALID_ARG;
  }
  if (n == 0) return LV_OK;
  launch(k_gather_edge, (unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream)(argmax, n, edge_map, n_pix, edge);
  count_launch(1);
  return cuda_check(cudaGetLastError(), "lv_gather_edge");
}

extern "C" lv_status lv_debug_pairs(int64_t n, const lv_camera* cams, int n_views, const lv_raster_opts* opts,
                                    const void* workspace, size_t ws_bytes, int64_t pair_capacity, uint64_t* keys,
                                    uint32_t* voxel, uint32_t* ranges, void* stream) {
  if (!cams || !opts || !workspace || n_views < 1 || n_views > LV_MAX_VIEWS || n < 0) { set_error("bad arguments"); return LV_ERR_INVALID_ARG; }
  if (opts->tile != 8 && opts->tile != 16 && opts->tile != 32) { set_error("bad tile"); return LV_ERR_INVALID_ARG; }
  cudaStream_t s = (cudaStream_t)stream;
  ViewSet vs;
  int64_t tiles, pixels;
  make_views(cams, n_views, opts->tile, &vs, &tiles, &pixels);
  FwdWs w = carve_fwd((void*)workspace, n, n_views, tiles, pixels, pair_capacity);
  if (ws_bytes < w.bytes) { set_error("workspace too small"); return LV_ERR_WORKSPACE; }
  if (keys || voxel) {
    static std::atomic<unsigned long long> done{0};
    allow_long_smem(k_debug_pairs, done);
    launch(k_debug_pairs, 608, TS_THREADS, sizeof(TileLongSmem), s)(list_view(w), tiles, w.s_dkey, keys, voxel);
    count_launch(1);
  }
  if (ranges) cudaMemcpyAsync(ranges, w.ranges, sizeof(uint32_t) * 2 * tiles, cudaMemcpyDeviceToDevice, s);
  return cuda_check(cudaGetLastError(), "lv_debug_pairs");
}

extern "C" lv_status lv_render_pixels_f64(const lv_voxels* vox, const lv_camera* cams, int n_views,
                                          const lv_raster_opts* opts, const void* workspace, size_t ws_bytes,
                                          int64_t pair_capacity, const int64_t* pixels, int64_t n_px, double* rgb,
                                          double* T, void* stream) {
  lv_status st = check_common(vox, cams, n_views, opts);
  if (st != LV_OK) return st;
  if (n_px < 0 || (n_px > 0 && (!pixels || !rgb)) || !workspace) { set_error("bad arguments"); return LV_ERR_INVALID_ARG; }
  if (n_px == 0) return LV_OK;
  cudaStream_t s = (cudaStream_t)stream;
  ViewSet vs;
  int64_t tiles, npix;
  make_views(cams, n_views, opts->tile, &vs, &tiles, &npix);
  FwdWs w = carve_fwd((void*)workspace, vox->n, n_views, tiles, npix, pair_capacity);
  if (ws_bytes < w.bytes) { set_error("workspace too small"); return LV_ERR_WORKSPACE; }
  if (vox->density_dtype == LV_F32 && vox->sh_dtype == LV_F32)
    launch_render_f64<float, float>(vox, opts, vs, w, pixels, n_px, rgb, T, s);
  else if (vox->density_dtype == LV_F16 && vox->sh_dtype == LV_F32)
    launch_render_f64<__half, float>(vox, opts, vs, w, pixels, n_px, rgb, T, s);
  else if (vox->density_dtype == LV_F32 && vox->sh_dtype == LV_BF16)
    launch_render_f64<float, __nv_bfloat16>(vox, opts, vs, w, pixels, n_px, rgb, T, s);
  else
    launch_render_f64<__half, __nv_bfloat16>(vox, opts, vs, w, pixels, n_px, rgb, T, s);
  return cuda_check(cudaGetLastError(), "lv_render_pixels_f64");
}
