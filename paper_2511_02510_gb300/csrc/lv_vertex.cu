// lv_vertex.cu -- the shared grid-vertex density variant (sm_103a): voxels
// whose corners sit at the same point of the octree's finest grid read one
// density value, so the field is continuous across neighbouring voxels of any
// level whose corners coincide (the voxels still interpolate their own 8
// corners trilinearly, Eq. 2-4 are unchanged).
//
//   lv_build_vertex_index: corner -> vertex id.  Every corner's integer
//     coordinates on the finest grid (half-size units) form a 63-bit key.  The
//     distinct keys are found with a hash table, radix-sorted and numbered in
//     key order, so vertex ids are the ranks of the distinct corner points
//     (deterministic).
//   lv_vertex_gather: vertex values -> per-voxel corners [n][8] (FP32).
//   lv_vertex_scatter_add: per-voxel corner values [n][8] -> vertex sums
//     (atomics across the voxels sharing a vertex): turns the rasterizer's
//     per-corner density gradient into the vertex gradient, or averages
//     per-voxel corners into vertices with a count array.
#include <math.h>

#include <algorithm>

#include "lv_prims.cuh"

namespace lv {
namespace {

constexpr int TPB = 256;
constexpr int COORD_BITS = 21;
constexpr long long COORD_OFF = 1ll << (COORD_BITS - 1);  // coordinates in [-2^20, 2^20)

constexpr uint32_t COORD_MASK = (1u << COORD_BITS) - 1;
constexpr uint64_t TAKEN = 1ull << 63;  // set in an occupied table word: the table starts as zeros

struct VxWs {
  unsigned long long* counters;  // [0] distinct keys
  uint32_t* bounds;              // [3] largest coordinate, [3] COORD_MASK - smallest coordinate
  int32_t* status;
  uint64_t* table;               // [1 << bits] TAKEN | key, then the vertex id
  uint64_t *k0, *k1;             // [8n] distinct keys
  uint32_t *v0, *v1;             // [8n] their table slots
  void* sort_tmp;
  int bits;
  size_t bytes;
};

VxWs carve_vx(void* base, int64_t n) {
  VxWs w;
  Carve c(base);
  const int64_t m = 8 * n;
  w.bits = 10;
  while (w.bits < 32 && (1ll << w.bits) < m + m / 4) ++w.bits;  // at most 0.8 full, 0.1 to 0.2 in real scenes
  w.counters = c.take<unsigned long long>(4);
  w.bounds = c.take<uint32_t>(6);
  w.status = c.take<int32_t>(1);
  w.table = c.take<uint64_t>((size_t)1 << w.bits);
  w.k0 = c.take<uint64_t>(m);
  w.k1 = c.take<uint64_t>(m);
  w.v0 = c.take<uint32_t>(m);
  w.v1 = c.take<uint32_t>(m);
  w.sort_tmp = c.take<char>(sort_tmp_bytes(m));
  w.bytes = c.off + 256;
  return w;
}

// Grid coordinate of x + h (h signed) in units of 1 / inv_unit, COORD_OFF added;
// false if it is more than 1e-3 off the grid or out of range.  The definition
// is the FP64 one at the end; FP64 is slow on this part (24 coordinates a voxel
// in FP64 took 131 us for 300,000 voxels), so pairs of FP32 values, good to
// 2^-44 relative, decide wherever the distance is clear of the limit.
__device__ __forceinline__ bool grid_coord(float x, float h, double inv_unit, float ih, float il, uint32_t* q) {
  const float s = __fadd_rn(x, h), bb = __fsub_rn(s, x);
  const float e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, bb)), __fsub_rn(h, bb));  // s + e == x + h exactly
  const float p = __fmul_rn(s, ih);
  const float lo = __fmaf_rn(e, ih, __fmaf_rn(s, il, __fmaf_rn(s, ih, -p)));
  const float rf = rintf(p);
  if (fabsf(__fadd_rn(__fsub_rn(p, rf), lo)) <= 9.9e-4f && fabsf(rf) < (float)COORD_OFF) {
    *q = (uint32_t)((int)rf + (int)COORD_OFF);
    return true;
  }
  const double xd = ((double)x + (double)h) * inv_unit;
  const double r = rint(xd);
  *q = (uint32_t)((uint64_t)((long long)r + COORD_OFF) & COORD_MASK);
  return fabs(xd - r) <= 1e-3 && r >= -(double)COORD_OFF && r < (double)COORD_OFF;
}

// The corners' keys entered in the table, a corner per thread (a voxel per
// thread, its eight probes one after another, took 81 us for 300,000 voxels):
// vidx gets each corner's table slot, a key's first finder appends it to the
// distinct keys, and the coordinates' bounds are reduced.  Octree neighbours
// share corners, so the distinct keys are a fraction of the corners: sorting only
// those, and reading each corner's id from the table, replaced eight 64-bit sort
// passes over all corners (the whole index of 300,000 voxels: 404 -> 176 us, of
// which this kernel is 40 and the sort 95, bound by its passes' latencies).
__global__ void __launch_bounds__(TPB) k_vx_hash(const float4* __restrict__ geom, int64_t n, double inv_unit,
                                                unsigned long long* table, int bits, uint32_t* vidx,
                                                uint64_t* keys, uint32_t* slots,
                                                unsigned long long* count, uint32_t* bounds, int32_t* status) {
  grid_begin();
  __shared__ uint32_t s_b[6], s_n;
  __shared__ unsigned long long s_at;
  if (threadIdx.x < 6) s_b[threadIdx.x] = 0u;
  if (threadIdx.x == 0) s_n = 0u;
  __syncthreads();
  const int64_t i = blockIdx.x * (int64_t)TPB + threadIdx.x;
  const int lane = threadIdx.x & 31, c = (int)(i & 7);
  const float ih = (float)inv_unit, il = (float)(inv_unit - (double)ih);
  uint32_t q[3] = {0u, 0u, 0u}, mn[3] = {0u, 0u, 0u}, slot = 0;
  uint64_t key = 0;
  bool fresh = false;
  if (i < 8 * n) {
    const float4 g = geom[i >> 3];
    bool ok = grid_coord(g.x, c & 1 ? g.w : -g.w, inv_unit, ih, il, &q[0]);
    ok &= grid_coord(g.y, c & 2 ? g.w : -g.w, inv_unit, ih, il, &q[1]);
    ok &= grid_coord(g.z, c & 4 ? g.w : -g.w, inv_unit, ih, il, &q[2]);
    if (!ok) report(status, LV_ERR_INVALID_ARG);
    key = TAKEN | (uint64_t)q[0] | (uint64_t)q[1] << COORD_BITS | (uint64_t)q[2] << (2 * COORD_BITS);
    slot = (uint32_t)((key * 0x9e3779b97f4a7c15ull) >> (64 - bits));
    // the table is never full, so a probe meets its key or an empty word
    uint64_t cur = __ldcg(table + slot);
    while (cur != key) {
      if (cur == 0ull) {
        cur = atomicCAS(table + slot, 0ull, (unsigned long long)key);
        fresh = cur == 0ull;
        if (fresh) break;
      } else {
        slot = (slot + 1u) & (uint32_t)((1ull << bits) - 1ull);
        cur = __ldcg(table + slot);
      }
    }
    vidx[i] = slot;
#pragma unroll
    for (int a = 0; a < 3; ++a) mn[a] = COORD_MASK - q[a];
  }
  // one atomic per block on the count (same-address atomics serialise: one per warp cost 25 us)
  const uint32_t who = __ballot_sync(FULL, fresh);
  uint32_t rank = 0;
  if (lane == 0 && who) rank = atomicAdd(&s_n, __popc(who));
  rank = __shfl_sync(FULL, rank, 0) + __popc(who & ((1u << lane) - 1u));
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const uint32_t x = __reduce_max_sync(FULL, q[a]), y = __reduce_max_sync(FULL, mn[a]);
    if (lane == 0) {
      atomicMax(&s_b[a], x);
      atomicMax(&s_b[3 + a], y);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && s_n) s_at = atomicAdd(count, (unsigned long long)s_n);
  // the bounds settle after a few blocks: most need no atomic
  if (threadIdx.x < 6 && s_b[threadIdx.x] > __ldcg(&bounds[threadIdx.x])) atomicMax(&bounds[threadIdx.x], s_b[threadIdx.x]);
  __syncthreads();
  if (fresh) {
    keys[s_at + rank] = key & ~TAKEN;
    slots[s_at + rank] = slot;
  }
}

// The distinct keys packed: each coordinate less its smallest value, in just the
// bits its range needs.  The order stays, and the sort's passes over the high
// bytes, all zero, are plain copies.
__global__ void __launch_bounds__(TPB) k_vx_pack(uint64_t* keys, const unsigned long long* count,
                                                const uint32_t* bounds) {
  grid_begin();
  const int64_t m = (int64_t)*count;
  uint32_t lo[3];
  int sh[3], at = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = COORD_MASK - bounds[3 + a];
    sh[a] = at;
    at += 32 - __clz(bounds[a] - lo[a]);
  }
  for (int64_t i = blockIdx.x * (int64_t)TPB + threadIdx.x; i < m; i += (int64_t)gridDim.x * TPB) {
    const uint64_t k = keys[i];
    uint64_t r = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) r |= (uint64_t)(((uint32_t)(k >> (COORD_BITS * a)) & COORD_MASK) - lo[a]) << sh[a];
    keys[i] = r;
  }
}

// a vertex's id is its key's rank
__global__ void __launch_bounds__(TPB) k_vx_rank(const uint32_t* slots, const unsigned long long* count,
                                                uint64_t* table, int64_t* n_vert) {
  grid_begin();
  const int64_t m = (int64_t)*count;
  for (int64_t i = blockIdx.x * (int64_t)TPB + threadIdx.x; i < m; i += (int64_t)gridDim.x * TPB)
    table[slots[i]] = (uint64_t)i;
  if (blockIdx.x == 0 && threadIdx.x == 0) *n_vert = m;
}

// four corners per thread
__global__ void __launch_bounds__(TPB) k_vx_assign(const uint64_t* table, int64_t n4,
                                                  uint32_t* vidx) {
  grid_begin();
  const int64_t i = blockIdx.x * (int64_t)TPB + threadIdx.x;
  if (i >= n4) return;
  uint32_t* p = vidx + 4 * i;
  if (((uintptr_t)vidx & 15) == 0) {  // grid-uniform
    const uint4 s = *(const uint4*)p;
    *(uint4*)p = make_uint4((uint32_t)table[s.x], (uint32_t)table[s.y], (uint32_t)table[s.z], (uint32_t)table[s.w]);
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) p[c] = (uint32_t)table[p[c]];
  }
}

template <typename DT>
__global__ void k_vx_gather(const uint32_t* __restrict__ vidx, int64_t m, const DT* __restrict__ vals,
                            float* __restrict__ out) {
  grid_begin();
  const int64_t i = blockIdx.x * (int64_t)TPB + threadIdx.x;
  if (i < m) out[i] = to_f32(vals[vidx[i]]);
}

// zero rows (voxels the views never reached) cost one 32-byte read and no atomics
__global__ void k_vx_scatter(const uint32_t* __restrict__ vidx, int64_t n, const float4* __restrict__ corner,
                             float* __restrict__ out, float* __restrict__ count) {
  grid_begin();
  const int64_t v = blockIdx.x * (int64_t)TPB + threadIdx.x;
  if (v >= n) return;
  const float4 a = corner[2 * v], b = corner[2 * v + 1];
  const float x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  const uint4 i0 = *(const uint4*)(vidx + 8 * v), i1 = *(const uint4*)(vidx + 8 * v + 4);
  const uint32_t id[8] = {i0.x, i0.y, i0.z, i0.w, i1.x, i1.y, i1.z, i1.w};
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    if (x[c] != 0.f) atomicAdd(out + id[c], x[c]);
    if (count) atomicAdd(count + id[c], 1.f);
  }
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

}  // namespace
}  // namespace lv

using namespace lv;

extern "C" size_t lv_vertex_index_workspace_size(int64_t n) {
  if (n < 0 || n > (0x7fffffffLL >> 3)) return 0;
  return carve_vx(nullptr, n).bytes;
}

extern "C" lv_status lv_build_vertex_index(const float* geom, int64_t n, double unit, uint32_t* vidx,
                                           int64_t* d_n_vert, void* workspace, size_t ws_bytes, int32_t* d_status,
                                           void* stream) {
  if (n < 0 || n > (0x7fffffffLL >> 3) || !(unit > 0.0) || (n > 0 && (!geom || !vidx)) || !d_n_vert) {
    set_error("bad arguments");
    return LV_ERR_INVALID_ARG;
  }
  if (!workspace || ((uintptr_t)workspace & 255)) { set_error("workspace must be non-null and 256-byte aligned"); return LV_ERR_INVALID_ARG; }
  VxWs w = carve_vx(workspace, n);
  if (ws_bytes < w.bytes) { set_error("workspace %zu < %zu bytes", ws_bytes, w.bytes); return LV_ERR_WORKSPACE; }
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t m = 8 * n;
  if (n == 0) {
    cudaMemsetAsync(d_n_vert, 0, sizeof(int64_t), s);
    return cuda_check(cudaGetLastError(), "lv_build_vertex_index");
  }
  int32_t* st = d_status ? d_status : w.status;
  zero_async(s, w.table, sizeof(uint64_t) << w.bits, w.counters, sizeof(unsigned long long), w.bounds,
             6 * sizeof(uint32_t), d_status ? nullptr : w.status, sizeof(int32_t));
  chain(k_vx_hash, (unsigned)((m + TPB - 1) / TPB), TPB, 0, s)((const float4*)geom, n, 1.0 / unit,
                                                            (unsigned long long*)w.table, w.bits, vidx, w.k0, w.v0,
                                                            w.counters, w.bounds, st);
  const unsigned grid = (unsigned)std::min<int64_t>((m + TPB - 1) / TPB, 8 * 152);  // the count is on the device
  chain(k_vx_pack, grid, TPB, 0, s)(w.k0, w.counters, w.bounds);
  const int which = radix_sort_pairs(w.k0, w.v0, w.k0, w.v0, w.k1, w.v1, w.sort_tmp, w.counters, m,
                                     3 * COORD_BITS, st, s);
  chain(k_vx_rank, grid, TPB, 0, s)(which ? w.v1 : w.v0, w.counters, w.table, d_n_vert);
  chain(k_vx_assign, (unsigned)((m / 4 + TPB - 1) / TPB), TPB, 0, s)(w.table, m / 4, vidx);
  count_launch(4);
  return cuda_check(cudaGetLastError(), "lv_build_vertex_index");
}

extern "C" lv_status lv_vertex_gather(const uint32_t* vidx, int64_t n, const void* vertex_values, lv_dtype dtype,
                                      float* corners, void* stream) {
  if (n < 0 || (n > 0 && (!vidx || !vertex_values || !corners))) { set_error("bad arguments"); return LV_ERR_INVALID_ARG; }
  if (dtype != LV_F32 && dtype != LV_F16) { set_error("vertex dtype must be F32 or F16"); return LV_ERR_INVALID_ARG; }
  if (n == 0) return LV_OK;
  const int64_t m = 8 * n;
  const unsigned blocks = (unsigned)((m + TPB - 1) / TPB);
  cudaStream_t s = (cudaStream_t)stream;
  if (dtype == LV_F32) launch(k_vx_gather<float>, blocks, TPB, 0, s)(vidx, m, (const float*)vertex_values, corners);
  else launch(k_vx_gather<__half>, blocks, TPB, 0, s)(vidx, m, (const __half*)vertex_values, corners);
  count_launch(1);
  return cuda_check(cudaGetLastError(), "lv_vertex_gather");
}

extern "C" lv_status lv_vertex_scatter_add(const uint32_t* vidx, int64_t n, const float* corners, float* vertex_sum,
                                           float* vertex_count, void* stream) {
  if (n < 0 || (n > 0 && (!vidx || !corners || !vertex_sum))) { set_error("bad arguments"); return LV_ERR_INVALID_ARG; }
  if (!aligned16(vidx) || !aligned16(corners)) { set_error("vidx and corners must be 16-byte aligned"); return LV_ERR_INVALID_ARG; }
  if (n == 0) return LV_OK;
  launch(k_vx_scatter, (unsigned)((n + TPB - 1) / TPB), TPB, 0, (cudaStream_t)stream)(
      vidx, n, (const float4*)corners, vertex_sum, vertex_count);
  count_launch(1);
  return cuda_check(cudaGetLastError(), "lv_vertex_scatter_add");
}
