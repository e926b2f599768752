// lv_loss.cu -- low-frequency-weighted photometric loss (LiteVoxel Sec. IV-B,
// Eq. 7-10 and Eq. 18) for sm_103a.  Per view: Sobel magnitude of the ground
// truth luma (stop-gradient), exact nearest-rank percentile normalisation by a
// radix select, inverse-Sobel weight (eps + 1 - s)^gamma, mean normalisation,
// weighted squared error and its gradient.  Sums are accumulated in FP64.
#include <mutex>

#include "lv_prims.cuh"

namespace lv {

namespace {

constexpr int TPB = 256;

// Every step runs all views in one launch (a launch per view cost about 8 us
// each however small the view): the blocks of a step are dealt out to the views
// by their pixels, block range [blk[v], blk[v + 1]) for view v.  With the
// selection by 14 + 9 + 9 bits, sixteen views of 14.6 Mpixel in all went from
// 701 to 285 us: Sobel 143 -> 79, selection 181 -> 33, weights 150 -> 61 (powf),
// loss 230 -> 86 (585 MB, the memory rate).
struct ViewPix {
  int n;
  int W[LV_MAX_VIEWS];
  int H[LV_MAX_VIEWS];
  long long off[LV_MAX_VIEWS + 1];
  uint32_t k[LV_MAX_VIEWS];    // nearest-rank index of the percentile
  int tile[LV_MAX_VIEWS + 1];  // first Sobel tile of each view
  int blk[LV_MAX_VIEWS + 1];   // first block of each view in the per-pixel steps
};

// The percentile is selected by the magnitudes' bits, digit by digit from the
// top: 14 bits (the highest, the sign, is always 0), then 9 and 9.  The first digit is
// wide so that the few octaves an image's gradients span fall into hundreds of
// counters: with 11 bits about 24 counters took all the shared-memory atomics.  It is counted where the magnitudes are
// computed, and no group array is read, as a block's pixels are one view's.
constexpr int D1_SHIFT = 18, D1_BINS = 1 << (31 - D1_SHIFT);
constexpr int D2_SHIFT = 9, D2_BINS = 1 << (D1_SHIFT - D2_SHIFT);
constexpr int D3_BINS = 1 << D2_SHIFT;
constexpr int HIST_WORDS = D1_BINS + D2_BINS + D3_BINS;  // a view's counters

struct LfPick {
  uint32_t prefix;  // digits chosen so far
  uint32_t k;       // rank among the keys that share them
};

struct LfWs {
  LfPick* pick;   // [2][views] after the first and the second digit
  double* wsum;   // [views]
  double* lsum;   // [LF_SLOTS][views]
  float2* view_k; // [views] mean weight, gradient scale
  uint32_t* done; // [views] blocks that have added to wsum
  uint32_t* hist; // [views][HIST_WORDS]
  uint32_t* mkey; // [pixels] bits of three times the Sobel magnitude
  float* w;       // [pixels] unnormalised weight
  size_t bytes;
};

LfWs carve_lf(void* base, int nv, int64_t pixels) {
  LfWs w;
  Carve c(base);
  w.pick = c.take<LfPick>(2 * LV_MAX_VIEWS);
  w.wsum = c.take<double>(LV_MAX_VIEWS);
  w.lsum = c.take<double>(LF_SLOTS * LV_MAX_VIEWS);
  w.view_k = c.take<float2>(LV_MAX_VIEWS);
  w.done = c.take<uint32_t>(LV_MAX_VIEWS);
  w.hist = c.take<uint32_t>((size_t)nv * HIST_WORDS);
  w.mkey = c.take<uint32_t>(pixels);
  w.w = c.take<float>(pixels);
  // The size asked for never falls below 10 bytes a pixel and the scratch of a 64-query select, the
  // layout that the allocation-free call's limit of about 1.6 million pixels comes from.
  Carve f(nullptr);
  f.take<SelectQuery>(SELECT_MAX_QUERIES);
  f.take<char>(select_tmp_bytes(SELECT_MAX_QUERIES));
  f.take<double>(LV_MAX_VIEWS);
  f.take<double>(LV_MAX_VIEWS);
  f.take<uint16_t>(pixels);
  f.take<uint32_t>(pixels);
  f.take<float>(pixels);
  w.bytes = (c.off > f.off ? c.off : f.off) + 256;
  return w;
}

// view of block b among the block ranges `first`
__device__ __forceinline__ int view_of_block(const int* first, int n, int b) {
  int v = 0;
  while (v + 1 < n && b >= first[v + 1]) ++v;
  return v;
}


// Eq. 7 input: |Sobel(Y)| with replicated border, and the first digit's counts.
// A block takes `per` tiles of 32 x 32 pixels; a tile's channel sums (three times
// the luma) with a border of one pixel are computed once into shared memory
// (1.13 pixels read per pixel; nine neighbours' three channels each from the
// caches before), and the next tile's pixels are loaded while this one is worked on.
constexpr int ST = 32, SP = ST + 2;
__global__ void __launch_bounds__(TPB) k_lf_sobel(const float* __restrict__ gt, const __grid_constant__ ViewPix vp,
                                                 int per, uint32_t* mkey, uint32_t* hist) {
  grid_wait();
  __shared__ uint32_t s_h[D1_BINS];
  __shared__ float s_y[SP * SP];
  const int t = threadIdx.x;
  for (int i = t; i < D1_BINS; i += TPB) s_h[i] = 0u;
  const int t0 = blockIdx.x * per, t1 = min(t0 + per, vp.tile[vp.n]);
  int v = view_of_block(vp.tile, vp.n, t0);
  constexpr int LD = (SP * SP + TPB - 1) / TPB;
  float ahead[LD][3];
  auto load = [&](int tile, int view) {
    const int W = vp.W[view], H = vp.H[view], tx = (W - 1) / ST + 1, loc = tile - vp.tile[view];
    const int x0 = loc % tx * ST, y0 = loc / tx * ST;
#pragma unroll
    for (int k = 0; k < LD; ++k) {
      const int i = min(t + k * TPB, SP * SP - 1), ly = i / SP, lx = i - ly * SP;
      const int x = max(x0 + min(lx - 1, W - 1 - x0), 0), y = max(y0 + min(ly - 1, H - 1 - y0), 0);
      const float* g = gt + 3 * (vp.off[view] + (long long)y * W + x);
      ahead[k][0] = g[0];
      ahead[k][1] = g[1];
      ahead[k][2] = g[2];
    }
  };
  if (t0 < t1) load(t0, v);
  for (int tile = t0; tile < t1; ++tile) {  // block-uniform
    const int W = vp.W[v], H = vp.H[v], tx = (W - 1) / ST + 1, loc = tile - vp.tile[v];
    const int x0 = loc % tx * ST, y0 = loc / tx * ST;
    __syncthreads();  // the last tile's sums are read
#pragma unroll
    for (int k = 0; k < LD; ++k)
      if (t + k * TPB < SP * SP) s_y[t + k * TPB] = ahead[k][0] + ahead[k][1] + ahead[k][2];
    __syncthreads();
    if (tile + 1 < t1) load(tile + 1, tile + 1 < vp.tile[v + 1] ? v : v + 1);
    const int lx = t % ST;
#pragma unroll
    for (int r = 0; r < ST * ST / TPB; ++r) {
      const int ly = t / ST + r * (TPB / ST);
      if (lx < W - x0 && ly < H - y0) {
#define Y_(a, b) s_y[(ly + (b)) * SP + lx + (a)]
        const float gx = (Y_(2, 0) + 2.f * Y_(2, 1) + Y_(2, 2)) - (Y_(0, 0) + 2.f * Y_(0, 1) + Y_(0, 2));
        const float gy = (Y_(0, 2) + 2.f * Y_(1, 2) + Y_(2, 2)) - (Y_(0, 0) + 2.f * Y_(1, 0) + Y_(2, 0));
#undef Y_
        // three times the magnitude (only its ratio to the percentile counts); bit order == value order
        const uint32_t key = __float_as_uint(sqrtf(gx * gx + gy * gy)) & 0x7fffffffu;
        mkey[vp.off[v] + (long long)(y0 + ly) * W + x0 + lx] = key;
        atomicAdd(&s_h[key >> D1_SHIFT], 1u);
      }
    }
    if (tile + 1 == t1 || tile + 1 == vp.tile[v + 1]) {  // the block's last tile of this view
      __syncthreads();
      uint32_t* h = hist + (size_t)v * HIST_WORDS;
      for (int i = t; i < D1_BINS; i += TPB) {
        const uint32_t c = s_h[i];
        if (c) {
          atomicAdd(&h[i], c);
          s_h[i] = 0u;
        }
      }
      ++v;
    }
  }
}

// The digit that holds the k-th key among NB counters, and the rank among its
// keys; the whole block calls, every thread gets both.  A warp sums its share of
// the counters 32 at a time (coalesced), one thread per 32 scans the sums, and
// the warp of the group that holds the key finds it there.
template <int NB>
__device__ __forceinline__ LfPick block_pick(const uint32_t* h, uint32_t k) {
  constexpr int PER = NB / TPB;  // groups of 32 counters per warp
  static_assert(PER >= 1 && PER <= 32, "a lane for each of a warp's groups");
  __shared__ uint32_t s_part[TPB / 32];
  __shared__ LfPick s_pick;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint32_t* hw = h + warp * (32 * PER);
  uint32_t c[PER], sum = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) c[i] = hw[32 * i + lane];
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const uint32_t r = __reduce_add_sync(FULL, c[i]);
    if (lane == i) sum = r;  // lane i: group i of the warp
  }
  uint32_t x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_part[warp] = x;
  __syncthreads();
  uint32_t before = x - sum;
  for (int w = 0; w < warp; ++w) before += s_part[w];
  const uint32_t who = __ballot_sync(FULL, before < k && k <= before + sum);
  if (who) {  // one warp: the counts add up to the view's pixels
    const int grp = __ffs(who) - 1;
    before = __shfl_sync(FULL, before, grp);
    const uint32_t own = hw[32 * grp + lane];
    uint32_t y = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t z = __shfl_up_sync(FULL, y, o);
      if (lane >= o) y += z;
    }
    before += y - own;
    if (before < k && k <= before + own) {
      s_pick.prefix = (uint32_t)(warp * (32 * PER) + 32 * grp + lane);
      s_pick.k = k - before;
    }
  }
  __syncthreads();
  return s_pick;
}

// Counts of the second digit (the keys with the first digit picked here) or,
// LAST, of the third.  Every block picks for its view; the view's first block
// leaves the pick for the next step.
template <bool LAST>
__global__ void __launch_bounds__(TPB) k_lf_digit(const uint32_t* mkey, const __grid_constant__ ViewPix vp,
                                                 uint32_t* hist, LfPick* pick) {
  grid_wait();
  constexpr int NB = LAST ? D3_BINS : D2_BINS;
  __shared__ uint32_t s_h[NB];
  const int t = threadIdx.x, v = view_of_block(vp.blk, vp.n, blockIdx.x);
  uint32_t* h = hist + (size_t)v * HIST_WORDS;
  for (int i = t; i < NB; i += TPB) s_h[i] = 0u;
  LfPick p;
  if (!LAST) {
    p = block_pick<D1_BINS>(h, vp.k[v]);
  } else {
    const LfPick p1 = pick[v];
    p = block_pick<D2_BINS>(h + D1_BINS, p1.k);
    p.prefix |= p1.prefix << (D1_SHIFT - D2_SHIFT);
  }
  const int b0 = vp.blk[v], nb = vp.blk[v + 1] - b0;
  if (t == 0 && (int)blockIdx.x == b0) pick[(LAST ? LV_MAX_VIEWS : 0) + v] = p;
  constexpr int SHIFT = LAST ? 0 : D2_SHIFT, ITEMS = 8;
  const long long lo = vp.off[v], hi = vp.off[v + 1];
  for (long long q = lo + (blockIdx.x - b0) * (long long)(TPB * ITEMS) + t; q < hi; q += (long long)nb * (TPB * ITEMS)) {
    uint32_t key[ITEMS];
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) key[u] = q + u * TPB < hi ? mkey[q + u * TPB] : ~0u;  // no key: top bit clear
#pragma unroll
    for (int u = 0; u < ITEMS; ++u)
      if (key[u] >> (LAST ? D2_SHIFT : D1_SHIFT) == p.prefix) atomicAdd(&s_h[(key[u] >> SHIFT) & (NB - 1)], 1u);
  }
  __syncthreads();
  uint32_t* out = h + D1_BINS + (LAST ? D2_BINS : 0);
  for (int i = t; i < NB; i += TPB) {
    const uint32_t c = s_h[i];
    if (c) atomicAdd(&out[i], c);
  }
}

__device__ __forceinline__ void block_add_f64(double v, double* dst) {
  __shared__ double sred[TPB / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  if (lane == 0) sred[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < TPB / 32 ? sred[lane] : 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    if (lane == 0 && v != 0.0) atomicAdd(dst, v);
  }
  __syncthreads();
}

// Eq. 7: w = (eps + 1 - s)^gamma, s = clip(|grad| / P, 0, 1); blocks never span views.
// Grid-stride over the view's pixels with a bounded block count: one FP64
// atomic per block (a per-256-pixel atomic would serialise at the L2).
__global__ void __launch_bounds__(TPB) k_lf_weight(const uint32_t* mkey, const uint32_t* hist,
                                                  const LfPick* pick,
                                                  const __grid_constant__ ViewPix vp, float eps, float gamma,
                                                  float* w, double* wsum, float2* view_k, uint32_t* done,
                                                  float* edge_out) {
  grid_wait();
  const int v = view_of_block(vp.blk, vp.n, blockIdx.x);
  const int b0 = vp.blk[v], nb = vp.blk[v + 1] - b0;
  const long long lo = vp.off[v], hi = vp.off[v + 1];
  // the view's gradient scale 2 / (3 |P|), rounded to FP32 from FP64
  if ((int)blockIdx.x == b0 && threadIdx.x == 0) view_k[v].y = (float)(2.0 / (3.0 * (double)(hi - lo)));
  const LfPick p2 = pick[LV_MAX_VIEWS + v];
  const LfPick p3 = block_pick<D3_BINS>(hist + (size_t)v * HIST_WORDS + D1_BINS + D2_BINS, p2.k);
  const float P = __uint_as_float(p2.prefix << D2_SHIFT | p3.prefix);
  const bool norm = P > 0.f;
  // a thread sums four pixels in FP32, and those sums and the blocks' in FP64 (the GPU's FP64
  // rate is low, so no per-pixel FP64 arithmetic)
  constexpr int ITEMS = 4;
  double acc = 0.0;
  for (long long p = lo + (blockIdx.x - b0) * (long long)(TPB * ITEMS) + threadIdx.x; p < hi;
       p += (long long)nb * (TPB * ITEMS)) {
    uint32_t key[ITEMS];
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) key[u] = p + u * TPB < hi ? mkey[p + u * TPB] : 0u;
    float part = 0.f;
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
      if (p + u * TPB >= hi) break;
      float s = 0.f;
      if (norm) s = fminf(fmaxf(__uint_as_float(key[u]) / P, 0.f), 1.f);
      if (edge_out) edge_out[p + u * TPB] = s;
      const float wv = gamma == 0.f ? 1.f : powf(eps + 1.f - s, gamma);
      w[p + u * TPB] = wv;
      part += wv;
    }
    acc += (double)part;
  }
  block_add_f64(acc, &wsum[v]);
  // the view's mean weight <w>, rounded to FP32 from FP64, once, by its last block (FP64 division is slow on
  // this part: not in every block that uses it)
  if (threadIdx.x == 0) {  // the thread that added
    __threadfence();
    if (atomicAdd(&done[v], 1u) == (uint32_t)nb - 1u) {
      __threadfence();
      view_k[v].x = (float)(__ldcg(&wsum[v]) / (double)(hi - lo));
    }
  }
}

// Eq. 8 + Eq. 18: w~ = w / <w>, L = 1/|P| sum w~ mean_c r^2, dL/drgb = 2/(3|P|) w~ r
__global__ void k_lf_loss(const float* __restrict__ rgb, const float* __restrict__ gt, const float* __restrict__ w,
                          const __grid_constant__ ViewPix vp, const float2* view_k, double* lsum,
                          float* __restrict__ grad) {
  grid_wait();
  const int v = view_of_block(vp.blk, vp.n, blockIdx.x);
  const int b0 = vp.blk[v], nb = vp.blk[v + 1] - b0;
  const long long lo = vp.off[v], hi = vp.off[v + 1];
  const float2 vk = view_k[v];
  const float mean = vk.x, gscale = vk.y;
  double acc = 0.0;  // sum of w~ (r0^2 + r1^2 + r2^2) over this thread's pixels; the 1/3 is applied at the end
  for (long long p = lo + (blockIdx.x - b0) * (long long)TPB + threadIdx.x; p < hi; p += (long long)nb * TPB) {
    const float wt = w[p] / mean;
    const float r0 = rgb[3 * p] - gt[3 * p], r1 = rgb[3 * p + 1] - gt[3 * p + 1], r2 = rgb[3 * p + 2] - gt[3 * p + 2];
    acc += (double)(wt * (r0 * r0 + r1 * r1 + r2 * r2));
    if (grad) {
      const float c = gscale * wt;
      grad[3 * p] = c * r0;
      grad[3 * p + 1] = c * r1;
      grad[3 * p + 2] = c * r2;
    }
  }
  block_add_f64(acc, &lsum[v]);  // few blocks: the first slot
}

// k_lf_loss over groups of four pixels: three 16-byte loads of rgb and of gt,
// one of w, three 16-byte stores of the gradient.  The pixels of the view
// before the first group boundary (global pixel index a multiple of 4) and
// after the last one go through the scalar path of thread 0 of its first block.  The
// per-pixel arithmetic is that of k_lf_loss; only the summation order of the
// partial sums differs.
__global__ void k_lf_loss4(const float* __restrict__ rgb, const float* __restrict__ gt, const float* __restrict__ w,
                           const __grid_constant__ ViewPix vp, const float2* view_k, double* lsum,
                           float* __restrict__ grad) {
  grid_wait();
  const int v = view_of_block(vp.blk, vp.n, blockIdx.x);
  const int b0 = vp.blk[v], nb = vp.blk[v + 1] - b0;
  const long long lo = vp.off[v], hi = vp.off[v + 1];
  const float2 vk = view_k[v];
  const float mean = vk.x, gscale = vk.y;
  const long long g0 = (lo + 3) >> 2, g1 = hi >> 2;  // whole groups [4 g0, 4 g1)
  double acc = 0.0;  // four pixels' terms are summed in FP32
  auto one = [&](long long p) {
    const float wt = w[p] / mean;
    const float r0 = rgb[3 * p] - gt[3 * p], r1 = rgb[3 * p + 1] - gt[3 * p + 1], r2 = rgb[3 * p + 2] - gt[3 * p + 2];
    acc += (double)(wt * (r0 * r0 + r1 * r1 + r2 * r2));
    if (grad) {
      const float c = gscale * wt;
      grad[3 * p] = c * r0;
      grad[3 * p + 1] = c * r1;
      grad[3 * p + 2] = c * r2;
    }
  };
  if ((int)blockIdx.x == b0 && threadIdx.x == 0) {
    if (g1 <= g0) {
      for (long long p = lo; p < hi; ++p) one(p);
    } else {
      for (long long p = lo; p < 4 * g0; ++p) one(p);
      for (long long p = 4 * g1; p < hi; ++p) one(p);
    }
  }
  const float4* r4 = (const float4*)rgb;
  const float4* t4 = (const float4*)gt;
  const float4* w4 = (const float4*)w;
  float4* d4 = (float4*)grad;
  for (long long g = g0 + (blockIdx.x - b0) * (long long)TPB + threadIdx.x; g < g1; g += (long long)nb * TPB) {
    const float4 a0 = r4[3 * g], a1 = r4[3 * g + 1], a2 = r4[3 * g + 2];
    const float4 b0 = t4[3 * g], b1 = t4[3 * g + 1], b2 = t4[3 * g + 2];
    const float4 wv = w4[g];
    const float r[12] = {a0.x - b0.x, a0.y - b0.y, a0.z - b0.z, a0.w - b0.w, a1.x - b1.x, a1.y - b1.y,
                         a1.z - b1.z, a1.w - b1.w, a2.x - b2.x, a2.y - b2.y, a2.z - b2.z, a2.w - b2.w};
    const float wt[4] = {wv.x / mean, wv.y / mean, wv.z / mean, wv.w / mean};
    float part = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) part += wt[k] * (r[3 * k] * r[3 * k] + r[3 * k + 1] * r[3 * k + 1] + r[3 * k + 2] * r[3 * k + 2]);
    acc += (double)part;
    if (grad) {
      float o[12];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float c = gscale * wt[k];
        o[3 * k] = c * r[3 * k];
        o[3 * k + 1] = c * r[3 * k + 1];
        o[3 * k + 2] = c * r[3 * k + 2];
      }
      d4[3 * g] = make_float4(o[0], o[1], o[2], o[3]);
      d4[3 * g + 1] = make_float4(o[4], o[5], o[6], o[7]);
      d4[3 * g + 2] = make_float4(o[8], o[9], o[10], o[11]);
    }
  }
  block_add_f64(acc, &lsum[v]);  // few blocks: the first slot
}

// clear: the sums are zeroed once read (the fused backward's sums start from zero next time)
__global__ void k_lf_finish(const __grid_constant__ ViewPix vp, double* lsum, float* loss, bool clear) {
  grid_begin();
  int v = threadIdx.x;
  if (v < vp.n) {
    const long long np = vp.off[v + 1] - vp.off[v];
    double sum = 0.0;
#pragma unroll
    for (unsigned k = 0; k < LF_SLOTS; ++k) sum += lsum[k * LV_MAX_VIEWS + v];
    loss[v] = np > 0 ? (float)(sum / (3.0 * (double)np)) : 0.f;
    if (clear)
#pragma unroll
      for (unsigned k = 0; k < LF_SLOTS; ++k) lsum[k * LV_MAX_VIEWS + v] = 0.0;
  }
}

constexpr int STEP_BLOCKS = 8 * 152;
constexpr int SOBEL_BLOCKS = 6 * 152;

bool make_viewpix(const int32_t* widths, const int32_t* heights, int nv, int32_t pctl_ppm, ViewPix* vp) {
  if (nv < 1 || nv > LV_MAX_VIEWS || !widths || !heights) return false;
  vp->n = nv;
  long long off = 0;
  for (int v = 0; v < nv; ++v) {
    if (widths[v] < 1 || heights[v] < 1) return false;
    vp->W[v] = widths[v];
    vp->H[v] = heights[v];
    vp->off[v] = off;
    const long long np = (long long)widths[v] * heights[v];
    unsigned long long k = ((unsigned long long)pctl_ppm * (unsigned long long)np + 999999ull) / 1000000ull;
    if (k < 1) k = 1;
    if (k > (unsigned long long)np) k = np;
    vp->k[v] = (uint32_t)k;
    off += np;
  }
  vp->off[nv] = off;
  if (off >= 0xffffffffLL) return false;
  // about four pixels per thread, more where that would make over STEP_BLOCKS blocks
  const long long px = off / STEP_BLOCKS > 4 * TPB ? off / STEP_BLOCKS : 4 * TPB;
  vp->tile[0] = vp->blk[0] = 0;
  for (int v = 0; v < nv; ++v) {
    const long long np = vp->off[v + 1] - vp->off[v];
    vp->tile[v + 1] = vp->tile[v] + ((vp->W[v] - 1) / ST + 1) * ((vp->H[v] - 1) / ST + 1);
    vp->blk[v + 1] = vp->blk[v] + (int)((np + px - 1) / px);
  }
  return true;
}

}  // namespace

}  // namespace lv

using namespace lv;

extern "C" float lv_lf_gamma(float t, const lv_lf_params* p) {
  if (!p) return 0.f;
  if (t < p->t0) return 0.f;
  if (t < p->t1) return p->gamma_max * (t - p->t0) / (p->t1 - p->t0);
  return p->gamma_max;
}

extern "C" size_t lv_lf_workspace_size(const int32_t* widths, const int32_t* heights, int n_views) {
  ViewPix vp;
  if (!make_viewpix(widths, heights, n_views, 990000, &vp)) return 0;
  return carve_lf(nullptr, n_views, vp.off[n_views]).bytes;
}

namespace {
bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

lv_status lf_setup(const int32_t* widths, const int32_t* heights, int n_views, int32_t pctl_ppm, void* workspace,
                   size_t ws_bytes, ViewPix* vp, LfWs* w) {
  if (!make_viewpix(widths, heights, n_views, pctl_ppm, vp)) { set_error("bad view sizes"); return LV_ERR_INVALID_ARG; }
  if (!workspace || ((uintptr_t)workspace & 255)) { set_error("workspace must be non-null and 256-byte aligned"); return LV_ERR_INVALID_ARG; }
  *w = carve_lf(workspace, n_views, vp->off[n_views]);
  if (ws_bytes < w->bytes) { set_error("workspace %zu < %zu bytes", ws_bytes, w->bytes); return LV_ERR_WORKSPACE; }
  return LV_OK;
}
}  // namespace

extern "C" lv_status lv_lf_weights(const float* gt, const int32_t* widths, const int32_t* heights, int n_views,
                                   float t, const lv_lf_params* p, void* workspace, size_t ws_bytes, void* stream) {
  if (!gt || !p) { set_error("null argument"); return LV_ERR_INVALID_ARG; }
  if (p->pctl_ppm < 0 || p->pctl_ppm > 1000000) { set_error("pctl_ppm must be in [0, 1e6]"); return LV_ERR_INVALID_ARG; }
  if (!(p->eps > 0.f) || !(p->t1 > p->t0) || !(p->gamma_max >= 0.f)) { set_error("need eps > 0, t1 > t0, gamma_max >= 0"); return LV_ERR_INVALID_ARG; }
  ViewPix vp;
  LfWs w;
  lv_status e = lf_setup(widths, heights, n_views, p->pctl_ppm, workspace, ws_bytes, &vp, &w);
  if (e != LV_OK) return e;
  cudaStream_t s = (cudaStream_t)stream;
  const float gamma = lv_lf_gamma(t, p);
  // the weight sums, the loss sums a backward with the fused loss accumulates, and the counters
  zero_async(s, w.wsum, sizeof(double) * LV_MAX_VIEWS, w.lsum, sizeof(double) * LF_SLOTS * LV_MAX_VIEWS, w.hist,
             sizeof(uint32_t) * HIST_WORDS * (size_t)n_views, w.done, sizeof(uint32_t) * LV_MAX_VIEWS);
  // a block clears and adds up all the counters, so it takes several tiles once there are enough
  const int tiles = vp.tile[n_views], per = (tiles + SOBEL_BLOCKS - 1) / SOBEL_BLOCKS;
  chain(k_lf_sobel, (unsigned)((tiles + per - 1) / per), TPB, 0, s)(gt, vp, per, w.mkey, w.hist);
  const unsigned blocks = (unsigned)vp.blk[n_views];
  chain(k_lf_digit<false>, blocks, TPB, 0, s)(w.mkey, vp, w.hist, w.pick);
  chain(k_lf_digit<true>, blocks, TPB, 0, s)(w.mkey, vp, w.hist, w.pick);
  chain(k_lf_weight, blocks, TPB, 0, s)(w.mkey, w.hist, w.pick, vp, p->eps, gamma, w.w, w.wsum, w.view_k, w.done,
                                       p->edge_out);
  count_launch(4);
  return cuda_check(cudaGetLastError(), "lv_lf_weights");
}

extern "C" lv_status lv_lf_loss_from_weights(const float* rgb, const float* gt, const int32_t* widths,
                                             const int32_t* heights, int n_views, float* loss, float* dL_drgb,
                                             void* workspace, size_t ws_bytes, void* stream) {
  if (!rgb || !gt || !loss) { set_error("null argument"); return LV_ERR_INVALID_ARG; }
  ViewPix vp;
  LfWs w;
  lv_status e = lf_setup(widths, heights, n_views, 990000, workspace, ws_bytes, &vp, &w);
  if (e != LV_OK) return e;
  cudaStream_t s = (cudaStream_t)stream;
  zero_async(s, w.lsum, sizeof(double) * LF_SLOTS * LV_MAX_VIEWS);
  // four pixels (three 16-byte words of rgb, gt and dL_drgb) per step where the buffers allow it
  const bool vec = aligned16(rgb) && aligned16(gt) && aligned16(w.w) && (!dL_drgb || aligned16(dL_drgb));
  const unsigned blocks = (unsigned)vp.blk[n_views];
  if (vec) chain(k_lf_loss4, blocks, TPB, 0, s)(rgb, gt, w.w, vp, w.view_k, w.lsum, dL_drgb);
  else chain(k_lf_loss, blocks, TPB, 0, s)(rgb, gt, w.w, vp, w.view_k, w.lsum, dL_drgb);
  chain(k_lf_finish, 1, LV_MAX_VIEWS, 0, s)(vp, w.lsum, loss, false);
  count_launch(2);
  return cuda_check(cudaGetLastError(), "lv_lf_loss_from_weights");
}

extern "C" lv_status lv_lf_loss_finish(const int32_t* widths, const int32_t* heights, int n_views, float* loss,
                                       void* workspace, size_t ws_bytes, void* stream) {
  if (!loss) { set_error("null argument"); return LV_ERR_INVALID_ARG; }
  ViewPix vp;
  LfWs w;
  lv_status e = lf_setup(widths, heights, n_views, 990000, workspace, ws_bytes, &vp, &w);
  if (e != LV_OK) return e;
  launch(k_lf_finish, 1, LV_MAX_VIEWS, 0, (cudaStream_t)stream)(vp, w.lsum, loss, true);
  count_launch(1);
  return cuda_check(cudaGetLastError(), "lv_lf_loss_finish");
}

namespace lv {
lv_status lf_fused_buffers(const int32_t* widths, const int32_t* heights, int n_views, void* workspace,
                           size_t ws_bytes, const float** w_out, const double** wsum, const float2** view_k,
                           double** lsum) {
  ViewPix vp;
  LfWs w;
  lv_status e = lf_setup(widths, heights, n_views, 990000, workspace, ws_bytes, &vp, &w);
  if (e != LV_OK) return e;
  *w_out = w.w;
  *wsum = w.wsum;
  *view_k = w.view_k;
  *lsum = w.lsum;
  return LV_OK;
}
}  // namespace lv

extern "C" lv_status lv_lf_weighted_loss(const float* rgb, const float* gt, const int32_t* widths,
                                         const int32_t* heights, int n_views, float t, const lv_lf_params* p,
                                         float* loss, float* dL_drgb, void* workspace, size_t ws_bytes,
                                         void* stream) {
  if (!rgb || !gt || !p || !loss) { set_error("null argument"); return LV_ERR_INVALID_ARG; }
  lv_status e = lv_lf_weights(gt, widths, heights, n_views, t, p, workspace, ws_bytes, stream);
  if (e != LV_OK) return e;
  return lv_lf_loss_from_weights(rgb, gt, widths, heights, n_views, loss, dL_drgb, workspace, ws_bytes, stream);
}

// ---------------------------------------------------------------- allocation-free variant
// For callers that cannot allocate device memory themselves: the scratch that
// lv_lf_weighted_loss takes from a caller workspace comes from this fixed
// array instead.  Every device that loads the library holds it until exit.
static __device__ __align__(256) unsigned char g_lf_scratch[LV_LF_NOALLOC_SCRATCH_BYTES];

namespace {
std::mutex g_lf_scratch_mu;
void* g_lf_scratch_ptr[256] = {};  // device address of g_lf_scratch per device ordinal

// The array's name is a host-side stand-in in host code; its device address is
// looked up once per device, with that device current.
lv_status lf_scratch_address(void** out) {
  int dev = 0;
  lv_status e = cuda_check(cudaGetDevice(&dev), "lv_lf_weighted_loss_noalloc: cudaGetDevice");
  if (e != LV_OK) return e;
  if (dev < 0 || dev >= 256) { set_error("lv_lf_weighted_loss_noalloc: device ordinal %d unsupported", dev); return LV_ERR_UNSUPPORTED; }
  std::lock_guard<std::mutex> lock(g_lf_scratch_mu);
  if (!g_lf_scratch_ptr[dev]) {
    void* ptr = nullptr;
    e = cuda_check(cudaGetSymbolAddress(&ptr, g_lf_scratch), "lv_lf_weighted_loss_noalloc: cudaGetSymbolAddress");
    if (e != LV_OK) return e;
    g_lf_scratch_ptr[dev] = ptr;
  }
  *out = g_lf_scratch_ptr[dev];
  return LV_OK;
}
}  // namespace

extern "C" lv_status lv_lf_weighted_loss_noalloc(const float* rgb, const float* gt, const int32_t* widths,
                                                 const int32_t* heights, int n_views, float t, const lv_lf_params* p,
                                                 float* loss, float* dL_drgb, void* stream) {
  const size_t need = lv_lf_workspace_size(widths, heights, n_views);
  if (need == 0) { set_error("lv_lf_weighted_loss_noalloc: bad view sizes"); return LV_ERR_INVALID_ARG; }
  if (need > sizeof(g_lf_scratch)) {
    set_error("lv_lf_weighted_loss_noalloc: these views need %zu bytes of scratch, the fixed array holds %zu "
              "(about 1.6 million pixels); use lv_lf_weighted_loss with a workspace instead",
              need, sizeof(g_lf_scratch));
    return LV_ERR_INVALID_ARG;
  }
  void* scratch = nullptr;
  lv_status e = lf_scratch_address(&scratch);
  if (e != LV_OK) return e;
  // lv_lf_weighted_loss clears its accumulators and selection histograms in the
  // scratch at the start of every call, so nothing else has to be zeroed here.
  return lv_lf_weighted_loss(rgb, gt, widths, heights, n_views, t, p, loss, dL_drgb, scratch, sizeof(g_lf_scratch),
                             stream);
}
