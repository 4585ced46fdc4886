// Preprocessing phase:
//   1. cull + count: every primitive -> number of tiles its rectangle covers (0 = culled): depth test on the mean, then
//      (attributes beyond the mean are only loaded for primitives in front of the camera) a lateral test from the scales
//      alone, and the covariance only for those that pass it;
//   2. scan of the counts (single-pass decoupled look-back) -> ascending list of visible primitives (the row map),
//      exclusive prefix of their tile counts (instance offsets), totals V and M, touched bitmask.  For scenes of up to
//      some 150,000 primitives 1 and 2 are one kernel, for larger ones 2 goes by the bitmask that 1 leaves;
//   3. rows: one thread per VISIBLE primitive recomputes the (deterministic) geometry and writes the compact record,
//      evaluates the SH colour and the opacity.
// At 2-30 % visibility recomputing the geometry of the visible rows is far cheaper than carrying per-primitive state
// through the block-wide scan.
#include "geom.cuh"
#include "layout.cuh"
#include "tilespan.cuh"

namespace {

struct Footprint {
  float u, v, depth, cA, cB, cC;
  int rad, x0, y0, x1, y1;
  uint32_t tiles;
};

// How the tile rectangle is chosen.  binning 0: the rectangle of the radius.  binning 1 (an optimised-pipeline variant
// in the sense of Sec. 5: same primitive ids, same image): additionally cut to the axis-aligned extent of the region in
// which alpha = opacity * exp(-q / 2) can reach alpha_min, q = d^T Sigma'^-1 d <= k = 2 ln(opacity / alpha_min), whose
// half extents are sqrt(k Sigma'_xx), sqrt(k Sigma'_yy) (widened by 1e-4 relative + 1e-3 pixels).  No pixel outside it
// passes the skip test of the blend kernels, so the instances that disappear never contributed.
struct BinRule {
  float dilation, radius_sigmas, alpha_min;
  int binning;
};

// Conic, radius and tile rectangle of one primitive.  Plain IEEE arithmetic (this file is compiled without fused
// multiply-add contraction): the integer results must not depend on which kernel evaluates them.
__device__ __forceinline__ Footprint project_footprint(const CamParams& cam, const BinRule& rule,
                                                      const float* __restrict__ means,
                                                      const float* __restrict__ log_scales,
                                                      const float4* __restrict__ quats,
                                                      const float* __restrict__ opacity_logit, size_t p) {
  const float dilation = rule.dilation, radius_sigmas = rule.radius_sigmas;
  Footprint f;
  f.tiles = 0; f.u = f.v = f.depth = f.cA = f.cB = f.cC = 0.f; f.rad = f.x0 = f.y0 = f.x1 = f.y1 = 0;
  SplatGeom g;
  odin_camera_space(cam, means[3 * p], means[3 * p + 1], means[3 * p + 2], g.t);
  if (!(g.t[2] > cam.znear && g.t[2] < cam.zfar)) return f;
  const float ls[3] = {log_scales[3 * p], log_scales[3 * p + 1], log_scales[3 * p + 2]};
  odin_splat_geometry(cam, dilation, ls, quats[p], g);
  if (!(g.det > 0.f)) return f;
  f.cA = g.c / g.det; f.cB = -g.b / g.det; f.cC = g.a / g.det;
  const float mid = (g.a + g.c) / 2.f;
  const float lam = mid + sqrtf(fmaxf(0.1f, mid * mid - g.det));
  const float radf = ceilf(radius_sigmas * sqrtf(lam));
  f.u = cam.fx * g.t[0] / g.t[2] + cam.cx;
  f.v = cam.fy * g.t[1] / g.t[2] + cam.cy;
  f.depth = g.t[2];
  const float ftx = (float)cam.TX, fty = (float)cam.TY;
  f.x0 = (int)fminf(ftx, fmaxf(0.f, floorf((f.u - radf) / 16.f)));
  f.x1 = (int)fminf(ftx, fmaxf(0.f, ceilf((f.u + radf) / 16.f)));
  f.y0 = (int)fminf(fty, fmaxf(0.f, floorf((f.v - radf) / 16.f)));
  f.y1 = (int)fminf(fty, fmaxf(0.f, ceilf((f.v + radf) / 16.f)));
  if (rule.binning == 1) {
    const float opac = 1.f / (1.f + expf(-opacity_logit[p]));
    if (!(opac >= rule.alpha_min)) {
      f.x1 = f.x0;  // never reaches alpha_min anywhere
    } else {
      const float k = 2.f * logf(opac / rule.alpha_min);
      const float ex = sqrtf(k * g.a) * 1.0001f + 1e-3f, ey = sqrtf(k * g.c) * 1.0001f + 1e-3f;
      // tiles that hold a pixel centre (i + 0.5) within [u - ex, u + ex]
      const int tx0 = (int)fminf(ftx, fmaxf(0.f, floorf((f.u - ex - 0.5f) / 16.f)));
      const int tx1 = (int)fminf(ftx, fmaxf(0.f, floorf((f.u + ex - 0.5f) / 16.f) + 1.f));
      const int ty0 = (int)fminf(fty, fmaxf(0.f, floorf((f.v - ey - 0.5f) / 16.f)));
      const int ty1 = (int)fminf(fty, fmaxf(0.f, floorf((f.v + ey - 0.5f) / 16.f) + 1.f));
      f.x0 = max(f.x0, tx0); f.x1 = max(f.x0, min(f.x1, tx1));
      f.y0 = max(f.y0, ty0); f.y1 = max(f.y0, min(f.y1, ty1));
    }
  }
  f.tiles = (uint32_t)(f.x1 - f.x0) * (uint32_t)(f.y1 - f.y0);
  f.rad = (int)fminf(radf, 2.0e9f);
  return f;
}

// packed look-back value: rows in the upper 28 bits, tile instances in the lower 34 bits
constexpr int PACK_SHIFT = 34;
constexpr uint64_t PACK_LOW = (1ull << PACK_SHIFT) - 1;
constexpr int SCAN_THREADS = 256;

// Cheap part of the footprint, for every primitive in front of the camera (t: camera-space mean, l: log scales): a
// lateral pre-test.  false = the exact rectangle is certainly empty.
// The lateral pre-test (most primitives of a large scene end up with no tile): a primitive in front of the camera whose
// centre lies farther from the image than a bound on its radius cannot touch a tile, and the bound needs neither the
// quaternion nor the covariance.  With T = J W (W a rotation) the projected covariance satisfies
// lambda_max(T Sigma T^T) <= |J|_F^2 s_max^2, |J|_F^2 <= (fx/z)^2 (1 + limx^2) + (fy/z)^2 (1 + limy^2), and the radius
// formula adds at most sqrt(0.1) to the larger eigenvalue; the bound is then widened by 1 % + 2 pixels, far beyond
// rounding.  Only primitives for which the exact rectangle is certainly empty leave here, so the result is unchanged.
__device__ __forceinline__ bool cull_survives(const CamParams& cam, const BinRule& rule, const float* t, float l0,
                                              float l1, float l2) {
  // hardware approximations (relative error ~1e-6) are enough here: the bound carries 1 % + 2 pixels of slack
  const float iz = __fdividef(1.f, t[2]);
  const float uc = cam.fx * t[0] * iz + cam.cx, vc = cam.fy * t[1] * iz + cam.cy;
  const float smax = __expf(fmaxf(l0, fmaxf(l1, l2)));
  const float jx = cam.fx * iz, jy = cam.fy * iz;
  const float jn2 = jx * jx * (1.f + cam.limx * cam.limx) + jy * jy * (1.f + cam.limy * cam.limy);
  float root;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(root) : "f"(jn2 * smax * smax + rule.dilation + 0.32f));
  const float rb = rule.radius_sigmas * root * 1.01f + 2.f;
  return !(uc + rb < 0.f || uc - rb > 16.f * (float)cam.TX || vc + rb < 0.f || vc - rb > 16.f * (float)cam.TY);
}

// Exact binning (binning 2): of the rectangle only the tiles the splat's alpha >= alpha_min region reaches
// (tilespan.cuh).  Called by all 32 lanes (f.tiles = 0 for lanes without a primitive): a lane counts a rectangle of few
// tile rows by itself; the tall ones of the warp are counted by all 32 lanes together.
__device__ __forceinline__ uint32_t exact_tiles_warp(const Footprint& f, const BinRule& rule,
                                                     const float* __restrict__ opacity_logit, size_t p) {
  const unsigned lane = threadIdx.x & 31;
  uint32_t tiles = f.tiles;
  SpanConic e;
  e.k = -1.f;
  if (tiles != 0) {
    const float opac = 1.f / (1.f + expf(-opacity_logit[p]));
    e = odin_span_conic(f.u, f.v, f.cA, f.cB, f.cC, opac, rule.alpha_min);
  }
  const bool tall = tiles != 0 && f.y1 - f.y0 > 4;
  if (tiles != 0 && !tall) {
    uint32_t kept = 0;
    for (int ty = f.y0; ty < f.y1; ++ty) {
      int xa, xb;
      odin_row_span(e, ty, f.x0, f.x1, xa, xb);
      kept += (uint32_t)(xb - xa);
    }
    tiles = kept;
  }
  uint32_t todo = __ballot_sync(0xffffffffu, tall);
  while (todo) {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    const SpanConic c = odin_span_conic_bcast(e, src);
    const uint32_t kept =
        odin_rect_kept_warp(c, __shfl_sync(0xffffffffu, f.x0, src), __shfl_sync(0xffffffffu, f.y0, src),
                            __shfl_sync(0xffffffffu, f.x1, src), __shfl_sync(0xffffffffu, f.y1, src));
    if ((int)lane == src) tiles = kept;
  }
  return tiles;
}

// Counting kernel for large scenes.  A warp takes 32 x CULL_ITEMS consecutive primitives: the cheap tests of all of them first,
// their loads in flight together (means -> depth test -> log scales of those in front of the camera -> lateral test); the
// survivors are listed in shared memory and taken 32 at a time through the covariance code, so its lanes are full.  What bounds
// it: the stream of means and scales where few primitives are visible, that code where many are (1 M, 32 % visible: 69 % of
// the issue slots, DRAM 25 %; 2.8 M, 28 % visible: 75 %, 29 %).  Before, with one primitive per
// thread, nearly every warp went through it for a fifth of its lanes.  Measured, before -> now: 5 M primitives of which 16 % are
// visible 101 -> 54 us; 20 M, 2 % visible 105 -> 85; 1 M, 33 % visible 26 -> 21; 2.8 M in runs all visible or all not 33 -> 35.
// Two primitives per lane leave the lists short (5 M: 70 us), eight leave too few warps to even out the work (1 M: 23,
// 400 k: 35); blocks of 256 end later than blocks of 128, blocks of 64 are too many for 20 M (97).
constexpr int CULL_ITEMS = 4, CULL_THREADS = 128, CULL_WARPS = CULL_THREADS / 32;
static_assert(256 % (32 * CULL_ITEMS) == 0, "a warp's primitives are of one group of 256");

template <bool EXACT>
__global__ void __launch_bounds__(CULL_THREADS, 10)
project_cull_kernel(const float* __restrict__ means, const float* __restrict__ log_scales, const float4* __restrict__ quats,
                    const float* __restrict__ opacity_logit, uint32_t n, CamParams cam, BinRule rule,
                    uint32_t* __restrict__ tiles_touched, unsigned long long* __restrict__ group_total,
                    unsigned long long* __restrict__ chunk_total, uint32_t groups_per_chunk, uint32_t* __restrict__ visible_mask) {
  odin_after_predecessor();
  __shared__ uint32_t s_tiles[CULL_WARPS][32 * CULL_ITEMS];
  __shared__ uint8_t s_lists[CULL_WARPS][32 * CULL_ITEMS];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* s_t = s_tiles[warp];
  uint8_t* s_list = s_lists[warp];
  const uint32_t base = (blockIdx.x * CULL_WARPS + warp) * (32 * CULL_ITEMS);
  if (base >= n) return;
  float c[CULL_ITEMS][3];  // mean, then camera-space mean
#pragma unroll
  for (int j = 0; j < CULL_ITEMS; ++j) {
    const uint32_t p = base + 32 * j + lane;
    c[j][0] = c[j][1] = c[j][2] = 0.f;
    if (p < n) { c[j][0] = means[3 * (size_t)p]; c[j][1] = means[3 * (size_t)p + 1]; c[j][2] = means[3 * (size_t)p + 2]; }
  }
  float l[CULL_ITEMS][3];
  bool front[CULL_ITEMS];
#pragma unroll
  for (int j = 0; j < CULL_ITEMS; ++j) {
    const uint32_t p = base + 32 * j + lane;
    const float mx = c[j][0], my = c[j][1], mz = c[j][2];
    odin_camera_space(cam, mx, my, mz, c[j]);
    front[j] = p < n && c[j][2] > cam.znear && c[j][2] < cam.zfar;
    l[j][0] = l[j][1] = l[j][2] = 0.f;
    if (front[j]) { l[j][0] = log_scales[3 * (size_t)p]; l[j][1] = log_scales[3 * (size_t)p + 1]; l[j][2] = log_scales[3 * (size_t)p + 2]; }
  }
  uint32_t listed = 0;
#pragma unroll
  for (int j = 0; j < CULL_ITEMS; ++j) {
    const bool alive = front[j] && cull_survives(cam, rule, c[j], l[j][0], l[j][1], l[j][2]);
    const uint32_t b = __ballot_sync(0xffffffffu, alive);
    if (alive) s_list[listed + __popc(b & ((1u << lane) - 1u))] = (uint8_t)(32 * j + lane);
    listed += __popc(b);
    s_t[32 * j + lane] = 0;
  }
  __syncwarp();
  for (uint32_t i0 = 0; i0 < listed; i0 += 32) {
    const bool have = i0 + lane < listed;
    const uint32_t q = have ? s_list[i0 + lane] : 0u, p = base + q;
    Footprint f = {};
    if (have) f = project_footprint(cam, rule, means, log_scales, quats, opacity_logit, p);
    if (EXACT) f.tiles = exact_tiles_warp(f, rule, opacity_logit, p);
    if (have) s_t[q] = f.tiles;
  }
  __syncwarp();
  uint32_t rows = 0, inst = 0;  // instances: at most 2^20 per primitive, 2^27 per warp
#pragma unroll
  for (int j = 0; j < CULL_ITEMS; ++j) {
    const uint32_t p = base + 32 * j + lane, t = s_t[32 * j + lane];
    if (p < n) tiles_touched[p] = t;
    // (32 primitives are one word of the mask that the list is made from)
    const uint32_t visible = __ballot_sync(0xffffffffu, t != 0);
    if (lane == 0 && base + 32 * j < n) visible_mask[(base + 32 * j) >> 5] = visible;
    rows += __popc(visible);
    inst += t;
  }
  // what the list needs to start anywhere without waiting: the packed (rows, instances) total of every 256 primitives and the
  // exact totals of the share they belong to, added up by the warps that have something to add (both zeroed before the
  // launch; no block barrier, so a warp with a long covariance path holds nobody up)
  if (rows == 0) return;
  inst = __reduce_add_sync(0xffffffffu, inst);
  if (lane == 0) {
    atomicAdd(&group_total[base / 256], ((unsigned long long)rows << PACK_SHIFT) | (unsigned long long)inst);
    const size_t g = base / 256 / groups_per_chunk;
    atomicAdd(&chunk_total[2 * g], (unsigned long long)rows);
    atomicAdd(&chunk_total[2 * g + 1], (unsigned long long)inst);
  }
}

// Position of the set bit of w in front of which there are r others.
__device__ __forceinline__ uint32_t nth_bit(uint32_t w, uint32_t r) {
  uint32_t pos = 0;
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    const uint32_t c = __popc(w & ((1u << s) - 1u));
    if (r >= c) {
      r -= c;
      pos += s;
      w >>= s;
    }
  }
  return pos;
}

// Row map and instance offsets behind project_cull_kernel.  A block takes `rounds` x 2048 primitives; the packed totals of every
// 256 primitives and the exact totals of every block's share are there, so its base is a sum over the shares in front of it
// and nothing is waited for.  A warp takes `rounds` consecutive groups of 256, a word of their visible mask per lane, and goes
// through the visible ones 64 at a time: lane i looks up set bits i and 32 + i, and the writes are side by side.
// What bounds it: a few dependent loads per block.  Next to no shared memory on purpose: the kernels behind are started
// while this one ends, on SMs that keep its division of their memory into shared memory and cache (with a list of the
// visible primitives in 33 KB, the whole step took 1,073 instead of 1,033 us for 2.8 M primitives).  All tile counts read,
// round after round of 256 per warp, and one warp summing the shares, took 47 us for 20 M primitives, 2 % of them visible;
// this way 27 (5 M: 27 -> 13; 2.8 M, 30 % visible: 13 -> 17, hidden behind the kernel in front: the step is the same).
constexpr int LIST_THREADS = 256, LIST_WARPS = LIST_THREADS / 32, LIST_MAX_ROUNDS = 4, LIST_WIDE = 2;
static_assert(LIST_WARPS * 256 == (int)PROJECT_TILE && LIST_MAX_ROUNDS * 8 <= 32, "a warp's mask words are one per lane at most");

__global__ void __launch_bounds__(LIST_THREADS)
project_list_kernel(uint32_t n, const uint32_t* __restrict__ tiles_touched, const uint32_t* __restrict__ visible_mask,
                    uint32_t capacity, uint32_t* __restrict__ prim_id, uint32_t* __restrict__ tile_offset,
                    uint32_t* __restrict__ num_rows, uint64_t* __restrict__ num_instances,
                    const uint64_t* __restrict__ group_total, const uint64_t* __restrict__ chunk_total, int* status, int rounds) {
  odin_after_predecessor();  // launched behind the counting kernel
  __shared__ uint64_t s_rows[LIST_WARPS], s_inst[LIST_WARPS], s_tot[LIST_WARPS * LIST_MAX_ROUNDS];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tile = blockIdx.x, groups = (n + 255) / 256, n_words = (n + 31) / 32;
  const uint32_t word0 = (tile * LIST_WARPS + warp) * 8 * rounds;  // the warp's first mask word
  const uint32_t w = (int)lane < 8 * rounds && word0 + lane < n_words ? visible_mask[word0 + lane] : 0u;
  // the block's base: all shares in front of it
  const ulonglong2* shares = reinterpret_cast<const ulonglong2*>(chunk_total);
  uint64_t rows = 0, inst = 0;
  for (uint32_t c = threadIdx.x; c < tile; c += LIST_THREADS) {
    const ulonglong2 x = shares[c];
    rows += x.x;
    inst += x.y;
  }
  if (threadIdx.x < LIST_WARPS * rounds) {
    const uint32_t g = tile * LIST_WARPS * rounds + threadIdx.x;
    s_tot[threadIdx.x] = g < groups ? group_total[g] : 0ull;
  }
  uint32_t upto = __popc(w);  // visible primitives up to and with the lane's word
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, upto, o);
    if ((int)lane >= o) upto += x;
  }
  const uint32_t listed = __shfl_sync(0xffffffffu, upto, 31);
  uint32_t p[LIST_WIDE], t[LIST_WIDE];  // of the next entries, on their way while others are scanned
  auto fetch = [&](uint32_t i0) {
#pragma unroll
    for (int h = 0; h < LIST_WIDE; ++h) {
      const uint32_t i = i0 + 32 * h + lane;
      uint32_t at = 0;  // lanes whose words end in front of entry i
#pragma unroll
      for (int s = 16; s > 0; s >>= 1)
        if (__shfl_sync(0xffffffffu, upto, at + s - 1) <= i) at += s;
      const uint32_t word = __shfl_sync(0xffffffffu, w, at), end = __shfl_sync(0xffffffffu, upto, at);
      p[h] = t[h] = 0;
      if (i < listed) {
        p[h] = (word0 + at) * 32 + nth_bit(word, i - (end - __popc(word)));
        t[h] = tiles_touched[p[h]];
      }
    }
  };
  fetch(0);
  for (int o = 16; o > 0; o >>= 1) {
    rows += __shfl_xor_sync(0xffffffffu, rows, o);
    inst += __shfl_xor_sync(0xffffffffu, inst, o);
  }
  if (lane == 0) { s_rows[warp] = rows; s_inst[warp] = inst; }
  __syncthreads();
  rows = inst = 0;
#pragma unroll
  for (int k = 0; k < LIST_WARPS; ++k) { rows += s_rows[k]; inst += s_inst[k]; }
  // 2^32 instances or more are an error by definition: the packed base is saturated so that the row field stays intact and
  // every write stays inside the caller's capacities (the row guard below)
  uint64_t run = (rows << PACK_SHIFT) | (inst < (1ull << 32) ? inst : ((1ull << 32) - 1));
  if (tile == gridDim.x - 1 && threadIdx.x == 0) {  // last block: totals
    rows += shares[tile].x;
    inst += shares[tile].y;
    *num_rows = (uint32_t)(rows < capacity ? rows : capacity);
    *num_instances = inst;
    if (rows > capacity || inst >= (1ull << 32)) odin_set_error(status, ODIN_ERR_CAPACITY);
  }
  if (listed == 0) return;
  uint64_t front = (int)lane < (int)warp * rounds ? s_tot[lane] : 0ull;  // the block's groups in front of the warp's
  for (int o = 16; o > 0; o >>= 1) front += __shfl_xor_sync(0xffffffffu, front, o);
  run += front;
  for (uint32_t i0 = 0; i0 < listed; i0 += 32 * LIST_WIDE) {
    uint32_t prim[LIST_WIDE], tiles[LIST_WIDE], inc[LIST_WIDE];
#pragma unroll
    for (int h = 0; h < LIST_WIDE; ++h) { prim[h] = p[h]; inc[h] = tiles[h] = t[h]; }  // (32 x 2^20 fits)
    if (i0 + 32 * LIST_WIDE < listed) fetch(i0 + 32 * LIST_WIDE);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
      for (int h = 0; h < LIST_WIDE; ++h) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, inc[h], o);
        if ((int)lane >= o) inc[h] += x;
      }
#pragma unroll
    for (int h = 0; h < LIST_WIDE; ++h) {
      const uint64_t e = run + ((uint64_t)lane << PACK_SHIFT) + (inc[h] - tiles[h]), r = e >> PACK_SHIFT;
      if (i0 + 32 * h + lane < listed && r < capacity) {
        prim_id[r] = prim[h];
        tile_offset[r] = (uint32_t)(e & PACK_LOW);
      }
      run += ((uint64_t)32 << PACK_SHIFT) + __shfl_sync(0xffffffffu, inc[h], 31);
    }
  }
}

// Counting and scan in one kernel, for scenes of no more primitives than there are resident threads, where a kernel launch and a
// pass over the counts are what there is to save.  A block takes 256 consecutive primitives by ticket, one per thread, so that
// the 32 primitives of a warp are one word of the touched bitmask.
//   A. the tile counts: depth test on the mean, lateral test with the scales, then the exact footprint;
//   B. packed (rows, instances) total of the block, ONE decoupled look-back;
//   C. ranks by population count and a 32-bit scan -> row map, instance offsets, touched bitmask.
template <bool EXACT>  // binning 2
__global__ void __launch_bounds__(SCAN_THREADS, EXACT ? 3 : 4)
project_scan_kernel(const float* __restrict__ means, const float* __restrict__ log_scales,
                    const float4* __restrict__ quats, const float* __restrict__ opacity_logit, uint32_t n, CamParams cam,
                    BinRule rule, uint32_t* tiles_touched, uint32_t capacity, uint32_t* __restrict__ prim_id,
                    uint32_t* __restrict__ tile_offset, uint32_t* __restrict__ num_rows,
                    uint64_t* __restrict__ num_instances, uint32_t* ticket, uint64_t* state,
                    int* status, int spin_limit, uint32_t* __restrict__ touched_mask) {
  odin_after_predecessor();
  __shared__ uint32_t s_tile;
  __shared__ uint64_t s_warp[SCAN_THREADS / 32];  // rows and instances of the warps
  __shared__ uint64_t s_inst[SCAN_THREADS / 32];
  __shared__ uint64_t s_base;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long* exact_instances = reinterpret_cast<unsigned long long*>(ticket + 2);  // zeroed with the ticket
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
  __syncthreads();
  const uint32_t tile = s_tile, p = tile * SCAN_THREADS + threadIdx.x;
  // ---- A
  Footprint f = {};
  if (p < n) {
    float c[3];
    odin_camera_space(cam, means[3 * (size_t)p], means[3 * (size_t)p + 1], means[3 * (size_t)p + 2], c);
    if (c[2] > cam.znear && c[2] < cam.zfar &&
        cull_survives(cam, rule, c, log_scales[3 * (size_t)p], log_scales[3 * (size_t)p + 1], log_scales[3 * (size_t)p + 2]))
      f = project_footprint(cam, rule, means, log_scales, quats, opacity_logit, p);
  }
  if (EXACT) f.tiles = exact_tiles_warp(f, rule, opacity_logit, p);
  const uint32_t t = f.tiles;
  if (p < n) tiles_touched[p] = t;
  const uint32_t visible = __ballot_sync(0xffffffffu, t != 0);
  if (touched_mask && lane == 0 && p < n) touched_mask[p >> 5] = visible;
  uint32_t inc = t;  // (32 x 2^20 fits)
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= (unsigned)o) inc += y;
  }
  if (lane == 31) {
    s_warp[warp] = __popc(visible);
    s_inst[warp] = inc;
  }

  // ---- B.  The instance field of the packed value holds 34 bits and there are up to 2^10 blocks of up to 2^8 x 2^20
  // instances, so the packed sums can carry into the row field when the view has 2^32 instances or more (an error by
  // definition).  That case is caught on a counter of its own: every block adds its exact instance count (kept apart
  // in 64 bits, the packed copy saturated) to a 64-bit total, and whoever sees that total reach 2^32 reports
  // ODIN_ERR_CAPACITY.  The outputs of such a view are meaningless but every write stays inside the caller's
  // capacities (the row guard below).
  __syncthreads();
  if (threadIdx.x < 32) {
    uint64_t total = (lane < SCAN_THREADS / 32) ? s_warp[lane] : 0ull;
    uint64_t total_inst = (lane < SCAN_THREADS / 32) ? s_inst[lane] : 0ull;
    for (int o = 16; o > 0; o >>= 1) {
      total += __shfl_xor_sync(0xffffffffu, total, o);
      total_inst += __shfl_xor_sync(0xffffffffu, total_inst, o);
    }
    if (lane == 0 && total_inst != 0) {
      const unsigned long long seen = atomicAdd(exact_instances, (unsigned long long)total_inst);
      if (seen + total_inst >= (1ull << 32)) odin_set_error(status, ODIN_ERR_CAPACITY);
    }
    total = (total << PACK_SHIFT) | (total_inst < (1ull << 32) ? total_inst : ((1ull << 32) - 1));
    const uint64_t base = odin_lookback_u64(state, tile, total, status, spin_limit);
    if (lane == 0) {
      s_base = base;
      if (tile == gridDim.x - 1) {  // last block: totals
        const uint64_t all = base + total;
        const uint64_t rows = all >> PACK_SHIFT, inst = all & PACK_LOW;
        *num_rows = (uint32_t)(rows < capacity ? rows : capacity);
        *num_instances = inst;
        if (rows > capacity || inst >= (1ull << 32)) odin_set_error(status, ODIN_ERR_CAPACITY);
      }
    }
  }
  __syncthreads();

  // ---- C
  if (t == 0) return;
  uint64_t run = s_base;
  for (int w = 0; w < (int)warp; ++w) run += (s_warp[w] << PACK_SHIFT) + s_inst[w];
  const uint64_t e = run + ((uint64_t)__popc(visible & ((1u << lane) - 1u)) << PACK_SHIFT) + (inc - t), r = e >> PACK_SHIFT;
  if (r < capacity) {
    prim_id[r] = p;
    tile_offset[r] = (uint32_t)(e & PACK_LOW);
  }
}

template <int DEG>
__global__ void __launch_bounds__(128)
project_rows_kernel(const float* __restrict__ means, const float* __restrict__ log_scales, const float4* __restrict__ quats,
                    const float* __restrict__ opacity_logit, const float* __restrict__ sh, CamParams cam, BinRule rule,
                    odin_projected out, uint32_t n, float* __restrict__ grad2d, uint8_t* __restrict__ row_active) {
  odin_after_predecessor();
  constexpr int K = (DEG + 1) * (DEG + 1);
  const uint32_t V = min(*out.num_rows, out.capacity);
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t r0 = blockIdx.x * blockDim.x + threadIdx.x - lane; r0 < V; r0 += gridDim.x * blockDim.x) {
    const uint32_t r = r0 + lane;
    if (grad2d) {  // a view step: the sums of the backward pass start at zero (the warp's 32 rows are consecutive words)
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const size_t w = (size_t)r0 * 9 + 32 * k + lane;
        if (w < (size_t)V * 9) grad2d[w] = 0.f;
      }
      if (row_active && r < V) row_active[r] = 0;
    }
    if (r >= V) break;
    const size_t p = min(out.prim_id[r], n - 1);  // in range even if the scan gave up and left part of the map unwritten
    const Footprint f = project_footprint(cam, rule, means, log_scales, quats, opacity_logit, p);
    reinterpret_cast<float2*>(out.xy)[r] = make_float2(f.u, f.v);
    out.depth[r] = f.depth;
    const float o = 1.f / (1.f + expf(-opacity_logit[p]));
    reinterpret_cast<float4*>(out.conic_opacity)[r] = make_float4(f.cA, f.cB, f.cC, o);
    out.radius[r] = f.rad;
    reinterpret_cast<ushort4*>(out.rect)[r] =
        make_ushort4((unsigned short)f.x0, (unsigned short)f.y0, (unsigned short)f.x1, (unsigned short)f.y1);
    // colour
    float dx = means[3 * p] - cam.pos[0], dy = means[3 * p + 1] - cam.pos[1], dz = means[3 * p + 2] - cam.pos[2];
    const float len = sqrtf(dx * dx + dy * dy + dz * dz);
    dx /= len; dy /= len; dz /= len;
    float Y[16];
    odin_sh_basis<DEG>(dx, dy, dz, Y);
    float acc[3] = {0.f, 0.f, 0.f};
    const float* row = sh + p * (3 * K);
    if ((3 * K) % 4 == 0) {  // 12 or 48 floats: 16-byte loads
      const float4* row4 = reinterpret_cast<const float4*>(row);
#pragma unroll
      for (int i = 0; i < 3 * K / 4; ++i) {
        const float4 c = row4[i];
        const float e[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int w = 4 * i + j;
          acc[w % 3] += Y[w / 3] * e[j];
        }
      }
    } else {
#pragma unroll
      for (int w = 0; w < 3 * K; ++w) acc[w % 3] += Y[w / 3] * row[w];
    }
    uint8_t flags = 0;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      acc[ch] += 0.5f;
      if (acc[ch] < 0.f) { acc[ch] = 0.f; flags |= (uint8_t)(1u << ch); }
    }
    out.rgb[3 * (size_t)r] = acc[0]; out.rgb[3 * (size_t)r + 1] = acc[1]; out.rgb[3 * (size_t)r + 2] = acc[2];
    out.clamp_flags[r] = flags;
  }
}

}  // namespace

extern "C" int odin_project(odin_ctx* ctx, const odin_scene* scene, const odin_camera* cam, odin_projected* out, void* ws,
                            size_t ws_bytes, void* stream) {
  if (!ctx || !out) return ODIN_ERR_NULL;
  int rc = odin_check_scene(scene);
  if (rc != ODIN_OK) return rc;
  rc = odin_check_camera(cam);
  if (rc != ODIN_OK) return rc;
  if (!out->num_rows || !out->num_instances) return ODIN_ERR_NULL;
  if (out->capacity > 0 && (!out->prim_id || !out->xy || !out->depth || !out->conic_opacity || !out->rgb || !out->radius ||
                            !out->rect || !out->tile_offset || !out->clamp_flags))
    return ODIN_ERR_NULL;
  if (!odin_aligned(out->xy, 8) || !odin_aligned(out->conic_opacity, 16) || !odin_aligned(out->rect, 8) ||
      !odin_aligned(out->num_instances, 8))
    return ODIN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const uint32_t n = scene->n;
  if (n == 0) {
    odin_chain_break(ctx);
    ODIN_CUDA(cudaMemsetAsync(out->num_rows, 0, 4, st));
    ODIN_CUDA(cudaMemsetAsync(out->num_instances, 0, 8, st));
    return ODIN_OK;
  }
  if (!out->tiles_touched) return ODIN_ERR_NULL;
  const size_t need = project_ws_bytes(n);
  if (!ws || !odin_aligned(ws, 256) || ws_bytes < need) return ODIN_ERR_WORKSPACE;
  ODIN_CUDA(odin_zero(ctx, ws, project_ws_mask_offset(n), st));
  uint32_t* ticket = reinterpret_cast<uint32_t*>(ws);
  const CamParams cp = odin_cam_params(cam, ctx->cfg);
  const float4* q4 = reinterpret_cast<const float4*>(scene->quats);
  const BinRule rule = {ctx->cfg.dilation, ctx->cfg.radius_sigmas, ctx->cfg.alpha_min, ctx->cfg.binning};
  // Scenes of one primitive per thread of the blocks that are resident at once take the kernel that counts and scans; larger ones
  // a counting kernel at full occupancy and the list from its mask.  (With up to eight primitives per thread in the fused
  // kernel, that is up to 1.2 M primitives, each warp went through a chain of eight rounds of its survivors: 1 M primitives
  // 26 us against 20 + 4, 273 k 18 against 8 + 2; 1,024 primitives 18.3 us against 8.8 with one per thread.)
  const bool fused = n <= (uint32_t)ctx->sm_count * 4u * SCAN_THREADS;
  if (fused) {
    OdinKernelScope ks(ctx, K_PROJECT, st);
    auto kernel = rule.binning == 2 ? project_scan_kernel<true> : project_scan_kernel<false>;
    uint64_t* states = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(ws) + project_ws_group_offset(n));  // one per block
    ODIN_CUDA(odin_launch(ctx, false, kernel, dim3((n + SCAN_THREADS - 1) / SCAN_THREADS), dim3(SCAN_THREADS), 0, st, scene->means,
                          scene->log_scales, q4, scene->opacity_logit, n, cp, rule, out->tiles_touched, out->capacity,
                          out->prim_id, out->tile_offset, out->num_rows, out->num_instances, ticket, states, ctx->d_status,
                          ctx->spin_limit, out->touched_mask));
  } else {
    // few shares to sum, about one wave of blocks; at most a mask word per lane of a warp
    const int most = scan_rounds_for(n, ctx->sm_count), rounds = most < LIST_MAX_ROUNDS ? most : LIST_MAX_ROUNDS;
    const uint32_t share = PROJECT_TILE * (uint32_t)rounds;
    uint64_t* group_total = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(ws) + project_ws_group_offset(n));
    uint64_t* chunk_total = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(ws) + project_ws_chunk_offset(n));
    // the mask of the visible primitives, in the workspace if the caller does not want it
    uint32_t* visible = out->touched_mask ? out->touched_mask : reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(ws) + project_ws_mask_offset(n));
    {
      OdinKernelScope ks(ctx, K_PROJECT, st);
      auto kernel = rule.binning == 2 ? project_cull_kernel<true> : project_cull_kernel<false>;
      ODIN_CUDA(odin_launch(ctx, false, kernel, dim3((n + CULL_THREADS * CULL_ITEMS - 1) / (CULL_THREADS * CULL_ITEMS)),
                            dim3(CULL_THREADS), 0, st, scene->means, scene->log_scales, q4, scene->opacity_logit, n, cp, rule,
                            out->tiles_touched, reinterpret_cast<unsigned long long*>(group_total),
                            reinterpret_cast<unsigned long long*>(chunk_total), share / 256, visible));
    }
    OdinKernelScope ks(ctx, K_PROJECT_SCAN, st);
    ODIN_CUDA(odin_launch(ctx, true, project_list_kernel, dim3((n + share - 1) / share), dim3(LIST_THREADS), 0, st, n,
                          out->tiles_touched, visible, out->capacity, out->prim_id, out->tile_offset, out->num_rows,
                          out->num_instances, group_total, chunk_total, ctx->d_status, rounds));
  }
  if (out->capacity == 0) return odin_launch_status();
  const uint32_t blocks_cap = (out->capacity + 127) / 128;
  const uint32_t grid = blocks_cap < (uint32_t)ctx->sm_count * 16 ? blocks_cap : (uint32_t)ctx->sm_count * 16;
  OdinKernelScope ks(ctx, K_PROJECT_ROWS, st);
#define LAUNCH(D)                                                                                                      \
  ODIN_CUDA(odin_launch(ctx, true, project_rows_kernel<D>, dim3(grid), dim3(128), 0, st, scene->means,                 \
                        scene->log_scales, q4, scene->opacity_logit, scene->sh, cp, rule, *out, n, ctx->view_grad2d, ctx->view_row_active))
  switch (scene->sh_degree) {
    case 0: LAUNCH(0); break;
    case 1: LAUNCH(1); break;
    case 2: LAUNCH(2); break;
    default: LAUNCH(3); break;
  }
#undef LAUNCH
  return odin_launch_status();
}
