// Shared by the compositing kernels and their backward: how a tile is divided among warps, segments of long lists, and the
// per-row quantities that all of them must evaluate with exactly the same arithmetic (so that skip / clamp decisions agree).
//
// Per row of a tile's sorted list and pixel, with (dx, dy) = row centre - pixel centre,
//     p = (sA dx^2 + lo) + dy (sB dx + sC dy)          (see BlendRow),   alpha = min(alpha_max, 2^p),
// and alpha = 0 where a skip test fails: what follows is straight-line code in which such a pixel changes nothing (where
// something is not a number: blend_tame).  These kernels are bound by instruction issue, so everything between the exponent
// and the sums runs on packed fp32x2 registers (two pixels of a column, or two rows at one pixel): fma.rn.f32x2 rounds each
// half as the scalar instruction does and takes one issue slot.
//
// Division of work.  A tile is four STRIPS of 16 x 4 pixels, a strip two CELLS of 8 x 4.
//   Images of BLEND_FULL_TILES tiles and more fill the GPU with large regions, whose warps load a row and its terms once for
//   many pixels: the forward head kernel takes half tiles (four pixels per lane), the backward kernel whole tiles (eight).
//   In a smaller image, and beyond BLEND_HEAD entries of any list, the chain of dependent work per warp decides: forward
//   cells (one pixel per lane, two warps per strip), backward strips (two pixels per lane).  A row is evaluated by a warp
//   only if its ellipse reaches the warp's region, so small regions also skip more.
// Measured (with the one-warp-per-tile kernels before): 64 x 64 pixels, lists of up to 400: forward 104 -> 21 us, backward
// 141 -> 42; 320 x 180, lists of up to 9,000: 591 -> 298 and 208 -> 110; 800 x 600: 105 -> 75 and 178 -> 106; 1600 x 1066 with
// splats of some thirty tiles: 203 -> 173 and 330 -> 240; 1920 x 1080 with splats of a few pixels: 346 -> 271 and 470 -> 421.
#pragma once
#include "common.cuh"

// Long lists.  Forward: where half tiles are taken, what is still live after BLEND_HEAD list entries goes to the tail kernel
// strip by strip, the per-pixel state travelling through the output images.  All kernels evaluate dx and dy as one
// subtraction from the pixel centre, so a pixel sees bit-identical alpha in each of them.
// Backward: the list of a tile is cut into SEGMENTS of BLEND_HEAD entries (see below) that are replayed independently, one warp
// each, all in one launch.  What a segment needs is the state of every pixel at its END: the transmittance and the
// colour still to come behind it.  The forward tail and strip kernels leave exactly that in the workspace: for every
// BLEND_HEAD entries they walk beyond the first BLEND_HEAD they take a segment slot from a counter and store, for the 64
// pixels of the strip, the transmittance before those entries and the colour they added; when the strip is finished they walk
// its slots from the last to the first and replace "colour added" by the running sum "colour still to come" (summed from the back,
// small terms first, as the sequential replay would: a difference final colour - colour so far would lose the small
// suffixes of nearly saturated pixels to rounding).  So the backward pass has no sequential tail at all, and the
// workspace of odin_render_bwd must be the one the odin_render_fwd of the same view used.
constexpr uint32_t BLEND_HEAD = 256;
constexpr uint32_t BLEND_DONE_BIT = 0x80000000u;  // in n_contrib while a strip is between two forward kernels
constexpr int BLEND_STRIPS = 4;                   // strips of 16 x 4 pixels per tile
constexpr int BLEND_STRIP_PIXELS = 64;
// From here on whole tiles and half tiles.  Forward + backward with them / with strips, us, by tiles of the image:
//   400 k primitives, unbounded:   448: 170 / 128    700: 174 / 171    920: 188 / 198   1,170: 192 / 220   2,040: 209 / 339
//   100 k primitives, blob:        448: 203 / 151    700: 225 / 200    920: 229 / 226   1,170: 229 / 247   2,040: 242 / 366
//   2.8 M, city from the air:    1,170: 534 / 486  1,450: 532 / 519  2,040: 539 / 579   3,600: 612 / 722
//   2.8 M, city from the street: 1,450: 478 / 458  2,040: 475 / 452  2,800: 440 / 458   3,600: 422 / 472
constexpr int BLEND_FULL_TILES = 1024;
constexpr uint32_t BLEND_SPARES = 1024;           // blocks that hold a slot in advance, at most; as many pairs of warps, twice

// Segments.  Their length is the length of a chain: BLEND_HEAD entries keep the number of records down, but an image of few
// tiles has few strips, and its backward pass takes as long as one segment.  Images of up to BLEND_SMALL_TILES tiles cut the first
// BLEND_FINE_END entries of a list into segments of BLEND_FINE.  Backward and forward: 64 x 64 pixels 41 -> 22 us and 17 -> 18;
// 206 x 105, lists of up to 4,100, 61 -> 44 and 41 -> 49; 238 x 123 34 -> 24 and 13 -> 14.  From some 200 tiles on the
// records cost more than the shorter chains give: 256 x 256 66 -> 57 and 48 -> 60; 320 x 180 148 -> 162 and 206 -> 217.
constexpr int BLEND_SMALL_TILES = 128;
constexpr uint32_t BLEND_FINE = 64, BLEND_FINE_END = 1024;
__host__ __device__ inline bool blend_fine(int n_tiles) { return n_tiles <= BLEND_SMALL_TILES; }
// length of the segment that begins at entry `off`; first entry of segment k; segment that begins at entry `off`
__host__ __device__ inline uint32_t blend_seg_length(uint32_t off, bool fine) { return fine && off < BLEND_FINE_END ? BLEND_FINE : BLEND_HEAD; }
__host__ __device__ inline uint32_t blend_seg_begin(uint32_t k, bool fine) {
  if (!fine) return k * BLEND_HEAD;
  constexpr uint32_t F = BLEND_FINE_END / BLEND_FINE;
  return k < F ? k * BLEND_FINE : BLEND_FINE_END + (k - F) * BLEND_HEAD;
}
__host__ __device__ inline uint32_t blend_seg_at(uint32_t off, bool fine) {
  if (!fine) return off / BLEND_HEAD;
  constexpr uint32_t F = BLEND_FINE_END / BLEND_FINE;
  return off < BLEND_FINE_END ? off / BLEND_FINE : F + (off - BLEND_FINE_END) / BLEND_HEAD;
}

// Workspace of the render calls (every region 256-byte aligned):
//   [256 B: u32 [0] ticket of the forward kernel, [1] work ticket of the backward kernel, [2] segment slots taken,
//           [3] ticket of the forward tail kernel, [4..7] strips queued for it in each of four classes
//           of list length, [8..23] items in each of the sixteen classes of the backward kernel's work order,
//           [24] ticket of the forward strip kernel behind the tail kernel, [25] strips queued for it]
//   [tile_work: u32 x tiles    rows evaluated by the tile's head warps, and how many of them are done]
//   [strip_first: u32 x strips 1 + slot of the strip's second segment (0 = none)]
//   [tail_queue: u32 x 4 x strips  strips the tail kernel takes over, one region per class, longest lists first;
//                              behind the third class's: those that it hands on to the strip kernel]
//   [bwd_queue: u32 x 16 x items  all items (tiles, or strips) in sixteen classes of rows evaluated: work order of the
//                              backward kernel]
//   [seg_strip: uint2 x S      (strip, k): the slot holds the state before segment k of that strip's list]
//   [seg_link: uint2 x S       1 + slot of the same strip's segment k + 1, of segment k - 1 (0 = none)]
//   [ckpt: BlendRecord x 64 x S   per pixel (32 * cell + lane of the cell's warp): T, colour to come (3)]
// S, the number of segment slots, follows from the size of the workspace the caller passes; the minimum size holds
// 2 x tiles + 4096 records of a whole tile's four strips (and a slot for every block that takes one in advance, and what the
// shorter segments of a small image need on top).
// Work order of the backward kernel over the first segments: sixteen classes by the number of rows the forward kernel
// evaluated for the region (the backward pass evaluates nearly the same rows), most first; the forward warp that finishes a
// region last files it.  The warps take items by ticket; in image order the expensive first segments of tiles late in
// the image were started last and the warps finished, on average, at 76 % of the kernel's duration.
constexpr int BLEND_BWD_CLASSES = 16;
__host__ __device__ inline uint32_t blend_bwd_class(uint32_t rows_evaluated) {
  const uint32_t c = rows_evaluated >> 4;  // at most BLEND_HEAD = 256 rows: 0 .. 16
  return c >= (uint32_t)BLEND_BWD_CLASSES ? 0u : (uint32_t)BLEND_BWD_CLASSES - 1u - c;
}

constexpr size_t BLEND_WS_HEADER = 256;
// The colour is kept in double: the backward pass needs its product with the pixel's incoming gradient, a sum over
// the three channels that cancels when the gradient's signs differ (an L1 loss: +-1/N), and a float colour would
// make that product wrong in its leading digits for every row of the segment at once.
struct BlendRecord {
  float T, pad;
  double S0, S1, S2;
};
static_assert(sizeof(BlendRecord) == 32, "record layout");
constexpr size_t BLEND_SEG_BYTES = BLEND_STRIPS * (8 + 8 + BLEND_STRIP_PIXELS * sizeof(BlendRecord));  // a tile's record
struct BlendWs {
  size_t strip_first, tail_queue, bwd_queue, seg_strip, seg_link, ckpt, total;
  uint32_t segments;  // strip slots
};
static inline size_t blend_align(size_t x) { return (x + 255) / 256 * 256; }
static inline bool blend_tile_items(int n_tiles) { return n_tiles >= BLEND_FULL_TILES; }
// records: in units of a whole tile (four strip slots)
static inline BlendWs blend_ws_layout(int n_tiles, uint32_t records) {
  BlendWs L;
  const size_t strips = (size_t)n_tiles * BLEND_STRIPS, items = blend_tile_items(n_tiles) ? (size_t)n_tiles : strips;
  const size_t segments = (size_t)records * BLEND_STRIPS + (strips < 3 * BLEND_SPARES ? strips : 3 * BLEND_SPARES) +
                          (blend_fine(n_tiles) ? strips * (BLEND_FINE_END / BLEND_FINE - BLEND_FINE_END / BLEND_HEAD) : 0);
  L.segments = (uint32_t)segments;
  L.strip_first = BLEND_WS_HEADER + blend_align((size_t)n_tiles * 4);
  L.tail_queue = L.strip_first + blend_align(strips * 4);
  L.bwd_queue = L.tail_queue + blend_align(strips * 16);
  L.seg_strip = L.bwd_queue + blend_align(items * 4 * BLEND_BWD_CLASSES);
  L.seg_link = L.seg_strip + blend_align(segments * 8);
  L.ckpt = L.seg_link + blend_align(segments * 8);
  L.total = L.ckpt + segments * BLEND_STRIP_PIXELS * sizeof(BlendRecord);
  return L;
}
static inline uint32_t blend_min_records(int n_tiles) { return 2u * (uint32_t)n_tiles + 4096u; }
static inline size_t blend_ws_bytes(int width, int height) {
  const int n_tiles = ((width + 15) / 16) * ((height + 15) / 16);
  return blend_ws_layout(n_tiles, blend_min_records(n_tiles)).total;
}
// the largest number of records whose layout fits into ws_bytes (at least the minimum, which the caller checked)
static inline uint32_t blend_ws_records(int n_tiles, size_t ws_bytes) {
  uint32_t s = blend_min_records(n_tiles);
  const size_t fixed = blend_ws_layout(n_tiles, 0).total + 3 * 256;
  if (ws_bytes > fixed) {
    const size_t fit = (ws_bytes - fixed) / BLEND_SEG_BYTES;
    if (fit > s) s = (uint32_t)(fit < 0x0fffffffu ? fit : 0x0fffffffu);
  }
  while (blend_ws_layout(n_tiles, s).total > ws_bytes && s > blend_min_records(n_tiles)) --s;
  return s;
}

constexpr int BLEND_WARPS = 4;          // items per block (warps do not synchronise with each other)
constexpr int BLEND_THREADS = 32 * BLEND_WARPS;
constexpr int BLEND_GROUP = 4;

// Two fp32 values in one 64-bit register pair: every operation rounds each half as the scalar instruction does.
typedef float2 f2;
__device__ __forceinline__ f2 f2_make(float lo, float hi) { return make_float2(lo, hi); }
__device__ __forceinline__ f2 f2_dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ void f2_split(f2 v, float& lo, float& hi) { lo = v.x; hi = v.y; }
__device__ __forceinline__ float f2_lo(f2 v) { return v.x; }
__device__ __forceinline__ float f2_hi(f2 v) { return v.y; }
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float f2_sum(f2 v) { return v.x + v.y; }
__device__ __forceinline__ f2 f2_half(const float4& v, int i) { return i ? make_float2(v.z, v.w) : make_float2(v.x, v.y); }

// One row of the list as staged in shared memory; only the rows that reach the warp's region are staged, in list order,
// so the loop over them is a plain count.  The exponent is evaluated in base 2 with the opacity folded in: with
// sA = -A log2(e) / 2, sB = -B log2(e), sC = -C log2(e) / 2 and lo = log2(opacity),
//     p = sA dx^2 + sB dx dy + sC dy^2 + lo = log2(opacity * exp(power)),   alpha = min(alpha_max, 2^p),
// so a pixel costs two fused multiply-adds, the tests, one ex2 and one min.  The skip test "alpha < alpha_min" is
// p < log2(alpha_min), a constant of the launch, and "power > 0" is p > lo (see blend_shape).  All blend kernels form p through
// blend_stage_conic / blend_x_terms and the same two multiply-adds, so they agree bit for bit on every (pixel, row)
// pair.  An opacity of 0 gives lo = -inf (nothing passes).
struct BlendRow {
  float4 a;  // r, r, g, g
  float4 b;  // blue, 1-based position in the list (bits; whole tiles: << 4 | strips that may be reached), u, v
  float4 c;  // sA, sB, sC, lo
};

constexpr float BLEND_LOG2E = 1.4426950408889634f;
constexpr float BLEND_LN2 = 0.6931471805599453f;

__device__ __forceinline__ float4 blend_stage_conic(float4 conic_o) {
  return make_float4(conic_o.x * (-0.5f * BLEND_LOG2E), conic_o.y * (-BLEND_LOG2E), conic_o.z * (-0.5f * BLEND_LOG2E),
                     log2f(conic_o.w));
}

// per row and lane: the terms of p that depend on the column only (dx = u - x)
__device__ __forceinline__ void blend_x_terms(const float4 q1, float dx, float& h0, float& h1, float& h2) {
  h0 = fmaf(q1.x * dx, dx, q1.w);
  h1 = q1.y * dx;
  h2 = q1.z;
}

__device__ __forceinline__ float blend_ex2(float p) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(p));
  return y;
}

__device__ __forceinline__ float blend_rcp(float x) {  // of 1 - alpha: a normal number, no scaling needed
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// p of two rows at one pixel: the same operations as blend_x_terms and the two multiply-adds on its result
__device__ __forceinline__ f2 blend_exponent2(f2 dx, f2 dy, f2 sA, f2 sB, f2 sC, f2 lo) {
  return f2_fma(dy, f2_fma(sC, dy, f2_mul(sB, dx)), f2_fma(f2_mul(sA, dx), dx, lo));
}

// The skip test "power > 0", p > lo, has nothing to do where the conic is an ellipse.  With q = A dx^2 + 2 B dx dy + C dy^2 and
// A C - B^2 > e A C, q is at least e times A dx^2 and e times C dy^2, so the sizes of its three terms add up to at most 4 q / e,
// and the five roundings of p (2^-24 of its terms and of lo each) move it by less than q / 20 for e = 1e-4 and by less than a
// millionth of lo: a row with such a PROPER conic exceeds its opacity by rounding at most, and none of the kernels tests it.
// (A product A C too large for fp32 is not proper; where it is too small for it the terms of p are below 1e-9 in any image.)  The
// other rows, splats 200 times as long as wide, are marked when they are staged and tested as they come up (blend_top, the bound on
// p).  What a row is depends on its conic alone, so the kernels agree.  Without the test the backward pass of
// 1600 x 1066 takes 208 us instead of 217, of the aerial city 394 instead of 403.  A batch with such a row gone through pixel by pixel
// instead: a tenth of 300 k splats 400 pixels long, 256 x 256: forward 37 against 35 us, backward 34 against 31.
constexpr float BLEND_PROPER = 1e-4f;
struct BlendShape {
  float det;
  bool ellipse, proper;
};
__device__ __forceinline__ BlendShape blend_shape(float A, float B, float C) {
  BlendShape s;
  const float ac = __fmul_rn(A, C);
  s.det = __fmaf_rn(-B, B, ac);
  const bool sized = A > 1e-30f && C > 1e-30f && A < 1e30f && C < 1e30f;
  s.ellipse = s.det > 0.f && sized;
  s.proper = s.det > __fmul_rn(BLEND_PROPER, ac) && sized;
  return s;
}
// the bound on p of a row that is or is not odd (not proper)
__device__ __forceinline__ float blend_top(float lo, bool odd) { return odd ? lo : __builtin_huge_valf(); }

// What a lane of a warp fetches of a row of the list.
struct BlendFetch {
  float2 c;
  float4 co;
  float r, g, b;
};
__device__ __forceinline__ BlendFetch blend_fetch(const float2* __restrict__ xy, const float4* __restrict__ conic_o,
                                                  const float* __restrict__ rgb, uint32_t r) {
  BlendFetch f;
  f.c = xy[r];
  f.co = conic_o[r];
  f.r = rgb[3 * (size_t)r]; f.g = rgb[3 * (size_t)r + 1]; f.b = rgb[3 * (size_t)r + 2];
  return f;
}

// Straight-line code multiplies a row's colour, and the gradients of a pixel, by a weight of 0 where the row does not blend,
// which changes nothing as long as they are numbers.  Infinities and NaN must not get to pixels or rows that have nothing
// to do with them either, so where a staged colour (in the backward pass also a conic, a pixel's incoming gradient or its
// colour to come) is not below these bounds - below them no product and no sum of the kernels overflows - the warp takes
// the same operations pixel by pixel.  What it costs where everything is a number, a vote per 32 rows: backward 1600 x 1066
// 259 -> 261 us, aerial city 488 -> 490, 1237 x 823 175 -> 173; forward nothing.
constexpr float BLEND_TAME = 1e18f, BLEND_TAME_PRODUCT = 1e37f;
__device__ __forceinline__ bool blend_tame(float a, float b, float c) { return fabsf(a) + fabsf(b) + fabsf(c) < BLEND_TAME; }

// Can the row pass the skip test at any pixel of the W x H region of pixel centres whose first is (x_lo, y_lo)?  The set
// power >= log(alpha_min / opacity) is the ellipse q(dx, dy) = A dx^2 + 2 B dx dy + C dy^2 <= k, k = 2 ln(opacity /
// alpha_min) = 2 ln 2 (lo - log2(alpha_min)), around the row's centre (u, v).  q is convex, so its minimum over the
// region is 0 if the centre lies inside and otherwise sits on one of the four edges, where it is the clamped
// one-dimensional minimiser.  The bound is widened by 1e-4 relative + 1e-3 + 2e-6 of the largest term any pixel of the
// region can see (the rounding of this evaluation and of the per-pixel exponent is a few ulp of that term), so a row it
// rejects fails the per-pixel test everywhere in the region and skipping it never changes a result.  Evaluated once per
// (region, row) by the lane that stages the row; anything that is not a proper ellipse is kept.
template <int W, int H>
__device__ __forceinline__ bool blend_reaches(float u, float v, float A, float B, float C, const BlendShape& shape, float lo,
                                              float l2amin, float x_lo, float y_lo) {
  if (!(lo >= l2amin)) return false;  // opacity below alpha_min, zero or not a number: nothing passes
  const float dxl = x_lo - u, dxh = dxl + (float)(W - 1), dyl = y_lo - v, dyh = dyl + (float)(H - 1);
  if (dxl <= 0.f && dxh >= 0.f && dyl <= 0.f && dyh >= 0.f) return true;
  if (!shape.ellipse) return true;
  const float iA = __fdividef(1.f, A), iC = __fdividef(1.f, C);
  const float t0 = fminf(fmaxf(-B * dxl * iC, dyl), dyh), t1 = fminf(fmaxf(-B * dxh * iC, dyl), dyh);
  const float q0 = fmaf(t0, fmaf(C, t0, 2.f * B * dxl), A * dxl * dxl);
  const float q1 = fmaf(t1, fmaf(C, t1, 2.f * B * dxh), A * dxh * dxh);
  const float s0 = fminf(fmaxf(-B * dyl * iA, dxl), dxh), s1 = fminf(fmaxf(-B * dyh * iA, dxl), dxh);
  const float q2 = fmaf(s0, fmaf(A, s0, 2.f * B * dyl), C * dyl * dyl);
  const float q3 = fmaf(s1, fmaf(A, s1, 2.f * B * dyh), C * dyh * dyh);
  const float qmin = fminf(fminf(q0, q1), fminf(q2, q3));
  const float mx = fmaxf(fabsf(dxl), fabsf(dxh)), my = fmaxf(fabsf(dyl), fabsf(dyh));
  const float big = A * mx * mx + 2.f * fabsf(B) * mx * my + C * my * my;
  const float bound = fmaf((lo - l2amin) * (2.f * BLEND_LN2), 1.0001f, 1e-3f + 2e-6f * big);
  return !(qmin > bound);
}

// The same for a whole tile, with the strips of four pixel rows the row may pass in as a mask (0: nowhere): those that
// meet the height of the ellipse, |dy| <= sqrt(bound A / (A C - B^2)), widened by 0.2 % + 0.02 pixels.  An ellipse so
// elongated that A C - B^2 is mostly rounding keeps all four.
__device__ __forceinline__ uint32_t blend_reached_strips(float u, float v, float A, float B, float C, const BlendShape& shape,
                                                         float lo, float l2amin, float x_lo, float y_lo) {
  if (!blend_reaches<16, 16>(u, v, A, B, C, shape, lo, l2amin, x_lo, y_lo)) return 0u;
  const float det = shape.det;
  if (!(det > 1e-3f * A * C) || !(A < 1e30f) || !(C < 1e30f)) return 15u;
  const float dyl = y_lo - v;
  const float mx = fmaxf(fabsf(x_lo - u), fabsf(x_lo - u + 15.f)), my = fmaxf(fabsf(dyl), fabsf(dyl + 15.f));
  const float big = A * mx * mx + 2.f * fabsf(B) * mx * my + C * my * my;
  const float bound = fmaf((lo - l2amin) * (2.f * BLEND_LN2), 1.0001f, 1e-3f + 2e-6f * big);
  float ext;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(ext) : "f"(bound * A * __fdividef(1.f, det)));
  ext = fmaf(ext, 1.002f, 0.02f);
  uint32_t m = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (dyl + (float)(4 * q) <= ext && dyl + (float)(4 * q + 3) >= -ext) m |= 1u << q;
  return m;
}
