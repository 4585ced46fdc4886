// Rendering phase: front-to-back alpha compositing.  Images of enough tiles: the first BLEND_HEAD entries of a tile's list
// by two warps of 16 x 8 pixels, four pixels per lane (head kernel), what is still live behind them by cells, one warp per 8 x 4
// pixels (tail kernel), and behind FWD_DEEP entries by strips, a block each (strip kernel).  Smaller images by strips from the
// start.  Rows are tested against the warp's region when they are staged through shared memory; warp-ballot early exit once
// every pixel of the region has terminated.  Also the L1 image loss.
#include <type_traits>

#include "blend.cuh"

namespace {

struct FwdArgs {
  const float2* xy;
  const float4* conic_o;
  const float* rgb;
  const uint32_t* vals;
  const uint2* ranges;
  int W, H, TX, n_tiles;
  float bg0, bg1, bg2, alpha_min, alpha_max, t_min;
  float* out;
  float* final_T;
  uint32_t* n_contrib;
  uint32_t* strip_first;
  uint32_t* header;
  uint32_t* tail_queue;
  uint32_t* bwd_queue;
  uint32_t* tile_work;
  uint2* seg_strip;
  uint2* seg_link;
  BlendRecord* ckpt;
  uint32_t seg_cap;
  int* status;
  uint32_t row_cap;
};

constexpr float FWD_DEAD = __builtin_huge_valf();  // cut of a pixel that accumulates no more: no exponent reaches it
constexpr int FWD_HEAD_BLOCKS = 7, FWD_TAIL_BLOCKS = 5;  // resident blocks per SM

// A slot of the segment records, for lane 0 (without a branch: the warp stays together).
__device__ __forceinline__ uint32_t fwd_take(uint32_t* counter, uint32_t old, unsigned lane) {
  asm volatile("{\n .reg .pred p;\n setp.eq.u32 p, %1, 0;\n @p atom.global.add.u32 %0, [%2], 1;\n}"
               : "+r"(old) : "r"(lane), "l"(counter) : "memory");
  return old;
}

// Head kernel: the first BLEND_HEAD entries of a tile's list for half a tile (16 x 8 pixels) per warp.  Lane l handles
// column l % 16; its slot s = 0 .. 3 is pixel row 2 s + l / 16, and the two slots of a strip are the two halves of packed
// registers.  Four pixels per lane: the loads and the terms of a row that do not depend on the pixel row are shared.  Two rows at
// a time: only their transmittances depend on one another, so four exponent chains cover each other's latency at 28 warps per
// SM, and one vote tells whether a pixel stops.  What bounds it: the issue of instructions.  One row / two rows at a time, us:
// 1600 x 1066 142 / 137, 1920 x 1080 with large splats 162 / 154, aerial city 160 / 150, 1237 x 823 93 / 88; three rows 148, 161,
// 161, 92; two rows with six or eight blocks per SM 142 and 140 in the first.
__global__ void __launch_bounds__(BLEND_THREADS, FWD_HEAD_BLOCKS)
render_fwd_head_kernel(FwdArgs A) {
  odin_after_predecessor();
  constexpr int Q = 2;  // strips per warp
  constexpr int G = 2;  // rows at a time
  __shared__ BlendRow s_rows[BLEND_WARPS][32 + G - 1];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  BlendRow* s_row = s_rows[warp];
  const float l2amin = log2f(A.alpha_min);
  const uint32_t n_items = (uint32_t)A.n_tiles * (BLEND_STRIPS / Q), n_strips = (uint32_t)A.n_tiles * BLEND_STRIPS;
  const size_t plane = (size_t)A.W * A.H;
  const f2 minus1 = f2_dup(-1.f);
  // Warps never synchronise with each other.  Each one keeps taking items from a ticket counter until none is left:
  // lists differ in length by orders of magnitude between tiles, and a fixed tile-to-warp map would leave most of the
  // GPU idle while the longest ones finish.
  while (true) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(A.header, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_items) return;
    const int tile = (int)(item / (BLEND_STRIPS / Q));
    const uint32_t strip0 = item * Q;
    const int px = (tile % A.TX) * 16 + (int)(lane & 15), y0 = (tile / A.TX) * 16 + 4 * (int)(strip0 % BLEND_STRIPS);
    const int py0 = y0 + (int)(lane >> 4);
    const float fx = (float)px + 0.5f;
    const float x_lo = (float)((tile % A.TX) * 16) + 0.5f, y_lo = (float)y0 + 0.5f;
    const uint2 rg = A.ranges[tile];
    const uint32_t start = rg.x, len = min(rg.y - rg.x, BLEND_HEAD);

    f2 T[Q], C0[Q], C1[Q], C2[Q], nfy[Q];
    float cut[2 * Q];  // log2(alpha_min), FWD_DEAD once the pixel has stopped
    uint32_t last[2 * Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      T[q] = f2_dup(1.f); C0[q] = C1[q] = C2[q] = f2_dup(0.f);
      const float y = (float)(py0 + 4 * q) + 0.5f;
      nfy[q] = f2_make(-y, -(y + 2.f));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        last[2 * q + h] = 0;
        cut[2 * q + h] = (px < A.W && py0 + 4 * q + 2 * h < A.H) ? l2amin : FWD_DEAD;
      }
    }
    uint32_t n_eval = 0;  // rows evaluated
    uint32_t r = lane < len ? min(A.vals[start + lane], A.row_cap - 1) : 0u;  // in range whatever the list holds
    for (uint32_t off = 0; off < len; off += 32) {
      if (!__any_sync(0xffffffffu, fminf(fminf(cut[0], cut[1]), fminf(cut[2], cut[3])) < FWD_DEAD)) break;
      BlendFetch f = {};
      if (off + lane < len) f = blend_fetch(A.xy, A.conic_o, A.rgb, r);
      const float4 q4 = blend_stage_conic(f.co);
      const BlendShape shape = blend_shape(f.co.x, f.co.y, f.co.z);
      const bool reach = off + lane < len && blend_reaches<16, 8>(f.c.x, f.c.y, f.co.x, f.co.y, f.co.z, shape, q4.w, l2amin, x_lo, y_lo);
      const uint32_t m = __ballot_sync(0xffffffffu, reach);
      const int cnt = __popc(m);
      const bool some_odd = __any_sync(0xffffffffu, reach && !(blend_tame(f.r, f.g, f.b) && shape.proper));
      float low = 1.f;
      uint32_t odd = 0;  // staged rows whose conic is not proper: the only ones whose exponent is tested against their opacity
      n_eval += (uint32_t)cnt;
      __syncwarp();  // the previous batch has been read
      if (reach) {
        BlendRow* d = s_row + __popc(m & ((1u << lane) - 1u));
        d->a = make_float4(f.r, f.r, f.g, f.g);
        d->b = make_float4(f.b, __uint_as_float(off + lane + 1), f.c.x, f.c.y);
        d->c = q4;
      }
      __syncwarp();
      if (some_odd) {
        // (colours that are not tame: every row of the batch pixel by pixel, as where a pixel stops)
        if (__any_sync(0xffffffffu, reach && !blend_tame(f.r, f.g, f.b))) low = -1.f;
        odd = __reduce_or_sync(0xffffffffu, reach && !shape.proper ? 1u << __popc(m & ((1u << lane) - 1u)) : 0u);
      }
      r = off + 32 + lane < len ? min(A.vals[start + off + 32 + lane], A.row_cap - 1) : 0u;  // on its way meanwhile
      if (cnt % G) {  // whole groups: the last row passes nowhere
        if (lane == 0) {
          s_row[cnt].a = s_row[cnt].b = make_float4(0.f, 0.f, 0.f, 0.f);
          s_row[cnt].c = make_float4(0.f, 0.f, 0.f, -__builtin_huge_valf());
        }
        __syncwarp();
      }
      for (int j = 0; j < cnt; j += G) {
        f2 w[G][Q], Tn[Q];
        bool k[G][2 * Q];
        auto weights = [&](auto test) {
          float p[G][2 * Q];
#pragma unroll
          for (int u = 0; u < G; ++u) {
            const float4 rc = s_row[j + u].c;
            const float2 uv = *reinterpret_cast<const float2*>(&s_row[j + u].b.z);
            float h0, h1, h2;
            blend_x_terms(rc, uv.x - fx, h0, h1, h2);
            const f2 H0 = f2_dup(h0), H1 = f2_dup(h1), H2 = f2_dup(h2), V = f2_dup(uv.y);
            const float top = blend_top(rc.w, odd >> (j + u) & 1u);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
              const f2 dy = f2_add(V, nfy[q]);
              f2_split(f2_fma(dy, f2_fma(H2, dy, H1), H0), p[u][2 * q], p[u][2 * q + 1]);
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                k[u][2 * q + h] = p[u][2 * q + h] >= cut[2 * q + h];
                if (decltype(test)::value) k[u][2 * q + h] = k[u][2 * q + h] && p[u][2 * q + h] <= top;
              }
              const float a0 = fminf(A.alpha_max, blend_ex2(p[u][2 * q])), a1 = fminf(A.alpha_max, blend_ex2(p[u][2 * q + 1]));
              w[u][q] = f2_make(k[u][2 * q] ? a0 : 0.f, k[u][2 * q + 1] ? a1 : 0.f);  // alpha = 0 where a skip test fails
            }
          }
        };
        if (odd == 0) weights(std::false_type{});
        else weights(std::true_type{});
        float lowest = low;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          Tn[q] = T[q];
#pragma unroll
          for (int u = 0; u < G; ++u) {
            w[u][q] = f2_mul(w[u][q], Tn[q]);
            Tn[q] = f2_fma(w[u][q], minus1, Tn[q]);
          }
          lowest = fminf(lowest, fminf(f2_lo(Tn[q]), f2_hi(Tn[q])));
        }
        // the transmittance only falls: one test for both rows
        if (__any_sync(0xffffffffu, lowest < A.t_min)) {
          // some pixel stops in front of one of these rows (once per pixel): pixel by pixel, with the same operations
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            float t[2], x[2], y[2], z[2];
            f2_split(T[q], t[0], t[1]); f2_split(C0[q], x[0], x[1]); f2_split(C1[q], y[0], y[1]); f2_split(C2[q], z[0], z[1]);
#pragma unroll
            for (int u = 0; u < G; ++u) {
              const float4 ra = s_row[j + u].a, rb = s_row[j + u].b;
              float ww[2];
              f2_split(w[u][q], ww[0], ww[1]);  // (up to the stop the weights are right)
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const float tn = fmaf(ww[h], -1.f, t[h]);
                if (!k[u][2 * q + h] || cut[2 * q + h] == FWD_DEAD) continue;
                if (tn < A.t_min) {
                  cut[2 * q + h] = FWD_DEAD;
                } else {
                  x[h] = fmaf(ra.x, ww[h], x[h]); y[h] = fmaf(ra.z, ww[h], y[h]); z[h] = fmaf(rb.x, ww[h], z[h]);
                  t[h] = tn;
                  last[2 * q + h] = __float_as_uint(rb.y);
                }
              }
            }
            T[q] = f2_make(t[0], t[1]); C0[q] = f2_make(x[0], x[1]); C1[q] = f2_make(y[0], y[1]); C2[q] = f2_make(z[0], z[1]);
          }
        } else {
#pragma unroll
          for (int u = 0; u < G; ++u) {
            const float4 ra = s_row[j + u].a, rb = s_row[j + u].b;
            const f2 red = f2_make(ra.x, ra.y), green = f2_make(ra.z, ra.w), blue = f2_dup(rb.x);
            const uint32_t ord = __float_as_uint(rb.y);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
              C0[q] = f2_fma(red, w[u][q], C0[q]); C1[q] = f2_fma(green, w[u][q], C1[q]); C2[q] = f2_fma(blue, w[u][q], C2[q]);
              if (k[u][2 * q]) last[2 * q] = ord;
              if (k[u][2 * q + 1]) last[2 * q + 1] = ord;
            }
          }
#pragma unroll
          for (int q = 0; q < Q; ++q) T[q] = Tn[q];
        }
      }
    }
    // strips in which some pixel is still live go on in the tail kernel when entries remain
    uint32_t more = 0;
#pragma unroll
    for (int q = 0; q < Q; ++q)
      if (rg.y - rg.x > len && __any_sync(0xffffffffu, fminf(cut[2 * q], cut[2 * q + 1]) < FWD_DEAD)) more |= 1u << q;
    if (lane < Q) {
      A.strip_first[strip0 + lane] = 0u;
      if (more >> lane & 1u) {  // queue of the tail kernel, longest lists first (four classes)
        const uint32_t all = rg.y - rg.x;
        const uint32_t cls = all > 8 * BLEND_HEAD ? 0u : (all > 4 * BLEND_HEAD ? 1u : (all > 2 * BLEND_HEAD ? 2u : 3u));
        A.tail_queue[cls * n_strips + atomicAdd(A.header + 4 + cls, 1u)] = strip0 + lane;
      }
    }
    if (lane == 0) {
      // The warp that finishes last of its tile files the tile for the backward pass: the rows that the two evaluated, on
      // average, say what its first segment costs.  (tile_work: rows in the upper bits, warps done in the lowest two.)
      const uint32_t add = (n_eval << 2) + 1u, done = atomicAdd(A.tile_work + tile, add) + add;
      if ((done & 3u) == (uint32_t)(BLEND_STRIPS / Q)) {
        const uint32_t bc = blend_bwd_class((done >> 2) / (BLEND_STRIPS / Q));
        A.bwd_queue[bc * (uint32_t)A.n_tiles + atomicAdd(A.header + 8 + bc, 1u)] = (uint32_t)tile;
      }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      float t[2], c0[2], c1[2], c2[2];
      f2_split(T[q], t[0], t[1]); f2_split(C0[q], c0[0], c0[1]); f2_split(C1[q], c1[0], c1[1]); f2_split(C2[q], c2[0], c2[1]);
      const bool go_on = more >> q & 1u;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int py = py0 + 4 * q + 2 * h;
        if (px < A.W && py < A.H) {
          const size_t pix = (size_t)py * A.W + px;
          const float tb = go_on ? 0.f : t[h];  // the background is added by whoever finishes the pixel
          A.out[pix] = c0[h] + tb * A.bg0;
          A.out[plane + pix] = c1[h] + tb * A.bg1;
          A.out[2 * plane + pix] = c2[h] + tb * A.bg2;
          A.final_T[pix] = t[h];
          A.n_contrib[pix] = last[2 * q + h] | ((go_on && cut[2 * q + h] == FWD_DEAD) ? BLEND_DONE_BIT : 0u);
        }
      }
    }
    __syncwarp();  // the staging array is reused by the next item
  }
}

constexpr int FWD_GROUP = 4;  // rows per group
constexpr int FWD_BATCH = 2;  // list entries per lane and batch
constexpr int FWD_ROWS = 32 * FWD_BATCH + FWD_GROUP;
static_assert(BLEND_HEAD % (32 * FWD_BATCH) == 0, "segments are whole batches");

// The staged rows of a warp, one array per quantity so that a group's values are wide loads.
struct __align__(16) FwdCellRows {
  float u[FWD_ROWS], v[FWD_ROWS], sA[FWD_ROWS], sB[FWD_ROWS], sC[FWD_ROWS], lo[FWD_ROWS];
  float r[FWD_ROWS], g[FWD_ROWS], b[FWD_ROWS];
  uint32_t ord[FWD_ROWS];  // 1-based position in the list; FWD_ODD: the conic is not proper
};
static_assert(sizeof(FwdCellRows) % 16 == 0 && FWD_ROWS % 4 == 0, "wide loads of every warp's arrays");
constexpr uint32_t FWD_ODD = 1u << 31;  // (lists are shorter than 2^30)

// The rows of a batch of 32 FWD_BATCH list entries, the first of them at position `off` of the list of `len` entries.  r: the
// lane's row ids, entry off + 32 u + lane.
__device__ __forceinline__ void fwd_fetch(const FwdArgs& A, const uint32_t (&r)[FWD_BATCH], uint32_t off, uint32_t len,
                                          unsigned lane, BlendFetch (&f)[FWD_BATCH]) {
#pragma unroll
  for (int u = 0; u < FWD_BATCH; ++u) {
    f[u] = BlendFetch{};
    if (off + 32 * u + lane < len) f[u] = blend_fetch(A.xy, A.conic_o, A.rgb, r[u]);
  }
}

// The fetched batch -> shared memory: only the rows that reach the cell, in list order.  Returns their number; behind the
// last one stand FWD_GROUP - 1 rows that pass nowhere.  tame: all of them are, and proper.
__device__ __forceinline__ int fwd_stage(const BlendFetch (&f)[FWD_BATCH], uint32_t off, uint32_t len, float l2amin, float x_lo,
                                         float y_lo, FwdCellRows& s, unsigned lane, bool& tame) {
  __syncwarp();  // the previous batch has been read
  int cnt = 0;
  bool wild = false;
#pragma unroll
  for (int u = 0; u < FWD_BATCH; ++u) {
    const float4 q = blend_stage_conic(f[u].co);
    const uint32_t ord = off + 32 * u + lane + 1;
    const BlendShape shape = blend_shape(f[u].co.x, f[u].co.y, f[u].co.z);
    const bool reach = ord <= len && blend_reaches<8, 4>(f[u].c.x, f[u].c.y, f[u].co.x, f[u].co.y, f[u].co.z, shape, q.w, l2amin, x_lo, y_lo);
    const uint32_t m = __ballot_sync(0xffffffffu, reach);
    wild = wild || (reach && !(blend_tame(f[u].r, f[u].g, f[u].b) && shape.proper));
    if (reach) {
      const int d = cnt + __popc(m & ((1u << lane) - 1u));
      s.u[d] = f[u].c.x; s.v[d] = f[u].c.y; s.sA[d] = q.x; s.sB[d] = q.y; s.sC[d] = q.z; s.lo[d] = q.w;
      s.r[d] = f[u].r; s.g[d] = f[u].g; s.b[d] = f[u].b;
      s.ord[d] = shape.proper ? ord : ord | FWD_ODD;
    }
    cnt += __popc(m);
  }
  if (lane < FWD_GROUP - 1) {
    const int d = cnt + lane;
    s.u[d] = s.v[d] = s.sA[d] = s.sB[d] = s.sC[d] = s.r[d] = s.g[d] = s.b[d] = 0.f;
    s.lo[d] = -__builtin_huge_valf();
  }
  tame = !__any_sync(0xffffffffu, wild);
  __syncwarp();
  return cnt;
}

// row ids of a batch (0 behind the end of the list)
__device__ __forceinline__ void fwd_ids(const FwdArgs& A, uint32_t start, uint32_t off, uint32_t len, unsigned lane,
                                        uint32_t (&r)[FWD_BATCH]) {
#pragma unroll
  for (int u = 0; u < FWD_BATCH; ++u) {
    const uint32_t i = off + 32 * u + lane;
    r[u] = i < len ? min(A.vals[start + i], A.row_cap - 1) : 0u;  // in range whatever the list holds
  }
}

struct FwdCellPixel {
  float T, C0, C1, C2;
  float cut;  // log2(alpha_min), FWD_DEAD once the pixel has stopped
  uint32_t last;
  double D[3];  // colour the segment has added
};

// The staged rows, a group at a time: exponents and skip tests of the group first (independent work, two rows per packed
// instruction), then its transmittances.  The transmittance only falls, so one test behind the group tells whether some
// pixel stops inside it (once per pixel); only then the group's weights are gone through again one by one.  The
// colour the rows add is also summed in double, for the segment records.  WILD: some colour is not tame or some conic not proper; the same operations, but
// the colour only where the row blends (see blend_tame), and the exponent tested where blend_top says so.
template <bool WILD>
__device__ __forceinline__ void fwd_rows(const FwdCellRows& s, const double (*s_cd)[FWD_ROWS], int cnt, f2 nfx, f2 nfy, float alpha_max,
                                         float t_min, FwdCellPixel& P) {
  for (int j = 0; j < cnt; j += FWD_GROUP) {
    float w[FWD_GROUP];
    bool k[FWD_GROUP];
#pragma unroll
    for (int h = 0; h < FWD_GROUP; h += 4) {
      const float4 u4 = *reinterpret_cast<const float4*>(s.u + j + h), v4 = *reinterpret_cast<const float4*>(s.v + j + h);
      const float4 a4 = *reinterpret_cast<const float4*>(s.sA + j + h), b4 = *reinterpret_cast<const float4*>(s.sB + j + h);
      const float4 c4 = *reinterpret_cast<const float4*>(s.sC + j + h), l4 = *reinterpret_cast<const float4*>(s.lo + j + h);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const f2 lo = f2_half(l4, i);
        const f2 p = blend_exponent2(f2_add(f2_half(u4, i), nfx), f2_add(f2_half(v4, i), nfy), f2_half(a4, i), f2_half(b4, i),
                                     f2_half(c4, i), lo);
        float p0, p1;
        f2_split(p, p0, p1);
        k[h + 2 * i] = p0 >= P.cut;
        k[h + 2 * i + 1] = p1 >= P.cut;
        if (WILD) {
          k[h + 2 * i] = k[h + 2 * i] && p0 <= blend_top(lo.x, s.ord[j + h + 2 * i] & FWD_ODD);
          k[h + 2 * i + 1] = k[h + 2 * i + 1] && p1 <= blend_top(lo.y, s.ord[j + h + 2 * i + 1] & FWD_ODD);
        }
        const float e0 = fminf(alpha_max, blend_ex2(p0)), e1 = fminf(alpha_max, blend_ex2(p1));
        w[h + 2 * i] = k[h + 2 * i] ? e0 : 0.f;  // alpha, 0 where a skip test fails
        w[h + 2 * i + 1] = k[h + 2 * i + 1] ? e1 : 0.f;
      }
    }
    float Tn = P.T;
#pragma unroll
    for (int u = 0; u < FWD_GROUP; ++u) {
      w[u] *= Tn;
      Tn -= w[u];
    }
    if (__any_sync(0xffffffffu, Tn < t_min)) {
      Tn = P.T;
#pragma unroll
      for (int u = 0; u < FWD_GROUP; ++u) {
        // (up to the stop the weights are right; w = 0 where the row does not blend)
        const float tn = Tn - w[u];
        if (tn < t_min) P.cut = FWD_DEAD;  // the pixel stops in front of this row
        if (P.cut == FWD_DEAD) { w[u] = 0.f; k[u] = false; }
        else Tn = tn;
      }
    }
    P.T = Tn;
    if (WILD) {
#pragma unroll
      for (int u = 0; u < FWD_GROUP; ++u) {
        if (!k[u]) continue;
        P.C0 = fmaf(s.r[j + u], w[u], P.C0); P.C1 = fmaf(s.g[j + u], w[u], P.C1); P.C2 = fmaf(s.b[j + u], w[u], P.C2);
        P.last = s.ord[j + u] & ~FWD_ODD;
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) P.D[ch] = fma(s_cd[ch][j + u], (double)w[u], P.D[ch]);
      }
      continue;
    }
#pragma unroll
    for (int h = 0; h < FWD_GROUP; h += 4) {
      const float4 r4 = *reinterpret_cast<const float4*>(s.r + j + h), g4 = *reinterpret_cast<const float4*>(s.g + j + h);
      const float4 b4 = *reinterpret_cast<const float4*>(s.b + j + h);
      const uint4 o4 = *reinterpret_cast<const uint4*>(s.ord + j + h);
      P.C0 = fmaf(r4.x, w[h], P.C0); P.C1 = fmaf(g4.x, w[h], P.C1); P.C2 = fmaf(b4.x, w[h], P.C2);
      P.C0 = fmaf(r4.y, w[h + 1], P.C0); P.C1 = fmaf(g4.y, w[h + 1], P.C1); P.C2 = fmaf(b4.y, w[h + 1], P.C2);
      P.C0 = fmaf(r4.z, w[h + 2], P.C0); P.C1 = fmaf(g4.z, w[h + 2], P.C1); P.C2 = fmaf(b4.z, w[h + 2], P.C2);
      P.C0 = fmaf(r4.w, w[h + 3], P.C0); P.C1 = fmaf(g4.w, w[h + 3], P.C1); P.C2 = fmaf(b4.w, w[h + 3], P.C2);
      if (k[h]) P.last = o4.x;
      if (k[h + 1]) P.last = o4.y;
      if (k[h + 2]) P.last = o4.z;
      if (k[h + 3]) P.last = o4.w;
    }
    {
      double wd[FWD_GROUP];
#pragma unroll
      for (int u = 0; u < FWD_GROUP; ++u) wd[u] = (double)w[u];
#pragma unroll
      for (int ch = 0; ch < 3; ++ch)
#pragma unroll
        for (int u = 0; u < FWD_GROUP; u += 2) {
          const double2 c = *reinterpret_cast<const double2*>(s_cd[ch] + j + u);
          P.D[ch] = fma(c.x, wd[u], P.D[ch]);
          P.D[ch] = fma(c.y, wd[u + 1], P.D[ch]);
        }
    }
  }
}

// What the head kernel left, up to entry FWD_DEEP of the list: one warp per cell, two per strip.  The warps of a pair walk
// their own rows of the list and meet every BLEND_HEAD entries, where a segment record of the strip is opened as long as one of
// them has a live pixel (see blend.cuh).  These strips are many and most of them end soon, however long the list: ten of them
// in flight per SM count for more than how fast each one is.  What is live even behind FWD_DEEP goes on in the strip kernel.
constexpr uint32_t FWD_DEEP = 4 * BLEND_HEAD;  // (the queue's first two classes have longer lists)
__global__ void __launch_bounds__(BLEND_THREADS, FWD_TAIL_BLOCKS)
render_fwd_tail_kernel(FwdArgs A) {
  odin_after_predecessor();
  __shared__ __align__(16) FwdCellRows s_rows[BLEND_WARPS];
  // the row's colour in double, converted once when the row is staged
  __shared__ __align__(16) double s_cds[BLEND_WARPS][3][FWD_ROWS];
  __shared__ uint32_t s_item[BLEND_WARPS / 2], s_slot[BLEND_WARPS / 2], s_live[BLEND_WARPS], s_slots[BLEND_WARPS / 2][4];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, pair = warp >> 1, half = warp & 1;
  auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + pair) : "memory"); };
  FwdCellRows& s = s_rows[warp];
  double(*s_cd)[FWD_ROWS] = s_cds[warp];
  const float l2amin = log2f(A.alpha_min);
  const uint32_t n_strips = (uint32_t)A.n_tiles * BLEND_STRIPS;
  const size_t plane = (size_t)A.W * A.H;
  uint32_t c[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) c[k] = A.header[4 + k];
  uint32_t spare = 0xffffffffu;  // (first warp of the pair, lane 0) a slot taken in advance, see the strip kernel
  bool have_spare = false;
  auto take_spare = [&]() {
    if (half == 0 && !have_spare) {
      spare = fwd_take(A.header + 2, spare, lane);
      have_spare = true;
    }
  };
  while (true) {
    if (half == 0 && lane == 0) s_item[pair] = atomicAdd(A.header + 3, 1u);
    pair_sync();
    uint32_t item = s_item[pair];
    if (item >= c[0] + c[1] + c[2] + c[3]) break;  // (both warps of the pair)
    // The duration of this kernel is that of its longest lists, so their class comes first.
    uint32_t cls = 0;
    while (cls < 3 && item >= c[cls]) { item -= c[cls]; ++cls; }
    const uint32_t strip = min(A.tail_queue[cls * n_strips + min(item, n_strips - 1)], n_strips - 1);
    const int tile = (int)(strip / BLEND_STRIPS);
    const int x0 = (tile % A.TX) * 16 + 8 * (int)half, y0 = (tile / A.TX) * 16 + 4 * (int)(strip % BLEND_STRIPS);
    const int px = x0 + (int)(lane & 7), py = y0 + (int)(lane >> 3);
    const bool inside = px < A.W && py < A.H;
    const size_t pix = (size_t)py * A.W + px;
    const f2 nfx = f2_dup(-((float)px + 0.5f)), nfy = f2_dup(-((float)py + 0.5f));
    const float x_lo = (float)x0 + 0.5f, y_lo = (float)y0 + 0.5f;
    const uint2 rg = A.ranges[tile];
    const uint32_t start = rg.x, all = rg.y - rg.x, len = min(all, FWD_DEEP);
    FwdCellPixel P;
    P.T = 1.f; P.C0 = P.C1 = P.C2 = 0.f; P.last = 0u;
    P.cut = inside ? l2amin : FWD_DEAD;
    P.D[0] = P.D[1] = P.D[2] = 0.0;
    if (inside) {
      P.T = A.final_T[pix];
      P.C0 = A.out[pix]; P.C1 = A.out[plane + pix]; P.C2 = A.out[2 * plane + pix];
      const uint32_t nc = A.n_contrib[pix];
      P.last = nc & ~BLEND_DONE_BIT;
      if (nc & BLEND_DONE_BIT) P.cut = FWD_DEAD;
    }
    uint32_t first_slot = 0, cur_slot = 0;  // 1 + slot; 0 = none
    int records = 0;
    uint32_t off = BLEND_HEAD;
    if (off < all) take_spare();
    uint32_t r[FWD_BATCH];
    BlendFetch f[FWD_BATCH];
    fwd_ids(A, start, off, len, lane, r);
    fwd_fetch(A, r, off, len, lane, f);
    fwd_ids(A, start, off + 32 * FWD_BATCH, len, lane, r);
    while (off < len) {
      {
        const bool live = __any_sync(0xffffffffu, P.cut < FWD_DEAD);
        if (lane == 0) s_live[warp] = live;
        pair_sync();
        if (!(s_live[warp] | s_live[warp ^ 1])) break;  // (both warps)
        // the record of segment k: the transmittance before entry k * BLEND_HEAD (where the backward replay of segment
        // k - 1 begins) and, once its entries are done, the colour they added
        if (half == 0 && lane == 0) s_slot[pair] = spare;
        if (cur_slot) {
          BlendRecord* q = A.ckpt + (size_t)(cur_slot - 1) * BLEND_STRIP_PIXELS + 32 * half + lane;
          q->S0 = P.D[0]; q->S1 = P.D[1]; q->S2 = P.D[2];
        }
        pair_sync();
        const uint32_t slot = s_slot[pair];
        have_spare = false;
        if (off + BLEND_HEAD < all) take_spare();
        if (slot < A.seg_cap) {
          if (half == 0 && lane == 0) {
            s_slots[pair][records & 3] = slot;
            A.seg_strip[slot] = make_uint2(strip, off / BLEND_HEAD);
            A.seg_link[slot] = make_uint2(0u, cur_slot);
            if (cur_slot) A.seg_link[cur_slot - 1].x = slot + 1;
          }
          if (!first_slot) first_slot = slot + 1;
          cur_slot = slot + 1;
          ++records;
          A.ckpt[(size_t)slot * BLEND_STRIP_PIXELS + 32 * half + lane].T = P.T;
          P.D[0] = P.D[1] = P.D[2] = 0.0;
        } else if (lane == 0) {
          odin_set_error(A.status, ODIN_ERR_CAPACITY);  // the backward pass will miss this strip's later segments
        }
      }
      const uint32_t seg_end = min(len, off + BLEND_HEAD);
      for (; off < seg_end; off += 32 * FWD_BATCH) {
        if (!__any_sync(0xffffffffu, P.cut < FWD_DEAD)) break;
        bool tame;
        const int cnt = fwd_stage(f, off, len, l2amin, x_lo, y_lo, s, lane, tame);
        // the next batch's rows and the ids behind them are on their way while this batch is blended
        fwd_fetch(A, r, off + 32 * FWD_BATCH, len, lane, f);
        fwd_ids(A, start, off + 64 * FWD_BATCH, len, lane, r);
        for (int i = lane; i < cnt + FWD_GROUP - 1; i += 32) {  // (the padding's too)
          s_cd[0][i] = (double)s.r[i]; s_cd[1][i] = (double)s.g[i]; s_cd[2][i] = (double)s.b[i];
        }
        __syncwarp();
        if (__builtin_expect(tame, 1)) fwd_rows<false>(s, s_cd, cnt, nfx, nfy, A.alpha_max, A.t_min, P);
        else fwd_rows<true>(s, s_cd, cnt, nfx, nfy, A.alpha_max, A.t_min, P);
      }
      off = seg_end;
    }
    const bool live_end = __any_sync(0xffffffffu, P.cut < FWD_DEAD);
    if (lane == 0) s_live[warp] = live_end;
    pair_sync();  // (the slots are written)
    const bool go_on = all > FWD_DEEP && (s_live[warp] | s_live[warp ^ 1]);
    if (inside) {
      const float tb = go_on ? 0.f : P.T;  // the background is added by whoever finishes the pixel
      A.out[pix] = P.C0 + tb * A.bg0;
      A.out[plane + pix] = P.C1 + tb * A.bg1;
      A.out[2 * plane + pix] = P.C2 + tb * A.bg2;
      A.final_T[pix] = P.T;
      A.n_contrib[pix] = P.last | (go_on && P.cut == FWD_DEAD ? BLEND_DONE_BIT : 0u);
    }
    if (go_on) {
      if (cur_slot) {
        BlendRecord* q = A.ckpt + (size_t)(cur_slot - 1) * BLEND_STRIP_PIXELS + 32 * half + lane;
        q->S0 = P.D[0]; q->S1 = P.D[1]; q->S2 = P.D[2];
      }
      // (the queue's third class is followed by room for the first two's strips)
      if (half == 0 && lane == 0) A.tail_queue[2 * n_strips + c[2] + atomicAdd(A.header + 25, 1u)] = strip;
    }
    // colour added by a segment -> colour still to come at its start, summed from the strip's last record to its first
    // (a lane rewrites its own words)
    if (cur_slot && !go_on) {
      double B[3] = {(double)P.T * (double)A.bg0, (double)P.T * (double)A.bg1, (double)P.T * (double)A.bg2};
      for (int k = records - 1; k >= 0; --k) {  // (at most three: the queue's lists are that short)
        BlendRecord* q = A.ckpt + (size_t)s_slots[pair][k & 3] * BLEND_STRIP_PIXELS + 32 * half + lane;
        const bool latest = k == records - 1;
        B[0] += latest ? P.D[0] : q->S0; B[1] += latest ? P.D[1] : q->S1; B[2] += latest ? P.D[2] : q->S2;
        q->S0 = B[0]; q->S1 = B[1]; q->S2 = B[2];
      }
    }
    if (half == 0 && lane == 0) A.strip_first[strip] = first_slot;
    pair_sync();  // s_item, s_live and the slots may be written again
  }
  if (have_spare && lane == 0 && spare < A.seg_cap) A.seg_strip[spare] = make_uint2(0xffffffffu, 0u);  // no strip's
}

// Strips with warps of two kinds, a block per strip (two cells of 8 x 4 pixels).  MAKERS warps fetch the list, a batch of 32
// entries each, test the rows against the two cells and evaluate the alphas of the cells' pixels; one more warp per cell takes
// the alphas of the step before and composites them, one pixel per lane.  What bounds it is the chain of dependent work
// along the longest list, so everything that does not depend on the transmittance is taken out of the warp that has to go
// through the list in order (256 x 256, all strips: 46 % of the issue slots while an SM has work, waits at the step's barrier and
// for the chain; behind the tail kernel, city from the street: an SM has work 21 % of the time, the longest lists).  (One warp per cell doing all of it, as in the tail kernel, against this: 64 x 64 pixels 20.7 ->
// 16.6 us; 320 x 180, lists of up to 9,900: 348 -> 193; 852 x 501, lists of up to 19,000, behind the head kernel: 720 -> 330.
// Lists of a few hundred entries gain nothing: 256 x 256, 46.5 -> 47.)  Shared memory, 45 KB, holds four blocks per SM; four
// makers, 90 KB and two blocks, are faster where few strips go deep (159 against 193 us, 330 against 370 in the examples) and
// slower where all strips run (62 against 47).  Behind the head kernel everything up to FWD_DEEP entries stays with the tail
// kernel: with lists of that length taken by blocks from the start 1600 x 1066 pixels took 25 -> 36 us and the aerial city
// 110 -> 133.
constexpr int FWD_PAD = 36;     // a maker's rows and the padding of its last group
constexpr int FWD_SLOTS = 128;  // records of a strip whose slots are kept at hand
template <bool DEEP>
struct FwdDivision {
  static constexpr int MAKERS = DEEP ? 4 : 2, STEP = 32 * MAKERS;  // list entries per step
  static constexpr int THREADS = 32 * (MAKERS + 2), BLOCKS = DEEP ? 2 : 4;
  static_assert((DEEP ? BLEND_HEAD : BLEND_FINE) % STEP == 0, "segments are whole steps");
};

template <int MAKERS>
struct FwdStep {  // what the makers leave of a step, by cell and maker; rows in list order, 32 places per maker
  float alpha[2][32 * MAKERS][32];                         // per pixel; sign bit set: the row fails a skip test there
  float4 colour[2][32 * MAKERS];                           // r, g, b, 1-based position in the list
  double wide[2][3][32 * MAKERS];                          // the colour in double (behind the first segment only)
  int count[2][MAKERS];                                    // (negative: not all of the rows' colours are tame)
};
struct FwdRows {  // a maker's rows of one cell, one array per quantity so that a group's values are wide loads
  float u[FWD_PAD], v[FWD_PAD], sA[FWD_PAD], sB[FWD_PAD], sC[FWD_PAD], lo[FWD_PAD];
};
template <int MAKERS>
struct FwdShared {
  FwdStep<MAKERS> step[2];
  FwdRows rows[MAKERS];
  uint32_t item, slot, live[2][2], eval[2];
  uint32_t slots[FWD_SLOTS];  // of the strip's first records
};

// A maker's share of a step: the rows of its 32 entries that reach a cell, and their alphas at the cell's pixels.
// (x, y): the strip's first pixel centre; f: the lane's row, entry off + lane of the list.
template <int MAKERS>
__device__ __forceinline__ void fwd_make(const FwdArgs& A, const BlendFetch& f, uint32_t off, uint32_t len, float l2amin, float x,
                                         float y, bool live0, bool live1, bool rec, FwdStep<MAKERS>& S, FwdRows& s, int maker, unsigned lane) {
  const float4 q = blend_stage_conic(f.co);
  const uint32_t ord = off + lane + 1;
  const BlendShape shape = blend_shape(f.co.x, f.co.y, f.co.z);
  const bool tame = blend_tame(f.r, f.g, f.b);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const float x_lo = x + 8.f * c;
    const bool reach = (c ? live1 : live0) && ord <= len &&
                       blend_reaches<8, 4>(f.c.x, f.c.y, f.co.x, f.co.y, f.co.z, shape, q.w, l2amin, x_lo, y);
    const uint32_t m = __ballot_sync(0xffffffffu, reach);
    const int cnt = __popc(m);
    const bool rare = __any_sync(0xffffffffu, reach && !(tame && shape.proper));
    if (lane == 0) S.count[c][maker] = cnt;
    __syncwarp();  // the rows of the cell before have been read
    if (reach) {
      const int d = __popc(m & ((1u << lane) - 1u)), e = 32 * maker + d;
      s.u[d] = f.c.x; s.v[d] = f.c.y; s.sA[d] = q.x; s.sB[d] = q.y; s.sC[d] = q.z; s.lo[d] = q.w;
      S.colour[c][e] = make_float4(f.r, f.g, f.b, __uint_as_float(ord));
      if (rec) { S.wide[c][0][e] = (double)f.r; S.wide[c][1][e] = (double)f.g; S.wide[c][2][e] = (double)f.b; }
    }
    const int pad = (cnt + 3) & ~3;  // rows that pass nowhere
    if (cnt + (int)lane < pad) {
      const int d = cnt + lane, e = 32 * maker + d;
      s.u[d] = s.v[d] = s.sA[d] = s.sB[d] = s.sC[d] = 0.f;
      s.lo[d] = -__builtin_huge_valf();
      S.colour[c][e] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (rec) S.wide[c][0][e] = S.wide[c][1][e] = S.wide[c][2][e] = 0.0;
    }
    __syncwarp();
    uint32_t odd = 0;  // rows whose conic is not proper
    if (rare) {
      if (__any_sync(0xffffffffu, reach && !tame) && lane == 0) S.count[c][maker] = -cnt;
      odd = __reduce_or_sync(0xffffffffu, reach && !shape.proper ? 1u << __popc(m & ((1u << lane) - 1u)) : 0u);
    }
    const f2 nfx = f2_dup(-(x_lo + (float)(lane & 7))), nfy = f2_dup(-(y + (float)(lane >> 3)));
    float(*out)[32] = S.alpha[c] + 32 * maker;
    auto alphas = [&](auto some) {
      for (int j = 0; j < cnt; j += 4) {
        const float4 u4 = *reinterpret_cast<const float4*>(s.u + j), v4 = *reinterpret_cast<const float4*>(s.v + j);
        const float4 a4 = *reinterpret_cast<const float4*>(s.sA + j), b4 = *reinterpret_cast<const float4*>(s.sB + j);
        const float4 c4 = *reinterpret_cast<const float4*>(s.sC + j), l4 = *reinterpret_cast<const float4*>(s.lo + j);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const f2 lo = f2_half(l4, i);
          const f2 p = blend_exponent2(f2_add(f2_half(u4, i), nfx), f2_add(f2_half(v4, i), nfy), f2_half(a4, i), f2_half(b4, i),
                                       f2_half(c4, i), lo);
          float p0, p1;
          f2_split(p, p0, p1);
          bool k0 = p0 >= l2amin, k1 = p1 >= l2amin;
          if (decltype(some)::value) {
            k0 = k0 && p0 <= blend_top(lo.x, odd >> (j + 2 * i) & 1u);
            k1 = k1 && p1 <= blend_top(lo.y, odd >> (j + 2 * i + 1) & 1u);
          }
          const float e0 = fminf(A.alpha_max, blend_ex2(p0)), e1 = fminf(A.alpha_max, blend_ex2(p1));
          out[j + 2 * i][lane] = k0 ? e0 : -0.f;
          out[j + 2 * i + 1][lane] = k1 ? e1 : -0.f;
        }
      }
    };
    if (__builtin_expect(odd == 0, 1)) alphas(std::false_type{});
    else alphas(std::true_type{});
  }
}

struct FwdPixel {
  float T, C0, C1, C2;
  float stopped;   // transmittance at which the pixel stopped; T is 0 from there on, so that every weight is
  float t_min;     // -1 once the pixel has stopped
  int pass;        // an alpha whose bits are at least this passed the tests and the pixel has not stopped
  uint32_t last;
  double D[3];     // (REC) colour the segment has added
  __device__ __forceinline__ bool dead() const { return pass != 0; }
  __device__ __forceinline__ float transmittance() const { return dead() ? stopped : T; }
  __device__ __forceinline__ void stop() { stopped = T; T = 0.f; t_min = -1.f; pass = 0x7fffffff; }
};

// The rows of a step, four at a time.  The transmittance only falls, so one test behind the four tells whether some pixel stops
// among them (once per pixel); only then they are gone through again one by one.  REC: the colour the rows add is also
// summed in double, for the segment records.  WILD: only where the row blends (see blend_tame).
template <bool REC, bool WILD, int MAKERS>
__device__ __forceinline__ void fwd_blend_rows(const FwdStep<MAKERS>& S, int c, int first, int cnt, unsigned lane, FwdPixel& P) {
  for (int j = first; j < first + cnt; j += 4) {
    float a[4], w[4];
    float4 col[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) { a[u] = S.alpha[c][j + u][lane]; col[u] = S.colour[c][j + u]; }
    const int pass = P.pass;  // (of a pixel that stops among these rows: up to the stop)
    float T = P.T;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      w[u] = a[u] * T;
      T -= w[u];
    }
    if (__any_sync(0xffffffffu, T < P.t_min)) {
      if (!P.dead()) {
        T = P.T;
#pragma unroll
        for (int u = 0; u < 4; ++u) {  // (up to the stop the weights are right)
          const float tn = T - w[u];
          if (!P.dead() && tn < P.t_min) {
            P.T = T;
            P.stop();  // in front of this row
            T = 0.f;
          }
          if (P.dead()) { w[u] = 0.f; a[u] = -0.f; }
          else T = tn;
        }
      }
    }
    P.T = T;
    if (WILD) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (__float_as_int(a[u]) < pass) continue;
        P.C0 = fmaf(col[u].x, w[u], P.C0); P.C1 = fmaf(col[u].y, w[u], P.C1); P.C2 = fmaf(col[u].z, w[u], P.C2);
        P.last = __float_as_uint(col[u].w);
        if (REC)
#pragma unroll
          for (int ch = 0; ch < 3; ++ch) P.D[ch] = fma(S.wide[c][ch][j + u], (double)w[u], P.D[ch]);
      }
      continue;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      P.C0 = fmaf(col[u].x, w[u], P.C0); P.C1 = fmaf(col[u].y, w[u], P.C1); P.C2 = fmaf(col[u].z, w[u], P.C2);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (__float_as_int(a[u]) >= pass) P.last = __float_as_uint(col[u].w);
    if (REC) {
      double wd[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) wd[u] = (double)w[u];
#pragma unroll
      for (int u = 0; u < 4; u += 2)
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
          const double2 d = *reinterpret_cast<const double2*>(S.wide[c][ch] + j + u);
          P.D[ch] = fma(d.x, wd[u], P.D[ch]);
          P.D[ch] = fma(d.y, wd[u + 1], P.D[ch]);
        }
    }
  }
}

template <bool REC, int MAKERS>
__device__ __forceinline__ void fwd_blend(const FwdStep<MAKERS>& S, int c, unsigned lane, FwdPixel& P) {
  for (int m = 0; m < MAKERS; ++m) {
    const int cnt = S.count[c][m];  // (negative: rows that are not tame)
    if (cnt >= 0) fwd_blend_rows<REC, false>(S, c, 32 * m, cnt, lane, P);
    else fwd_blend_rows<REC, true>(S, c, 32 * m, -cnt, lane, P);
  }
}

// DEEP: the strips that the tail kernel queued, from entry FWD_DEEP of the list on, state from the output images; otherwise
// all strips from the start.  Where a segment behind the first begins a record of the strip is opened as long as one
// of its pixels is live (see blend.cuh).  The image keeps its one sequential sum per pixel, so it does not depend on where
// the steps and segments fall.
template <bool DEEP>
__global__ void __launch_bounds__(FwdDivision<DEEP>::THREADS, FwdDivision<DEEP>::BLOCKS)
render_fwd_strip_kernel(FwdArgs A) {
  odin_after_predecessor();
  extern __shared__ __align__(16) uint8_t fwd_smem[];
  constexpr int MAKERS = FwdDivision<DEEP>::MAKERS, STEP = FwdDivision<DEEP>::STEP;
  FwdShared<MAKERS>& S = *reinterpret_cast<FwdShared<MAKERS>*>(fwd_smem);
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool maker = warp < MAKERS;
  const int cell = (int)warp - MAKERS;  // (of a compositing warp)
  // A segment slot is taken from the counter well before it is needed (the atomic's way there and back would stand in the chain
  // of the list once per segment); one that a strip did not need after all goes to the block's next strip.
  uint32_t spare = 0xffffffffu;  // (first compositing warp, lane 0)
  bool have_spare = false;
  auto take_spare = [&]() {
    if (cell == 0 && !have_spare) {
      spare = fwd_take(A.header + 2, spare, lane);
      have_spare = true;
    }
  };
  auto pair_sync = [&]() { asm volatile("bar.sync 1, 64;" ::: "memory"); };  // the two compositing warps
  const bool fine = !DEEP && blend_fine(A.n_tiles);
  const uint32_t second = blend_seg_length(0u, fine);  // where the second segment begins
  const float l2amin = log2f(A.alpha_min);
  const uint32_t n_strips = (uint32_t)A.n_tiles * BLEND_STRIPS;
  const size_t plane = (size_t)A.W * A.H;
  const uint32_t items = DEEP ? min(A.header[25], n_strips) : n_strips;
  if (DEEP && items == 0) return;
  const uint32_t* queue = A.tail_queue + 2 * (size_t)n_strips + (DEEP ? min(A.header[6], n_strips - items) : 0u);
  while (true) {
    if (threadIdx.x == 0) S.item = atomicAdd(A.header + (DEEP ? 24 : 0), 1u);
    __syncthreads();
    const uint32_t item = S.item;
    if (item >= items) break;
    const uint32_t strip = DEEP ? min(queue[item], n_strips - 1) : item;
    const int tile = (int)(strip / BLEND_STRIPS);
    const int x0 = (tile % A.TX) * 16, y0 = (tile / A.TX) * 16 + 4 * (int)(strip % BLEND_STRIPS);
    const uint2 rg = A.ranges[tile];
    const uint32_t start = rg.x, len = rg.y - rg.x, first = DEEP ? FWD_DEEP : 0u;
    const uint32_t steps = len > first ? (len - first + STEP - 1) / STEP : 0u;

    if (maker) {
      const float x = (float)x0 + 0.5f, y = (float)y0 + 0.5f;
      bool live0 = true, live1 = true;
      auto id = [&](uint32_t i) { return i < len ? min(A.vals[start + i], A.row_cap - 1) : 0u; };  // in range whatever the list holds
      auto fetch = [&](uint32_t i, uint32_t r) {
        BlendFetch f = {};
        if (i < len) f = blend_fetch(A.xy, A.conic_o, A.rgb, r);
        return f;
      };
      const uint32_t at = first + 32 * warp + lane;
      uint32_t r = id(at);
      BlendFetch f = fetch(at, r);
      r = id(at + STEP);
      for (uint32_t i = 0;; ++i) {
        if (i < steps) {
          const uint32_t off = first + i * STEP + 32 * warp;
          const BlendFetch now = f;
          // the next step's row and the id behind it are on their way while this step is evaluated
          f = fetch(off + STEP + lane, r);
          r = id(off + 2 * STEP + lane);
          fwd_make(A, now, off, len, l2amin, x, y, live0, live1, off >= second, S.step[i & 1], S.rows[warp], (int)warp, lane);
        }
        __syncthreads();
        if (i == steps) break;
        if (i > 0) {
          live0 = S.live[i & 1][0]; live1 = S.live[i & 1][1];
          if (!live0 && !live1) break;
        }
      }
      continue;
    }

    const int px = x0 + 8 * cell + (int)(lane & 7), py = y0 + (int)(lane >> 3);
    const bool inside = px < A.W && py < A.H;
    const size_t pix = (size_t)py * A.W + px;
    FwdPixel P;
    P.T = 1.f; P.C0 = P.C1 = P.C2 = 0.f; P.last = 0u;
    P.stopped = 0.f; P.t_min = A.t_min; P.pass = 0;
    P.D[0] = P.D[1] = P.D[2] = 0.0;
    if (!inside) P.stop();
    if (DEEP && inside) {
      P.T = A.final_T[pix];
      P.C0 = A.out[pix]; P.C1 = A.out[plane + pix]; P.C2 = A.out[2 * plane + pix];
      const uint32_t nc = A.n_contrib[pix];
      P.last = nc & ~BLEND_DONE_BIT;
      if (nc & BLEND_DONE_BIT) P.stop();
    }
    uint32_t n_eval = 0;  // rows evaluated in the first segment
    uint32_t first_slot = 0, cur_slot = 0;  // 1 + slot; 0 = none
    int records = 0;
    if (len > max(first, second)) take_spare();
    if (DEEP) {  // the records that the tail kernel opened
      first_slot = A.strip_first[strip];
      for (uint32_t s1 = first_slot; s1 != 0 && records < FWD_SLOTS; s1 = A.seg_link[s1 - 1].x) {
        if (cell == 0 && lane == 0) S.slots[records] = s1 - 1;
        cur_slot = s1;
        ++records;
      }
    }
    for (uint32_t i = 0;; ++i) {  // composites the step in front of the one that is being made
      if (i > 0) {
        const uint32_t off = first + (i - 1) * STEP;
        const FwdStep<MAKERS>& step = S.step[(i - 1) & 1];
        if (off < second) {
          for (int m = 0; m < MAKERS; ++m) n_eval += (uint32_t)abs(step.count[cell][m]);
          fwd_blend<false, MAKERS>(step, cell, lane, P);
        } else {
          if (off % blend_seg_length(off, fine) == 0) {
            // the record of segment k: the transmittance before its first entry (where the backward replay of segment
            // k - 1 begins) and, once its entries are done, the colour they added
            if (cell == 0 && lane == 0) S.slot = spare;
            if (cur_slot && off > first) {  // (the tail kernel has filled in its last one)
              BlendRecord* q = A.ckpt + (size_t)(cur_slot - 1) * BLEND_STRIP_PIXELS + 32 * cell + lane;
              q->S0 = P.D[0]; q->S1 = P.D[1]; q->S2 = P.D[2];
            }
            pair_sync();
            const uint32_t slot = S.slot;
            have_spare = false;
            if (off + blend_seg_length(off, fine) < len) take_spare();
            if (slot < A.seg_cap) {
              if (cell == 0 && lane == 0) {
                if (records < FWD_SLOTS) S.slots[records] = slot;
                A.seg_strip[slot] = make_uint2(strip, blend_seg_at(off, fine));
                A.seg_link[slot] = make_uint2(0u, cur_slot);
                if (cur_slot) A.seg_link[cur_slot - 1].x = slot + 1;
              }
              if (!first_slot) first_slot = slot + 1;
              cur_slot = slot + 1;
              ++records;
              A.ckpt[(size_t)slot * BLEND_STRIP_PIXELS + 32 * cell + lane].T = P.transmittance();
              P.D[0] = P.D[1] = P.D[2] = 0.0;
            } else if (lane == 0) {
              odin_set_error(A.status, ODIN_ERR_CAPACITY);  // the backward pass will miss this strip's later segments
            }
          }
          fwd_blend<true, MAKERS>(step, cell, lane, P);
        }
        const bool live = __any_sync(0xffffffffu, !P.dead());
        if (lane == 0) S.live[i & 1][cell] = live;
      }
      __syncthreads();
      if (i == steps || (i > 0 && !S.live[i & 1][0] && !S.live[i & 1][1])) break;
    }
    const float T = P.transmittance();
    if (inside) {
      A.out[pix] = P.C0 + T * A.bg0;
      A.out[plane + pix] = P.C1 + T * A.bg1;
      A.out[2 * plane + pix] = P.C2 + T * A.bg2;
      A.final_T[pix] = T;
      A.n_contrib[pix] = P.last;
    }
    // colour added by a segment -> colour still to come at its start, summed from the strip's last record to its first
    // (a lane rewrites its own words)
    if (lane == 0) S.eval[cell] = n_eval;
    pair_sync();  // the counts and the links are written
    if (cur_slot) {
      double B[3] = {(double)T * (double)A.bg0, (double)T * (double)A.bg1, (double)T * (double)A.bg2};
      BlendRecord* mine = A.ckpt + 32 * cell + lane;
      auto close = [&](uint32_t slot, double d0, double d1, double d2) {
        BlendRecord* q = mine + (size_t)slot * BLEND_STRIP_PIXELS;
        B[0] += d0; B[1] += d1; B[2] += d2;
        q->S0 = B[0]; q->S1 = B[1]; q->S2 = B[2];
      };
      close(cur_slot - 1, P.D[0], P.D[1], P.D[2]);
      int k = records - 2;
      for (uint32_t s1 = cur_slot; k >= FWD_SLOTS; --k) {  // records whose slots are only linked
        s1 = A.seg_link[s1 - 1].y;
        const BlendRecord* q = mine + (size_t)(s1 - 1) * BLEND_STRIP_PIXELS;
        close(s1 - 1, q->S0, q->S1, q->S2);
      }
      for (; k >= 0; k -= 4) {  // the others: four records on their way at a time
        double d[4][3];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const BlendRecord* q = mine + (size_t)S.slots[max(k - u, 0)] * BLEND_STRIP_PIXELS;
          d[u][0] = q->S0; d[u][1] = q->S1; d[u][2] = q->S2;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (k - u >= 0) close(S.slots[k - u], d[u][0], d[u][1], d[u][2]);
      }
    }
    if (cell == 0 && lane == 0) {
      A.strip_first[strip] = first_slot;
      if (!DEEP) {
        const uint32_t bc = blend_bwd_class((S.eval[0] + S.eval[1]) / 2);
        A.bwd_queue[bc * n_strips + atomicAdd(A.header + 8 + bc, 1u)] = strip;
      }
    }
  }
  if (have_spare && lane == 0 && spare < A.seg_cap) A.seg_strip[spare] = make_uint2(0xffffffffu, 0u);  // no strip's
}

// Measurement aid (not part of the view step): how many (pixel, list entry) pairs the compositing of a view consists
// of.  One block per tile, one pixel per thread, the same tests as the forward kernels.  counts[0]: pairs inside the
// pixel's walked prefix (entries up to the last one that contributed to the pixel); counts[1]: those that blend (pass
// the skip tests): the pairs the backward pass differentiates.
__global__ void __launch_bounds__(256)
count_pairs_kernel(const float2* __restrict__ xy, const float4* __restrict__ conic_o, const uint32_t* __restrict__ vals,
                   const uint2* __restrict__ ranges, int W, int H, int TX, float alpha_min, float alpha_max,
                   const uint32_t* __restrict__ n_contrib, uint32_t row_cap, unsigned long long* __restrict__ counts) {
  const int tile = blockIdx.x;
  const int px = (tile % TX) * 16 + (int)(threadIdx.x & 15), py = (tile / TX) * 16 + (int)(threadIdx.x >> 4);
  unsigned long long walked = 0, blended = 0;
  if (px < W && py < H) {
    const uint32_t start = ranges[tile].x;
    const uint32_t n = min(n_contrib[(size_t)py * W + px], ranges[tile].y - start);
    const float fx = (float)px + 0.5f, fy = (float)py + 0.5f;
    walked = n;
    for (uint32_t k = 0; k < n; ++k) {
      const uint32_t r = min(vals[start + k], row_cap - 1);
      const float2 c = xy[r];
      const float4 q = conic_o[r];
      const float dx = c.x - fx, dy = c.y - fy;
      const float power = -0.5f * (q.x * dx * dx + q.z * dy * dy) - q.y * dx * dy;
      if (power > 0.f) continue;
      if (fminf(alpha_max, q.w * __expf(power)) < alpha_min) continue;
      ++blended;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    walked += __shfl_xor_sync(0xffffffffu, walked, o);
    blended += __shfl_xor_sync(0xffffffffu, blended, o);
  }
  if ((threadIdx.x & 31) == 0 && walked) {
    atomicAdd(&counts[0], walked);
    atomicAdd(&counts[1], blended);
  }
}

constexpr int LB = 256;

__global__ void __launch_bounds__(LB)
l1_loss_kernel(const float* __restrict__ out, const float* __restrict__ target, size_t count, float inv, double* loss_acc,
               float* __restrict__ dL, double inv_count, float* __restrict__ loss, size_t vec4) {
  odin_after_predecessor();
  // vec4: number of leading float4 groups (0 when the three images are not 16-byte aligned); the rest one by one
  float acc = 0.f;
  const size_t tid = (size_t)blockIdx.x * LB + threadIdx.x, stride = (size_t)gridDim.x * LB;
  for (size_t i = tid; i < vec4; i += stride) {
    const float4 a = reinterpret_cast<const float4*>(out)[i], b = reinterpret_cast<const float4*>(target)[i];
    const float d0 = a.x - b.x, d1 = a.y - b.y, d2 = a.z - b.z, d3 = a.w - b.w;
    acc += (fabsf(d0) + fabsf(d1)) + (fabsf(d2) + fabsf(d3));
    reinterpret_cast<float4*>(dL)[i] = make_float4(d0 > 0.f ? inv : (d0 < 0.f ? -inv : 0.f), d1 > 0.f ? inv : (d1 < 0.f ? -inv : 0.f),
                                                   d2 > 0.f ? inv : (d2 < 0.f ? -inv : 0.f), d3 > 0.f ? inv : (d3 < 0.f ? -inv : 0.f));
  }
  for (size_t i = vec4 * 4 + tid; i < count; i += stride) {
    const float d = out[i] - target[i];
    acc += fabsf(d);
    dL[i] = d > 0.f ? inv : (d < 0.f ? -inv : 0.f);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  __shared__ float s[LB / 32];
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int i = 0; i < LB / 32; ++i) t += (double)s[i];
    atomicAdd(loss_acc, t);
    // the block that arrives last turns the sum into the mean (no second launch)
    __threadfence();
    uint32_t* arrivals = reinterpret_cast<uint32_t*>(loss_acc + 1);
    if (atomicAdd(arrivals, 1u) == gridDim.x - 1u) {
      __threadfence();
      *loss = (float)(atomicAdd(loss_acc, 0.0) * inv_count);
      *loss_acc = 0.0;
      *arrivals = 0u;
    }
  }
}

}  // namespace

extern "C" int odin_render_workspace_bytes(const odin_ctx* ctx, int width, int height, size_t* bytes) {
  if (!ctx || !bytes) return ODIN_ERR_NULL;
  if (width <= 0 || height <= 0 || width > 16384 || height > 16384) return ODIN_ERR_INVALID_ARG;
  *bytes = blend_ws_bytes(width, height);
  return ODIN_OK;
}

extern "C" int odin_render_fwd(odin_ctx* ctx, const odin_projected* proj, const uint32_t* d_vals,
                               const uint32_t* d_tile_ranges, const odin_camera* cam, float* d_rgb, float* d_final_T,
                               uint32_t* d_n_contrib, void* ws, size_t ws_bytes, void* stream) {
  if (!ctx || !proj || !d_tile_ranges || !d_rgb || !d_final_T || !d_n_contrib) return ODIN_ERR_NULL;
  const int rc = odin_check_camera(cam);
  if (rc != ODIN_OK) return rc;
  if (proj->capacity > 0 && (!proj->xy || !proj->conic_opacity || !proj->rgb || !d_vals)) return ODIN_ERR_NULL;
  if (!odin_aligned(proj->xy, 8) || !odin_aligned(proj->conic_opacity, 16) || !odin_aligned(d_tile_ranges, 8))
    return ODIN_ERR_INVALID_ARG;
  const int TX = (cam->width + 15) / 16, TY = (cam->height + 15) / 16;
  const int n_tiles = TX * TY;
  if (!ws || !odin_aligned(ws, 256) || ws_bytes < blend_ws_bytes(cam->width, cam->height)) return ODIN_ERR_WORKSPACE;
  const BlendWs L = blend_ws_layout(n_tiles, blend_ws_records(n_tiles, ws_bytes));
  char* base = reinterpret_cast<char*>(ws);
  uint32_t* header = reinterpret_cast<uint32_t*>(base);
  cudaStream_t st = (cudaStream_t)stream;
  const bool tiles = blend_tile_items(n_tiles);
  // tickets, segments taken, the class counts of the two queues; where tiles are filed, their counters right behind
  ODIN_CUDA(odin_zero(ctx, header, BLEND_WS_HEADER + (tiles ? (size_t)n_tiles * 4 : 0), st));
  FwdArgs A;
  A.xy = reinterpret_cast<const float2*>(proj->xy); A.conic_o = reinterpret_cast<const float4*>(proj->conic_opacity);
  A.rgb = proj->rgb; A.vals = d_vals; A.ranges = reinterpret_cast<const uint2*>(d_tile_ranges);
  A.W = cam->width; A.H = cam->height; A.TX = TX; A.n_tiles = n_tiles;
  A.bg0 = cam->bg[0]; A.bg1 = cam->bg[1]; A.bg2 = cam->bg[2];
  A.alpha_min = ctx->cfg.alpha_min; A.alpha_max = ctx->cfg.alpha_max; A.t_min = ctx->cfg.t_min;
  A.out = d_rgb; A.final_T = d_final_T; A.n_contrib = d_n_contrib;
  A.strip_first = reinterpret_cast<uint32_t*>(base + L.strip_first); A.header = header;
  A.tile_work = reinterpret_cast<uint32_t*>(base + BLEND_WS_HEADER);
  A.tail_queue = reinterpret_cast<uint32_t*>(base + L.tail_queue); A.bwd_queue = reinterpret_cast<uint32_t*>(base + L.bwd_queue);
  A.seg_strip = reinterpret_cast<uint2*>(base + L.seg_strip); A.seg_link = reinterpret_cast<uint2*>(base + L.seg_link);
  A.ckpt = reinterpret_cast<BlendRecord*>(base + L.ckpt); A.seg_cap = L.segments; A.status = ctx->d_status;
  A.row_cap = proj->capacity;
  // resident warps pull their work: half tiles (head) or strips (two warps each)
  // resident warps pull their work: half tiles (head, one warp each), strips (strip kernel, a block each), strips (tail kernel,
  // two warps each)
  auto blocks = [&](size_t items, size_t per_block, int resident) {
    const size_t all = (items + per_block - 1) / per_block, most = (size_t)ctx->sm_count * resident;
    return dim3((unsigned)(all < most ? all : most));
  };
  const size_t strips = (size_t)n_tiles * BLEND_STRIPS;
  auto launch_strips = [&](auto deep, bool dependent) {
    constexpr bool DEEP = decltype(deep)::value;
    typedef FwdDivision<DEEP> D;
    const int smem = (int)sizeof(FwdShared<D::MAKERS>);
    const cudaError_t e = cudaFuncSetAttribute(render_fwd_strip_kernel<DEEP>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return odin_launch(ctx, dependent, render_fwd_strip_kernel<DEEP>, blocks(strips, 1, D::BLOCKS), dim3(D::THREADS), smem, st, A);
  };
  if (!tiles) {
    OdinKernelScope ks(ctx, K_FWD, st);
    ODIN_CUDA(launch_strips(std::false_type{}, false));
    return odin_launch_status();
  }
  {
    OdinKernelScope ks(ctx, K_FWD, st);
    ODIN_CUDA(odin_launch(ctx, false, render_fwd_head_kernel, blocks(strips / 2, BLEND_WARPS, FWD_HEAD_BLOCKS), dim3(BLEND_THREADS), 0, st, A));
  }
  OdinKernelScope ks(ctx, K_FWD_TAIL, st);
  ODIN_CUDA(odin_launch(ctx, true, render_fwd_tail_kernel, blocks(strips, BLEND_WARPS / 2, FWD_TAIL_BLOCKS), dim3(BLEND_THREADS), 0, st, A));
  ODIN_CUDA(launch_strips(std::true_type{}, true));
  return odin_launch_status();
}

extern "C" int odin_count_blend_pairs(odin_ctx* ctx, const odin_projected* proj, const uint32_t* d_vals,
                                      const uint32_t* d_tile_ranges, const odin_camera* cam, const uint32_t* d_n_contrib,
                                      uint64_t* d_counts, void* stream) {
  if (!ctx || !proj || !d_tile_ranges || !d_n_contrib || !d_counts) return ODIN_ERR_NULL;
  const int rc = odin_check_camera(cam);
  if (rc != ODIN_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  odin_chain_break(ctx);
  ODIN_CUDA(cudaMemsetAsync(d_counts, 0, 16, st));
  if (proj->capacity == 0) return ODIN_OK;
  if (!proj->xy || !proj->conic_opacity || !d_vals) return ODIN_ERR_NULL;
  const int TX = (cam->width + 15) / 16, TY = (cam->height + 15) / 16;
  count_pairs_kernel<<<TX * TY, 256, 0, st>>>(
      reinterpret_cast<const float2*>(proj->xy), reinterpret_cast<const float4*>(proj->conic_opacity), d_vals,
      reinterpret_cast<const uint2*>(d_tile_ranges), cam->width, cam->height, TX, ctx->cfg.alpha_min, ctx->cfg.alpha_max,
      d_n_contrib, proj->capacity, reinterpret_cast<unsigned long long*>(d_counts));
  return odin_launch_status();
}

extern "C" int odin_l1_loss(odin_ctx* ctx, const float* d_rgb, const float* d_target, int width, int height,
                            float* d_loss, float* d_dL_drgb, void* stream) {
  if (!ctx || !d_rgb || !d_target || !d_loss || !d_dL_drgb) return ODIN_ERR_NULL;
  if (width <= 0 || height <= 0) return ODIN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t count = (size_t)3 * width * height;
  // the accumulator (8 bytes) and the arrival counter of the blocks (4 bytes behind it) live behind the status word in
  // the context's device block; the last block leaves both at zero for the next call
  double* acc = reinterpret_cast<double*>(reinterpret_cast<char*>(ctx->d_status) + 64);
  const bool aligned = odin_aligned(d_rgb, 16) && odin_aligned(d_target, 16) && odin_aligned(d_dL_drgb, 16);
  const size_t vec4 = aligned ? count / 4 : 0;
  size_t blocks = (count / 4 + LB - 1) / LB + 1;
  if (blocks > (size_t)ctx->sm_count * 8) blocks = (size_t)ctx->sm_count * 8;
  OdinKernelScope ks(ctx, K_L1, st);
  ODIN_CUDA(odin_launch(ctx, false, l1_loss_kernel, dim3((unsigned)blocks), dim3(LB), 0, st, d_rgb, d_target, count, (float)(1.0 / (double)count), acc, d_dL_drgb,
                                                  1.0 / (double)count, d_loss, vec4));
  return odin_launch_status();
}
