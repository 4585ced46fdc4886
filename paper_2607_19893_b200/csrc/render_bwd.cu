// Backward phase: (a) back-to-front replay of the compositing, one warp per segment of a region's list, per-lane
// accumulation over the lane's pixels, sums over the lanes for several rows at a time through shared memory and one
// global atomic per (segment, row, word); (b) per-row chain rule through the projection into compact gradient rows.
#include <type_traits>

#include "blend.cuh"
#include "geom.cuh"

namespace {

__global__ void zero_rows_kernel(float* __restrict__ g2d, uint8_t* __restrict__ row_active,
                                 const uint32_t* __restrict__ num_rows, uint32_t capacity, uint32_t* __restrict__ ticket) {
  odin_after_predecessor();
  if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0u;
  const uint32_t V = min(*num_rows, capacity);
  const size_t count = (size_t)V * 9;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
    g2d[i] = 0.f;
    if (row_active && i < V) row_active[i] = 0;
  }
}

struct BwdArgs {
  const float2* xy;
  const float4* conic_o;
  const float* rgb;
  const uint32_t* vals;
  const uint2* ranges;
  int W, H, TX, n_tiles;
  float bg0, bg1, bg2, alpha_min, alpha_max;
  const uint32_t* strip_first;
  const uint32_t* seg_count;
  const uint2* seg_strip;
  const uint2* seg_link;
  const BlendRecord* ckpt;
  uint32_t seg_cap;
  const float* final_T;
  const uint32_t* n_contrib;
  const float* dL;
  float* g2d;
  uint32_t* ticket;
  uint8_t* row_active;
  uint32_t row_cap;
  const uint32_t* bwd_count;
  const uint32_t* bwd_queue;
};

// Sums over the lanes.  A row that contributes leaves nine partial sums per lane; BWD_PEND rows are collected in shared
// memory, two lines of 32 four-word entries and one of 32 words per row, and then every lane adds up half of one wide line
// and an eighth of two narrow ones and issues the global atomics: three stores per row and some ninety instructions per
// BWD_PEND rows, where a transposing reduction by shuffles takes some fifty per row and a line per word nine stores and
// fifteen.  BWD_WIDE and BWD_LINE set the lines apart so that the wide loads of a quarter warp meet all banks.  The nine sums
// are those of dL/dpower times dx, dy, dx^2, dx dy, dy^2 and 1 and of the three colour weights; the row's constants are applied
// to the totals.
constexpr int BWD_PEND = 8;
constexpr int BWD_WIDE = 34;  // four-word entries
constexpr int BWD_LINE = 36;  // words
constexpr int BWD_ROWS = 32;
struct BwdWarp {
  BlendRow row[BWD_ROWS];
  float2 aux[BWD_ROWS];  // row id (bits), 1 / opacity (negative: the row is not plain, see bwd_plain)
  float4 wide[BWD_PEND][2][BWD_WIDE];  // sums with dx, dy, 1, dx^2; dx dy, dy^2, and the weights for red, green
  float blue[BWD_PEND][BWD_LINE];
  float4 pend_conic[BWD_PEND];  // sA, sB, sC, 1 / opacity
  uint32_t pend_row[BWD_PEND];
};

__device__ __forceinline__ void bwd_flush(BwdWarp& s, int pending, float* __restrict__ g2d, unsigned lane) {
  __syncwarp();
  // four lanes per row: lane c of them takes every other entry of wide line c / 2 and then two words of the line
  const unsigned row = lane >> 2, c = lane & 3;
  const float4* line = s.wide[row][c >> 1] + (c & 1);
  f2 a[2] = {f2_dup(0.f), f2_dup(0.f)}, b[2] = {a[0], a[0]};
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float4 v = line[2 * i];
    a[i & 1] = f2_add(a[i & 1], f2_half(v, 0));
    b[i & 1] = f2_add(b[i & 1], f2_half(v, 1));
  }
  const f2 lo = f2_add(a[0], a[1]), hi = f2_add(b[0], b[1]);
  const f2 send = c & 1 ? lo : hi, keep = c & 1 ? hi : lo;
  const f2 t = f2_add(keep, f2_make(__shfl_xor_sync(0xffffffffu, send.x, 1), __shfl_xor_sync(0xffffffffu, send.y, 1)));
  const float4 v0 = reinterpret_cast<const float4*>(s.blue[row])[c], v1 = reinterpret_cast<const float4*>(s.blue[row])[c + 4];
  float t2 = f2_sum(f2_add(f2_add(f2_half(v0, 0), f2_half(v0, 1)), f2_add(f2_half(v1, 0), f2_half(v1, 1))));
  t2 += __shfl_xor_sync(0xffffffffu, t2, 1);
  t2 += __shfl_xor_sync(0xffffffffu, t2, 2);
  if ((int)row < pending) {
    const float4 q = s.pend_conic[row];
    float t0 = t.x, t1 = t.y;
    // the staged conic is (-A log2(e) / 2, -B log2(e), -C log2(e) / 2): -(A gdx + B gdy) = ln 2 (2 sA gdx + sB gdy)
    if (c == 0) {
      t0 = BLEND_LN2 * fmaf(2.f * q.x, t.x, q.y * t.y);
      t1 = BLEND_LN2 * fmaf(2.f * q.z, t.y, q.y * t.x);
    } else if (c < 3) {
      t0 *= c == 1 ? q.w : -1.f;
      t1 *= -0.5f;
    }
    float* g = g2d + (size_t)s.pend_row[row] * 9;
    if (t0 != 0.f) atomicAdd(g + (c == 1 ? 5 : c == 2 ? 3 : 2 * c), t0);
    if (t1 != 0.f) atomicAdd(g + (c == 1 ? 2 : c == 2 ? 4 : 2 * c + 1), t1);
    if (c == 2 && t2 != 0.f) atomicAdd(g + 8, t2);
  }
  __syncwarp();
}

// A row's partial sums of this lane; flushes when BWD_PEND rows have come together.  j: the row's place in the staged batch
template <bool TRACK>
__device__ __forceinline__ void bwd_pend(const BwdArgs& P, BwdWarp& s, int& pending, int j, float4 conic, float gx, float gy, float gxx,
                                         float gxy, float gyy, float gp, float ar, float ag, float ab, unsigned lane) {
  s.wide[pending][0][lane] = make_float4(gx, gy, gp, gxx);
  s.wide[pending][1][lane] = make_float4(gxy, gyy, ar, ag);
  s.blue[pending][lane] = ab;
  const float2 aux = s.aux[j];
  if (lane == 0) {
    s.pend_row[pending] = __float_as_uint(aux.x);
    s.pend_conic[pending] = make_float4(conic.x, conic.y, conic.z, fabsf(aux.y));
  }
  if (TRACK) {
    if (lane == 2) P.row_active[__float_as_uint(aux.x)] = 1;  // realized-active: blended into at least one pixel
  }
  if (++pending == BWD_PEND) {
    bwd_flush(s, BWD_PEND, P.g2d, lane);
    pending = 0;
  }
}

// A row is PLAIN when its alpha cannot reach alpha_max: 2^p is at most its opacity (of a proper conic, see blend.cuh; the margin covers the
// rounding).  Nothing is clamped then, which are six of some 38 instructions per pair of pixels.  With this and the wide lines
// above 1600 x 1066 took 234 -> 217 us (159 -> 138 M warp instructions), the aerial city 422 -> 403, 1237 x 823 167 -> 153.
__device__ __forceinline__ bool bwd_plain(float lo, const BlendShape& shape, float l2amax) { return lo <= l2amax - 1e-3f && shape.proper; }

// Both kinds of item replay a segment back to front from the state at its END: that of the next segment's record, or the
// final state of the pixel when nothing behind the segment contributed.  Per pixel the transmittance T behind the row and
// A, the colour to come behind the row times the pixel's incoming gradient and over T, are carried: with the row's
// colour times that gradient cg, dL/dalpha = T_front (cg - A) and A becomes A + alpha (cg - A) in front of the row, a
// convex combination (no difference of sums, and one reciprocal, that of 1 - alpha, per pixel).
// TRACK: also flag the rows that contributed (realized active set).

// A pixel's state at the end of a segment from the record of the one behind it.
__device__ __forceinline__ void bwd_from_record(const BlendRecord* __restrict__ c, float g0, float g1, float g2, float& T, float& A) {
  const BlendRecord r = *c;
  T = r.T;
  A = (float)(fma(r.S2, (double)g2, fma(r.S1, (double)g1, r.S0 * (double)g0)) / (double)r.T);
}

// Of a pair, the halves at which the row blends (og: opacity * exp(power), 0 elsewhere), and 0: for rows and pixels with something
// that is not a number (WILD, see blend_tame; for a whole batch and all that follow, as it stays in the pixels' A).
__device__ __forceinline__ f2 bwd_where(f2 og, f2 x) { return f2_make(og.x > 0.f ? x.x : 0.f, og.y > 0.f ? x.y : 0.f); }

// Where a pixel of a strip stands in the strip's record: two cells of 8 x 4 pixels (the forward pass's warps).
__device__ __forceinline__ uint32_t bwd_record_index(uint32_t slot, int x, int y) {  // x, y inside the strip
  return slot * BLEND_STRIP_PIXELS + 32 * (x >> 3) + 8 * y + (x & 7);
}

// A strip's segment, two pixels per lane: lane l handles column l % 16, pixel rows l / 16 and l / 16 + 2 of the strip, in the
// two halves of packed registers.  Two rows at a time: what is independent of the state before them is evaluated together.
template <bool TRACK>
__device__ __forceinline__ void bwd_strip(const BwdArgs& P, BwdWarp& s, uint32_t strip, uint32_t seg, uint32_t next, float l2amin, float l2amax,
                                          unsigned lane) {
  constexpr int G = 2;
  const bool fine = blend_fine(P.n_tiles);
  const uint32_t seg_base = blend_seg_begin(seg, fine), seg_end = seg_base + blend_seg_length(seg_base, fine);
  const int tile = (int)(strip / BLEND_STRIPS);
  const int px = (tile % P.TX) * 16 + (int)(lane & 15), y0 = (tile / P.TX) * 16 + 4 * (int)(strip % BLEND_STRIPS);
  const int py0 = y0 + (int)(lane >> 4);
  const float fx = (float)px + 0.5f, fy = (float)py0 + 0.5f;
  const float x_lo = (float)((tile % P.TX) * 16) + 0.5f, y_lo = (float)y0 + 0.5f;
  const f2 nfy = f2_make(-fy, -(fy + 2.f)), minus1 = f2_dup(-1.f), one = f2_dup(1.f);
  const uint2 rg = P.ranges[tile];
  const size_t plane = (size_t)P.W * P.H;
  float t[2], a[2], g[2][3];
  uint32_t last[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int py = py0 + 2 * h;
    t[h] = 1.f; g[h][0] = g[h][1] = g[h][2] = 0.f; last[h] = 0;
    if (px < P.W && py < P.H) {
      const size_t pix = (size_t)py * P.W + px;
      t[h] = P.final_T[pix];
      last[h] = P.n_contrib[pix];
      g[h][0] = P.dL[pix]; g[h][1] = P.dL[plane + pix]; g[h][2] = P.dL[2 * plane + pix];
    }
    a[h] = P.bg0 * g[h][0] + P.bg1 * g[h][1] + P.bg2 * g[h][2];  // behind everything: the background
  }
  uint32_t total = __reduce_max_sync(0xffffffffu, max(last[0], last[1]));  // list entries any pixel of the strip used
  if (total <= seg_base) return;                                          // nothing in this segment contributed
  if (total > seg_end) {
    total = seg_end;
    // next == 0: the record is missing (the segment slots ran out, which the forward call reported, or n_contrib is not
    // the forward pass's own); the final state stands in, exact for the pixels that end inside this segment
    if (next != 0) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
        bwd_from_record(P.ckpt + bwd_record_index(next - 1, (int)(lane & 15), 2 * h + (int)(lane >> 4)), g[h][0], g[h][1], g[h][2], t[h], a[h]);
    }
  }
  bool wild = __any_sync(0xffffffffu, !(blend_tame(g[0][0], g[0][1], g[0][2]) && blend_tame(g[1][0], g[1][1], g[1][2]) &&
                                        fmaxf(fabsf(a[0]), fabsf(a[1])) < BLEND_TAME_PRODUCT && a[0] == a[0] && a[1] == a[1]));
  f2 T = f2_make(t[0], t[1]), A = f2_make(a[0], a[1]);
  const f2 g0 = f2_make(g[0][0], g[1][0]), g1 = f2_make(g[0][1], g[1][1]), g2 = f2_make(g[0][2], g[1][2]);
  total = min(total, rg.y - rg.x) - min(seg_base, rg.y - rg.x);  // entries of this segment to walk
  const uint32_t seg_start = rg.x + seg_base;
  int pending = 0;
  // walk the entries back to front, 32 at a time; the rows of the next batch are fetched while one is replayed
  const int nb = (int)((total + 31) / 32);
  BlendFetch f = {};
  uint32_t rid = 0, rid_next = 0;
  if (nb > 0) {
    const uint32_t i = (uint32_t)(nb - 1) * 32 + lane;
    if (i < total) { rid = min(P.vals[seg_start + i], P.row_cap - 1); f = blend_fetch(P.xy, P.conic_o, P.rgb, rid); }
    if (nb > 1) rid_next = min(P.vals[seg_start + i - 32], P.row_cap - 1);
  }
  for (int bi = nb - 1; bi >= 0; --bi) {
    const uint32_t b = (uint32_t)bi * 32;
    const float4 conic = blend_stage_conic(f.co);
    const BlendShape shape = blend_shape(f.co.x, f.co.y, f.co.z);
    const bool reach = b + lane < total && blend_reaches<16, 4>(f.c.x, f.c.y, f.co.x, f.co.y, f.co.z, shape, conic.w, l2amin, x_lo, y_lo);
    const uint32_t m = __ballot_sync(0xffffffffu, reach);
    const int cnt = __popc(m);
    const bool tame = blend_tame(f.r, f.g, f.b);
    uint32_t odd = 0;  // staged rows whose conic is not proper: the only ones whose exponent is tested against their opacity
    if (__any_sync(0xffffffffu, reach && !(tame && shape.proper))) {
      wild |= __any_sync(0xffffffffu, reach && !tame);
      odd = __reduce_or_sync(0xffffffffu, reach && !shape.proper ? 1u << __popc(m & ((1u << lane) - 1u)) : 0u);
    }
    __syncwarp();
    if (reach) {
      const int pos = __popc(m & ((1u << lane) - 1u));
      s.row[pos].a = make_float4(f.r, f.r, f.g, f.g);
      s.row[pos].b = make_float4(f.b, __uint_as_float(seg_base + b + lane + 1), f.c.x, f.c.y);
      s.row[pos].c = conic;
      s.aux[pos] = make_float2(__uint_as_float(rid), (bwd_plain(conic.w, shape, l2amax) ? 1.f : -1.f) / f.co.w);
    }
    __syncwarp();
    const uint32_t plain = __ballot_sync(0xffffffffu, (int)lane < cnt && s.aux[lane].y > 0.f);
    if (bi > 0) {
      rid = rid_next;
      f = blend_fetch(P.xy, P.conic_o, P.rgb, rid);
      if (bi > 1) rid_next = min(P.vals[seg_start + b - 64 + lane], P.row_cap - 1);
    }
    auto rows = [&](int j0, auto where, auto kind, auto test) {
      constexpr bool WILD = decltype(where)::value, PLAIN = decltype(kind)::value, TEST = decltype(test)::value;
      f2 dy[G], al[G], inv[G], cg[G], og[G];
      float dx[G];
      float4 rc[G];
#pragma unroll
      for (int u = 0; u < G; ++u) {
        const int j = max(j0 - u, 0);
        const float4 ra = s.row[j].a, rb = s.row[j].b;
        rc[u] = s.row[j].c;
        dx[u] = rb.z - fx;
        float h0, h1, h2;
        blend_x_terms(rc[u], dx[u], h0, h1, h2);
        dy[u] = f2_add(f2_dup(rb.w), nfy);
        float p0, p1;
        f2_split(f2_fma(dy[u], f2_fma(f2_dup(h2), dy[u], f2_dup(h1)), f2_dup(h0)), p0, p1);
        const uint32_t ord = j0 - u >= 0 ? __float_as_uint(rb.y) : 0xffffffffu;
        bool k0 = ord <= last[0] && p0 >= l2amin, k1 = ord <= last[1] && p1 >= l2amin;
        if (TEST) {
          const float top = blend_top(rc[u].w, odd >> j & 1u);
          k0 = k0 && p0 <= top;
          k1 = k1 && p1 <= top;
        }
        og[u] = f2_make(k0 ? blend_ex2(p0) : 0.f, k1 ? blend_ex2(p1) : 0.f);  // opacity * exp(power), 0 where it does not blend
        al[u] = PLAIN ? og[u] : f2_make(fminf(P.alpha_max, og[u].x), fminf(P.alpha_max, og[u].y));
        const f2 om = f2_fma(al[u], minus1, one);
        inv[u] = f2_make(blend_rcp(om.x), blend_rcp(om.y));
        cg[u] = f2_fma(f2_dup(rb.x), g2, f2_fma(f2_make(ra.z, ra.w), g1, f2_mul(f2_make(ra.x, ra.y), g0)));
      }
#pragma unroll
      for (int u = 0; u < G; ++u) {
        const f2 Tb = f2_mul(T, inv[u]);  // transmittance in front of the row
        auto at = [&](f2 x) { return WILD ? bwd_where(og[u], x) : x; };
        const f2 w = f2_mul(al[u], Tb), d = at(f2_fma(A, minus1, cg[u]));
        A = f2_fma(al[u], d, A);
        T = Tb;
        if (!__any_sync(0xffffffffu, fmaxf(og[u].x, og[u].y) > 0.f)) continue;  // the row blends nowhere in the strip
        // dL/dpower; dL/dopacity is this over the opacity.  A clamped alpha passes no gradient to opacity or geometry.
        const f2 gp = f2_mul(PLAIN ? w : f2_make(og[u].x <= P.alpha_max ? w.x : 0.f, og[u].y <= P.alpha_max ? w.y : 0.f), d);
        const f2 gy = f2_mul(gp, dy[u]);
        const float gpsum = f2_sum(gp), m1y = f2_sum(gy), gd = dx[u] * gpsum;
        bwd_pend<TRACK>(P, s, pending, max(j0 - u, 0), rc[u], gd, m1y, dx[u] * gd, dx[u] * m1y, f2_sum(f2_mul(gy, dy[u])), gpsum,
                        f2_sum(f2_mul(w, at(g0))), f2_sum(f2_mul(w, at(g1))), f2_sum(f2_mul(w, at(g2))), lane);
      }
    };
    if (__builtin_expect(!wild && odd == 0, 1)) {
      for (int j0 = cnt - 1; j0 >= 0; j0 -= G) {  // (the row that fills up the last pair is row 0 again)
        if (j0 > 0 ? (plain >> (j0 - 1) & 3u) == 3u : (plain & 1u) != 0u) rows(j0, std::false_type{}, std::true_type{}, std::false_type{});
        else rows(j0, std::false_type{}, std::false_type{}, std::false_type{});
      }
    } else if (!wild) {  // (a loop of its own: with the third kind in the one above 256 x 256 takes 1 % longer)
      for (int j0 = cnt - 1; j0 >= 0; j0 -= G) rows(j0, std::false_type{}, std::false_type{}, std::true_type{});
    } else {
      for (int j0 = cnt - 1; j0 >= 0; j0 -= G) rows(j0, std::true_type{}, std::false_type{}, std::true_type{});
    }
  }
  if (pending) bwd_flush(s, pending, P.g2d, lane);
}

// The first segment of a whole tile, eight pixels per lane: lane l handles column l % 16; its slot s is pixel row
// 2 s + l / 16, and the two slots of a strip of four pixel rows are the two halves of packed registers.  For every row the
// lane accumulates, over its own pixels, the colour weights and the moments of dL/dpower in dy; dx is constant per lane.
template <bool TRACK>
__device__ __forceinline__ void bwd_tile(const BwdArgs& P, BwdWarp& s, int tile, float l2amin, float l2amax, unsigned lane) {
  constexpr int Q = 4;
  const int tx = tile % P.TX, ty = tile / P.TX;
  const int px = tx * 16 + (int)(lane & 15);
  const int py0 = ty * 16 + (int)(lane >> 4);
  const float fx = (float)px + 0.5f;
  const float x_lo = (float)(tx * 16) + 0.5f, y_lo = (float)(ty * 16) + 0.5f;
  const uint2 rg = P.ranges[tile];
  const size_t plane = (size_t)P.W * P.H;
  const f2 minus1 = f2_dup(-1.f), one = f2_dup(1.f);

  f2 T[Q], SA[Q], g0[Q], g1[Q], g2[Q];
  uint32_t last[2 * Q];
  uint32_t total = 0;  // list entries any pixel of the tile used
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    float t[2], a[2][3];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int py = py0 + 4 * q + 2 * h;
      t[h] = 1.f; a[h][0] = a[h][1] = a[h][2] = 0.f; last[2 * q + h] = 0;
      if (px < P.W && py < P.H) {
        const size_t pix = (size_t)py * P.W + px;
        t[h] = P.final_T[pix];
        last[2 * q + h] = P.n_contrib[pix];
        a[h][0] = P.dL[pix]; a[h][1] = P.dL[plane + pix]; a[h][2] = P.dL[2 * plane + pix];
      }
      total = max(total, last[2 * q + h]);
    }
    T[q] = f2_make(t[0], t[1]);
    g0[q] = f2_make(a[0][0], a[1][0]); g1[q] = f2_make(a[0][1], a[1][1]); g2[q] = f2_make(a[0][2], a[1][2]);
    SA[q] = f2_make(P.bg0 * a[0][0] + P.bg1 * a[0][1] + P.bg2 * a[0][2], P.bg0 * a[1][0] + P.bg1 * a[1][1] + P.bg2 * a[1][2]);
  }
  total = __reduce_max_sync(0xffffffffu, total);
  if (total > BLEND_HEAD) {
    total = BLEND_HEAD;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      // no record: no pixel of the strip was live there (or see bwd_strip)
      const uint32_t next = P.strip_first[(uint32_t)tile * BLEND_STRIPS + q];
      if (next == 0 || next > P.seg_cap) continue;
      float t[2], a[2], ga[2], gb[2], gc[2];
      f2_split(g0[q], ga[0], ga[1]); f2_split(g1[q], gb[0], gb[1]); f2_split(g2[q], gc[0], gc[1]);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        bwd_from_record(P.ckpt + bwd_record_index(next - 1, (int)(lane & 15), 2 * h + (int)(lane >> 4)), ga[h], gb[h], gc[h], t[h], a[h]);
      T[q] = f2_make(t[0], t[1]);
      SA[q] = f2_make(a[0], a[1]);
    }
  }
  bool wild = false;  // (see bwd_strip)
#pragma unroll
  for (int q = 0; q < Q; ++q)
    wild = wild || !(blend_tame(g0[q].x, g1[q].x, g2[q].x) && blend_tame(g0[q].y, g1[q].y, g2[q].y) &&
                     fmaxf(fabsf(SA[q].x), fabsf(SA[q].y)) < BLEND_TAME_PRODUCT && SA[q].x == SA[q].x && SA[q].y == SA[q].y);
  wild = __any_sync(0xffffffffu, wild);
  total = min(total, rg.y - rg.x);
  int pending = 0;
  // walk the entries back to front, 32 at a time
  const int nb = (int)((total + 31) / 32);
  for (int bi = nb - 1; bi >= 0; --bi) {
    const uint32_t b = (uint32_t)bi * 32;
    uint32_t strips = 0, rid = 0;
    BlendFetch f = {};
    float4 conic;
    BlendShape shape = {};
    if (b + lane < total) {
      rid = min(P.vals[rg.x + b + lane], P.row_cap - 1);
      f = blend_fetch(P.xy, P.conic_o, P.rgb, rid);
      conic = blend_stage_conic(f.co);
      shape = blend_shape(f.co.x, f.co.y, f.co.z);
      strips = blend_reached_strips(f.c.x, f.c.y, f.co.x, f.co.y, f.co.z, shape, conic.w, l2amin, x_lo, y_lo);
    }
    const uint32_t m = __ballot_sync(0xffffffffu, strips != 0);
    const int cnt = __popc(m);
    const bool tame = blend_tame(f.r, f.g, f.b) && blend_tame(f.co.x, f.co.y, f.co.z);
    uint32_t odd = 0;  // staged rows whose conic is not proper
    if (__any_sync(0xffffffffu, strips && !(tame && shape.proper))) {
      wild |= __any_sync(0xffffffffu, strips && !tame);
      odd = __reduce_or_sync(0xffffffffu, strips && !shape.proper ? 1u << __popc(m & ((1u << lane) - 1u)) : 0u);
    }
    __syncwarp();
    if (strips) {
      const int pos = __popc(m & ((1u << lane) - 1u));
      s.row[pos].a = make_float4(f.r, f.r, f.g, f.g);
      s.row[pos].b = make_float4(f.b, __uint_as_float((b + lane + 1) << 4 | strips), f.c.x, f.c.y);
      s.row[pos].c = conic;
      s.aux[pos] = make_float2(__uint_as_float(rid), (bwd_plain(conic.w, shape, l2amax) ? 1.f : -1.f) / f.co.w);
    }
    __syncwarp();
    const uint32_t plain = __ballot_sync(0xffffffffu, (int)lane < cnt && s.aux[lane].y > 0.f);
    // which of the staged rows reach which strip, in registers every lane shares
    uint32_t reach[Q];
    {
      const uint32_t tag = (int)lane < cnt ? __float_as_uint(s.row[lane].b.y) : 0u;
#pragma unroll
      for (int q = 0; q < Q; ++q) reach[q] = __ballot_sync(0xffffffffu, tag >> q & 1u);
    }
    auto rows = [&](auto where) {
      constexpr bool WILD = decltype(where)::value;
      for (int j = cnt - 1; j >= 0; --j) {
        const float4 ra = s.row[j].a, rb = s.row[j].b, rc = s.row[j].c;
        const float dx = rb.z - fx;
        float h0, h1, h2;
        blend_x_terms(rc, dx, h0, h1, h2);
        const f2 H0 = f2_dup(h0), H1 = f2_dup(h1), H2 = f2_dup(h2);
        const f2 red = f2_make(ra.x, ra.y), green = f2_make(ra.z, ra.w), blue = f2_dup(rb.x);
        const uint32_t ord = __float_as_uint(rb.y) >> 4;
        const bool is_plain = plain >> j & 1u;
        const float top = blend_top(rc.w, odd >> j & 1u);
        f2 ar, ag, ab, gps, m1, m2;
        bool some = false;
        // kind: the row is plain.  first: nothing has been added up yet.  test: the exponent is tested
        auto strip = [&](int q, auto kind, auto first, auto test) {
          constexpr bool PLAIN = decltype(kind)::value, FIRST = decltype(first)::value, TEST = decltype(test)::value;
          const float y = (float)(py0 + 4 * q) + 0.5f;
          const f2 dy = f2_make(rb.w - y, rb.w - (y + 2.f));
          float p0, p1;
          f2_split(f2_fma(dy, f2_fma(H2, dy, H1), H0), p0, p1);
          bool k0 = ord <= last[2 * q] && p0 >= l2amin, k1 = ord <= last[2 * q + 1] && p1 >= l2amin;
          if (TEST) { k0 = k0 && p0 <= top; k1 = k1 && p1 <= top; }
          const float o0 = k0 ? blend_ex2(p0) : 0.f, o1 = k1 ? blend_ex2(p1) : 0.f;  // opacity * exp(power)
          if (TRACK || WILD) some = some || k0 || k1;
          const f2 og = f2_make(o0, o1), al = PLAIN ? og : f2_make(fminf(P.alpha_max, o0), fminf(P.alpha_max, o1));
          float i0, i1;
          f2_split(f2_fma(al, minus1, one), i0, i1);
          const f2 Tb = f2_mul(T[q], f2_make(blend_rcp(i0), blend_rcp(i1)));  // transmittance in front of the row
          const f2 w = f2_mul(al, Tb);
          auto at = [&](f2 x) { return WILD ? bwd_where(og, x) : x; };
          auto add = [&](f2 x, f2 y, f2& sum) { sum = FIRST ? f2_mul(x, y) : f2_fma(x, y, sum); };
          add(w, at(g0[q]), ar); add(w, at(g1[q]), ag); add(w, at(g2[q]), ab);
          const f2 cg = f2_fma(blue, g2[q], f2_fma(green, g1[q], f2_mul(red, g0[q])));
          const f2 t = at(f2_fma(SA[q], minus1, cg));
          SA[q] = f2_fma(al, t, SA[q]);
          T[q] = Tb;
          float w0, w1;
          f2_split(w, w0, w1);
          const f2 gp = f2_mul(PLAIN ? w : f2_make(o0 <= P.alpha_max ? w0 : 0.f, o1 <= P.alpha_max ? w1 : 0.f), t);
          const f2 gy = f2_mul(gp, dy);
          gps = FIRST ? gp : f2_add(gps, gp);
          m1 = FIRST ? gy : f2_add(m1, gy);
          add(gy, dy, m2);
        };
        constexpr std::true_type yes{};
        constexpr std::false_type no{};
        const bool is_odd = odd >> j & 1u;
        if (!WILD && !is_odd && (reach[0] & reach[1] & reach[2] & reach[3]) >> j & 1u) {  // (uniform) straight through
          if (is_plain) {  // (rows that may be clamped strip by strip instead: opaque splats, 1237 x 823, 89 us instead of 82)
            strip(0, yes, yes, no);
#pragma unroll
            for (int q = 1; q < Q; ++q) strip(q, yes, no, no);
          } else {
            strip(0, no, yes, no);
#pragma unroll
            for (int q = 1; q < Q; ++q) strip(q, no, no, no);
          }
        } else {
          ar = ag = ab = gps = m1 = m2 = f2_dup(0.f);
          if (!WILD && is_plain) {  // two strips in one stretch where the row reaches both: their chains overlap
#pragma unroll
            for (int q = 0; q < Q; q += 2) {
              if ((reach[q] & reach[q + 1]) >> j & 1u) {
                strip(q, yes, no, no);
                strip(q + 1, yes, no, no);
              } else if (reach[q] >> j & 1u) {
                strip(q, yes, no, no);
              } else if (reach[q + 1] >> j & 1u) {
                strip(q + 1, yes, no, no);
              }
            }
          } else {
#pragma unroll
            for (int q = 0; q < Q; ++q)
              if (reach[q] >> j & 1u) strip(q, no, no, yes);
          }
        }
        if ((TRACK || WILD) && !__any_sync(0xffffffffu, some)) continue;  // the row blends nowhere in the tile
        const float gpsum = f2_sum(gps), m1y = f2_sum(m1), gd = dx * gpsum;
        bwd_pend<TRACK>(P, s, pending, j, rc, gd, m1y, dx * gd, dx * m1y, f2_sum(m2), gpsum, f2_sum(ar), f2_sum(ag), f2_sum(ab), lane);
      }
    };
    if (__builtin_expect(!wild, 1)) rows(std::false_type{});
    else rows(std::true_type{});
  }
  if (pending) bwd_flush(s, pending, P.g2d, lane);
}

// TILES: first segments are taken by whole tiles, otherwise by strips (see blend.cuh).
constexpr int BWD_BLOCKS = 4;  // resident blocks per SM: 128 registers keep four straight-line strips in flight without spills
template <bool TILES, bool TRACK>
__global__ void __launch_bounds__(BLEND_THREADS, BWD_BLOCKS)
render_bwd_blend_kernel(BwdArgs P) {
  odin_after_predecessor();  // launched behind zero_rows_kernel
  __shared__ __align__(16) BwdWarp s_warp[BLEND_WARPS];
  const unsigned lane = threadIdx.x & 31;
  BwdWarp& s = s_warp[threadIdx.x >> 5];
  const uint32_t n_seg = min(*P.seg_count, P.seg_cap);
  const float l2amin = log2f(P.alpha_min), l2amax = log2f(P.alpha_max);
  const uint32_t n_strips = (uint32_t)P.n_tiles * BLEND_STRIPS, n_items = TILES ? (uint32_t)P.n_tiles : n_strips;
  // warps never synchronise with each other; each keeps taking work items from a ticket counter (see the forward
  // kernel).  The recorded segments come first.  A workspace that is not the forward call's own must not lead anywhere:
  // records, queue entries and links are checked before use.
  while (true) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(P.ticket, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item < n_seg) {
      const uint2 st = P.seg_strip[item];
      uint32_t next = P.seg_link[item].x;
      if (st.x >= n_strips || st.y >= (1u << 23)) continue;
      if (next > P.seg_cap) next = 0;
      bwd_strip<TRACK>(P, s, st.x, st.y, next, l2amin, l2amax, lane);
    } else {
      uint32_t pos = item - n_seg;
      if (pos >= n_items) return;
      // the items in the order the forward pass filed them: classes of rows evaluated, most first (the class counts
      // add up to the number of items; whatever else the words hold, pos stays below it and the item is clamped)
      uint32_t cls = 0;
      while (cls + 1 < (uint32_t)BLEND_BWD_CLASSES && pos >= P.bwd_count[cls]) { pos -= P.bwd_count[cls]; ++cls; }
      const uint32_t it = min(P.bwd_queue[cls * n_items + min(pos, n_items - 1)], n_items - 1);
      if (TILES) {
        bwd_tile<TRACK>(P, s, (int)it, l2amin, l2amax, lane);
      } else {
        uint32_t next = P.strip_first[it];
        if (next > P.seg_cap) next = 0;
        bwd_strip<TRACK>(P, s, it, 0u, next, l2amin, l2amax, lane);
      }
    }
  }
}

// ----------------------------------------------------------------------------------------------------------------
// A warp looks at 32 rows at a time and lists those with a gradient; where 32 have come together (or its rows have come to an
// end) it takes them through the chain rule, a lane each.  The SH rows of the listed primitives are copied to shared memory, lanes side
// by side along a row, while the geometry is worked out, and the gradient rows go back the same way.  What bounds it: DRAM where most
// rows blend (431 k rows of an aerial city, 221 MB: 34 us at the copy bandwidth), the chain of dependent loads where few do.
// Measured against a thread per row, whose lanes each went along a line of their own, all 32 as soon as one had a gradient: the
// aerial city 63 -> 48 us, 328 k rows of which 8 k blend 22 -> 17; one group of rows at a time instead of BP_AHEAD: 819 k rows 21 -> 23.
constexpr int BP_THREADS = 128, BP_WARPS = BP_THREADS / 32;
constexpr int BP_BLOCKS = 5;  // resident blocks per SM, up to 96 registers (six spill, and are no faster)
constexpr int BP_AHEAD = 4;   // groups of 32 rows a warp looks at together
constexpr uint32_t BP_LIST = 256;
static_assert(31 + 32 * BP_AHEAD <= BP_LIST, "listed rows of a warp");
template <int DEG>
struct ProjectRows {
  static constexpr int FLOATS = 3 * (DEG + 1) * (DEG + 1);
  static constexpr int VEC = FLOATS % 4 == 0 ? 4 : 1;  // floats of a piece
  static constexpr int PITCH = DEG == 3 ? 52 : DEG == 0 ? 1 : FLOATS;  // of 48 floats a quarter warp's pieces would meet in two banks
  static constexpr int PIECES = FLOATS / VEC;
  float sh[BP_WARPS][32 * PITCH];
  uint2 list[BP_WARPS][BP_LIST];  // row, primitive
  // all pieces of the 32 rows, lanes side by side along a row: three pieces per lane are 96 / PIECES rows, or a row at a time
  template <class F>
  static __device__ __forceinline__ void for_pieces(unsigned lane, F&& at) {
    if (VEC == 4) {
#pragma unroll
      for (int phase = 0; phase < 3; ++phase) {
        const int k = phase * 32 + (int)lane;
#pragma unroll
        for (int i = 0; i < PIECES / 3; ++i) at(k / PIECES + i * (96 / PIECES), k % PIECES);
      }
    } else {
#pragma unroll 8
      for (int row = 0; row < 32; ++row) at(row, (int)lane);
    }
  }
  // Gradient rows of zeros: those of [first, first + 32) whose bit of `zeros` is set.  The 32 rows lie behind one another in every
  // array, so the lanes go through them side by side, whichever row a piece belongs to.  Bound by the bytes.  What writing 320 k
  // such rows adds to the kernel, a lane per row and word by word / now, us: degree 3 101 / 18, degree 2 51 / 12, degree 1 20 / 7.
  static __device__ __forceinline__ void write_zeros(uint32_t first, uint32_t zeros, unsigned lane, float* __restrict__ g_means,
                                                     float* __restrict__ g_ls, float4* __restrict__ g_quats,
                                                     float* __restrict__ g_opac, float* __restrict__ g_sh) {
    if (zeros == 0) return;  // (uniform)
    asm volatile("" : "+r"(lane));  // (what follows from the lane is worked out here and not kept all along: no spills)
    if (zeros >> lane & 1u) {
      g_quats[first + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
      g_opac[first + lane] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const uint32_t w = 32 * i + lane;
      if (zeros >> (w / 3) & 1u) {
        g_means[3 * (size_t)first + w] = 0.f;
        g_ls[3 * (size_t)first + w] = 0.f;
      }
    }
    float* const out = g_sh + (size_t)first * FLOATS;
#pragma unroll
    for (int i = 0; i < PIECES; ++i) {
      const uint32_t k = 32 * i + lane;
      if (zeros >> (k / PIECES) & 1u) {
        if (VEC == 4) reinterpret_cast<float4*>(out)[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        else out[k] = 0.f;
      }
    }
  }
};

template <int DEG>
__global__ void __launch_bounds__(BP_THREADS, BP_BLOCKS)
render_bwd_project_kernel(const float* __restrict__ means, const float* __restrict__ log_scales,
                          const float4* __restrict__ quats, const float* __restrict__ opacity_logit,
                          const float* __restrict__ sh, CamParams cam, float dilation, const uint32_t* __restrict__ prim_id,
                          const uint8_t* __restrict__ clamp_flags, const uint32_t* __restrict__ num_rows, uint32_t capacity,
                          const float* __restrict__ g2d, float* __restrict__ g_means, float* __restrict__ g_ls,
                          float4* __restrict__ g_quats, float* __restrict__ g_opac, float* __restrict__ g_sh,
                          uint8_t* __restrict__ row_zero, uint32_t n) {
  odin_after_predecessor();
  constexpr int K = (DEG + 1) * (DEG + 1);
  typedef ProjectRows<DEG> Rows;
  __shared__ __align__(16) Rows s;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* const s_sh = s.sh[warp];
  uint2* const list = s.list[warp];
  const uint32_t V = min(*num_rows, capacity);
  const uint32_t stride = gridDim.x * BP_THREADS;
  uint32_t next = (blockIdx.x * BP_WARPS + warp) * 32, head = 0, listed = 0;
  while (true) {
    while (listed < 32 && next < V) {
      // the nine words of BP_AHEAD groups are on their way together
      float g[BP_AHEAD][9];
      uint32_t prim[BP_AHEAD], zeros = 0;  // lane k: rows of group k that are zero
#pragma unroll
      for (int k = 0; k < BP_AHEAD; ++k) {
        const uint32_t r = next + k * stride + lane;
        prim[k] = 0;
#pragma unroll
        for (int i = 0; i < 9; ++i) g[k][i] = 0.f;
        if (r < V) {
          prim[k] = min(prim_id[r], n - 1);
#pragma unroll
          for (int i = 0; i < 9; ++i) g[k][i] = g2d[(size_t)r * 9 + i];
        }
      }
#pragma unroll
      for (int k = 0; k < BP_AHEAD; ++k) {
        const uint32_t r = next + k * stride + lane;
        // The chain rule is linear in these nine words.  Most touched rows never blend into a pixel (they are occluded)
        // and arrive with all nine at zero: their gradient row is zero and needs neither the scene nor any arithmetic.
        bool some = false;
#pragma unroll
        for (int i = 0; i < 9; ++i) some = some || g[k][i] != 0.f;
        // the caller takes a flag instead of a row of zeros (the optimizer then reads no gradient for it), or the zeros below
        if (row_zero && r < V) row_zero[r] = some ? 0 : 1;
        const uint32_t none = __ballot_sync(0xffffffffu, r < V && !some);
        if (lane == (unsigned)k) zeros = none;
        const uint32_t m = __ballot_sync(0xffffffffu, some);
        if (some) list[(head + listed + __popc(m & ((1u << lane) - 1u))) % BP_LIST] = make_uint2(r, prim[k]);
        listed += __popc(m);
      }
      if (!row_zero) {
#pragma unroll 1
        for (int k = 0; k < BP_AHEAD; ++k)
          Rows::write_zeros(next + k * stride, __shfl_sync(0xffffffffu, zeros, k), lane, g_means, g_ls, g_quats, g_opac, g_sh);
      }
      next += BP_AHEAD * stride;
    }
    if (listed == 0) return;
    __syncwarp();
    const uint32_t cnt = min(listed, 32u);
    const bool on = lane < cnt;  // (the other lanes work on the last row as well and write nothing)
    const uint2 row_prim = list[(head + min(lane, cnt - 1)) % BP_LIST];
    const uint32_t r = row_prim.x;
    const size_t p = row_prim.y;
    const float* gg = g2d + (size_t)r * 9;
    const float gu = gg[0], gv = gg[1], gA = gg[2], gB = gg[3], gC = gg[4], go = gg[5];
    const float grgb[3] = {gg[6], gg[7], gg[8]};
    const float mx = means[3 * p], my = means[3 * p + 1], mz = means[3 * p + 2];
    const float ls[3] = {log_scales[3 * p], log_scales[3 * p + 1], log_scales[3 * p + 2]};
    const float4 quat = quats[p];
    const float logit = opacity_logit[p];
    const uint8_t flags = clamp_flags[r];
    if (DEG > 0) {
      Rows::for_pieces(lane, [&](int row, int piece) {
        const uint32_t prim = __shfl_sync(0xffffffffu, (uint32_t)p, row);
        if (row < (int)cnt && piece < Rows::PIECES)
          odin_copy_async<4 * Rows::VEC>(s_sh + row * Rows::PITCH + piece * Rows::VEC, sh + (size_t)prim * (3 * K) + piece * Rows::VEC);
      });
    }
    SplatGeom g;
    odin_camera_space(cam, mx, my, mz, g.t);
    odin_splat_geometry(cam, dilation, ls, quat, g);
    // conic -> 2D covariance
    const float a = g.a, b = g.b, c = g.c, D = g.det * g.det;
    const float ga = (-c * c * gA + b * c * gB - b * b * gC) / D;
    const float gb = (2.f * b * c * gA - (a * c + b * b) * gB + 2.f * a * b * gC) / D;
    const float gc = (-b * b * gA + a * b * gB - a * a * gC) / D;
    const float Gs[4] = {ga, 0.5f * gb, 0.5f * gb, gc};
    float GT[6];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) GT[3 * i + j] = Gs[2 * i] * g.Tm[j] + Gs[2 * i + 1] * g.Tm[3 + j];
    const float S[9] = {g.Sig[0], g.Sig[1], g.Sig[2], g.Sig[1], g.Sig[3], g.Sig[4], g.Sig[2], g.Sig[4], g.Sig[5]};
    float gSig[9], gTm[6];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) gSig[3 * i + j] = g.Tm[i] * GT[j] + g.Tm[3 + i] * GT[3 + j];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) gTm[3 * i + j] = 2.f * (GT[3 * i] * S[j] + GT[3 * i + 1] * S[3 + j] + GT[3 * i + 2] * S[6 + j]);
    // dL/dJ = dL/dTm R_c^T; only J00, J02, J11, J12 depend on t
    const float gJ00 = gTm[0] * cam.R[0] + gTm[1] * cam.R[1] + gTm[2] * cam.R[2];
    const float gJ02 = gTm[0] * cam.R[6] + gTm[1] * cam.R[7] + gTm[2] * cam.R[8];
    const float gJ11 = gTm[3] * cam.R[3] + gTm[4] * cam.R[4] + gTm[5] * cam.R[5];
    const float gJ12 = gTm[3] * cam.R[6] + gTm[4] * cam.R[7] + gTm[5] * cam.R[8];
    const float tx = g.t[0], ty = g.t[1], tz = g.t[2];
    const float iz = 1.f / tz, iz2 = iz * iz, iz3 = iz2 * iz;
    float gt0 = 0.f, gt1 = 0.f, gt2 = -(gJ00 * cam.fx + gJ11 * cam.fy) * iz2;
    if (g.clampx) gt2 += gJ02 * cam.fx * g.Lx * iz2;
    else { gt0 += -gJ02 * cam.fx * iz2; gt2 += 2.f * gJ02 * cam.fx * tx * iz3; }
    if (g.clampy) gt2 += gJ12 * cam.fy * g.Ly * iz2;
    else { gt1 += -gJ12 * cam.fy * iz2; gt2 += 2.f * gJ12 * cam.fy * ty * iz3; }
    gt0 += gu * cam.fx * iz; gt2 += -gu * cam.fx * tx * iz2;
    gt1 += gv * cam.fy * iz; gt2 += -gv * cam.fy * ty * iz2;
    float gmu[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) gmu[j] = cam.R[j] * gt0 + cam.R[3 + j] * gt1 + cam.R[6 + j] * gt2;
    // Sigma = M M^T
    float gM[9], gR[9], gls[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        gM[3 * i + j] = 2.f * (gSig[3 * i] * g.M[j] + gSig[3 * i + 1] * g.M[3 + j] + gSig[3 * i + 2] * g.M[6 + j]);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      float gs = 0.f;
#pragma unroll
      for (int i = 0; i < 3; ++i) { gs += g.Rm[3 * i + j] * gM[3 * i + j]; gR[3 * i + j] = gM[3 * i + j] * g.s[j]; }
      gls[j] = g.s[j] * gs;
    }
    const float w = g.qn[0], x = g.qn[1], y = g.qn[2], z = g.qn[3];
    float gq[4];
    gq[0] = 2.f * (-z * gR[1] + y * gR[2] + z * gR[3] - x * gR[5] - y * gR[6] + x * gR[7]);
    gq[1] = 2.f * (y * gR[1] + z * gR[2] + y * gR[3] - 2.f * x * gR[4] - w * gR[5] + z * gR[6] + w * gR[7] - 2.f * x * gR[8]);
    gq[2] = 2.f * (-2.f * y * gR[0] + x * gR[1] + w * gR[2] + x * gR[3] + z * gR[5] - w * gR[6] + z * gR[7] - 2.f * y * gR[8]);
    gq[3] = 2.f * (-2.f * z * gR[0] - w * gR[1] + x * gR[2] + w * gR[3] - 2.f * z * gR[4] + y * gR[5] + x * gR[6] + y * gR[7]);
    const float qd = w * gq[0] + x * gq[1] + y * gq[2] + z * gq[3];
    const float iq = 1.f / g.qlen;
    const float o = 1.f / (1.f + expf(-logit));
    if (on) {
      g_ls[3 * (size_t)r] = gls[0]; g_ls[3 * (size_t)r + 1] = gls[1]; g_ls[3 * (size_t)r + 2] = gls[2];
      g_quats[r] = make_float4((gq[0] - w * qd) * iq, (gq[1] - x * qd) * iq, (gq[2] - y * qd) * iq, (gq[3] - z * qd) * iq);
      g_opac[r] = o * (1.f - o) * go;
    }
    // colour
    float dvx = mx - cam.pos[0], dvy = my - cam.pos[1], dvz = mz - cam.pos[2];
    const float len = sqrtf(dvx * dvx + dvy * dvy + dvz * dvz);
    const float d0 = dvx / len, d1 = dvy / len, d2 = dvz / len;
    float Y[16], dY[16][3];
    odin_sh_basis<DEG>(d0, d1, d2, Y);
    odin_sh_basis_grad<DEG>(d0, d1, d2, dY);
    float gch[3];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) gch[ch] = (flags & (1u << ch)) ? 0.f : grgb[ch];
    float gd[3] = {0.f, 0.f, 0.f};
    if (DEG > 0) {
      odin_copies_landed();
      __syncwarp();  // all lanes' copies
      float* const mine = s_sh + lane * Rows::PITCH;
#pragma unroll
      for (int i = 0; i < Rows::PIECES; ++i) {  // the gradient takes the place of the coefficients
        float e[Rows::VEC];
        if (Rows::VEC == 4) *reinterpret_cast<float4*>(e) = reinterpret_cast<const float4*>(mine)[i];
        else e[0] = mine[i];
#pragma unroll
        for (int j = 0; j < Rows::VEC; ++j) {
          const int w = Rows::VEC * i + j, k = w / 3, ch = w % 3;
          if (k > 0) {
            const float wgt = e[j] * gch[ch];
            gd[0] += dY[k][0] * wgt; gd[1] += dY[k][1] * wgt; gd[2] += dY[k][2] * wgt;
          }
          e[j] = Y[k] * gch[ch];
        }
        if (Rows::VEC == 4) reinterpret_cast<float4*>(mine)[i] = *reinterpret_cast<const float4*>(e);
        else mine[i] = e[0];
      }
      __syncwarp();
      Rows::for_pieces(lane, [&](int row, int piece) {
        const uint32_t to_row = __shfl_sync(0xffffffffu, r, row);
        if (row < (int)cnt && piece < Rows::PIECES) {
          const float* from = s_sh + row * Rows::PITCH + piece * Rows::VEC;
          float* to = g_sh + (size_t)to_row * (3 * K) + piece * Rows::VEC;
          if (Rows::VEC == 4) *reinterpret_cast<float4*>(to) = *reinterpret_cast<const float4*>(from);
          else *to = *from;
        }
      });
    } else if (on) {
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) g_sh[3 * (size_t)r + ch] = Y[0] * gch[ch];
    }
    const float dd = d0 * gd[0] + d1 * gd[1] + d2 * gd[2];
    gmu[0] += (gd[0] - d0 * dd) / len; gmu[1] += (gd[1] - d1 * dd) / len; gmu[2] += (gd[2] - d2 * dd) / len;
    if (on) {
      g_means[3 * (size_t)r] = gmu[0]; g_means[3 * (size_t)r + 1] = gmu[1]; g_means[3 * (size_t)r + 2] = gmu[2];
    }
    head += cnt;
    listed -= cnt;
    __syncwarp();  // shared memory and list are free again
  }
}

}  // namespace

extern "C" int odin_render_bwd(odin_ctx* ctx, const odin_scene* scene, const odin_camera* cam, const odin_projected* proj,
                               const uint32_t* d_vals, const uint32_t* d_tile_ranges, const float* d_final_T,
                               const uint32_t* d_n_contrib, const float* d_dL_drgb, float* d_grad2d, odin_scene* grad_rows,
                               uint8_t* d_row_active, uint8_t* d_row_zero, void* ws, size_t ws_bytes, void* stream) {
  if (!ctx || !proj || !grad_rows) return ODIN_ERR_NULL;
  int rc = odin_check_scene(scene);
  if (rc != ODIN_OK) return rc;
  rc = odin_check_camera(cam);
  if (rc != ODIN_OK) return rc;
  rc = odin_check_scene(grad_rows);
  if (rc != ODIN_OK) return rc;
  if (grad_rows->sh_degree != scene->sh_degree) return ODIN_ERR_INVALID_ARG;
  if (proj->capacity == 0 || scene->n == 0) return ODIN_OK;
  if (grad_rows->n < proj->capacity) return ODIN_ERR_INVALID_ARG;
  if (!d_vals || !d_tile_ranges || !d_final_T || !d_n_contrib || !d_dL_drgb || !d_grad2d || !proj->xy ||
      !proj->conic_opacity || !proj->rgb || !proj->prim_id || !proj->clamp_flags || !proj->num_rows)
    return ODIN_ERR_NULL;
  cudaStream_t st = (cudaStream_t)stream;
  const int TX = (cam->width + 15) / 16, TY = (cam->height + 15) / 16;
  if (!ws || !odin_aligned(ws, 256) || ws_bytes < blend_ws_bytes(cam->width, cam->height)) return ODIN_ERR_WORKSPACE;
  const int n_tiles = TX * TY;
  const BlendWs L = blend_ws_layout(n_tiles, blend_ws_records(n_tiles, ws_bytes));
  char* base = reinterpret_cast<char*>(ws);
  uint32_t* header = reinterpret_cast<uint32_t*>(base);
  uint32_t* ticket = header + 1;
  const uint32_t zgrid = (uint32_t)ctx->sm_count * 8;
  // (inside a view step the projection has zeroed the rows, and the ticket with the rest of the header is still at zero)
  if (!ctx->view_grad2d || ctx->view_grad2d != d_grad2d || ctx->view_row_active != d_row_active) {
    OdinKernelScope ks(ctx, K_ZERO_ROWS, st);
    ODIN_CUDA(odin_launch(ctx, false, zero_rows_kernel, dim3(zgrid), dim3(256), 0, st, d_grad2d, d_row_active, proj->num_rows,
                          proj->capacity, ticket));
  }
  {
    OdinKernelScope ks(ctx, K_BWD_BLEND, st);
    BwdArgs P;
    P.xy = reinterpret_cast<const float2*>(proj->xy); P.conic_o = reinterpret_cast<const float4*>(proj->conic_opacity);
    P.rgb = proj->rgb; P.vals = d_vals; P.ranges = reinterpret_cast<const uint2*>(d_tile_ranges);
    P.W = cam->width; P.H = cam->height; P.TX = TX; P.n_tiles = n_tiles;
    P.bg0 = cam->bg[0]; P.bg1 = cam->bg[1]; P.bg2 = cam->bg[2];
    P.alpha_min = ctx->cfg.alpha_min; P.alpha_max = ctx->cfg.alpha_max;
    P.strip_first = reinterpret_cast<const uint32_t*>(base + L.strip_first); P.seg_count = header + 2;
    P.seg_strip = reinterpret_cast<const uint2*>(base + L.seg_strip);
    P.seg_link = reinterpret_cast<const uint2*>(base + L.seg_link);
    P.ckpt = reinterpret_cast<const BlendRecord*>(base + L.ckpt); P.seg_cap = L.segments;
    P.final_T = d_final_T; P.n_contrib = d_n_contrib; P.dL = d_dL_drgb; P.g2d = d_grad2d; P.ticket = ticket;
    P.row_active = d_row_active; P.row_cap = proj->capacity; P.bwd_count = header + 8;
    P.bwd_queue = reinterpret_cast<const uint32_t*>(base + L.bwd_queue);
    const int blocks = ctx->sm_count * BWD_BLOCKS;  // resident warps pull work
    const bool tiles = blend_tile_items(n_tiles);
#define LAUNCH_BLEND(TILES, TRACK) \
  ODIN_CUDA(odin_launch(ctx, true, render_bwd_blend_kernel<TILES, TRACK>, dim3(blocks), dim3(BLEND_THREADS), 0, st, P))
    if (d_row_active) { if (tiles) LAUNCH_BLEND(true, true); else LAUNCH_BLEND(false, true); }
    else { if (tiles) LAUNCH_BLEND(true, false); else LAUNCH_BLEND(false, false); }
#undef LAUNCH_BLEND
  }
  const CamParams cp = odin_cam_params(cam, ctx->cfg);
  const uint32_t blocks_cap = (proj->capacity + BP_THREADS - 1) / BP_THREADS, resident = (uint32_t)ctx->sm_count * BP_BLOCKS;
  const uint32_t pgrid = blocks_cap < resident ? blocks_cap : resident;
#define LAUNCH(D)                                                                                                       \
  ODIN_CUDA(odin_launch(ctx, true, render_bwd_project_kernel<D>, dim3(pgrid), dim3(BP_THREADS), 0, st,                         \
      scene->means, scene->log_scales, reinterpret_cast<const float4*>(scene->quats), scene->opacity_logit, scene->sh,  \
      cp, ctx->cfg.dilation, proj->prim_id, proj->clamp_flags, proj->num_rows, proj->capacity, d_grad2d,                \
      grad_rows->means, grad_rows->log_scales, reinterpret_cast<float4*>(grad_rows->quats), grad_rows->opacity_logit,    \
      grad_rows->sh, d_row_zero, scene->n))
  OdinKernelScope ks(ctx, K_BWD_PROJECT, st);
  switch (scene->sh_degree) {
    case 0: LAUNCH(0); break;
    case 1: LAUNCH(1); break;
    case 2: LAUNCH(2); break;
    default: LAUNCH(3); break;
  }
#undef LAUNCH
  return odin_launch_status();
}
