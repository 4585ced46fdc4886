// Optimizer update restricted to the touched rows: bandwidth-bound gather / scatter Adam.
// The gradient side is read fully coalesced (consecutive threads, consecutive floats of the compact rows); the
// parameter side touches, per row, one contiguous span per attribute array (192 B for degree-3 SH = six full sectors).
#include "common.cuh"

namespace {

// A row whose gradient and both moments are zero is left alone: m' = v' = 0 and theta' = theta - step * 0 / (0 + eps) =
// theta bit for bit (eps > 0), so neither the parameter is read nor anything written.  Most touched rows of a view are
// occluded (zero gradient), and until a primitive has been active in some view its moments are zero too: for those
// rows the update costs the two moment reads only.  (skip_idle is off when eps == 0, where 0 / 0 would be the result.)
struct AdamK {
  int skip_idle;
  float beta1, beta2, omb1, omb2, eps;
  float step_size[6];  // lr_g / (1 - beta1^t)
  float inv_bc2s;      // 1 / sqrt(1 - beta2^t)
};

// The square root and the division are the hardware approximations (relative error ~1e-7 each, far inside the bar
// on the updated parameter): the correctly rounded forms are ~20 instructions per scalar, which made these kernels
// issue-bound next to their memory traffic.
__device__ __forceinline__ float adam_sqrt(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void adam_one(float& th, float& m, float& v, float g, float step_size, const AdamK& k) {
  m = k.beta1 * m + k.omb1 * g;
  v = k.beta2 * v + k.omb2 * g * g;
  th = th - __fdividef(step_size * m, adam_sqrt(v) * k.inv_bc2s + k.eps);
}

// Flags of the primitives whose moments may be non-zero (live[p] == 0: every moment of p, in every attribute, is zero).
// With them a row that has no gradient and no history costs its index and two bytes instead of a read of both moments.
__device__ __forceinline__ bool adam_cold(const uint8_t* live, size_t prim, const AdamK& k) {
  return live && k.skip_idle && live[prim] == 0;
}
// Called by a thread that is about to write moments that may be non-zero.
__device__ __forceinline__ void adam_mark_live(uint8_t* live, size_t prim, bool cold, const AdamK& k) {
  if (live && (cold || !k.skip_idle)) live[prim] = 1;
}

// The kernel gives a warp 32 consecutive rows of the list at a time.  The warp first looks at the rows themselves
// (index, row flag, primitive flag: three coalesced or nearly coalesced loads), drops the rows with nothing to do - no
// gradient and no history, or an index out of range - and leaves the others, in order, in shared memory; the elements
// of the remaining rows are then spread over the lanes.  Where most rows of a view are occluded a warp so works on full
// loads of the few rows that matter instead of running the whole chain of dependent loads for one live lane in eight.
constexpr int ADAM_WARPS = 8;

// returns the number of rows kept; s_prim[i] = primitive, s_info[i] = place in the group | zero << 8 | cold << 9
__device__ __forceinline__ uint32_t adam_stage_rows(uint32_t grp, uint32_t V, const uint32_t* __restrict__ idx,
                                                    const uint8_t* __restrict__ row_zero, const uint8_t* live,
                                                    uint32_t n_prims, const AdamK& k, uint32_t* s_prim, uint32_t* s_info,
                                                    unsigned lane) {
  const uint32_t r = grp * 32 + lane;
  uint32_t prim = 0;
  bool zero = false, cold = false, act = false;
  if (r < V) {
    prim = idx[r];
    if (prim < n_prims) {  // (an index list that is not a view's own, e.g. after a timed-out scan: no write)
      zero = row_zero && row_zero[r];  // the gradient row was not written: it is zero
      // cold: the primitive's flag says that all of its moments are zero, so they are not read
      cold = adam_cold(live, prim, k);
      act = !(cold && zero);
    }
  }
  const uint32_t mask = __ballot_sync(0xffffffffu, act);
  __syncwarp();  // the previous group's entries have been read
  if (act) {
    const uint32_t pos = __popc(mask & ((1u << lane) - 1u));
    s_prim[pos] = prim;
    s_info[pos] = lane | (zero ? 256u : 0u) | (cold ? 512u : 0u);
  }
  __syncwarp();
  return (uint32_t)__popc(mask);
}

// One element of VEC words: the update, unless there is neither a gradient nor history.  The parameters are fetched together
// with the moments where the primitive flags are in use (a row that gets this far then nearly always has work).
template <int VEC>
struct AdamWords { float w[VEC]; };
template <int VEC>
__device__ __forceinline__ AdamWords<VEC> adam_load(const float* __restrict__ a, bool on) {
  AdamWords<VEC> r;
  if (VEC == 4) {
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (on) x = *reinterpret_cast<const float4*>(a);
    r.w[0] = x.x; r.w[VEC > 1 ? 1 : 0] = VEC > 1 ? x.y : x.x; r.w[VEC > 2 ? 2 : 0] = VEC > 2 ? x.z : x.x; r.w[VEC > 3 ? 3 : 0] = VEC > 3 ? x.w : x.x;
  } else {
    r.w[0] = on ? *a : 0.f;
  }
  return r;
}
template <int VEC>
__device__ __forceinline__ void adam_store(float* __restrict__ a, const AdamWords<VEC>& x) {
  if (VEC == 4) *reinterpret_cast<float4*>(a) = make_float4(x.w[0], x.w[VEC > 1 ? 1 : 0], x.w[VEC > 2 ? 2 : 0], x.w[VEC > 3 ? 3 : 0]);
  else *a = x.w[0];
}

struct AdamBlock {  // one attribute: parameters, moments, compact gradient rows
  float* p; float* m; float* v; const float* g;
};

// Elements of one attribute of WIDTH words in elements of VEC, the rows' elements spread over the lanes, UNROLL per lane: first
// all of them are fetched, later updated.  SH: words 0 .. 2 of a row take step size 4, the others 5; otherwise all take `group`.
template <int WIDTH, int VEC, int UNROLL, bool SH>
struct AdamBatch {
  static constexpr uint32_t EPR = WIDTH / VEC;  // elements per row
  AdamWords<VEC> gg[UNROLL], mm[UNROLL], vv[UNROLL], pp[UNROLL];

  __device__ __forceinline__ void load(const AdamBlock& B, uint32_t q0, uint32_t kept, uint32_t row0, const uint32_t* s_prim,
                                       const uint32_t* s_info, bool eager) {
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const uint32_t q = q0 + 32 * u, slot = q / EPR, j = q - slot * EPR;
      const bool in = q < kept * EPR;
      const uint32_t prim = in ? s_prim[slot] : 0u, info = in ? s_info[slot] : 0u;
      const size_t at = (size_t)prim * WIDTH + (size_t)j * VEC;
      gg[u] = adam_load<VEC>(B.g + (size_t)(row0 + (info & 255u)) * WIDTH + (size_t)j * VEC, in && !(info & 256u));
      mm[u] = adam_load<VEC>(B.m + at, in && !(info & 512u));
      vv[u] = adam_load<VEC>(B.v + at, in && !(info & 512u));
      pp[u] = adam_load<VEC>(B.p + at, in && eager);
    }
  }
  __device__ __forceinline__ void update(const AdamBlock& B, uint32_t q0, uint32_t kept, const uint32_t* s_prim, const uint32_t* s_info,
                                         const AdamK& k, int group, bool eager, uint8_t* live) {
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const uint32_t q = q0 + 32 * u, slot = q / EPR, j = q - slot * EPR;
      if (q >= kept * EPR) continue;
      const uint32_t prim = s_prim[slot];
      const bool cold = s_info[slot] & 512u;
      bool gzero = true, mzero = true;
#pragma unroll
      for (int i = 0; i < VEC; ++i) {
        gzero = gzero && gg[u].w[i] == 0.f;
        mzero = mzero && mm[u].w[i] == 0.f && vv[u].w[i] == 0.f;
      }
      if (gzero && (cold || (k.skip_idle && mzero))) continue;
      adam_mark_live(live, prim, cold, k);
      const size_t at = (size_t)prim * WIDTH + (size_t)j * VEC;
      if (!eager) pp[u] = adam_load<VEC>(B.p + at, true);
#pragma unroll
      for (int i = 0; i < VEC; ++i)
        adam_one(pp[u].w[i], mm[u].w[i], vv[u].w[i], gg[u].w[i], k.step_size[SH ? ((int)j * VEC + i < 3 ? 4 : 5) : group], k);
      adam_store<VEC>(B.p + at, pp[u]);
      adam_store<VEC>(B.m + at, mm[u]);
      adam_store<VEC>(B.v + at, vv[u]);
    }
  }
};

// All attributes in one kernel: a warp looks at its 32 rows once and then goes through them, the four small attributes together
// (all their words are on their way before the first is updated), then the colour coefficients; consecutive lanes on
// consecutive words.  What bounds it: scattered pieces of 4 to 192 bytes, i.e. DRAM accesses of 64 bytes and the latency of
// chains of dependent loads (list -> flags -> moments).  Degree 3, 104 k of 328 k touched rows of 1 M primitives with work:
// 83 us as two kernels that each walked the chain, four predicated lanes per row for the geometry; 68 attribute by attribute
// in one; 64 this way.  417 k rows of a 20 M aerial scene 177 -> 125 -> 122, 841 k rows of a street 272 -> 210 -> 204 (1.2 GB:
// 0.9 of the copy bandwidth).  All five attributes at once, or two blocks per SM: 67, 223 for the street.
template <int ROWF, int VEC>
__global__ void __launch_bounds__(ADAM_WARPS * 32, 3)
adam_kernel(AdamBlock means, AdamBlock scales, AdamBlock quats, AdamBlock opacity, AdamBlock sh, const uint32_t* __restrict__ idx,
            const uint32_t* __restrict__ count, uint32_t cap, AdamK k, const uint8_t* __restrict__ row_zero, uint32_t n_prims,
            uint8_t* live) {
  odin_after_predecessor();
  __shared__ uint32_t s_prim[ADAM_WARPS][32], s_info[ADAM_WARPS][32];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t V = min(*count, cap);
  const uint32_t groups = (V + 31) / 32;
  const bool eager = live != nullptr;
  for (uint32_t grp = blockIdx.x * ADAM_WARPS + warp; grp < groups; grp += gridDim.x * ADAM_WARPS) {
    const uint32_t kept = adam_stage_rows(grp, V, idx, row_zero, live, n_prims, k, s_prim[warp], s_info[warp], lane);
    if (kept == 0) continue;
    const uint32_t row0 = grp * 32;
    const uint32_t *sp = s_prim[warp], *si = s_info[warp];
    AdamBatch<4, 4, 1, false> q;
    AdamBatch<3, 1, 3, false> m, l;
    AdamBatch<1, 1, 1, false> o;
    q.load(quats, lane, kept, row0, sp, si, eager);
    m.load(means, lane, kept, row0, sp, si, eager);
    l.load(scales, lane, kept, row0, sp, si, eager);
    o.load(opacity, lane, kept, row0, sp, si, eager);
    AdamBatch<ROWF, VEC, 2, true> h;
    q.update(quats, lane, kept, sp, si, k, 2, eager, live);
    m.update(means, lane, kept, sp, si, k, 0, eager, live);
    l.update(scales, lane, kept, sp, si, k, 1, eager, live);
    o.update(opacity, lane, kept, sp, si, k, 3, eager, live);
    for (uint32_t q0 = lane; q0 < kept * (ROWF / VEC); q0 += 32 * 2) {
      h.load(sh, q0, kept, row0, sp, si, eager);
      h.update(sh, q0, kept, sp, si, k, 0, eager, live);
    }
  }
}

// Gradient rows of a task unit.  A warp takes 32 consecutive rows of the list.  Where that is the union of the two views'
// lists, which ascend like it, their members among these 32 primitives are among the 32 entries from the first one at or
// behind the first primitive on: one search per view and warp (32-way: three steps for a million rows), then every lane finds
// its primitive in the 32 entries by a binary search over the lanes.  (Other lists: warp_rows_of.)  The rows' words are then
// added flat, consecutive lanes on consecutive words.  (One warp per row, two searches each: 80 us for the 190 k rows of two
// views of 400 k primitives at degree 1; this way 22.)
struct RowsView {
  const float* means; const float* log_scales; const float* quats; const float* opacity_logit; const float* sh;
  const uint8_t* zero; const uint32_t* idx; const uint32_t* count; uint32_t cap;
};

__device__ __forceinline__ uint32_t warp_lower_bound(const uint32_t* __restrict__ idx, uint32_t n, uint32_t key, unsigned lane) {
  // first position of the ascending idx[0..n) whose entry is at least key (n if none); all lanes take part
  uint32_t lo = 0, hi = n;  // the answer lies in [lo, hi]
  while (hi - lo > 32) {
    const uint32_t step = (hi - lo + 31) / 32, probe = lo + lane * step;
    const bool below = probe < hi && idx[probe] < key;  // monotone: true for the first cnt lanes
    const uint32_t cnt = __popc(__ballot_sync(0xffffffffu, below));
    if (cnt == 0) return lo;                            // idx[lo] >= key (uniform over the warp)
    hi = min(hi, lo + cnt * step);
    lo += (cnt - 1) * step + 1;                         // idx[lo - 1] < key
  }
  return lo + __popc(__ballot_sync(0xffffffffu, lo + lane < hi && idx[lo + lane] < key));
}

// Row of the lane's primitive p in a view, -1 if the view does not list it or flagged it as zero instead of writing it.  A
// search settles every lane whose primitive lies in the span of the 32 entries it fetches; of a union's rows that is all of
// them (between the first and the last of 32 union rows a view lists 32 primitives at most).  A list that leaves members
// out, or that does not ascend, takes another search from the first lane that is left, which settles at least that lane.
__device__ __forceinline__ int warp_rows_of(const RowsView& a, uint32_t n, uint32_t p, bool valid, unsigned lane) {
  int r = -1;
  uint32_t open = __ballot_sync(0xffffffffu, valid);
  while (open) {
    const uint32_t first = __shfl_sync(0xffffffffu, p, __ffs(open) - 1);
    const uint32_t base = warp_lower_bound(a.idx, n, first, lane);
    const uint32_t e = base + lane < n ? a.idx[base + lane] : 0xffffffffu;
    uint32_t at = 0;  // entries below p among the first 31
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      const uint32_t x = __shfl_sync(0xffffffffu, e, at + s - 1);
      if (x < p) at += s;
    }
    const uint32_t x = __shfl_sync(0xffffffffu, e, at);
    const bool settled = p >= first && (x >= p || base + 32 >= n);  // neither in front of the entries nor behind them
    if ((open >> lane & 1u) && settled && x == p && base + at < n) r = (int)(base + at);
    open &= ~__ballot_sync(0xffffffffu, settled);
  }
  return r >= 0 && !(a.zero && a.zero[r]) ? r : -1;
}

constexpr int ACC_WARPS = 8;
__global__ void __launch_bounds__(ACC_WARPS * 32)
accumulate_rows_kernel(RowsView a, RowsView b, const uint32_t* __restrict__ idx_u, const uint32_t* __restrict__ count_u,
                       uint32_t cap_u, int sh_floats, float* __restrict__ o_means, float* __restrict__ o_ls,
                       float* __restrict__ o_q, float* __restrict__ o_op, float* __restrict__ o_sh) {
  __shared__ int2 s_rows[ACC_WARPS][32];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t U = min(*count_u, cap_u);
  const uint32_t na = min(*a.count, a.cap), nb = min(*b.count, b.cap);
  for (uint32_t r0 = (blockIdx.x * ACC_WARPS + warp) * 32; r0 < U; r0 += gridDim.x * ACC_WARPS * 32) {
    const bool valid = r0 + lane < U;
    const uint32_t p = idx_u[min(r0 + lane, U - 1)];
    const int ra = warp_rows_of(a, na, p, valid, lane), rb = warp_rows_of(b, nb, p, valid, lane);
    __syncwarp();
    s_rows[warp][lane] = make_int2(ra, rb);
    __syncwarp();
    const uint32_t rows = min(32u, U - r0);
    auto sum = [&](const float* __restrict__ xa, const float* __restrict__ xb, float* __restrict__ out, uint32_t width) {
      for (uint32_t e = lane; e < rows * width; e += 32) {
        const uint32_t row = e / width, i = e - row * width;
        const int2 r = s_rows[warp][row];
        float s = 0.f;
        if (r.x >= 0) s += xa[(size_t)r.x * width + i];
        if (r.y >= 0) s += xb[(size_t)r.y * width + i];
        out[(size_t)r0 * width + e] = s;
      }
    };
    sum(a.means, b.means, o_means, 3);
    sum(a.log_scales, b.log_scales, o_ls, 3);
    sum(a.quats, b.quats, o_q, 4);
    sum(a.opacity_logit, b.opacity_logit, o_op, 1);
    sum(a.sh, b.sh, o_sh, (uint32_t)sh_floats);
  }
}

// live[i / width] = 1 for every non-zero word a[i] (the flags are cleared first; one launch per attribute array)
__global__ void __launch_bounds__(256)
mark_nonzero_kernel(const float* __restrict__ a, size_t total, uint32_t width, uint8_t* __restrict__ live) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x)
    if (a[i] != 0.f) live[i / width] = 1;  // (a NaN counts as non-zero)
}

}  // namespace

extern "C" int odin_accumulate_rows(odin_ctx* ctx, const odin_scene* rows_a, const uint8_t* d_zero_a, const uint32_t* d_idx_a,
                                    const uint32_t* d_count_a, const odin_scene* rows_b, const uint8_t* d_zero_b,
                                    const uint32_t* d_idx_b, const uint32_t* d_count_b, const uint32_t* d_idx_u,
                                    const uint32_t* d_count_u, odin_scene* rows_u, void* stream) {
  if (!ctx || !d_count_a || !d_count_b || !d_count_u) return ODIN_ERR_NULL;
  int rc = odin_check_scene(rows_a);
  if (rc == ODIN_OK) rc = odin_check_scene(rows_b);
  if (rc == ODIN_OK) rc = odin_check_scene(rows_u);
  if (rc != ODIN_OK) return rc;
  if (rows_a->sh_degree != rows_u->sh_degree || rows_b->sh_degree != rows_u->sh_degree) return ODIN_ERR_INVALID_ARG;
  if (rows_u->n == 0) return ODIN_OK;
  if (!d_idx_u || (rows_a->n && !d_idx_a) || (rows_b->n && !d_idx_b)) return ODIN_ERR_NULL;
  const RowsView a = {rows_a->means, rows_a->log_scales, rows_a->quats, rows_a->opacity_logit, rows_a->sh, d_zero_a, d_idx_a,
                      d_count_a, rows_a->n};
  const RowsView b = {rows_b->means, rows_b->log_scales, rows_b->quats, rows_b->opacity_logit, rows_b->sh, d_zero_b, d_idx_b,
                      d_count_b, rows_b->n};
  const int K = (rows_u->sh_degree + 1) * (rows_u->sh_degree + 1);
  uint32_t grid = (rows_u->n + 32 * ACC_WARPS - 1) / (32 * ACC_WARPS);
  if (grid > (uint32_t)ctx->sm_count * 16) grid = (uint32_t)ctx->sm_count * 16;
  OdinKernelScope ks(ctx, K_ACCUMULATE, (cudaStream_t)stream);
  accumulate_rows_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(a, b, d_idx_u, d_count_u, rows_u->n, 3 * K, rows_u->means,
                                                                rows_u->log_scales, rows_u->quats, rows_u->opacity_logit,
                                                                rows_u->sh);
  return odin_launch_status();
}

extern "C" int odin_adam_live_refresh(odin_ctx* ctx, const odin_scene* m, const odin_scene* v, uint8_t* d_live,
                                     void* stream) {
  if (!ctx || !d_live) return ODIN_ERR_NULL;
  int rc = odin_check_scene(m);
  if (rc == ODIN_OK) rc = odin_check_scene(v);
  if (rc != ODIN_OK) return rc;
  if (m->n != v->n || m->sh_degree != v->sh_degree) return ODIN_ERR_INVALID_ARG;
  if (m->n == 0) return ODIN_OK;
  cudaStream_t st = (cudaStream_t)stream;
  odin_chain_break(ctx);
  ODIN_CUDA(cudaMemsetAsync(d_live, 0, m->n, st));
  const int K = (m->sh_degree + 1) * (m->sh_degree + 1);
  for (const odin_scene* s : {m, v}) {
    const float* arrays[5] = {s->means, s->log_scales, s->quats, s->opacity_logit, s->sh};
    const uint32_t widths[5] = {3, 3, 4, 1, (uint32_t)(3 * K)};
    for (int a = 0; a < 5; ++a) {
      const size_t total = (size_t)m->n * widths[a];
      size_t blocks = (total + 255) / 256;
      if (blocks > (size_t)ctx->sm_count * 16) blocks = (size_t)ctx->sm_count * 16;
      OdinKernelScope ks(ctx, K_ADAM_LIVE, st);
      mark_nonzero_kernel<<<(unsigned)blocks, 256, 0, st>>>(arrays[a], total, widths[a], d_live);
    }
  }
  return odin_launch_status();
}

extern "C" int odin_sparse_adam(odin_ctx* ctx, odin_scene* params, odin_scene* m, odin_scene* v,
                                const odin_scene* grad_rows, const uint8_t* d_row_zero, const uint32_t* d_idx,
                                const uint32_t* d_count, const float lr[6], float beta1, float beta2, float eps,
                                uint32_t step, void* stream) {
  return odin_sparse_adam_live(ctx, params, m, v, grad_rows, d_row_zero, d_idx, d_count, nullptr, lr, beta1, beta2, eps, step,
                               stream);
}

extern "C" int odin_sparse_adam_live(odin_ctx* ctx, odin_scene* params, odin_scene* m, odin_scene* v,
                                     const odin_scene* grad_rows, const uint8_t* d_row_zero, const uint32_t* d_idx,
                                     const uint32_t* d_count, uint8_t* d_live, const float lr[6], float beta1, float beta2,
                                     float eps, uint32_t step, void* stream) {
  if (!ctx || !lr || !d_count) return ODIN_ERR_NULL;
  int rc = odin_check_scene(params);
  if (rc == ODIN_OK) rc = odin_check_scene(m);
  if (rc == ODIN_OK) rc = odin_check_scene(v);
  if (rc == ODIN_OK) rc = odin_check_scene(grad_rows);
  if (rc != ODIN_OK) return rc;
  if (m->n != params->n || v->n != params->n || m->sh_degree != params->sh_degree || v->sh_degree != params->sh_degree ||
      grad_rows->sh_degree != params->sh_degree)
    return ODIN_ERR_INVALID_ARG;
  if (step == 0 || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) || !(eps >= 0.f))
    return ODIN_ERR_INVALID_ARG;
  if (params->n == 0 || grad_rows->n == 0) return ODIN_OK;
  if (!d_idx) return ODIN_ERR_NULL;
  AdamK k;
  k.beta1 = beta1; k.beta2 = beta2; k.omb1 = 1.f - beta1; k.omb2 = 1.f - beta2; k.eps = eps;
  k.skip_idle = eps > 0.f ? 1 : 0;
  const float bc1 = 1.f - (float)pow((double)beta1, (double)step);
  const float bc2s = (float)sqrt(1.0 - pow((double)beta2, (double)step));
  for (int i = 0; i < 6; ++i) k.step_size[i] = lr[i] / bc1;
  k.inv_bc2s = 1.f / bc2s;
  cudaStream_t st = (cudaStream_t)stream;
  const uint32_t cap = grad_rows->n;
  const int K = (params->sh_degree + 1) * (params->sh_degree + 1);
  // a warp per 32 rows of the list
  size_t blocks = ((size_t)cap + 32 * ADAM_WARPS - 1) / (32 * ADAM_WARPS);
  if (blocks > (size_t)ctx->sm_count * 16) blocks = (size_t)ctx->sm_count * 16;
  const AdamBlock means = {params->means, m->means, v->means, grad_rows->means};
  const AdamBlock scales = {params->log_scales, m->log_scales, v->log_scales, grad_rows->log_scales};
  const AdamBlock quats = {params->quats, m->quats, v->quats, grad_rows->quats};
  const AdamBlock opacity = {params->opacity_logit, m->opacity_logit, v->opacity_logit, grad_rows->opacity_logit};
  const AdamBlock sh = {params->sh, m->sh, v->sh, grad_rows->sh};
  OdinKernelScope ks(ctx, K_ADAM, st);
#define L2CH(ROWF, VEC)                                                                                               \
  ODIN_CUDA(odin_launch(ctx, false, adam_kernel<ROWF, VEC>, dim3((unsigned)blocks), dim3(ADAM_WARPS * 32), 0, st, means, scales, \
                        quats, opacity, sh, d_idx, d_count, cap, k, d_row_zero, params->n, d_live))
  switch (params->sh_degree) {
    case 0: L2CH(3, 1); break;
    case 1: L2CH(12, 4); break;
    case 2: L2CH(27, 1); break;
    default: L2CH(48, 4); break;
  }
#undef L2CH
  return odin_launch_status();
}
