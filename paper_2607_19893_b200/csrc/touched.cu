// Touched-set bitmask + ascending index list (single pass, decoupled look-back) and pairwise intersection counts.
#include <atomic>

#include "common.cuh"
#include "layout.cuh"
#include "pair_cost.h"

namespace {

constexpr int TS_THREADS = 256;
constexpr int TS_ITEMS = TOUCHED_TILE / TS_THREADS;  // 8 words of 32 primitives per warp

// A block takes `scan_rounds` x 2048 consecutive primitives by ticket; each of its eight warps owns a contiguous eighth
// of them.  Load q of lane l is primitive span_base + 32 q + l, so one ballot is one mask word and ranks inside the
// warp follow the primitive order.  The ballots are kept (word q in lane q % 32), so the list is written after the
// look-back without reading the counts a second time.
constexpr int TS_MAX_ROUNDS = 8;

__global__ void __launch_bounds__(TS_THREADS)
touched_set_kernel(const uint32_t* __restrict__ tiles_touched, uint32_t n, uint32_t* __restrict__ mask,
                   uint32_t* __restrict__ idx, uint32_t idx_capacity, uint32_t* __restrict__ count, uint32_t* ticket,
                   uint64_t* state, int* status, int scan_rounds, int spin_limit) {
  const uint32_t scan_chunk = TOUCHED_TILE * (uint32_t)scan_rounds;
  __shared__ uint32_t s_tile;
  __shared__ uint32_t s_warp[33];
  __shared__ uint64_t s_base;
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
  __syncthreads();
  const uint32_t tile = s_tile;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int words = scan_rounds * TS_ITEMS;  // mask words (ballots) per warp: 8 .. 64
  const uint32_t span_base = tile * scan_chunk + warp * (uint32_t)words * 32u;
  const uint32_t n_words = (n + 31) / 32;
  // pass A: ballots of the warp's span; word q stays in lane q % 32 of keep[q / 32]
  uint32_t keep[TS_MAX_ROUNDS * TS_ITEMS / 32] = {0u, 0u};
  uint32_t warp_count = 0;
#pragma unroll 8
  for (int q = 0; q < words; ++q) {
    const uint32_t p = span_base + 32u * (uint32_t)q + lane;
    const uint32_t bal = __ballot_sync(0xffffffffu, p < n && tiles_touched[p] > 0);
    warp_count += __popc(bal);
    if (lane == (unsigned)(q & 31)) keep[q >> 5] = bal;
  }
  // the mask words of the span: 32 consecutive words per store
  for (int h = 0; h * 32 < words; ++h) {
    const uint32_t word = span_base / 32 + h * 32 + lane;
    if ((int)(h * 32 + lane) < words && word < n_words) mask[word] = keep[h];
  }
  uint32_t chunk_total;
  const uint32_t scan = odin_block_exclusive_sum(lane == 0 ? warp_count : 0u, s_warp, &chunk_total);
  const uint32_t warp_off = __shfl_sync(0xffffffffu, scan, 0);
  if (threadIdx.x < 32) {
    const uint64_t ex = odin_lookback_u64(state, tile, (uint64_t)chunk_total, status, spin_limit);
    if (threadIdx.x == 0) s_base = ex;
  }
  __syncthreads();
  const uint64_t base = s_base;
  if (tile == (n + scan_chunk - 1) / scan_chunk - 1 && threadIdx.x == 0) {
    const uint64_t v = base + chunk_total;
    *count = (uint32_t)(v < idx_capacity ? v : idx_capacity);
    if (v > idx_capacity) odin_set_error(status, ODIN_ERR_CAPACITY);
  }
  // pass B: the ascending list from the kept ballots
  uint64_t pos = base + warp_off;
  const uint32_t lt = (1u << lane) - 1u;
  for (int q = 0; q < words; ++q) {
    const uint32_t bal = __shfl_sync(0xffffffffu, keep[q >> 5], q & 31);
    if (bal >> lane & 1u) {
      const uint64_t dst = pos + __popc(bal & lt);
      if (dst < idx_capacity) idx[dst] = span_base + 32u * (uint32_t)q + lane;
    }
    pos += __popc(bal);
  }
}

// The ascending list of the members of a bitmask.  A block takes ML_WORDS words by ticket, lane l of a warp the l-th of 32
// consecutive words; population counts, one look-back, and a word's members are written side by side, the places of eight words
// worked out together (a chain of exchanges from word to word before: with the memset, 400 k primitives of which half are members
// 13.7 -> 8.5 us, 5 M 19.5 -> 14.5, 20 M 33 -> 21; 2 % members 10.6 -> 8.5, 16.6 -> 14.2, 20.8 -> 20.5), except where few of the words have members: up to ML_FEW of 32 are taken
// one by one (0.1 to 0.6 % members, 100 k to 20 M primitives: 8.5 -> 6.5 to 18.8 -> 15.2).  What bounds it: ticket, load, look-back and
// stores behind one another.  Tried: one word per thread (20 M 27 us), four (400 k 12 us); all totals in front
// read side by side instead of a look-back (5 M with one word per thread 14 -> 12, but 20 M 24 and 120 M 118 against 83).
constexpr int ML_THREADS = 256;
constexpr int ML_ITEMS = 2;                               // words per thread
constexpr int ML_FEW = 6;                                 // words with members of 32 that are taken one by one
constexpr uint32_t ML_WORDS = ML_THREADS * ML_ITEMS;      // 16,384 primitives per look-back tile
static_assert(ML_WORDS * 32 >= TOUCHED_TILE, "the look-back words of touched_ws_bytes are enough");

__global__ void __launch_bounds__(ML_THREADS)
mask_to_list_kernel(const uint32_t* __restrict__ mask, uint32_t n, uint32_t* __restrict__ idx, uint32_t idx_capacity,
                    uint32_t* __restrict__ count, uint32_t* ticket, uint64_t* state, int* status, int spin_limit) {
  __shared__ uint32_t s_tile, s_warp[33];
  __shared__ uint64_t s_base;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
  __syncthreads();
  const uint32_t tile = s_tile, n_words = (n + 31) / 32;
  const uint32_t word0 = tile * ML_WORDS + warp * (32 * ML_ITEMS);
  uint32_t w[ML_ITEMS], c[ML_ITEMS];
#pragma unroll
  for (int k = 0; k < ML_ITEMS; ++k) {
    const uint32_t word = word0 + 32 * k + lane;
    w[k] = word < n_words ? mask[word] : 0u;
    if (word == n_words - 1 && (n & 31u)) w[k] &= (1u << (n & 31u)) - 1u;  // bits past n do not name primitives
    c[k] = __popc(w[k]);
  }
  uint32_t warp_count = 0;
#pragma unroll
  for (int k = 0; k < ML_ITEMS; ++k) warp_count += __reduce_add_sync(0xffffffffu, c[k]);
  uint32_t total;
  const uint32_t before = __shfl_sync(0xffffffffu, odin_block_exclusive_sum(lane == 0 ? warp_count : 0u, s_warp, &total), 0);
  if (warp == 0) {
    const uint64_t b = odin_lookback_u64(state, tile, (uint64_t)total, status, spin_limit);
    if (lane == 0) {
      s_base = b;
      if (tile == (n_words + ML_WORDS - 1) / ML_WORDS - 1) {
        const uint64_t v = b + total;
        *count = (uint32_t)(v < idx_capacity ? v : idx_capacity);
        if (v > idx_capacity) odin_set_error(status, ODIN_ERR_CAPACITY);
      }
    }
  }
  __syncthreads();
  uint64_t pos = s_base + before;
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
  for (int k = 0; k < ML_ITEMS; ++k) {
    uint32_t some = __ballot_sync(0xffffffffu, w[k] != 0);
    if (__popc(some) <= ML_FEW) {  // word by word
      while (some) {
        const int src = __ffs(some) - 1;
        some &= some - 1;
        const uint32_t bits = __shfl_sync(0xffffffffu, w[k], src);
        const uint64_t dst = pos + __popc(bits & lt);
        if ((bits >> lane & 1u) && dst < idx_capacity) idx[dst] = (word0 + 32 * k + src) * 32 + lane;
        pos += __popc(bits);
      }
      continue;
    }
    uint32_t upto = c[k];  // members in the words of the lanes up to and with this one
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, upto, o);
      if (lane >= (unsigned)o) upto += x;
    }
    uint32_t* const out = idx + pos;
    const uint32_t room = (uint32_t)(pos < idx_capacity ? min((uint64_t)idx_capacity - pos, (uint64_t)1024) : 0);
    const uint32_t id = (word0 + 32 * k) * 32 + lane;
#pragma unroll
    for (int g = 0; g < 32; g += 8) {  // eight words' exchanges at a time
      if (!(some >> g & 255u)) continue;
#pragma unroll
      for (int src = g; src < g + 8; ++src) {
        const uint32_t bits = __shfl_sync(0xffffffffu, w[k], src), first = __shfl_sync(0xffffffffu, upto - c[k], src);
        const uint32_t at = first + __popc(bits & lt);
        if ((bits >> lane & 1u) && at < room) out[at] = id + 32 * src;
      }
    }
    pos += __shfl_sync(0xffffffffu, upto, 31);
  }
}

constexpr int CC_THREADS = (int)PAIR_THREADS;

// One block column per pair (blockIdx.y); blocks of a column stride over the mask words four at a time.
__global__ void __launch_bounds__(CC_THREADS)
conflict_count_kernel(const uint32_t* __restrict__ masks, uint32_t stride_words, uint32_t words,
                      const uint32_t* __restrict__ pairs, uint32_t n_masks, unsigned long long* __restrict__ counts,
                      int* status) {
  odin_after_predecessor();
  const uint32_t pair = blockIdx.y;
  const uint32_t va = pairs[2 * pair], vb = pairs[2 * pair + 1];
  if (va >= n_masks || vb >= n_masks) {  // uniform over the block: a pair naming a missing view counts 0
    if (threadIdx.x == 0) odin_set_error(status, ODIN_ERR_INVALID_ARG);
    return;
  }
  const uint32_t* a = masks + (size_t)va * stride_words;
  const uint32_t* b = masks + (size_t)vb * stride_words;
  uint32_t c = 0;
  const uint32_t vec = words / 4;
  const uint4* a4 = reinterpret_cast<const uint4*>(a);
  const uint4* b4 = reinterpret_cast<const uint4*>(b);
  for (uint32_t i = blockIdx.x * CC_THREADS + threadIdx.x; i < vec; i += gridDim.x * CC_THREADS) {
    const uint4 x = a4[i], y = b4[i];
    c += __popc(x.x & y.x) + __popc(x.y & y.y) + __popc(x.z & y.z) + __popc(x.w & y.w);
  }
  if (blockIdx.x == 0)
    for (uint32_t i = vec * 4 + threadIdx.x; i < words; i += CC_THREADS) c += __popc(a[i] & b[i]);
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  __shared__ uint32_t s[CC_THREADS / 32];
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t tot = 0;
    for (int i = 0; i < CC_THREADS / 32; ++i) tot += s[i];
    if (tot) atomicAdd(&counts[pair], (unsigned long long)tot);
  }
}

// Many pairs over few masks: all intersections at once, as the product of the 0/1 matrix [mask][primitive] with its
// transpose on the tensor cores: tcgen05.mma kind::mxf4, e2m1 x e2m1 -> f32 with every block scale 1.  Products of 0 and 1 are exact, and so
// are their sums: none exceeds 2^23 (CG_BLOCK_WORDS).  Counting pair by pair reads both masks again for every pair and is bound by the
// population count (16 words a clock and SM).  All 8,128 pairs of 128 masks of 20 M primitives: pair by pair 2,080 us, as bytes on the integer
// tensor cores (twice the products and stores, one block-wide barrier per step) 330, here 126 (64 masks 170 -> 66, 200 masks of 8 M
// 487 -> 213).  What bounds it: three things about equal.  The products alone take 100 us, expansion and products with words from L2
// 117, the fetch alone 107 (128 rows 2.5 MB apart, 256 bytes of each at a time).  128 masks of 8 M: tensor pipe active 57 % of
// the cycles that an SM has work, the data pipe of shared memory 58 %, issue slots 47 %, DRAM 27 %.
//
// A block takes 128 masks against 128 (the same ones on the diagonal of the mask blocks, where one copy in shared memory is
// both operands) and a share of the words.  64 masks or 32 fill the 128 rows with two or four stretches of words each; their
// sums are then on the diagonal of the result.  Per step every expanding thread turns 4 words of one row into 16 bytes each: 32 KB, as
// K-major core matrices without swizzle (8 rows x 16 bytes, 128 bytes each; a warp's 32 rows are 512 consecutive bytes, so the stores
// have no bank conflicts; rows of 128 bytes in the 128-byte swizzle: the same).  Warps hand over by barriers of their own and are
// up to four steps ahead of the products.  Two warps issue these, every other step each into sums of its own, so that one waits
// while the other's products run (one warp: 168 us; two sets of sums for one warp: 164).  The order of the primitives within a
// word is that of the bit planes, which is as good as any: both operands share it.
constexpr int CG_EXPANDERS = 16;                         // warps that expand
constexpr int CG_ISSUERS = 2;                            // warps that issue the products, of every other step each
constexpr int CG_THREADS = 32 * (CG_EXPANDERS + CG_ISSUERS);
constexpr int CG_ROWS = 128;                             // rows of a side
constexpr int CG_STAGES = 4;                             // steps that are expanded or being multiplied; steps of a round
constexpr int CG_STAGE = CG_EXPANDERS * 32 * 64;         // bytes of a step: 4 words per thread, 16 bytes each
constexpr int CG_AHEAD = 3;                              // rounds whose words are there or on their way
constexpr int CG_ROUND = 32 * 16 * CG_STAGES;            // bytes of a warp's round: 64 of each of its rows
constexpr size_t CG_SMEM = CG_STAGES * CG_STAGE + CG_EXPANDERS * CG_AHEAD * CG_ROUND + 128;
constexpr uint32_t CG_TMEM = 512, CG_SCALE = CG_ISSUERS * CG_ROWS;  // columns: sums of each issuer; 16 of scales for each operand (4 are read)
// Words of a block off the diagonal; one on it gets up to twice as many (4 / 3 as many, rounded up to one block at worst), half of them
// in each issuer's sums: at most 2^18 words, 2^23 primitives a sum, where 2^24 would still be exact in fp32.
constexpr uint32_t CG_BLOCK_WORDS = 1u << 18;

// descriptor of an operand in shared memory: core matrices CG_ROWS * 16 bytes apart along K, 128 along the rows
__device__ __forceinline__ uint64_t gram_operand(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3fffu) | (uint64_t)(CG_ROWS * 16 >> 4) << 16 | (uint64_t)(128 >> 4) << 32 | 1ull << 46;
}

// A bounded wait for the phase of a barrier; false if it ran out.  The first look does not wait (a limit of 0 gives up at
// once), each further one for a while that the hardware sets.
__device__ __forceinline__ bool gram_wait(uint32_t mbar, uint32_t parity, int spin_limit) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
  for (int spins = 0; !done && spins < spin_limit; ++spins)
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
  return done != 0;
}

__global__ void __launch_bounds__(CG_THREADS, 1)
conflict_gram_kernel(const uint32_t* __restrict__ masks, uint32_t stride_words, uint32_t words, uint32_t n_masks,
                     const uint32_t* __restrict__ pairs, uint32_t n_pairs, unsigned long long* __restrict__ counts, int* status,
                     int side_log, int spin_limit) {  // 2^side_log masks fill a side: 32, 64 or 128
  odin_after_predecessor();
  extern __shared__ uint8_t gram_raw[];
  __shared__ __align__(8) uint64_t s_bar[2 * CG_STAGES];  // stage is full (one arrival per expanding warp), stage is free
  __shared__ uint32_t s_tmem;
  uint8_t* smem = gram_raw + ((128u - ((uint32_t)__cvta_generic_to_shared(gram_raw) & 127u)) & 127u);
  const uint32_t smem_addr = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t full = (uint32_t)__cvta_generic_to_shared(s_bar), free_ = full + 8 * CG_STAGES;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // pair of mask blocks: (0,0), (0,1), (1,1), (0,2), ...
  uint32_t mb = 0;
  for (uint32_t rest = blockIdx.y; rest > mb; rest -= mb) ++mb;
  const uint32_t ma = blockIdx.y - mb * (mb + 1) / 2, a0 = ma << side_log, b0 = mb << side_log;
  const bool diag = ma == mb;
  // off the diagonal a word costs the same products and twice the expansion: 4 blocks for 3
  const uint32_t parts = diag && gridDim.y > 1 ? max(1u, 3 * gridDim.x / 4) : gridDim.x;
  if (blockIdx.x >= parts) return;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(&s_tmem)), "n"(CG_TMEM) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < CG_STAGES; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8 * i), "n"(CG_EXPANDERS) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(free_ + 8 * i) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;
  if (warp < 4) {  // every scale is 1 (2^(127 - 127)), in whatever order the products read them
#pragma unroll
    for (uint32_t c = 0; c < 32; c += 8)
      asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};"
                   ::"r"(tmem + (32 * warp << 16) + CG_SCALE + c), "r"(0x7f7f7f7fu) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  const uint32_t groups = diag ? 4 : 2;  // threads of a row: 128 threads each of a side's rows
  const uint32_t row_words = groups * 4 * CG_STAGES, round_words = row_words * (CG_ROWS >> side_log), rounds = (words + round_words - 1) / round_words;
  bool late = false;
  if (warp < CG_EXPANDERS) {
    // The warp's rows (of side 0, or of side 1 off the diagonal) and its 16 words of each in a round, as pieces of 16 bytes:
    // neighbouring lanes fetch neighbouring pieces of a row; a piece lies in shared memory at a place that keeps the 8 rows a
    // quarter warp reads apart in banks.
    const uint32_t group = warp / 4, side = group / groups, in_side = group % groups, row0 = warp % 4 * 32;
    const uint32_t buf = smem_addr + CG_STAGES * CG_STAGE + warp * (CG_AHEAD * CG_ROUND), first_mask = side ? b0 : a0;
    auto place = [&](uint32_t r, uint32_t piece) { return r * 64 + ((piece ^ (r >> 1 & 3u)) << 4); };
    // piece k of the lane: its word of the round to come, and where that is; both move on by a round of this block
    const uint32_t step_words = parts * round_words;
    const uint32_t* src[4];
    uint32_t word[4], dst_fetch[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t r = 8 * k + lane / 4, piece = lane % 4, row = row0 + r, mask = first_mask + (row & ((1u << side_log) - 1u));
      word[k] = mask < n_masks ? blockIdx.x * round_words + (row >> side_log) * row_words + in_side * (4 * CG_STAGES) + 4 * piece : words;
      src[k] = masks + (mask < n_masks ? (size_t)mask * stride_words + word[k] : (size_t)0);
      dst_fetch[k] = buf + place(r, piece);
    }
    auto fetch = [&](uint32_t slot) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        // behind the last word: zeros (what is read lies within the row's stride)
        const uint32_t bytes = word[k] < words ? min(words - word[k], 4u) * 4u : 0u;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                     ::"r"(dst_fetch[k] + slot * CG_ROUND), "l"(bytes ? src[k] : masks), "r"(bytes) : "memory");
        word[k] = word[k] < words ? word[k] + step_words : words;
        src[k] += step_words;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    uint8_t* const dst = smem + group * (4 * CG_ROWS * 16) + (row0 + lane) * 16;
    uint32_t slot = 0, parity = 1;  // (the stages of a fresh barrier are free)
    for (uint32_t i = 0; i < CG_AHEAD; ++i) fetch(i);
    for (uint32_t round = blockIdx.x; round < rounds && !late; round += parts, parity ^= 1u) {
      asm volatile("cp.async.wait_group %0;" ::"n"(CG_AHEAD - 1) : "memory");
      __syncwarp();
#pragma unroll
      for (uint32_t q = 0; q < CG_STAGES; ++q) {
        uint32_t v[4];
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                     : "r"(buf + slot * CG_ROUND + place(lane, q)) : "memory");
        // the products that read this stage before (where the wait ran out they may still read it: nothing is written)
        if (!__all_sync(0xffffffffu, gram_wait(free_ + 8 * q, parity, spin_limit))) { late = true; break; }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t one = 0x22222222u;  // 1.0 in e2m1 is 2
          *reinterpret_cast<uint4*>(dst + q * CG_STAGE + k * (CG_ROWS * 16)) = make_uint4((v[k] << 1) & one, v[k] & one, (v[k] >> 1) & one, (v[k] >> 2) & one);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(full + 8 * q) : "memory");
      }
      if (late) break;
      fetch(slot);  // every lane has read the slot
      slot = slot + 1 == CG_AHEAD ? 0 : slot + 1;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    // The whole warp goes through the loop, so that what the products take is uniform; one lane issues them.
    // f32 += e2m1 x e2m1, both K-major, scales ue8m0
    constexpr uint32_t IDESC = 1u << 7 | 1u << 10 | (uint32_t)(CG_ROWS >> 3) << 17 | 1u << 23 | (uint32_t)(CG_ROWS >> 4) << 24;
    const uint32_t leader = lane == 0, issuer = warp - CG_EXPANDERS, sums = tmem + issuer * CG_ROWS;
    const uint64_t a = gram_operand(smem_addr + issuer * CG_STAGE), b = gram_operand(smem_addr + issuer * CG_STAGE + (diag ? 0u : groups * (4 * CG_ROWS * 16)));
    uint32_t parity = 0, more = 0, last = 0;
    for (uint32_t round = blockIdx.x; round < rounds && !late; round += parts, parity ^= 1u)
#pragma unroll
      for (uint32_t q = 0; q < CG_STAGES; q += CG_ISSUERS) {
        if (!__all_sync(0xffffffffu, gram_wait(full + 8 * (q + issuer), parity, spin_limit))) { late = true; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) {  // 64 primitives each
          if (k < 2 * groups)
            asm volatile(
                "{\n .reg .pred p, q;\n setp.ne.u32 p, %4, 0;\n setp.ne.u32 q, %7, 0;\n"
                " @q tcgen05.mma.cta_group::1.kind::mxf4.block_scale.block32 [%0], %1, %2, %3, [%5], [%6], p;\n}"
                ::"r"(sums), "l"(a + (q * CG_STAGE + k * (CG_ROWS * 32) >> 4)), "l"(b + (q * CG_STAGE + k * (CG_ROWS * 32) >> 4)), "r"(IDESC),
                  "r"(more + k), "r"(tmem + CG_SCALE), "r"(tmem + CG_SCALE + 16), "r"(leader) : "memory");
        }
        more = 1;
        last = 1 + 2 * (q + issuer) + parity;
        asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %1, 0;\n"
                     " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}"
                     ::"r"(free_ + 8 * (q + issuer)), "r"(leader) : "memory");
      }
    // The last products finish whatever becomes of this block, and until then the shared memory they read and the tensor
    // memory they write are theirs: this wait's limit is its own, not the caller's.
    if (last) late |= !gram_wait(free_ + 8 * (last - 1 >> 1), last - 1 & 1u, ODIN_DEFAULT_SPIN_LIMIT);
  }
  const bool whole = !__syncthreads_or(late);  // the block's share was gone through: its sums count
  if (!whole && threadIdx.x == 0) odin_set_error(status, ODIN_ERR_TIMEOUT);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  // sums to shared memory (rows one word apart in banks): a warp reads its quarter of the tensor memory's lanes, which are
  // the rows, and a quarter of the columns
  uint32_t* s_gram = reinterpret_cast<uint32_t*>(smem);
  const bool any = blockIdx.x < rounds;
  if (whole && any && warp < 16) {
    const uint32_t quarter = warp & 3u, col0 = (warp >> 2) * (CG_ROWS / 4);
#pragma unroll
    for (int c0 = 0; c0 < CG_ROWS / 4; c0 += 16) {
      uint32_t c[16] = {};
#pragma unroll
      for (int m = 0; m < CG_ISSUERS; ++m) {
        float r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
            : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]), "=f"(r[9]),
              "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
            : "r"(tmem + (32 * quarter << 16) + m * CG_ROWS + col0 + c0));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 16; ++i) c[i] += __float2uint_rn(r[i]);
      }
#pragma unroll
      for (int i = 0; i < 16; ++i) s_gram[(32 * quarter + lane) * (CG_ROWS + 1) + col0 + c0 + i] = c[i];
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(CG_TMEM) : "memory");
  // every pair that this pair of mask blocks answers
  for (uint32_t p = threadIdx.x; p < n_pairs; p += CG_THREADS) {
    const uint32_t va = pairs[2 * p], vb = pairs[2 * p + 1], lo = min(va, vb), hi = max(va, vb);
    if (hi >= n_masks) {  // a pair naming a missing view counts 0
      if (blockIdx.x == 0 && blockIdx.y == 0) odin_set_error(status, ODIN_ERR_INVALID_ARG);
      continue;
    }
    if (lo >> side_log != ma || hi >> side_log != mb || !any || !whole) continue;
    uint32_t c = 0;
    for (uint32_t r = 0; r < CG_ROWS; r += 1u << side_log) c += s_gram[(r + lo - a0) * (CG_ROWS + 1) + (r + hi - b0)];
    if (c) atomicAdd(&counts[p], (unsigned long long)c);
  }
}

}  // namespace

extern "C" int odin_touched_set(odin_ctx* ctx, const uint32_t* d_tiles_touched, uint32_t n, uint32_t* d_mask,
                                uint32_t* d_idx, uint32_t idx_capacity, uint32_t* d_count, void* ws, size_t ws_bytes,
                                void* stream) {
  if (!ctx || !d_count) return ODIN_ERR_NULL;
  cudaStream_t st = (cudaStream_t)stream;
  if (n >= (1u << 28)) return ODIN_ERR_INVALID_ARG;
  if (n == 0) {
    odin_chain_break(ctx);
    ODIN_CUDA(cudaMemsetAsync(d_count, 0, 4, st));
    return ODIN_OK;
  }
  if (!d_tiles_touched || !d_mask || (idx_capacity > 0 && !d_idx)) return ODIN_ERR_NULL;
  const size_t need = touched_ws_bytes(n);
  if (!ws || !odin_aligned(ws, 256) || ws_bytes < need) return ODIN_ERR_WORKSPACE;
  odin_chain_break(ctx);
  ODIN_CUDA(cudaMemsetAsync(ws, 0, need, st));
  uint32_t* ticket = reinterpret_cast<uint32_t*>(ws);
  uint64_t* state = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(ws) + 256);
  const int scan_rounds = scan_rounds_for(n, ctx->sm_count);
  const uint32_t scan_chunk = TOUCHED_TILE * (uint32_t)scan_rounds;
  const uint32_t grid = (n + scan_chunk - 1) / scan_chunk;
  OdinKernelScope ks(ctx, K_TOUCHED, st);
  touched_set_kernel<<<grid, TS_THREADS, 0, st>>>(d_tiles_touched, n, d_mask, d_idx, idx_capacity, d_count, ticket,
                                                         state, ctx->d_status, scan_rounds, ctx->spin_limit);
  return odin_launch_status();
}

extern "C" int odin_mask_to_list(odin_ctx* ctx, const uint32_t* d_mask, uint32_t n, uint32_t* d_idx, uint32_t idx_capacity,
                                 uint32_t* d_count, void* ws, size_t ws_bytes, void* stream) {
  if (!ctx || !d_count) return ODIN_ERR_NULL;
  cudaStream_t st = (cudaStream_t)stream;
  if (n >= (1u << 28)) return ODIN_ERR_INVALID_ARG;
  if (n == 0) {
    odin_chain_break(ctx);
    ODIN_CUDA(cudaMemsetAsync(d_count, 0, 4, st));
    return ODIN_OK;
  }
  if (!d_mask || (idx_capacity > 0 && !d_idx)) return ODIN_ERR_NULL;
  const size_t need = touched_ws_bytes(n);
  if (!ws || !odin_aligned(ws, 256) || ws_bytes < need) return ODIN_ERR_WORKSPACE;
  odin_chain_break(ctx);
  ODIN_CUDA(cudaMemsetAsync(ws, 0, 256 + (((size_t)n + 31) / 32 / ML_WORDS + 1) * 8, st));
  uint32_t* ticket = reinterpret_cast<uint32_t*>(ws);
  uint64_t* state = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(ws) + 256);
  const uint32_t grid = ((n + 31) / 32 + ML_WORDS - 1) / ML_WORDS;
  OdinKernelScope ks(ctx, K_TOUCHED, st);
  mask_to_list_kernel<<<grid, ML_THREADS, 0, st>>>(d_mask, n, d_idx, idx_capacity, d_count, ticket, state, ctx->d_status, ctx->spin_limit);
  return odin_launch_status();
}

// ---------------------------------------------------------------------------------------------------------------
// Touched set without any allocation.  Some users of this library are handed all of their GPU memory up front and may
// never allocate again: a component embedded in a host application that owns the memory pool, or a real-time loop in
// which an allocation could stall or fail at a bad moment.  They cannot call odin_create (it allocates the status word)
// nor size and allocate a workspace.  For them this entry point runs the same kernel as odin_touched_set with its
// scratch (tile ticket, deferred-status sink, look-back words) in a fixed array that is part of the loaded library:
// every GPU that loads libodin.so holds these 128.3 KB until the process exits.
constexpr uint32_t TS_STATIC_MAX_N = 1u << 25;  // 33,554,432 primitives
constexpr size_t TS_STATIC_HEADER = 256;        // [0] ticket, [64] status sink
constexpr size_t TS_STATIC_BYTES = TS_STATIC_HEADER + (size_t)(TS_STATIC_MAX_N / TOUCHED_TILE) * 8;
static __device__ __align__(256) unsigned char g_touched_static_scratch[TS_STATIC_BYTES];

// In host code the array's name is only a handle for the runtime, not a device address, so the address is asked for
// once per device (with that device current) and cached.  The cache entries are atomics: two host threads that make
// the first call on a device at the same time both look the address up and store the same value.
constexpr int TS_STATIC_MAX_DEVICES = 64;
static std::atomic<unsigned char*> g_touched_static_ptr[TS_STATIC_MAX_DEVICES];

extern "C" int odin_touched_set_static(const uint32_t* d_tiles_touched, uint32_t n, uint32_t* d_mask, uint32_t* d_idx,
                                       uint32_t idx_capacity, uint32_t* d_count, int* d_status, void* stream) {
  if (!d_count) return ODIN_ERR_NULL;
  if (n > TS_STATIC_MAX_N) return ODIN_ERR_INVALID_ARG;  // beyond the fixed scratch: use odin_touched_set
  cudaStream_t st = (cudaStream_t)stream;
  if (n == 0) {
    ODIN_CUDA(cudaMemsetAsync(d_count, 0, 4, st));
    return ODIN_OK;
  }
  if (!d_tiles_touched || !d_mask || (idx_capacity > 0 && !d_idx)) return ODIN_ERR_NULL;
  int device = -1;
  ODIN_CUDA(cudaGetDevice(&device));
  if (device < 0 || device >= TS_STATIC_MAX_DEVICES) return ODIN_ERR_UNSUPPORTED;
  unsigned char* scratch = g_touched_static_ptr[device].load(std::memory_order_acquire);
  if (!scratch) {  // first call on this device: resolve the array's device address (this may load the module)
    void* p = nullptr;
    ODIN_CUDA(cudaGetSymbolAddress(&p, g_touched_static_scratch));
    if (!p) return ODIN_ERR_CUDA;
    scratch = static_cast<unsigned char*>(p);
    g_touched_static_ptr[device].store(scratch, std::memory_order_release);
  }
  const uint32_t tiles = (n + TOUCHED_TILE - 1) / TOUCHED_TILE;
  // the array keeps whatever the previous call left: the ticket, the sink and the look-back words must start at zero
  ODIN_CUDA(cudaMemsetAsync(scratch, 0, TS_STATIC_HEADER + (size_t)tiles * 8, st));
  uint32_t* ticket = reinterpret_cast<uint32_t*>(scratch);
  int* status = d_status ? d_status : reinterpret_cast<int*>(scratch + 64);
  uint64_t* state = reinterpret_cast<uint64_t*>(scratch + TS_STATIC_HEADER);
  // no context here, so the SM count is not looked up: the block size is chosen for the 148 SMs of a B200 (any other
  // count only changes how many blocks share the work, never the result)
  const int scan_rounds = scan_rounds_for(n, 148);
  const uint32_t scan_chunk = TOUCHED_TILE * (uint32_t)scan_rounds;
  touched_set_kernel<<<(n + scan_chunk - 1) / scan_chunk, TS_THREADS, 0, st>>>(
      d_tiles_touched, n, d_mask, d_idx, idx_capacity, d_count, ticket, state, status, scan_rounds,
      ODIN_DEFAULT_SPIN_LIMIT);
  return odin_launch_status();
}

extern "C" int odin_conflict_count(odin_ctx* ctx, const uint32_t* d_masks, uint32_t n_masks, uint32_t mask_stride_words,
                                   uint32_t n_prims, const uint32_t* d_pairs, uint32_t n_pairs, uint64_t* d_counts,
                                   void* stream) {
  if (!ctx) return ODIN_ERR_NULL;
  if (n_pairs == 0) return ODIN_OK;
  if (!d_pairs || !d_counts) return ODIN_ERR_NULL;
  if (n_pairs > 65535) return ODIN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  ODIN_CUDA(odin_zero(ctx, d_counts, (size_t)n_pairs * 8, st));
  const uint32_t words = (n_prims + 31) / 32;
  if (words == 0) return ODIN_OK;
  if (!d_masks) return ODIN_ERR_NULL;
  if (n_masks == 0 || mask_stride_words < words || (mask_stride_words % 4) != 0 || !odin_aligned(d_masks, 16))
    return ODIN_ERR_INVALID_ARG;
  // All pairs of a set of masks (or a good part of them) go to the matrix kernel: its cost does not depend on their number.
  if (pair_by_matrix(words, n_masks, n_pairs, (uint32_t)ctx->sm_count)) {
    const PairSides sides = pair_sides(n_masks);
    const int side_log = sides.side_log;
    const uint32_t blocks_m = sides.blocks_m, block_pairs = sides.block_pairs;
    OdinKernelScope ks(ctx, K_CONFLICT, st);
    const uint32_t round = (blocks_m == 1 ? 4u : 2u) * 4 * CG_STAGES * (CG_ROWS >> side_log), rounds = (words + round - 1) / round;
    // one block per SM; those off the diagonal of the mask blocks get 4 for every 3 on it
    uint32_t gx = (uint32_t)ctx->sm_count;
    if (blocks_m > 1) gx = 4 * gx / (3 * blocks_m + 4 * (block_pairs - blocks_m));
    if (gx < (words + CG_BLOCK_WORDS - 1) / CG_BLOCK_WORDS) gx = (words + CG_BLOCK_WORDS - 1) / CG_BLOCK_WORDS;
    if (gx > rounds) gx = rounds;
    if (gx == 0) gx = 1;
    ODIN_CUDA(cudaFuncSetAttribute(conflict_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CG_SMEM));
    ODIN_CUDA(odin_launch(ctx, false, conflict_gram_kernel, dim3(gx, block_pairs), dim3(CG_THREADS), CG_SMEM, st, d_masks,
                          mask_stride_words, words, n_masks, d_pairs, n_pairs, reinterpret_cast<unsigned long long*>(d_counts),
                          ctx->d_status, side_log, ctx->spin_limit));
    return odin_launch_status();
  }
  const uint32_t gx = pair_grid(words, n_pairs, (uint32_t)ctx->sm_count);
  OdinKernelScope ks(ctx, K_CONFLICT, st);
  ODIN_CUDA(odin_launch(ctx, false, conflict_count_kernel, dim3(gx, n_pairs), dim3(CC_THREADS), 0, st, d_masks,
                        mask_stride_words, words, d_pairs, n_masks, reinterpret_cast<unsigned long long*>(d_counts),
                        ctx->d_status));
  return odin_launch_status();
}
