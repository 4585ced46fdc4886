// Tile binning and sort.  The order asked for is that of a stable least-significant-digit radix sort of the instance
// keys tile_id << 32 | depth bits.  All instances of a row share the row's depth, so the passes over the depth digits are
// taken on the ROWS (several times fewer than the instances): rows are sorted by depth, the instances are emitted in
// that order (load balanced over instances), and only the passes over the tile-id digits run on the instances.  The
// result is the very sequence the full-width sort produces: after the depth passes an instance list is ordered by
// (depth, row, position in the row's rectangle) either way.  Every pass is a onesweep pass with decoupled look-back
// (no library sort).  The per-tile ranges and the digit histograms of the instance passes come from per-tile instance
// counts that are accumulated from the rectangles (a difference array over the tile ids), not from the instances.
#include <type_traits>

#include "common.cuh"
#include "layout.cuh"
#include "tilespan.cuh"

namespace {

// ------------------------------------------------------------------------------------------------ row histograms
// Digit histograms of the depth bits of all rows for the first three passes over them, and their exclusive scans.  The third digit
// is the last one unless the bits above the first two span more than ROW_RADIX values: it is scanned from the smallest of them on,
// around the end, so that three passes order any depths that lie within a factor of 2^16, whatever the unit of length; *top
// tells whether the fourth pass, on the ROW_TOP_BITS that are left, is needed as well.  Also zeroes the look-back words of the passes, of the tiles that
// there are (the third pass those of the fourth).
// Plain shared atomics: aggregating the equal digits of a warp with match.any first (the high digits of a depth take
// few distinct values) was slower, 0.023 against 0.016 ms for 317 k rows - the match costs more than the conflicts.  The block
// that arrives last turns the histograms into exclusive scans, which saves a launch.
constexpr int RH_THREADS = 1024;
constexpr uint32_t ROW_TOP_SHIFT = 3 * ROW_RADIX_BITS, ROW_TOP_BITS = 32 - ROW_TOP_SHIFT;
constexpr uint32_t ROW_HIGH_SHIFT = 2 * ROW_RADIX_BITS, ROW_HIGHS = 1u << (32 - ROW_HIGH_SHIFT);  // of the bits above the first two digits
static_assert(ROW_TOP_BITS == 5, "a lane per digit of the fourth pass");
__global__ void __launch_bounds__(RH_THREADS)
row_hist_kernel(const uint32_t* __restrict__ depth_bits, const uint32_t* __restrict__ num_rows, uint32_t* __restrict__ hist,
                uint32_t* __restrict__ base, uint32_t* arrivals, uint32_t* __restrict__ top, uint32_t* __restrict__ range,
                uint32_t* __restrict__ states, uint32_t row_tile, uint32_t row_tiles) {
  constexpr int DIGITS = SORT_DEPTH_DIGITS - 1, BINS = DIGITS * (int)ROW_RADIX;
  static_assert(RH_THREADS >= (int)ROW_RADIX, "thread d scans digit d");
  __shared__ uint32_t s_hist[BINS];
  __shared__ uint32_t s_warp[33], s_flag, s_range[2];  // (range: ROW_HIGHS less the smallest value, the largest and one more)
  for (int i = threadIdx.x; i < BINS; i += RH_THREADS) s_hist[i] = 0;
  if (threadIdx.x < 2) s_range[threadIdx.x] = 0;
  odin_after_predecessor();
  __syncthreads();
  const uint32_t V = *num_rows;
  const uint32_t stride = gridDim.x * blockDim.x, tid = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t tiles = min((uint32_t)(((uint64_t)V + row_tile - 1) / row_tile), row_tiles);
  const size_t pass_words = (size_t)row_tiles * ROW_RADIX;
  for (int d = 0; d < DIGITS; ++d) {
    uint4* w = reinterpret_cast<uint4*>(states + d * pass_words);
    for (uint32_t i = tid; i < tiles * (ROW_RADIX / 4); i += stride) w[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  uint32_t below = 0, above = 0;
  for (uint32_t r = tid; r < V; r += stride) {
    const uint32_t key = depth_bits[r], high = key >> ROW_HIGH_SHIFT;
#pragma unroll
    for (int d = 0; d < DIGITS; ++d) atomicAdd(&s_hist[d * ROW_RADIX + (key >> (ROW_RADIX_BITS * d) & (ROW_RADIX - 1))], 1u);
    below = max(below, ROW_HIGHS - high);
    above = max(above, high + 1u);
  }
  below = __reduce_max_sync(0xffffffffu, below);
  above = __reduce_max_sync(0xffffffffu, above);
  if ((threadIdx.x & 31) == 0 && above) {
    atomicMax(&s_range[0], below);
    atomicMax(&s_range[1], above);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < BINS; i += RH_THREADS) {
    const uint32_t c = s_hist[i];
    if (c) atomicAdd(&hist[i], c);
  }
  if (threadIdx.x < 2 && s_range[threadIdx.x]) atomicMax(&range[threadIdx.x], s_range[threadIdx.x]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_flag = (atomicAdd(arrivals, 1u) == gridDim.x - 1u) ? 1u : 0u;
  __syncthreads();
  if (!s_flag) return;
  __threadfence();
  const uint32_t lowest = ROW_HIGHS - ld_volatile_u32(range), highs = ld_volatile_u32(range + 1) - lowest;
  const bool fourth = V != 0 && highs > ROW_RADIX;
  for (int d = 0; d < DIGITS; ++d) {
    const bool owner = threadIdx.x < ROW_RADIX;
    const uint32_t digit = (threadIdx.x + (d == DIGITS - 1 && !fourth ? lowest : 0u)) & (ROW_RADIX - 1);
    const uint32_t h = owner ? ld_volatile_u32(hist + d * ROW_RADIX + digit) : 0u;
    uint32_t total;
    const uint32_t e = odin_block_exclusive_sum(h, s_warp, &total);
    if (owner) base[d * ROW_RADIX + digit] = e;
  }
  if (threadIdx.x == 0 && fourth) *top = 1u;
}

// Lanes of the warp that hold the same digit: a ballot per bit (match.any, the single instruction for this, occupies its pipe
// longer than these sixteen or eighteen).
template <int BITS>
__device__ __forceinline__ uint32_t odin_match_digit(uint32_t d) {
  uint32_t peers = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < BITS; ++b) {
    const uint32_t vote = __ballot_sync(0xffffffffu, (d >> b) & 1u);
    peers &= ((d >> b) & 1u) ? vote : ~vote;
  }
  return peers;
}

// ------------------------------------------------------------------------------------------------ onesweep pass
constexpr int OS_THREADS = 512;                           // threads per block in the passes over the instances
constexpr int OS_ROW_ITEMS = 4;                           // keys per thread in the passes over the rows: a pass is one wave of tiles
                                                          // whose duration is the latency of a tile, so it is spread over many threads
constexpr int OS_INST_ITEMS = SORT_TILE / OS_THREADS;     // 8 in the passes over the instances
// Tiles of 2,048 rows on 512 threads, two per SM, while one wave of them has an SM each; tiles of 4,096 on 1,024 threads for larger
// buffers of rows: half as many predecessors to look back over.  Passes over the rows of a view in all, four of 8-bit digits and
// 2,048 rows / three (and the launch of the fourth) of 2,048 / of 4,096, us: 74 k rows 27 / 25 / 31; 93 k 27 / 25 / -; 328 k rows
// (buffer of 500 k) 42 / 37 / 34; 431 k (1.6 M) 44 / 41 / 36; 819 k (1.25 M) 66 / 61 / 54.  4,096 rows on 512 threads: 48, 52, 57 for
// the last three.  What the fourth pass adds where it is needed: 5 us for 9 k rows, 7 for 74 k, 10 for 328 k, 15 for 819 k; in all four
// passes are never slower than those of 8 bits except for few rows in a large buffer (9 k in 310 k, whole odin_bin_sort 48 -> 54).
static_assert(OS_THREADS >= (int)SORT_RADIX && ROW_SORT_TILE / OS_ROW_ITEMS >= ROW_RADIX, "thread d owns digit d");
constexpr int OS_INST_WINDOW = 6;                 // predecessors fetched per look-back step and digit (instances; with 2 the
                                                  // two passes over 4 M instances took 93.6 us, with 6 91.2)
constexpr int OS_ROW_WINDOW = 8;                  // ... and in the passes over the rows
constexpr int OS_RESIDENT = 1024;               // resident threads per SM
constexpr uint32_t OS_FLAG_AGG = 1u << 30, OS_FLAG_INC = 2u << 30, OS_VALUE = (1u << 30) - 1;
constexpr size_t os_smem_bytes(int items, int threads, bool rows) {  // (the warps' counts of the row passes are of 16 bits)
  const size_t radix = rows ? ROW_RADIX : SORT_RADIX;
  return (size_t)items * threads * 8 + (size_t)(threads / 32) * radix * (rows ? 2 : 4) + 2 * radix * 4 + 16;
}
// What a pass over the rows is told beside its shift.  Where the fourth pass is not needed the third one writes no keys and its
// values to their final place, and the fourth returns at once; otherwise the third counts the fourth's digits and zeroes its
// look-back words.
struct RowPass {
  int pass;
  const uint32_t* top;    // is the fourth pass needed
  uint32_t* final_vals;   // of the third pass
  uint32_t* top_counts;   // [32]
  uint32_t* top_states;
};

// One pass over one digit of 32-bit keys, 8 bits of a tile id or (ROWS) 9 of a row's key.  Persistent blocks take tiles of ITEMS * THREADS keys by ticket.  Per tile:
// warp-striped loads, per-warp digit ranking (stable; a ballot per key and bit), block
// digit counts published for look-back, exclusive global digit offsets by a per-digit look-back walk (thread d walks digit d), keys and values exchanged
// through shared memory so that the global scatter writes runs of consecutive addresses.
//   vals_in == nullptr: the values are the positions themselves (first pass over the rows)
//   keys_out == nullptr: the keys are not needed afterwards (last pass over the rows)
//   WIDE: the last pass over the instances may also write the full 64-bit key key << 32 | depth_bits[value]
//   the number of keys is *count32 if given, else min(*count64, capacity)
//   ITEMS keys per thread on THREADS threads: 8 x 512 for the instances, 4 x 512 or 1,024 for the rows, of which there are so few
//   that a pass is one wave of blocks and its duration is the latency of one tile (with 256 threads per tile the
//   ITEMS-long ranking chain and the write-out were twice as long: whole step 0.870 -> 0.855 ms at 317 k rows; the two
//   instance passes at 1.9 M instances 0.084 -> 0.075 ms)
template <bool ROWS, bool WIDE, int ITEMS, int WINDOW, int THREADS>
__global__ void __launch_bounds__(THREADS, OS_RESIDENT / THREADS)
onesweep_kernel(const uint32_t* __restrict__ keys_in, const uint32_t* __restrict__ vals_in, uint32_t* __restrict__ keys_out,
                uint32_t* __restrict__ vals_out, uint64_t* __restrict__ keys64_out, const uint32_t* __restrict__ depth_bits,
                const uint32_t* __restrict__ count32, const uint64_t* __restrict__ count64, uint64_t capacity, int shift,
                const uint32_t* __restrict__ digit_base, uint32_t* states, uint32_t* ticket, int* status,
                int spin_limit, uint32_t depth_rows, RowPass rp) {
  constexpr int BITS = ROWS ? ROW_RADIX_BITS : SORT_RADIX_BITS;
  constexpr uint32_t RADIX = 1u << BITS;
  using Count = typename std::conditional<ROWS, uint16_t, uint32_t>::type;  // of a digit's keys in a warp, and in front of one in a tile
  static_assert(!ROWS || ITEMS * THREADS < 65536, "counts of 16 bits");
  odin_after_predecessor();  // launched behind the histogram / the pass in front
  __shared__ uint32_t s_top[ROWS ? 1 << ROW_TOP_BITS : 1];  // third pass: counts of the fourth's digits; fourth: where they begin
  bool count_top = false;
  if (ROWS && rp.pass >= 2) {
    const bool fourth = *rp.top != 0u;
    if (rp.pass == 3 && !fourth) return;
    if (rp.pass == 2 && !fourth) { keys_out = nullptr; vals_out = rp.final_vals; }
    count_top = rp.pass == 2 && fourth;
    if (threadIdx.x < (1u << ROW_TOP_BITS)) {
      uint32_t c = 0;
      if (rp.pass == 3) {
        const uint32_t mine = rp.top_counts[threadIdx.x];
        c = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t x = __shfl_up_sync(0xffffffffu, c, o);
          if ((int)threadIdx.x >= o) c += x;
        }
        c -= mine;
      }
      s_top[threadIdx.x] = c;
    }
  }
  extern __shared__ __align__(16) unsigned char os_smem[];
  uint32_t* s_keys = reinterpret_cast<uint32_t*>(os_smem);
  constexpr uint32_t TILE = (uint32_t)ITEMS * THREADS;
  constexpr int OS_WARPS = THREADS / 32;
  const bool owner = threadIdx.x < RADIX;  // thread d owns digit d; the threads beyond the radix own none
  uint32_t* s_vals = s_keys + TILE;
  Count(*s_warp_hist)[RADIX] = reinterpret_cast<Count(*)[RADIX]>(s_vals + TILE);
  uint32_t* s_digit_start = reinterpret_cast<uint32_t*>(&s_warp_hist[0][0] + OS_WARPS * RADIX);
  uint32_t* s_global = s_digit_start + RADIX;
  uint32_t* s_misc = s_global + RADIX;  // [0] tile ticket
  __shared__ uint32_t s_scan[33];

  uint64_t M64;
  if (count32) {
    M64 = *count32;
  } else {
    const uint64_t M_all = *count64;
    M64 = M_all < capacity ? M_all : capacity;
  }
  const uint32_t M = (uint32_t)(M64 < (uint64_t)OS_VALUE ? M64 : (uint64_t)OS_VALUE);
  const uint32_t ntiles = (M + TILE - 1) / TILE;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt_mask = (1u << lane) - 1u;

  // The keys and values of the NEXT tile are requested as soon as the registers of the current one are free (after
  // the exchange through shared memory), so that their latency overlaps the global scatter of the current tile.
  uint32_t key[ITEMS];
  uint32_t val[ITEMS];
  auto load_tile = [&](uint32_t t) {
    const uint32_t wb = t * TILE + warp * (32 * ITEMS);
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const uint32_t i = wb + 32 * j + lane;
      const bool in = t < ntiles && i < M;
      key[j] = in ? keys_in[i] : ~0u;  // padding sorts to the end of the tile and is never written
      val[j] = in ? (vals_in ? vals_in[i] : i) : 0u;
    }
  };
  auto digit = [&](uint32_t k) -> uint32_t { return (k >> shift) & (RADIX - 1); };
  if (threadIdx.x == 0) s_misc[0] = atomicAdd(ticket, 1u);
  __syncthreads();
  uint32_t tile = s_misc[0];
  load_tile(tile);

  while (tile < ntiles) {
    for (int i = threadIdx.x; i < OS_WARPS * (int)RADIX * (int)sizeof(Count) / 4; i += THREADS) reinterpret_cast<uint32_t*>(s_warp_hist)[i] = 0;
    __syncthreads();
    const uint32_t tile_base = tile * TILE;
    const uint32_t tile_count = min(TILE, M - tile_base);

    if (ROWS && count_top) {  // (uniform; rare)
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) {
        const bool in = warp * (32 * ITEMS) + 32 * j + lane < tile_count;
        const uint32_t d = key[j] >> ROW_TOP_SHIFT, peers = __match_any_sync(0xffffffffu, in ? d : ~0u);
        if (in && (int)lane == __ffs(peers) - 1) atomicAdd(&s_top[d], (uint32_t)__popc(peers));
      }
      if (owner) rp.top_states[(size_t)tile * RADIX + threadIdx.x] = 0u;
    }
    uint32_t pos[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const uint32_t d = digit(key[j]);
      // (measured: ballots 0.060 against 0.064 ms with match.any for the four row passes at 317 k rows; no difference
      // in the passes over 1.9 M instances)
      const uint32_t peers = odin_match_digit<BITS>(d);
      const int leader = __ffs(peers) - 1;
      uint32_t old = 0;
      if ((int)lane == leader) {
        old = s_warp_hist[warp][d];
        s_warp_hist[warp][d] = (Count)(old + __popc(peers));
      }
      old = __shfl_sync(0xffffffffu, old, leader);
      pos[j] = old + __popc(peers & lt_mask);
      __syncwarp();
    }
    __syncthreads();

    // exclusive offsets of the warps inside the thread's digit, block totals published
    const uint32_t d = threadIdx.x;
    uint32_t cta_count = 0;
    if (owner) {
#pragma unroll
      for (int w = 0; w < OS_WARPS; ++w) {
        const uint32_t t = s_warp_hist[w][d];
        s_warp_hist[w][d] = (Count)cta_count;
        cta_count += t;
      }
      st_volatile_u32(states + (size_t)tile * RADIX + d, (tile == 0 ? OS_FLAG_INC : OS_FLAG_AGG) | cta_count);
    }
    uint32_t total;
    const uint32_t digit_start = odin_block_exclusive_sum(cta_count, s_scan, &total);
    if (owner) s_digit_start[d] = digit_start;
    uint32_t exclusive = 0;
    if (tile > 0 && owner) {
      // walk back over the predecessors
      int64_t t = (int64_t)tile - 1;
      int spins = 0;
      while (t >= 0) {
        bool stalled = true;  // cleared as soon as any predecessor word is consumed
        // a window of WINDOW predecessors is fetched at once: the walk is a chain of dependent L2 round
        // trips, and when a launch starts every resident tile has hundreds of aggregates in front of it
        uint32_t s[WINDOW];
#pragma unroll
        for (int k = 0; k < WINDOW; ++k) s[k] = t - k >= 0 ? ld_volatile_u32(states + (size_t)(t - k) * RADIX + d) : 0u;
#pragma unroll
        for (int k = 0; k < WINDOW; ++k) {
          if (t < 0) break;
          const uint32_t flag = s[k] >> 30;
          if (flag == 0) break;  // not published yet: use what precedes it, come back
          exclusive += s[k] & OS_VALUE;
          t = flag == 2 ? -1 : t - 1;
          stalled = false;
        }
        if (t >= 0 && stalled) {
          __nanosleep(32);
          if (++spins > spin_limit) { odin_set_error(status, ODIN_ERR_TIMEOUT); break; }
        }
      }
      st_volatile_u32(states + (size_t)tile * RADIX + d, OS_FLAG_INC | ((exclusive + cta_count) & OS_VALUE));
    }
    const uint32_t first = ROWS && rp.pass == 3 ? s_top[d & ((1u << ROW_TOP_BITS) - 1u)] : owner ? digit_base[d] : 0u;
    if (owner) s_global[d] = first + exclusive - digit_start;  // + slot index inside the tile = address
    __syncthreads();

#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const uint32_t dg = digit(key[j]);
      const uint32_t slot = s_digit_start[dg] + s_warp_hist[warp][dg] + pos[j];
      s_keys[slot] = key[j];
      s_vals[slot] = val[j];
    }
    if (threadIdx.x == 0) s_misc[0] = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t next = s_misc[0];
    load_tile(next);  // in flight while the current tile is written out
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const uint32_t slot = j * THREADS + threadIdx.x;
      if (slot < tile_count) {
        const uint32_t k = s_keys[slot];
        const uint32_t dst = s_global[digit(k)] + slot;
        if (dst < M) {
          const uint32_t v = s_vals[slot];
          if (keys_out) keys_out[dst] = k;
          vals_out[dst] = v;
          if (WIDE) {
            // (depth_rows: length of depth_bits; the clamp only matters for a list that an earlier timed-out pass left
            // partly unwritten)
            if (keys64_out) keys64_out[dst] = ((uint64_t)k << 32) | (uint64_t)depth_bits[min(v, depth_rows - 1)];
          }
        }
      }
    }
    tile = next;
    __syncthreads();
  }
  if (ROWS && count_top && threadIdx.x < (1u << ROW_TOP_BITS) && s_top[threadIdx.x])
    atomicAdd(&rp.top_counts[threadIdx.x], s_top[threadIdx.x]);
}

// ------------------------------------------------------------------------------------------------ few rows
// All passes over the rows at once, by one block in shared memory, where the buffers hold no more rows than fit: histogram and
// four passes are five launches of about 6 us however few rows there are (1,000 rows: 45 -> 13 us).  By the capacity of the row
// buffer, which the host knows, not by the rows in it.  Whole odin_bin_sort with five launches / one block: 256 rows
// 50 / 36 us, 1,024 74 / 60, 4,096 124 / 108, 8,192 123 / 120.  What bounds it: the one SM's barriers and shared memory (44 % of
// its issue slots).
// Position p of the list lies with warp p / (32 items), its load p / 32 % items, lane p % 32, so that the ranks are stable.
constexpr uint32_t ROW_SORT_SMALL = 8192;
constexpr int RS_THREADS = 1024, RS_WARPS = RS_THREADS / 32, RS_ITEMS = ROW_SORT_SMALL / RS_THREADS;
constexpr size_t RS_SMEM = (size_t)ROW_SORT_SMALL * 8 + (size_t)(RS_WARPS + 1) * SORT_RADIX * 4;

__global__ void __launch_bounds__(RS_THREADS, 1)
row_sort_small_kernel(const uint32_t* __restrict__ depth_bits, const uint32_t* __restrict__ num_rows, uint32_t capacity,
                      uint32_t* __restrict__ sorted_row) {
  extern __shared__ __align__(16) unsigned char rs_smem[];
  uint32_t* s_keys = reinterpret_cast<uint32_t*>(rs_smem);
  uint32_t* s_vals = s_keys + ROW_SORT_SMALL;
  uint32_t(*s_hist)[SORT_RADIX] = reinterpret_cast<uint32_t(*)[SORT_RADIX]>(s_vals + ROW_SORT_SMALL);
  uint32_t* s_start = &s_hist[0][0] + RS_WARPS * SORT_RADIX;
  __shared__ uint32_t s_scan[33];
  odin_after_predecessor();
  const uint32_t V = min(min(*num_rows, capacity), ROW_SORT_SMALL);
  if (V == 0) return;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt_mask = (1u << lane) - 1u;
  const int items = (int)((V + RS_THREADS - 1) / RS_THREADS);
  const uint32_t first = warp * 32 * items + lane;  // + 32 j
  uint32_t key[RS_ITEMS], val[RS_ITEMS], pos[RS_ITEMS];
#pragma unroll
  for (int j = 0; j < RS_ITEMS; ++j) {
    const uint32_t i = first + 32 * j;
    const bool in = j < items && i < V;
    key[j] = in ? depth_bits[i] : ~0u;  // (the positions behind the last row sort to the end and stay there)
    val[j] = i;
  }
  for (int shift = 0; shift < 32; shift += (int)SORT_RADIX_BITS) {
    for (int i = threadIdx.x; i < RS_WARPS * (int)SORT_RADIX; i += RS_THREADS) (&s_hist[0][0])[i] = 0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < RS_ITEMS; ++j) {
      if (j >= items) break;
      const uint32_t d = (key[j] >> shift) & (SORT_RADIX - 1), peers = odin_match_digit<SORT_RADIX_BITS>(d);
      const int leader = __ffs(peers) - 1;
      uint32_t old = 0;
      if ((int)lane == leader) {
        old = s_hist[warp][d];
        s_hist[warp][d] = old + __popc(peers);
      }
      old = __shfl_sync(0xffffffffu, old, leader);
      pos[j] = old + __popc(peers & lt_mask);
      __syncwarp();
    }
    __syncthreads();
    uint32_t c = 0;
    if (threadIdx.x < SORT_RADIX) {  // thread d: the warps' offsets inside digit d, and its count
#pragma unroll
      for (int w = 0; w < RS_WARPS; ++w) {
        const uint32_t t = s_hist[w][threadIdx.x];
        s_hist[w][threadIdx.x] = c;
        c += t;
      }
    }
    uint32_t total;
    const uint32_t start = odin_block_exclusive_sum(c, s_scan, &total);
    if (threadIdx.x < SORT_RADIX) s_start[threadIdx.x] = start;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < RS_ITEMS; ++j) {
      if (j >= items) break;
      const uint32_t d = (key[j] >> shift) & (SORT_RADIX - 1), slot = s_start[d] + s_hist[warp][d] + pos[j];
      s_keys[slot] = key[j];
      s_vals[slot] = val[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < RS_ITEMS; ++j) {
      if (j >= items) break;
      key[j] = s_keys[first + 32 * j];
      val[j] = s_vals[first + 32 * j];
    }
  }
#pragma unroll
  for (int j = 0; j < RS_ITEMS; ++j)
    if (j < items && first + 32 * j < V) sorted_row[first + 32 * j] = val[j];
}

// ------------------------------------------------------------------------------------------------ sorted offsets
// sorted_off[i] = number of instances of the rows in front of position i of the depth order: an exclusive scan of the
// rectangles' tile counts gathered through sorted_row.  2048 positions per block, one decoupled look-back per block,
// blocks ordered by ticket.
constexpr int RO_THREADS = 1024;
constexpr int RO_ITEMS = OFFSET_TILE / RO_THREADS;
// the instances are emitted in chunks of DUP_CHUNK consecutive slots (emit_instances_kernel)
constexpr int DUP_THREADS = 256;
constexpr int DUP_ITEMS = 8;
constexpr int DUP_CHUNK = DUP_THREADS * DUP_ITEMS;  // a chunk spans at most DUP_CHUNK rows

//
// The same kernel counts the instances per tile without touching a single instance: one tile row of a rectangle is a
// run of consecutive tile ids [t0, t1), which adds 1 at t0 and subtracts 1 at t1 in a difference array over the tile
// ids; tile_scan_block integrates it.  Only the first `capacity` instances of the depth order count.
// It also fills chunk_row[c] = the position (in depth order) of the row whose slots contain slot c * DUP_CHUNK: a row
// writes an entry for every chunk boundary that falls inside its slot range (usually none or one).
__global__ void __launch_bounds__(RO_THREADS)
sorted_offsets_kernel(const uint32_t* __restrict__ sorted_row, const ushort4* __restrict__ rect,
                      const uint32_t* __restrict__ num_rows, uint32_t capacity, int TX, uint32_t* __restrict__ sorted_off,
                      uint32_t* __restrict__ chunk_row, uint32_t chunks_cap, uint32_t* __restrict__ tile_diff,
                      uint32_t diff_words, uint32_t* ticket, uint64_t* state, int* status, int spin_limit) {
  // diff_words != 0: the block first accumulates its part of the difference array in shared memory (`diff_words` =
  // tiles + 1 words of dynamic shared memory) and adds the non-zero words to the global one at the end: a tile on which
  // thousands of rectangles pile up would otherwise serialise that many global reductions on one address.
  extern __shared__ uint32_t s_tdiff[];
  __shared__ uint32_t s_tile, s_base;
  __shared__ uint32_t s_warp[33];
  // (in front of the wait: the counter was zeroed further back than by the kernel in front)
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
  for (uint32_t i = threadIdx.x; i < diff_words; i += RO_THREADS) s_tdiff[i] = 0;
  odin_after_predecessor();
  const uint32_t V = *num_rows;
  const uint32_t ntiles = (V + OFFSET_TILE - 1) / OFFSET_TILE;
  __syncthreads();
  const uint32_t tile = s_tile;
  if (tile >= ntiles) return;  // uniform over the block; nobody waits for a tile past the end
  const uint32_t first = tile * OFFSET_TILE + threadIdx.x * RO_ITEMS;
  ushort4 rc[RO_ITEMS];
  uint32_t cnt[RO_ITEMS];
  uint32_t sum = 0;  // sums are taken modulo 2^32; the true totals fit (M >= 2^32 is an error raised by the projection)
#pragma unroll
  for (int k = 0; k < RO_ITEMS; ++k) {
    rc[k] = make_ushort4(0, 0, 0, 0);
    // (a row id is clamped to the rows of this view: it stays in range even if a pass of the row sort gave up and left
    // part of its output unwritten)
    if (first + k < V) rc[k] = rect[min(sorted_row[first + k], V - 1)];
    cnt[k] = ((uint32_t)rc[k].z - (uint32_t)rc[k].x) * ((uint32_t)rc[k].w - (uint32_t)rc[k].y);
    sum += cnt[k];
  }
  uint32_t total;
  const uint32_t before = odin_block_exclusive_sum(sum, s_warp, &total);
  if (threadIdx.x < 32) {
    const uint64_t b = odin_lookback_u64(state, tile, (uint64_t)total, status, spin_limit);
    if (threadIdx.x == 0) s_base = (uint32_t)b;
  }
  __syncthreads();
  uint32_t run = s_base + before;
#pragma unroll
  for (int k = 0; k < RO_ITEMS; ++k) {
    if (first + k < V) {
      sorted_off[first + k] = run;
      const uint64_t hi = (uint64_t)run + cnt[k];
      for (uint64_t c = ((uint64_t)run + DUP_CHUNK - 1) / DUP_CHUNK; c * DUP_CHUNK < hi && c < chunks_cap; ++c)
        chunk_row[c] = first + k;
    }
    // instances of this row that are emitted: those in front of the capacity
    uint32_t left = run < capacity ? min(cnt[k], capacity - run) : 0u;
    const uint32_t w = (uint32_t)rc[k].z - (uint32_t)rc[k].x;
    for (uint32_t y = rc[k].y; left != 0; ++y) {
      const uint32_t len = min(w, left);
      left -= len;
      const uint32_t t0 = y * (uint32_t)TX + (uint32_t)rc[k].x;
      uint32_t* diff = diff_words ? s_tdiff : tile_diff;
      atomicAdd(&diff[t0], 1u);
      atomicSub(&diff[t0 + len], 1u);
    }
    run += cnt[k];
  }
  if (diff_words) {
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < diff_words; i += RO_THREADS) {
      const uint32_t d = s_tdiff[i];
      if (d) atomicAdd(&tile_diff[i], d);
    }
  }
}

// Run by ONE block (all of its threads).  Integrates the difference array into the instance count of every tile (sums
// modulo 2^32; every prefix is a true count), writes the tile ranges [first, one past last) as the exclusive scan of
// the counts, and builds the digit histograms of the instances' tile ids and their exclusive scans (the digit bases of
// the instance passes).  Needs blockDim.x >= 256.
constexpr int TS_ITEMS = 4;

__device__ __forceinline__ void tile_scan_block(const uint32_t* __restrict__ tile_diff, uint32_t n_tiles, int tile_passes,
                                                uint32_t* __restrict__ ranges, uint32_t* __restrict__ base, uint32_t cap) {
  __shared__ uint32_t s_h[SORT_MAX_TILE_DIGITS][SORT_RADIX];
  __shared__ uint32_t s_warp[33];
  const unsigned lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < SORT_MAX_TILE_DIGITS * (int)SORT_RADIX; i += blockDim.x) (&s_h[0][0])[i] = 0;
  __syncthreads();
  uint32_t carry_count = 0, carry_off = 0;  // count of the tile in front of the batch; instances in front of the batch
  for (uint32_t b0 = 0; b0 < n_tiles; b0 += blockDim.x * TS_ITEMS) {
    const uint32_t t0 = b0 + threadIdx.x * TS_ITEMS;
    uint32_t c[TS_ITEMS];
    uint32_t run = 0;
#pragma unroll
    for (int k = 0; k < TS_ITEMS; ++k) {
      run += (t0 + k < n_tiles) ? tile_diff[t0 + k] : 0u;
      c[k] = run;  // inclusive prefix of the differences inside the thread
    }
    uint32_t total;
    const uint32_t before = carry_count + odin_block_exclusive_sum(run, s_warp, &total);
    uint32_t mine = 0;
#pragma unroll
    for (int k = 0; k < TS_ITEMS; ++k) {
      c[k] = (t0 + k < n_tiles) ? c[k] + before : 0u;  // instances of tile t0 + k
      mine += c[k];
    }
    carry_count += total;
    uint32_t total2;
    uint32_t off = carry_off + odin_block_exclusive_sum(mine, s_warp, &total2);
    carry_off += total2;
#pragma unroll
    for (int k = 0; k < TS_ITEMS; ++k) {
      const uint32_t t = t0 + k;
      if (t < n_tiles) {
        // never beyond the instance capacity (the counts already respect it unless a look-back gave up)
        reinterpret_cast<uint2*>(ranges)[t] = make_uint2(min(off, cap), min(off + c[k], cap));
        if (c[k]) atomicAdd(&s_h[0][t & (SORT_RADIX - 1)], c[k]);
        off += c[k];
      }
    }
    // higher digits: the 128 consecutive tiles of a warp share the digit unless they straddle a multiple of 256 (or
    // 65536), so the warp adds its sum once instead of 128 times to the same word
    for (int d = 1; d < tile_passes; ++d) {
      const int shift = (int)SORT_RADIX_BITS * d;
      const uint32_t first = __shfl_sync(0xffffffffu, t0, 0), last = __shfl_sync(0xffffffffu, t0 + TS_ITEMS - 1, 31);
      if ((first >> shift) == (last >> shift)) {
        const uint32_t sum = __reduce_add_sync(0xffffffffu, mine);
        if (lane == 0 && sum) atomicAdd(&s_h[d][(first >> shift) & (SORT_RADIX - 1)], sum);
      } else {
#pragma unroll
        for (int k = 0; k < TS_ITEMS; ++k)
          if (c[k]) atomicAdd(&s_h[d][((t0 + k) >> shift) & (SORT_RADIX - 1)], c[k]);
      }
    }
  }
  __syncthreads();
  for (int d = 0; d < tile_passes; ++d) {
    const uint32_t h = threadIdx.x < SORT_RADIX ? s_h[d][threadIdx.x] : 0u;
    uint32_t total;
    const uint32_t e = odin_block_exclusive_sum(h, s_warp, &total);
    if (threadIdx.x < SORT_RADIX) base[d * SORT_RADIX + threadIdx.x] = e;
  }
}

// ------------------------------------------------------------------------------------------------ emission

// Cooperative 256-ary upper bound: first r in [0, V) with off[r] > x (V if none).  All threads must call.
__device__ __forceinline__ uint32_t block_upper_bound(const uint32_t* __restrict__ off, uint32_t V, uint32_t x) {
  uint32_t lo = 0, hi = V;
  while (lo < hi) {
    const uint32_t span = hi - lo;
    const uint32_t step = (span + DUP_THREADS - 1) / DUP_THREADS;
    const uint32_t probe = lo + threadIdx.x * step;
    const int below = (probe < hi) && (off[probe] <= x);
    const uint32_t cnt = (uint32_t)__syncthreads_count(below);  // monotone predicate: the first cnt probes are <= x
    if (cnt == 0) { hi = lo; break; }
    const uint32_t new_lo = lo + (cnt - 1) * step + 1;
    const uint32_t new_hi = min(hi, lo + cnt * step);
    lo = new_lo; hi = new_hi;
  }
  return lo;
}

// Each chunk of DUP_CHUNK consecutive instance slots finds the positions of the depth order it overlaps, stages their
// offsets, row ids and rectangles in shared memory, and every thread expands its slots: slot i of a row is tile
// (y0 + k / w, x0 + k % w) with k = i - offset, w = x1 - x0.  Keys (tile ids) and values (row ids) are written fully
// coalesced.  The last block of the grid does something else at the same time: the scan over the tiles (ranges and
// digit bases), which is one block's work and would otherwise be a launch of its own on the critical path.
__global__ void __launch_bounds__(DUP_THREADS)
emit_instances_kernel(const uint32_t* __restrict__ sorted_off, const uint32_t* __restrict__ sorted_row,
                      const uint32_t* __restrict__ chunk_row, const ushort4* __restrict__ rect,
                      const uint32_t* __restrict__ num_rows, const uint64_t* __restrict__ num_instances, uint64_t capacity,
                      int TX, uint32_t* __restrict__ keys, uint32_t* __restrict__ vals, int* status,
                      const uint32_t* __restrict__ tile_diff, uint32_t n_tiles, int tile_passes,
                      uint32_t* __restrict__ ranges, uint32_t* __restrict__ tile_dbase) {
  odin_after_predecessor();
  if (blockIdx.x == 0) {  // block 0: it is scheduled first
    tile_scan_block(tile_diff, n_tiles, tile_passes, ranges, tile_dbase,
                    (uint32_t)(capacity < 0xffffffffull ? capacity : 0xffffffffull));
    return;
  }
  const uint32_t emit_blocks = gridDim.x - 1, emit_block = blockIdx.x - 1;
  __shared__ uint32_t s_off[DUP_CHUNK + 1];
  __shared__ ushort4 s_rect[DUP_CHUNK];
  __shared__ uint32_t s_row[DUP_CHUNK];
  __shared__ __align__(16) uint16_t s_map[DUP_CHUNK];  // slot of the chunk -> staged row of the chunk
  __shared__ uint32_t s_scan[DUP_THREADS / 32];
  const uint32_t V = *num_rows;
  const uint64_t M_all = *num_instances;
  const uint64_t M64 = M_all < capacity ? M_all : capacity;
  if (emit_block == 0 && threadIdx.x == 0 && M_all > capacity) odin_set_error(status, ODIN_ERR_CAPACITY);
  const uint32_t M = (uint32_t)(M64 < 0xffffffffull ? M64 : 0xffffffffull);
  const uint32_t chunks = V == 0 ? 0u : (M + DUP_CHUNK - 1) / DUP_CHUNK;
  const unsigned lane = threadIdx.x & 31;
  for (uint32_t chunk = emit_block; chunk < chunks; chunk += emit_blocks) {
    const uint32_t c0 = chunk * DUP_CHUNK;
    const uint32_t c1 = (M - c0 < (uint32_t)DUP_CHUNK) ? M : c0 + DUP_CHUNK;
    // first and last position of the chunk from the chunk table; only the last chunk has to search for its end
    // (every index taken from the tables is clamped: if a look-back gave up, parts of them were never written, and
    // the emission must still stay inside its buffers; with intact tables the clamps change nothing)
    const uint32_t row_lo = min(chunk_row[chunk], V - 1);
    uint32_t row_hi;
    if (chunk + 1 < chunks) {
      const uint32_t rn = min(chunk_row[chunk + 1], V - 1);  // position that holds slot c1
      row_hi = (sorted_off[rn] == c1 && rn > 0) ? rn - 1 : rn;
    } else {
      row_hi = max(block_upper_bound(sorted_off, V, c1 - 1), 1u) - 1;  // offset[0] = 0, so the bound is >= 1
    }
    row_hi = min(max(row_hi, row_lo), row_lo + (uint32_t)DUP_CHUNK - 1);
    const uint32_t nrows = row_hi - row_lo + 1;  // <= DUP_CHUNK: every row owns at least one slot
    for (uint32_t i = threadIdx.x; i < nrows; i += DUP_THREADS) {
      const uint32_t r = min(sorted_row[row_lo + i], V - 1);
      s_off[i] = sorted_off[row_lo + i];
      s_row[i] = r;
      s_rect[i] = rect[r];
    }
    if (threadIdx.x == 0) s_off[nrows] = (row_hi + 1 < V) ? sorted_off[row_hi + 1] : (uint32_t)M_all;
    for (int i = threadIdx.x; i < DUP_CHUNK; i += DUP_THREADS) s_map[i] = 0;
    __syncthreads();
    // slot -> staged row: every row marks its first slot, an inclusive max-scan fills the rest
    for (uint32_t i = threadIdx.x; i < nrows; i += DUP_THREADS)
      s_map[min(max(s_off[i], c0) - c0, (uint32_t)DUP_CHUNK - 1)] = (uint16_t)i;
    __syncthreads();
    {
      static_assert(DUP_ITEMS == 8, "a thread's slots are one 16-byte word of the map");
      uint4* map4 = reinterpret_cast<uint4*>(s_map) + threadIdx.x;
      const uint4 raw = *map4;
      const uint32_t rw[4] = {raw.x, raw.y, raw.z, raw.w};
      uint32_t m[DUP_ITEMS];
      uint32_t run = 0;
#pragma unroll
      for (int k = 0; k < DUP_ITEMS; ++k) {
        run = max(run, (rw[k >> 1] >> (16 * (k & 1))) & 0xffffu);
        m[k] = run;
      }
      uint32_t inc = run;  // inclusive max over the threads of the warp (values >= 0, so 0 is neutral)
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o, 32);
        if (lane >= (unsigned)o) inc = max(inc, y);
      }
      if (lane == 31) s_scan[threadIdx.x >> 5] = inc;
      __syncthreads();
      uint32_t before = __shfl_up_sync(0xffffffffu, inc, 1);
      if (lane == 0) before = 0;
      for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) before = max(before, s_scan[w]);
#pragma unroll
      for (int k = 0; k < DUP_ITEMS; ++k) m[k] = max(m[k], before);
      *map4 = make_uint4(m[0] | (m[1] << 16), m[2] | (m[3] << 16), m[4] | (m[5] << 16), m[6] | (m[7] << 16));
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < DUP_ITEMS; ++k) {
      const uint32_t i = c0 + k * DUP_THREADS + threadIdx.x;
      if (i < c1) {
        const uint32_t lo = s_map[i - c0];  // staged row that owns this slot
        const ushort4 rc = s_rect[lo];
        const uint32_t local = i - s_off[lo];
        const uint32_t w = (uint32_t)rc.z - (uint32_t)rc.x;
        const uint32_t dy = local / w, dx = local - dy * w;
        keys[i] = ((uint32_t)rc.y + dy) * (uint32_t)TX + (uint32_t)rc.x + dx;
        vals[i] = s_row[lo];
      }
    }
    __syncthreads();
  }
}


// ------------------------------------------------------------------------------------------------ counting scatter
// The instances never need a sort of their own.  With the rows in depth order, the list of a tile is the subsequence of
// rows whose rectangle covers it, so the final position of an instance is
//     first position of the tile + instances of the tile in earlier chunks of rows + rank of the row inside its chunk,
// and all three are cheap: the rectangles give the per-(chunk, tile) counts through a difference array (one block per
// chunk of OFFSET_TILE sorted rows), a scan over the chunks and one over the tiles give the first positions, and the
// rank inside a chunk is the order in which a lane per tile walks the chunk's rows (exact binning: set bits of a bit matrix, tile x
// row, in shared memory, read off in row order).  Three launches that together move 8V + 4M bytes plus the counters, against emission + two radix passes over
// 8-byte instances.

// One block per chunk, blocks ordered by ticket.  Writes the rectangles in depth order and the chunk's instance count for every
// tile.  The running instance offset is only needed for the capacity rule (the instances in front of `capacity` in depth order are
// the ones that exist), so only a view with more instances than that looks back
// for it and writes sorted_off.  (Looked back for in every view the kernel took 13.5 instead of 11.7 us for 328 k rows, 38 instead of 34 for 819 k.)
// EXACT (binning 2): a row's instances are the kept spans of its rectangle's tile rows (tilespan.cuh), recomputed here
// from the row's centre, conic and opacity, which are also written out in depth order for the scatter kernel.
// THREADS x ITEMS = OFFSET_TILE rows per block.
template <bool EXACT, int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS)
chunk_counts_kernel(const uint32_t* __restrict__ sorted_row, const ushort4* __restrict__ rect,
                    const float2* __restrict__ xy, const float4* __restrict__ conic_o, float alpha_min,
                    const uint32_t* __restrict__ num_rows, const uint64_t* __restrict__ num_instances, uint32_t capacity,
                    int TX, uint32_t n_tiles, uint32_t tiles_pad, uint32_t* __restrict__ sorted_off,
                    ushort4* __restrict__ sorted_rect, float4* __restrict__ sorted_geo4, float2* __restrict__ sorted_geo2,
                    uint32_t* __restrict__ counts, uint32_t* ticket, uint64_t* state, int* status, int spin_limit) {
  extern __shared__ __align__(16) uint32_t s_tdiff[];  // tiles_pad + 8 words
  __shared__ uint32_t s_tile, s_base;
  __shared__ uint32_t s_warp[33];
  // (in front of the wait: the counter was zeroed further back than by the kernel in front)
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
  for (uint32_t i = threadIdx.x; i < tiles_pad + 8; i += THREADS) s_tdiff[i] = 0;
  odin_after_predecessor();
  const uint32_t V = *num_rows;
  const uint32_t ntiles = (V + OFFSET_TILE - 1) / OFFSET_TILE;
  __syncthreads();
  const uint32_t tile = s_tile;
  if (tile >= ntiles) return;  // uniform over the block; nobody waits for a chunk past the end
  // only when the view has more instances than the caller's capacity can a row be denied some of its instances (those
  // at or behind `capacity` in depth order); otherwise the counts do not depend on the running offset
  const bool cut = *num_instances > (uint64_t)capacity;
  const uint32_t first = tile * OFFSET_TILE + threadIdx.x * ITEMS;
  ushort4 rc[ITEMS];
  uint32_t cnt[ITEMS];
  uint32_t sum = 0;
  // adds the run of tiles [t0, t0 + len) to the difference array
  auto add_run = [&](uint32_t t0, uint32_t len) {
    t0 = min(t0, n_tiles);  // (clamps: see emit_instances_kernel)
    atomicAdd(&s_tdiff[t0], 1u);
    atomicSub(&s_tdiff[min(t0 + len, n_tiles)], 1u);
  };
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    rc[k] = make_ushort4(0, 0, 0, 0);
    cnt[k] = 0;
    SpanConic e;
    e.k = -1.f;
    if (first + k < V) {
      const uint32_t r = min(sorted_row[first + k], V - 1);
      rc[k] = rect[r];
      if (EXACT) {
        const float2 c = xy[r];
        const float4 q = conic_o[r];
        e = odin_span_conic(c.x, c.y, q.x, q.y, q.z, q.w, alpha_min);
        sorted_geo4[first + k] = make_float4(e.u, e.v, e.A, e.B);
        sorted_geo2[first + k] = make_float2(e.C, e.k);
      } else {
        cnt[k] = ((uint32_t)rc[k].z - (uint32_t)rc[k].x) * ((uint32_t)rc[k].w - (uint32_t)rc[k].y);
      }
    }
    if (EXACT) {
      // a lane walks the tile rows of a low rectangle by itself; the tall rectangles of the warp are walked by all 32
      // lanes together (one tile row per lane and step)
      const int h = (int)rc[k].w - (int)rc[k].y;
      const bool tall = h > 4;
      if (h > 0 && !tall)
        for (int y = rc[k].y; y < (int)rc[k].w; ++y) {
          int xa, xb;
          odin_row_span(e, y, rc[k].x, rc[k].z, xa, xb);
          if (xb > xa) {
            cnt[k] += (uint32_t)(xb - xa);
            if (!cut) add_run((uint32_t)y * (uint32_t)TX + (uint32_t)xa, (uint32_t)(xb - xa));
          }
        }
      uint32_t todo = __ballot_sync(0xffffffffu, tall);
      while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const SpanConic q = odin_span_conic_bcast(e, src);
        const int qx0 = __shfl_sync(0xffffffffu, (int)rc[k].x, src), qy0 = __shfl_sync(0xffffffffu, (int)rc[k].y, src);
        const int qx1 = __shfl_sync(0xffffffffu, (int)rc[k].z, src), qy1 = __shfl_sync(0xffffffffu, (int)rc[k].w, src);
        uint32_t kept = 0;
        for (int y = qy0 + (int)(threadIdx.x & 31); y < qy1; y += 32) {
          int xa, xb;
          odin_row_span(q, y, qx0, qx1, xa, xb);
          if (xb > xa) {
            kept += (uint32_t)(xb - xa);
            if (!cut) add_run((uint32_t)y * (uint32_t)TX + (uint32_t)xa, (uint32_t)(xb - xa));
          }
        }
        kept = __reduce_add_sync(0xffffffffu, kept);
        if ((int)(threadIdx.x & 31) == src) cnt[k] = kept;
      }
    }
    sum += cnt[k];
  }
  uint32_t run = 0;
  if (cut) {
    uint32_t total;
    const uint32_t before = odin_block_exclusive_sum(sum, s_warp, &total);
    if (threadIdx.x < 32) {
      const uint64_t b = odin_lookback_u64(state, tile, (uint64_t)total, status, spin_limit);
      if (threadIdx.x == 0) s_base = (uint32_t)b;
    }
    __syncthreads();
    run = s_base + before;
  }
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    if (first + k < V) {
      if (cut) sorted_off[first + k] = run;
      sorted_rect[first + k] = rc[k];
    }
    if (!EXACT || cut) {
      // the instances of the row that exist: those in front of `capacity`, its tiles taken in row-major order
      uint32_t left = !cut ? cnt[k] : run < capacity ? min(cnt[k], capacity - run) : 0u;
      const uint32_t w = (uint32_t)rc[k].z - (uint32_t)rc[k].x;
      SpanConic e;
      if (EXACT && left != 0) {
        const float4 g4 = sorted_geo4[first + k];  // written above by this thread
        const float2 g2 = sorted_geo2[first + k];
        e.u = g4.x; e.v = g4.y; e.A = g4.z; e.B = g4.w; e.C = g2.x; e.k = g2.y;
      }
      for (uint32_t y = rc[k].y; left != 0 && y < (uint32_t)rc[k].w; ++y) {
        uint32_t x0 = rc[k].x, len = w;
        if (EXACT) {
          int xa, xb;
          odin_row_span(e, (int)y, rc[k].x, rc[k].z, xa, xb);
          x0 = (uint32_t)xa; len = (uint32_t)(xb - xa);
          if (len == 0) continue;
        }
        len = min(len, left);
        left -= len;
        add_run(y * (uint32_t)TX + x0, len);
      }
    }
    run += cnt[k];
  }
  __syncthreads();
  // integrate the difference array: instances of every tile in this chunk
  uint32_t* __restrict__ out = counts + (size_t)tile * tiles_pad;
  uint32_t carry = 0;
  for (uint32_t b0 = 0; b0 < n_tiles; b0 += THREADS * 4) {
    const uint32_t t0 = b0 + threadIdx.x * 4;
    uint4 d = make_uint4(0, 0, 0, 0);
    if (t0 < n_tiles) d = *reinterpret_cast<const uint4*>(s_tdiff + t0);  // padded: words past n_tiles are zero or unused
    const uint32_t c0 = d.x, c1 = c0 + d.y, c2 = c1 + d.z, c3 = c2 + d.w;
    uint32_t tot;
    const uint32_t base = carry + odin_block_exclusive_sum(c3, s_warp, &tot);
    if (t0 + 3 < n_tiles) {
      *reinterpret_cast<uint4*>(out + t0) = make_uint4(c0 + base, c1 + base, c2 + base, c3 + base);
    } else {
      if (t0 < n_tiles) out[t0] = c0 + base;
      if (t0 + 1 < n_tiles) out[t0 + 1] = c1 + base;
      if (t0 + 2 < n_tiles) out[t0 + 2] = c2 + base;
    }
    carry += tot;
  }
}

// counts[c][t] -> exclusive prefix over the chunks c; tile ranges.  A block owns TB_TILES tiles, taken by ticket; its warps split
// the chunks: each warp sums its share, the shares are combined in shared memory, then each warp rewrites its share.  A warp's
// counts of up to TB_HOLD chunks are fetched at once and kept in registers (beyond that in batches of eight, twice).  The first
// position of a block's tiles is the sum over all blocks in front of it, which publish their totals as soon as they have them
// and are read side by side, a thread each, so that nothing is a chain.  What bounds it: those few dependent trips to L2.
// Measured against eight warps that fetched the ragged end of their share one by one, and the block that arrives last scanning
// all totals: 100 x 67 tiles, 160 chunks 15 -> 6 us; 120 x 68, 400 chunks 22 -> 9; 78 x 52, 46 chunks 9.5 -> 4.  32 warps with 16 chunks
// in registers: 10, 11, 5.
constexpr int TB_THREADS = 512;
constexpr int TB_PARTS = TB_THREADS / 32;
constexpr int TB_HOLD = 24;

__global__ void __launch_bounds__(TB_THREADS)
tile_bases_kernel(uint32_t* __restrict__ counts, uint32_t tiles_pad, uint32_t n_tiles, const uint32_t* __restrict__ num_rows,
                  const uint64_t* __restrict__ num_instances, uint64_t capacity, uint64_t* state, uint32_t* __restrict__ ranges,
                  uint32_t* ticket, int* status, int spin_limit) {
  static_assert(TB_TILES == 32, "a lane per tile");
  __shared__ uint32_t s_part[TB_PARTS][32];
  __shared__ uint32_t s_warp[33];
  __shared__ uint32_t s_block;
  // (in front of the wait: the counter was zeroed further back than by the kernel in front)
  if (threadIdx.x == 0) s_block = atomicAdd(ticket, 1u);
  odin_after_predecessor();
  const uint32_t V = *num_rows;
  const uint32_t nchunks = (V + OFFSET_TILE - 1) / OFFSET_TILE;
  const unsigned lane = threadIdx.x & 31, part = threadIdx.x >> 5;
  __syncthreads();
  const uint32_t block = s_block, t = block * TB_TILES + lane;
  const uint32_t per = (nchunks + TB_PARTS - 1) / TB_PARTS;
  const uint32_t c_lo = min(part * per, nchunks), c_hi = t < n_tiles ? min(c_lo + per, nchunks) : 0u;
  uint32_t* __restrict__ col = counts + min(t, n_tiles - 1);
  const bool held = per <= TB_HOLD;
  uint32_t v[TB_HOLD], mine = 0;
  if (held) {
#pragma unroll
    for (int i = 0; i < TB_HOLD; ++i) v[i] = c_lo + i < c_hi ? col[(size_t)(c_lo + i) * tiles_pad] : 0u;
#pragma unroll
    for (int i = 0; i < TB_HOLD; ++i) mine += v[i];
  } else {
    for (uint32_t c = c_lo; c < c_hi; c += 8) {
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = c + i < c_hi ? col[(size_t)(c + i) * tiles_pad] : 0u;
#pragma unroll
      for (int i = 0; i < 8; ++i) mine += v[i];
    }
  }
  s_part[part][lane] = mine;
  __syncthreads();
  uint32_t acc = 0, all = 0;
#pragma unroll
  for (int q = 0; q < TB_PARTS; ++q) {
    const uint32_t x = s_part[q][lane];
    if (q < (int)part) acc += x;
    all += x;
  }
  uint32_t upto = all;  // the block's tiles up to and with the lane's
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, upto, o);
    if ((int)lane >= o) upto += x;
  }
  if (threadIdx.x == 31) st_volatile_u64(state + block, LB64_AGG | upto);
  if (held) {
#pragma unroll
    for (int i = 0; i < TB_HOLD; ++i) {
      if (c_lo + i < c_hi) col[(size_t)(c_lo + i) * tiles_pad] = acc;
      acc += v[i];
    }
  } else {
    for (uint32_t c = c_lo; c < c_hi; c += 8) {
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = c + i < c_hi ? col[(size_t)(c + i) * tiles_pad] : 0u;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (c + i < c_hi) col[(size_t)(c + i) * tiles_pad] = acc;
        acc += v[i];
      }
    }
  }
  // the blocks in front (all of them have started: tickets)
  uint32_t before = 0;
  int spins = 0;
  for (uint32_t b = threadIdx.x; b < block; b += TB_THREADS) {
    uint64_t x;
    while (((x = ld_volatile_u64(state + b)) >> LB64_FLAG_SHIFT) == 0) {
      if (++spins > spin_limit) { odin_set_error(status, ODIN_ERR_TIMEOUT); break; }
      __nanosleep(32);
    }
    before += (uint32_t)(x & LB64_VALUE);
  }
  uint32_t first;
  odin_block_exclusive_sum(before, s_warp, &first);
  if (block == 0 && threadIdx.x == 0 && *num_instances > capacity) odin_set_error(status, ODIN_ERR_CAPACITY);
  const uint32_t cap = (uint32_t)(capacity < 0xffffffffull ? capacity : 0xffffffffull);
  if (part == 0 && t < n_tiles) {
    const uint32_t end = first + upto;
    reinterpret_cast<uint2*>(ranges)[t] = make_uint2(min(end - all, cap), min(end, cap));
  }
}

// Exact binning (binning 2): writes every instance to its final place.  A work item is (chunk of OFFSET_TILE sorted rows, band
// of `band_rows` tile rows); blocks loop over the items.  The rows of the chunk whose rectangle meets the band are compacted in order,
// then handled SC_SUB at a time: every such row sets its bit in the bit vector of each tile it covers inside the band
// (word-major bit matrix [SC_SUB / 32][tiles of the band]), and every tile reads its bits off in order, which is the
// depth order, and writes the row ids behind the position it has reached.
constexpr int SC_THREADS = 256;
constexpr int SC_ITEMS = OFFSET_TILE / SC_THREADS;
constexpr int SC_SUB = 256;
constexpr int SC_WORDS = SC_SUB / 32;
constexpr uint32_t SC_BAND_TILES = SCATTER_MAX_TX;  // tiles of a band: band_rows * TX <= this
// (the rows kept for a band are staged SC_SUB at a time, straight from the registers that hold the chunk's rectangles:
// 32 KB of shared memory per block instead of 64, seven resident blocks instead of three)
constexpr size_t SC_SMEM = (size_t)SC_SUB * (8 + 4 + 4 + 4) + (size_t)SC_WORDS * SC_BAND_TILES * 4 + SC_BAND_TILES * 4;

// The tiles of a row inside a tile row are the kept span (tilespan.cuh), recomputed from the row's centre, conic and
// threshold as chunk_counts_kernel left them in depth order.
template <bool WIDE>
__global__ void __launch_bounds__(SC_THREADS)
scatter_spans_kernel(const ushort4* __restrict__ sorted_rect, const float4* __restrict__ sorted_geo4,
                         const float2* __restrict__ sorted_geo2, const uint32_t* __restrict__ sorted_row,
                         const uint32_t* __restrict__ sorted_off, const uint32_t* __restrict__ num_rows,
                         const uint64_t* __restrict__ num_instances, uint32_t capacity, int TX, int TY, int band_rows,
                         const uint32_t* __restrict__ counts, uint32_t tiles_pad, const uint2* __restrict__ ranges,
                         uint32_t* __restrict__ vals, uint64_t* __restrict__ keys64,
                         const uint32_t* __restrict__ depth_bits, uint32_t* __restrict__ item_ticket) {
  odin_after_predecessor();
  extern __shared__ __align__(16) unsigned char sc_smem[];
  ushort4* s_prect = reinterpret_cast<ushort4*>(sc_smem);                    // [SC_SUB] rectangles of the rows of the batch
  uint32_t* s_prow = reinterpret_cast<uint32_t*>(s_prect + SC_SUB);          // [SC_SUB] their row ids
  uint32_t* s_plim = s_prow + SC_SUB;                                        // [SC_SUB] instances they may emit
  uint32_t* s_pidx = s_plim + SC_SUB;                                        // [SC_SUB] place of the row in its chunk
  uint32_t* s_bits = s_pidx + SC_SUB;                                        // [SC_WORDS][band tiles]
  uint32_t* s_pos = s_bits + SC_WORDS * SC_BAND_TILES;                       // [band tiles] next position of the tile
  __shared__ uint32_t s_warp[33];
  const uint32_t V = *num_rows;
  const uint32_t nchunks = (V + OFFSET_TILE - 1) / OFFSET_TILE;
  const uint32_t nbands = ((uint32_t)TY + band_rows - 1) / band_rows;
  const uint32_t items = nchunks * nbands;
  const bool cut = *num_instances > (uint64_t)capacity;  // only then can a row be denied some of its instances
  __shared__ uint32_t s_item;
  while (true) {
    // items by ticket (they differ in cost by the number of rows of the chunk that meet the band)
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(item_ticket, 1u);
    __syncthreads();
    const uint32_t item = s_item;
    if (item >= items) break;
    const uint32_t chunk = item / nbands, band = item - chunk * nbands;  // neighbouring blocks share a chunk's rows
    const uint32_t by0 = band * band_rows, by1 = min((uint32_t)TY, by0 + band_rows);
    const uint32_t band_tiles = (by1 - by0) * (uint32_t)TX;
    const uint32_t first = chunk * OFFSET_TILE + threadIdx.x * SC_ITEMS;
    ushort4 rc[SC_ITEMS];
    uint32_t keep = 0;
#pragma unroll
    for (int k = 0; k < SC_ITEMS; ++k) {
      rc[k] = make_ushort4(0, 0, 0, 0);
      if (first + k < V) {
        rc[k] = sorted_rect[first + k];
        if ((uint32_t)rc[k].y < by1 && (uint32_t)rc[k].w > by0 && rc[k].z > rc[k].x) keep |= 1u << k;
      }
    }
    uint32_t npass;
    const uint32_t p0 = odin_block_exclusive_sum((uint32_t)__popc(keep), s_warp, &npass);  // (its barriers also fence
    if (npass == 0) continue;                                                             //  the reuse of s_pos; uniform)
    for (uint32_t t = threadIdx.x; t < band_tiles; t += SC_THREADS) {
      const uint32_t tile = by0 * (uint32_t)TX + t;
      s_pos[t] = ranges[tile].x + counts[(size_t)chunk * tiles_pad + tile];
    }
    __syncthreads();
    for (uint32_t sub = 0; sub < npass; sub += SC_SUB) {
      for (uint32_t i = threadIdx.x; i < SC_WORDS * band_tiles; i += SC_THREADS) s_bits[i] = 0;
      {
        // stage the rows of this batch: kept row number p0 + (kept rows of the thread in front of it)
        uint32_t p = p0;
#pragma unroll
        for (int k = 0; k < SC_ITEMS; ++k) {
          if (keep >> k & 1u) {
            if (p >= sub && p < sub + SC_SUB) {
              const uint32_t q = p - sub;
              s_prect[q] = rc[k];
              s_prow[q] = min(sorted_row[first + k], V - 1);
              uint32_t lim = 0xffffffffu;
              if (cut) {
                const uint32_t off = sorted_off[first + k];
                lim = off < capacity ? capacity - off : 0u;
              }
              s_plim[q] = lim;
              s_pidx[q] = threadIdx.x * SC_ITEMS + k;
            }
            ++p;
          }
        }
      }
      __syncthreads();
      {
        // Tile row by tile row of the band: the tiles of a row of the list inside one tile row are a run [xa, xa + len).
        // A lane sets the bits of a short run by itself; the long runs of a warp are then taken one at a time by all 32
        // lanes (one tile per lane and step), so that a splat as wide as the image costs the warp a few steps instead
        // of one lane a hundred.
        const uint32_t j = sub + threadIdx.x;
        const unsigned lane = threadIdx.x & 31;
        uint32_t* word = s_bits + (threadIdx.x >> 5) * band_tiles;  // the warp's 32 rows are the bits of these words
        uint32_t rx = 0, ry = 0, ry1 = 0, lim = 0, x1 = 0;
        SpanConic e;
        e.k = -1.f;
        if (j < npass) {
          const ushort4 r = s_prect[threadIdx.x];
          rx = r.x; ry = r.y; ry1 = r.w; lim = s_plim[threadIdx.x];
          x1 = min((uint32_t)r.z, (uint32_t)TX);
          const uint32_t gi = chunk * OFFSET_TILE + s_pidx[threadIdx.x];
          const float4 g4 = sorted_geo4[gi];
          const float2 g2 = sorted_geo2[gi];
          e.u = g4.x; e.v = g4.y; e.A = g4.z; e.B = g4.w; e.C = g2.x; e.k = g2.y;
        }
        for (uint32_t y = by0; y < by1; ++y) {
          uint32_t xa = 0, len = 0, k0 = 0;  // the lane's run in this tile row; k0: index of its first instance in the row
          if (j < npass && y >= ry && y < ry1) {
            int a, b;
            odin_row_span(e, (int)y, (int)rx, (int)x1, a, b);
            xa = (uint32_t)a; len = (uint32_t)(b - a);
            if (cut && len != 0)  // instances of the tile rows above (rare path: the view overflows the capacity)
              for (uint32_t yy = ry; yy < y; ++yy) {
                odin_row_span(e, (int)yy, (int)rx, (int)x1, a, b);
                k0 += (uint32_t)(b - a);
              }
          }
          uint32_t* line = word + (y - by0) * (uint32_t)TX;
          const bool large = len > 16;
          if (!large) {
            const uint32_t bit = 1u << lane;
            for (uint32_t i = 0; i < len; ++i)
              if (k0 + i < lim) atomicOr(line + xa + i, bit);  // other lanes of the warp may hold the same tile
          }
          uint32_t todo = __ballot_sync(0xffffffffu, large);
          __syncwarp();
          while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            const uint32_t q_xa = __shfl_sync(0xffffffffu, xa, src), q_len = __shfl_sync(0xffffffffu, len, src);
            const uint32_t q_k0 = __shfl_sync(0xffffffffu, k0, src), q_lim = __shfl_sync(0xffffffffu, lim, src);
            const uint32_t bit = 1u << src;
            for (uint32_t c = lane; c < q_len; c += 32)  // distinct tiles per lane: no two lanes share a word here
              if (q_k0 + c < q_lim) line[q_xa + c] |= bit;
            __syncwarp();
          }
        }
      }
      __syncthreads();
      for (uint32_t t = threadIdx.x; t < band_tiles; t += SC_THREADS) {
        uint32_t pos = s_pos[t];
#pragma unroll
        for (int wd = 0; wd < SC_WORDS; ++wd) {
          uint32_t bits = s_bits[wd * band_tiles + t];
          while (bits) {
            const int b = __ffs(bits) - 1;
            bits &= bits - 1;
            const uint32_t row = s_prow[wd * 32 + b];
            if (pos < capacity) {
              vals[pos] = row;
              if (WIDE) keys64[pos] = ((uint64_t)(by0 * (uint32_t)TX + t) << 32) | (uint64_t)depth_bits[row];
            }
            ++pos;
          }
        }
        s_pos[t] = pos;
      }
      __syncthreads();
    }
  }
}

// Writes every instance to its final place, a lane per tile.  A work item, one block each, is (chunk of OFFSET_TILE sorted rows,
// band of four tile rows).  The block lists the chunk's rows that meet the band, in depth order: span, tile rows of the band as
// bits, row id.  Its warps then take the band in units of 8 x 4 tiles.  For its unit a warp
//   1. turns the listed rows, one per lane, into words of 32 tiles and keeps those that are not empty, in order;
//   2. goes through the kept ones ST_BATCH at a time: every lane whose bit is set appends the row id to its ring in shared
//      memory ([place][lane]: a lane stays in its own bank; places follow the alignment of the list in memory);
//   3. writes every group of eight that is complete as one 32-byte store; the ends of a lane's run go word by word.
// What bounds it: the data pipe of loads and stores (71 % busy while an SM has work: the lists that the lanes walk, the rings, the stores of
// single sectors; 46 % of the issue slots, DRAM 21 %; 55 M instances of 168 k rows).  Units of 8 x 4 tiles and not 32 x 1, because a row
// of 18 x 18 tiles then touches 18 of them instead of 28 (105 against 131 us).  Measured against a bit matrix in shared memory read
// off tile by tile and, for rows of more than 96 tiles, runs collected by transposing bits: 10.5 M instances of 317 k rows
// (1600 x 1066) 127 -> 63 us, 272 M of 840 k (1920 x 1080) 930 -> 464, 2.9 M of 87 k (1237 x 823) 60 -> 25.
// Tried: the next item drawn and its rectangles fetched while this one is written (272 M: 520, few chunks 20 % slower: who draws
// early draws badly), the number of warps as a run-time value (10-15 % slower), batches of 24 rows (the same).  The one kind of view
// found in which the bit matrix was faster: all rectangles, of a tile or two, inside one unit of a wide image, which one warp per chunk
// walks (120 x 68 tiles, 70 k rows of a tile: whole odin_bin_sort 96 -> 104).
constexpr int ST_BAND = 4;      // tile rows of a band
constexpr int ST_BATCH = 16;
constexpr int ST_RING = 32;     // places per lane: up to 7 that wait for their group, and a batch
constexpr int ST_STAGE = 64;    // kept rows of a warp: fewer than a batch, and 32 more
static_assert(ST_RING >= ST_BATCH + 7 && ST_STAGE >= ST_BATCH + 32 && ST_STAGE % ST_BATCH == 0, "a batch never overruns");
static_assert(SCATTER_MAX_TX < 1024 && ST_BAND == 4, "fields of an entry, bits to bytes");
template <int WARPS>
struct ScatterSmem {
  uint32_t ring[WARPS][ST_RING][32];
  uint2 stage[WARPS][ST_STAGE];  // tiles of the 32 that the row covers, row id
  uint2 list[OFFSET_TILE + 34];  // first tile | end << 10 | tile rows of the band << 20, row id; behind the last 33 empty ones
  uint32_t cnt[OFFSET_TILE / 32], extra, item;
};
static_assert(OFFSET_TILE == 2048, "two counts per lane of the scan");
// Blocks of 8 or of 16 warps, four or two per SM (known on the device only: both kernels are launched, one returns at once, which
// with dependent launches costs about a microsecond): the kind that goes through its items in fewer rounds of units, counted as
// (items per resident block, at least one) x (units of a band per warp).  Where both take as many, what decides is the balance: items
// differ in cost, and up to ten per SM, or where rows cover hundreds of tiles, the longest are shorter with 16; many small ones are
// 3-6 % faster with 8.  Measured, whole odin_bin_sort with 8 / 16, us, by tiles of width, items, tiles per row:
//   8 wide, 392, 30: 119 / 176    50, 360, 33: 80 / 72      50, 1,288, 33: 113 / 124      78, 484, 72: 103 / 81      78, 880, 72: 119 / 101
//   78, 1,760, 72: 132 / 138      100, 660, 116: 111 / 89   100, 2,145, 30: 109 / 115     120, 748, 163: 123 / 98   120, 1,343, 163: 143 / 130
//   120, 2,414, 42: 121 / 126     160, 3,266, 69: 164 / 173 240, 340, 609: 149 / 118      240, 5,372, 609: 528 / 508
// The rule is 0.5 % from the better one on average over 117 views of 640 to 3,840 pixels' width (a bound of 600 items below
// 105 tiles of width and beyond 128: 2.2 %), and furthest, 21 %, with 1,012 items of 280 tiles per row in 160 tiles of width.
__device__ __forceinline__ int scatter_warps(uint32_t items, int TX, uint32_t rows, uint64_t instances, uint32_t sms) {
  const uint32_t units = ((uint32_t)TX + 7) / 8;
  const uint64_t rounds8 = (uint64_t)max(items, 4 * sms) * ((units + 7) / 8), rounds16 = 2ull * max(items, 2 * sms) * ((units + 15) / 16);
  if (rounds8 != rounds16) return rounds16 < rounds8 ? 16 : 8;
  return items <= 10 * sms || instances > (uint64_t)rows * 256u ? 16 : 8;
}

__device__ __forceinline__ uint32_t bit_run(uint32_t first, uint32_t len) {  // bits [first, first + len) of a word
  uint32_t m;
  asm("bmsk.clamp.b32 %0, %1, %2;" : "=r"(m) : "r"(first), "r"(len));
  return m;
}

template <bool WIDE, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 32 / WARPS)
scatter_tiles_kernel(const ushort4* __restrict__ sorted_rect, const uint32_t* __restrict__ sorted_row,
                     const uint32_t* __restrict__ sorted_off, const uint32_t* __restrict__ num_rows,
                     const uint64_t* __restrict__ num_instances, uint32_t capacity, int TX, int TY,
                     const uint32_t* __restrict__ counts, uint32_t tiles_pad, const uint2* __restrict__ ranges,
                     uint32_t* __restrict__ vals, uint64_t* __restrict__ keys64, const uint32_t* __restrict__ depth_bits,
                     uint32_t* __restrict__ item_ticket, uint32_t sms) {
  odin_after_predecessor();
  extern __shared__ __align__(16) unsigned char st_smem[];
  ScatterSmem<WARPS>& s = *reinterpret_cast<ScatterSmem<WARPS>*>(st_smem);
  constexpr int THREADS = 32 * WARPS, ITEMS = OFFSET_TILE / THREADS;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t V = *num_rows;
  const uint32_t nchunks = (V + OFFSET_TILE - 1) / OFFSET_TILE;
  const uint32_t nbands = ((uint32_t)TY + ST_BAND - 1) / ST_BAND, items = nchunks * nbands;
  if (scatter_warps(items, TX, V, *num_instances, sms) != WARPS) return;  // the other one's view
  const bool cut = *num_instances > (uint64_t)capacity;  // only then can a row be denied some of its instances
  const uint32_t lane_bit = 1u << lane;
  const uint32_t shift = (uint32_t)(reinterpret_cast<uintptr_t>(vals) >> 2) & 7u;  // place of vals[0] in its group of eight
  const uint32_t lane_ring = warp * (ST_RING * 128) + lane * 4;  // ring of the lane, bytes from the start of the rings
  uint2* const stage = s.stage[warp];
  const int cap_end = (int)(capacity + shift);
  while (true) {
    // items by ticket (they differ in cost by the number of rows of the chunk that meet the band)
    __syncthreads();
    if (threadIdx.x == 0) { s.item = atomicAdd(item_ticket, 1u); s.extra = 0u; }
    __syncthreads();
    const uint32_t item = s.item;
    if (item >= items) return;
    const uint32_t chunk = item / nbands, by0 = (item - chunk * nbands) * ST_BAND;  // neighbouring blocks share a chunk
    const uint32_t by1 = min((uint32_t)TY, by0 + ST_BAND);
    const uint32_t first = chunk * OFFSET_TILE;
    uint2 entry[ITEMS], partial = make_uint2(0, 0);
    uint32_t place[ITEMS];
    uint32_t keep = 0;
    {
      ushort4 rc[ITEMS];
#pragma unroll
      for (int k = 0; k < ITEMS; ++k) {
        const uint32_t i = first + k * THREADS + threadIdx.x;
        rc[k] = i < V ? sorted_rect[i] : make_ushort4(0, 0, 0, 0);
      }
#pragma unroll
      for (int k = 0; k < ITEMS; ++k) {
        const uint32_t i = first + k * THREADS + threadIdx.x;
        const uint32_t x0 = rc[k].x, x1 = min((uint32_t)rc[k].z, (uint32_t)TX), y0 = max((uint32_t)rc[k].y, by0);
        uint32_t y1 = min((uint32_t)rc[k].w, by1);
        bool meets = y1 > y0 && x1 > x0;
        if (cut && meets) {  // rare: of the row's instances, its tiles in row-major order, the first `lim` exist
          const uint32_t off = sorted_off[i], lim = off < capacity ? capacity - off : 0u, w = (uint32_t)rc[k].z - x0;
          const uint32_t ye = (uint32_t)rc[k].y + lim / w, rest = lim % w;  // whole up to tile row ye, of which `rest` tiles
          meets = lim != 0;
          if (ye < y1) {  // at most one row is cut in two: its last tile row is an entry of its own, the list's last
            if (meets && ye >= y0 && rest)
              partial = make_uint2(x0 | min(x0 + rest, x1) << 10 | 1u << (20 + ye - by0), min(sorted_row[i], V - 1));
            y1 = max(ye, y0);
          }
        }
        entry[k].x = x0 | x1 << 10 | (bit_run(y0 - by0, y1 - y0) & 15u) << 20;
        entry[k].y = i < V ? sorted_row[i] : 0u;
        const uint32_t m = __ballot_sync(0xffffffffu, meets);
        if (meets) keep |= 1u << k;
        place[k] = __popc(m & (lane_bit - 1u));
        if (lane == 0) s.cnt[k * WARPS + warp] = __popc(m);
      }
    }
    __syncthreads();
    uint32_t listed;
    {
      // every warp scans the counts itself
      const uint32_t a = s.cnt[2 * lane], b = s.cnt[2 * lane + 1];
      uint32_t inc = a + b;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= (unsigned)o) inc += y;
      }
      listed = __shfl_sync(0xffffffffu, inc, 31);
      const uint32_t ex = inc - a - b + (warp & 1u ? a : 0u);
#pragma unroll
      for (int k = 0; k < ITEMS; ++k) {
        const uint32_t e0 = __shfl_sync(0xffffffffu, ex, (k * WARPS + warp) >> 1);
        if (keep >> k & 1u) s.list[e0 + place[k]] = make_uint2(entry[k].x, min(entry[k].y, V - 1));
      }
      if (threadIdx.x < 33) s.list[listed + threadIdx.x] = make_uint2(0, 0);  // no tile rows: whole steps of 32 below
      if (cut) {
        __syncthreads();
        if (partial.x) { s.list[listed] = partial; s.extra = 1u; }
      }
    }
    __syncthreads();
    listed += s.extra;
    for (uint32_t u = warp; u < ((uint32_t)TX + 7) / 8; u += WARPS) {  // 8 tile columns of the band
      const uint32_t x = 8 * u + (lane & 7u), y = by0 + (lane >> 3);
      const bool mine = x < (uint32_t)TX && y < by1;
      const uint32_t tile = y * (uint32_t)TX + x;
      const int ca = -8 * (int)u;
      // (places in the list of all instances, counted from the group of eight that holds vals[0])
      const int start = (int)(min(mine ? ranges[tile].x + counts[(size_t)chunk * tiles_pad + tile] : 0u, capacity) + shift);
      int group = start & ~7;          // first place of the group that waits to be written
      uint32_t p = (uint32_t)start << 7;  // 128 times the next place
      // writes the lane's places of [group, group + 8) that lie in front of `end`
      auto write_group = [&](int end) {
        const uint32_t* r = reinterpret_cast<const uint32_t*>(st_smem + (((uint32_t)group << 7 & (ST_RING * 128 - 1)) | lane_ring));
        uint32_t v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = r[32 * k];
        uint32_t* out = vals + (group - (int)shift);
        if (!WIDE && group >= start && group + 8 <= min(end, cap_end)) {
          asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                       ::"l"(out), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
        } else {
          const uint32_t have = (uint32_t)(min(end, cap_end) - start);
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if ((uint32_t)(group - start + k) < have) {
              out[k] = v[k];
              if (WIDE) keys64[group - (int)shift + k] = ((uint64_t)tile << 32) | (uint64_t)depth_bits[v[k]];
            }
        }
        group += 8;
      };
      auto batch = [&](uint32_t at) {  // ST_BATCH kept rows
#pragma unroll
        for (int r = 0; r < ST_BATCH; r += 2) {
          const uint4 e = *reinterpret_cast<const uint4*>(stage + at + r);
          if (e.x & lane_bit) { *reinterpret_cast<uint32_t*>(st_smem + ((p & (ST_RING * 128 - 128)) | lane_ring)) = e.y; p += 128; }
          if (e.z & lane_bit) { *reinterpret_cast<uint32_t*>(st_smem + ((p & (ST_RING * 128 - 128)) | lane_ring)) = e.w; p += 128; }
        }
        while (true) {
          const bool full = p - ((uint32_t)group << 7) >= 1024u;
          if (!__any_sync(0xffffffffu, full)) break;
          if (full) write_group(group + 8);
        }
      };
      uint32_t head = 0, n = 0;  // kept rows: from head on, around the end of the stage
      for (uint32_t j0 = 0; j0 < listed; j0 += 32) {
        const uint2 e = s.list[j0 + lane];
        const int x0 = (int)(e.x & 1023u), x1 = (int)(e.x >> 10 & 1023u);
        const int a = max(x0 + ca, 0), b = max(x1 + ca, 0);
        // one bit per tile column, times one per tile row of the unit (from 4 neighbouring bits to 4 bytes)
        const uint32_t m = (bit_run((uint32_t)a, (uint32_t)(b - a)) & 255u) * (((e.x >> 20) * 0x00204081u) & 0x01010101u);
        const uint32_t kept = __ballot_sync(0xffffffffu, m != 0);
        if (m) stage[(head + n + __popc(kept & (lane_bit - 1u))) & (ST_STAGE - 1)] = make_uint2(m, e.y);
        n += __popc(kept);
        __syncwarp();
        while (n >= ST_BATCH) {
          batch(head);
          head = (head + ST_BATCH) & (ST_STAGE - 1);
          n -= ST_BATCH;
        }
        __syncwarp();
      }
      if (n) {
        if (lane >= n && lane < ST_BATCH) stage[head + lane] = make_uint2(0, 0);
        __syncwarp();
        batch(head);
        __syncwarp();
      }
      const int end = group + (int)((p - ((uint32_t)group << 7)) >> 7);  // less than a group is left
      if (end > max(group, start)) write_group(end);
    }
  }
}

int tile_digit_passes(uint32_t n_tiles) {
  int tile_bits = 0;
  while ((1ull << tile_bits) < (unsigned long long)n_tiles) ++tile_bits;
  const int p = (tile_bits + (int)SORT_RADIX_BITS - 1) / (int)SORT_RADIX_BITS;
  return p < 1 ? 1 : p;  // a one-tile image still takes one pass, which moves the emission into the outputs
}

}  // namespace

extern "C" int odin_bin_sort_workspace_bytes(const odin_ctx* ctx, uint32_t row_capacity, uint64_t max_instances, int width,
                                            int height, size_t* bytes) {
  if (!ctx || !bytes) return ODIN_ERR_NULL;
  if (width <= 0 || height <= 0 || width > 16384 || height > 16384) return ODIN_ERR_INVALID_ARG;
  const int TX = (width + 15) / 16, TY = (height + 15) / 16;
  const uint32_t n_tiles = (uint32_t)TX * (uint32_t)TY;
  if (ctx->cfg.instance_sort != 1 && scatter_eligible(TX, n_tiles)) *bytes = scatter_layout(row_capacity, n_tiles).total;
  else *bytes = binsort_ws_bytes(max_instances, row_capacity);
  return ODIN_OK;
}

namespace {
// The workspace as the call will use it, and what it wants zeroed: tickets, histograms, look-back words, and for the passes
// over the instances the used part of the difference array and the look-back words of the passes that run.
struct BinSortPlan {
  bool use_scatter;
  ScatterLayout F;
  BinSortLayout L;
  size_t zero_at[2], zero_bytes[2];
};
BinSortPlan bin_sort_plan(const odin_ctx* ctx, uint32_t rows, int TX, uint32_t n_tiles, uint64_t capacity, const void* ws, size_t ws_bytes) {
  BinSortPlan P;
  P.F = scatter_layout(rows, n_tiles);
  P.L = binsort_layout(capacity, rows);
  P.use_scatter = ctx->cfg.instance_sort != 1 && scatter_eligible(TX, n_tiles) && ws && ws_bytes >= P.F.total;
  P.zero_at[0] = 0;
  P.zero_bytes[0] = P.use_scatter ? P.F.row_states : P.L.tile_diff + ((size_t)n_tiles + 1) * 4;
  P.zero_at[1] = P.use_scatter ? 0 : P.L.scan_state;
  P.zero_bytes[1] = P.use_scatter ? 0 : P.L.inst_states + (size_t)tile_digit_passes(n_tiles) * P.L.tiles * SORT_RADIX * 4 - P.L.scan_state;
  return P;
}
}  // namespace

bool odin_bin_sort_scratch(const odin_ctx* ctx, const odin_projected* proj, int width, int height, uint64_t capacity, void* ws,
                           size_t ws_bytes, void** p, size_t* bytes) {
  if (!ws || width <= 0 || height <= 0 || width > 16384 || height > 16384 || capacity == 0 || capacity >= (1ull << 30) ||
      proj->capacity == 0 || proj->capacity >= (1u << 30))
    return false;
  const int TX = (width + 15) / 16;
  const BinSortPlan P = bin_sort_plan(ctx, proj->capacity, TX, (uint32_t)TX * (uint32_t)((height + 15) / 16), capacity, ws, ws_bytes);
  if (!P.use_scatter && ws_bytes < P.L.total) return false;
  for (int k = 0; k < 2; ++k) { p[k] = reinterpret_cast<char*>(ws) + P.zero_at[k]; bytes[k] = P.zero_bytes[k]; }
  return true;
}

extern "C" int odin_bin_sort(odin_ctx* ctx, const odin_projected* proj, int width, int height, uint64_t* d_keys,
                             uint32_t* d_vals, uint64_t capacity, uint32_t* d_tile_ranges, void* ws, size_t ws_bytes,
                             void* stream) {
  if (!ctx || !proj || !d_tile_ranges) return ODIN_ERR_NULL;
  if (width <= 0 || height <= 0 || width > 16384 || height > 16384) return ODIN_ERR_INVALID_ARG;
  if (!proj->num_rows || !proj->num_instances) return ODIN_ERR_NULL;
  if (capacity >= (1ull << 30) || proj->capacity >= (1u << 30)) return ODIN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int TX = (width + 15) / 16, TY = (height + 15) / 16;
  const uint32_t n_tiles = (uint32_t)TX * (uint32_t)TY;
  if (!odin_aligned(d_tile_ranges, 8)) return ODIN_ERR_INVALID_ARG;
  if (capacity == 0 || proj->capacity == 0) {
    odin_chain_break(ctx);
    ODIN_CUDA(cudaMemsetAsync(d_tile_ranges, 0, (size_t)n_tiles * 8, st));
    return ODIN_OK;
  }
  if (!d_vals || !proj->rect || !proj->depth) return ODIN_ERR_NULL;
  if ((d_keys && !odin_aligned(d_keys, 16)) || !odin_aligned(d_vals, 16) || !odin_aligned(proj->rect, 8))
    return ODIN_ERR_INVALID_ARG;
  const BinSortPlan plan = bin_sort_plan(ctx, proj->capacity, TX, n_tiles, capacity, ws, ws_bytes);
  const ScatterLayout& F = plan.F;
  const BinSortLayout& L = plan.L;
  const bool use_scatter = plan.use_scatter;
  const bool exact = ctx->cfg.binning == 2;
  if (exact && !use_scatter) return ODIN_ERR_UNSUPPORTED;  // the spans of exact binning exist in the scatter path only
  if (exact && (!proj->xy || !proj->conic_opacity)) return ODIN_ERR_NULL;
  if (!ws || !odin_aligned(ws, 256) || (!use_scatter && ws_bytes < L.total)) return ODIN_ERR_WORKSPACE;
  char* base = reinterpret_cast<char*>(ws);
  const int tile_passes = tile_digit_passes(n_tiles);
  // the regions both paths share (tickets, row histograms, look-back words of the row passes, ping-pong row buffers)
  const size_t o_hist = use_scatter ? F.hist : L.hist, o_dbase = use_scatter ? F.digit_base : L.digit_base;
  const size_t o_scan = use_scatter ? F.scan_state : L.scan_state, o_rstates = use_scatter ? F.row_states : L.row_states;
  const bool wide_rows = proj->capacity > (uint32_t)ctx->sm_count * ROW_SORT_TILE;
  const uint32_t row_tile = wide_rows ? 2 * ROW_SORT_TILE : ROW_SORT_TILE, row_tiles = (proj->capacity + row_tile - 1) / row_tile;
  for (int k = 0; k < 2; ++k) ODIN_CUDA(odin_zero(ctx, base + plan.zero_at[k], plan.zero_bytes[k], st));
  uint32_t* tickets = reinterpret_cast<uint32_t*>(base);
  uint32_t* hist = reinterpret_cast<uint32_t*>(base + o_hist);
  uint32_t* dbase = reinterpret_cast<uint32_t*>(base + o_dbase);
  uint64_t* scan_state = reinterpret_cast<uint64_t*>(base + o_scan);
  uint32_t* row_states = reinterpret_cast<uint32_t*>(base + o_rstates);
  uint32_t* row_keys[2], *row_vals[2];
  for (int b = 0; b < 2; ++b) {
    row_keys[b] = reinterpret_cast<uint32_t*>(base + (use_scatter ? F.row_keys[b] : L.row_keys[b]));
    row_vals[b] = reinterpret_cast<uint32_t*>(base + (use_scatter ? F.row_vals[b] : L.row_vals[b]));
  }
  uint32_t* sorted_off = reinterpret_cast<uint32_t*>(base + (use_scatter ? F.sorted_off : L.sorted_off));
  const uint32_t* depth_bits = reinterpret_cast<const uint32_t*>(proj->depth);
  const ushort4* rect = reinterpret_cast<const ushort4*>(proj->rect);
  const uint32_t sms = (uint32_t)ctx->sm_count;
  const uint32_t row_blocks = (proj->capacity + RH_THREADS - 1) / RH_THREADS;

  // ---- rows by depth
  const uint32_t* sorted_row = nullptr;
  constexpr size_t OS_SMEM = os_smem_bytes(OS_INST_ITEMS, OS_THREADS, false);
  if (proj->capacity <= ROW_SORT_SMALL) {
    OdinKernelScope ks(ctx, K_ROW_SORT, st);
    ODIN_CUDA(cudaFuncSetAttribute(row_sort_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RS_SMEM));
    ODIN_CUDA(odin_launch(ctx, false, row_sort_small_kernel, dim3(1), dim3(RS_THREADS), RS_SMEM, st, depth_bits, proj->num_rows,
                          proj->capacity, row_vals[1]));
    sorted_row = row_vals[1];
  } else {
    {
      OdinKernelScope ks(ctx, K_ROW_HIST, st);
      // one block per SM at most: every block ends with 1,500 global reductions onto the same 1,500 words
      ODIN_CUDA(odin_launch(ctx, false, row_hist_kernel, dim3(row_blocks < sms ? row_blocks : sms), dim3(RH_THREADS), 0, st,
                            depth_bits, proj->num_rows, hist, dbase, tickets + 9, tickets + 7, tickets + 13, row_states, row_tile, row_tiles));
    }
    // the third pass ends in row_vals[0] where it is the last one, otherwise it goes by way of sorted_off, which is not in use yet
    const uint32_t* kin[SORT_DEPTH_DIGITS] = {depth_bits, row_keys[0], row_keys[1], row_keys[0]};
    const uint32_t* vin[SORT_DEPTH_DIGITS] = {nullptr, row_vals[0], row_vals[1], sorted_off};
    uint32_t* kout[SORT_DEPTH_DIGITS] = {row_keys[0], row_keys[1], row_keys[0], nullptr};
    uint32_t* vout[SORT_DEPTH_DIGITS] = {row_vals[0], row_vals[1], sorted_off, row_vals[0]};
    for (int p = 0; p < SORT_DEPTH_DIGITS; ++p) {
      OdinKernelScope ks(ctx, K_ROW_SORT, st);
      const RowPass rp = {p, tickets + 7, row_vals[0], hist + 3 * ROW_RADIX, row_states + (size_t)3 * row_tiles * ROW_RADIX};
#define LAUNCH_ROWS(THREADS)                                                                                              \
  do {                                                                                                                  \
    constexpr size_t SMEM = os_smem_bytes(OS_ROW_ITEMS, THREADS, true);                                                 \
    const uint32_t resident = sms * (OS_RESIDENT / THREADS), grid = row_tiles < resident ? row_tiles : resident;        \
    const auto kernel = onesweep_kernel<true, false, OS_ROW_ITEMS, OS_ROW_WINDOW, THREADS>;                             \
    if (SMEM > 48 * 1024)                                                                                               \
      ODIN_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM));                  \
    ODIN_CUDA(odin_launch(ctx, true, kernel, dim3(grid), dim3(THREADS), SMEM, st, kin[p], vin[p], kout[p], vout[p], nullptr, nullptr, \
                          proj->num_rows, nullptr, 0, p * (int)ROW_RADIX_BITS, dbase + p * ROW_RADIX,                    \
                          row_states + (size_t)p * row_tiles * ROW_RADIX, tickets + p, ctx->d_status, ctx->spin_limit,  \
                          proj->capacity, rp));                                                                         \
  } while (0)
      if (wide_rows) LAUNCH_ROWS(1024);
      else LAUNCH_ROWS(512);
#undef LAUNCH_ROWS
    }
    sorted_row = row_vals[0];
  }
  if (use_scatter) {
    // ---- instances straight to their final places
    ushort4* sorted_rect = reinterpret_cast<ushort4*>(base + F.sorted_rect);
    uint64_t* base_state = reinterpret_cast<uint64_t*>(base + F.base_state);
    uint32_t* counts = reinterpret_cast<uint32_t*>(base + F.counts);
    float4* geo4 = reinterpret_cast<float4*>(base + F.sorted_geo4);
    float2* geo2 = reinterpret_cast<float2*>(base + F.sorted_geo2);
    const uint32_t cap32 = (uint32_t)capacity;
    {
      OdinKernelScope ks(ctx, K_ROW_OFFSETS, st);
      const size_t smem = ((size_t)F.tiles_pad + 8) * 4;
      const int max_smem = (int)(((size_t)SCATTER_MAX_TILES + 64 + 8) * 4);
      static_assert(RO_THREADS * RO_ITEMS == (int)OFFSET_TILE && 1024 * 2 == (int)OFFSET_TILE, "rows per chunk");
      ODIN_CUDA(cudaFuncSetAttribute(chunk_counts_kernel<false, 1024, 2>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
      ODIN_CUDA(cudaFuncSetAttribute(chunk_counts_kernel<true, 1024, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     max_smem));
#define LAUNCH_COUNTS(EXACT, THREADS, ITEMS)                                                                           \
  ODIN_CUDA(odin_launch(ctx, true, chunk_counts_kernel<EXACT, THREADS, ITEMS>, dim3(F.chunks), dim3(THREADS), smem, st, \
                        sorted_row, rect, reinterpret_cast<const float2*>(proj->xy),                                     \
                        reinterpret_cast<const float4*>(proj->conic_opacity), ctx->cfg.alpha_min, proj->num_rows,        \
                        proj->num_instances, cap32, TX, n_tiles, F.tiles_pad, sorted_off, sorted_rect, geo4, geo2,       \
                        counts, tickets + 8, scan_state, ctx->d_status, ctx->spin_limit))
      if (exact) LAUNCH_COUNTS(true, 1024, 2);
      else LAUNCH_COUNTS(false, 1024, 2);
#undef LAUNCH_COUNTS
    }
    {
      OdinKernelScope ks(ctx, K_TILE_BASES, st);
      ODIN_CUDA(odin_launch(ctx, true, tile_bases_kernel, dim3((n_tiles + TB_TILES - 1) / TB_TILES), dim3(TB_THREADS), 0, st, counts,
                            F.tiles_pad, n_tiles, proj->num_rows, proj->num_instances, capacity, base_state,
                            d_tile_ranges, tickets + 10, ctx->d_status, ctx->spin_limit));
    }
    if (exact) {
      OdinKernelScope ks(ctx, K_EMIT, st);
      // two tile rows per band: the bit matrix of a band is mostly empty (a depth-ordered batch of rows is scattered
      // over the image), and the words to clear and to read off grow with the band while the instances do not
      // (measured at 1600 x 1066 and 1920 x 1080: 1 / 2 / 3 / 7 rows -> 0.170 / 0.145 / 0.160 / 0.183 ms)
      int band_rows = (int)(SC_BAND_TILES / (uint32_t)TX);
      if (band_rows > 2) band_rows = 2;
      if (band_rows > TY) band_rows = TY;
      const uint64_t items_cap = (uint64_t)F.chunks * (((uint32_t)TY + band_rows - 1) / band_rows);
      const uint32_t grid = (uint32_t)(items_cap < (uint64_t)sms * 6 ? items_cap : (uint64_t)sms * 6);
#define LAUNCH_SCATTER(WIDE)                                                                                           \
  do {                                                                                                                 \
    ODIN_CUDA(cudaFuncSetAttribute(scatter_spans_kernel<WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                                   (int)SC_SMEM));                                                                     \
    ODIN_CUDA(odin_launch(ctx, true, scatter_spans_kernel<WIDE>, dim3(grid), dim3(SC_THREADS), SC_SMEM, st,  \
                          sorted_rect, geo4, geo2, sorted_row, sorted_off, proj->num_rows, proj->num_instances, cap32,  \
                          TX, TY, band_rows, counts, F.tiles_pad, reinterpret_cast<const uint2*>(d_tile_ranges), d_vals, \
                          d_keys, depth_bits, tickets + 11));                                                           \
  } while (0)
      if (d_keys) LAUNCH_SCATTER(true);
      else LAUNCH_SCATTER(false);
#undef LAUNCH_SCATTER
    } else {
      const uint64_t items_cap = (uint64_t)F.chunks * ((TY + ST_BAND - 1) / ST_BAND);
#define LAUNCH_TILES(WIDE, WARPS)                                                                                        \
  do {                                                                                                                  \
    OdinKernelScope ks(ctx, K_EMIT, st);                                                                                \
    const uint32_t grid = (uint32_t)(items_cap < (uint64_t)sms * (32 / WARPS) ? items_cap : (uint64_t)sms * (32 / WARPS)); \
    ODIN_CUDA(cudaFuncSetAttribute(scatter_tiles_kernel<WIDE, WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,       \
                                   (int)sizeof(ScatterSmem<WARPS>)));                                                   \
    ODIN_CUDA(odin_launch(ctx, true, scatter_tiles_kernel<WIDE, WARPS>, dim3(grid), dim3(32 * WARPS),                    \
                          sizeof(ScatterSmem<WARPS>), st, sorted_rect, sorted_row, sorted_off, proj->num_rows,           \
                          proj->num_instances, cap32, TX, TY, counts, F.tiles_pad,                                      \
                          reinterpret_cast<const uint2*>(d_tile_ranges), d_vals, d_keys, depth_bits, tickets + 12, sms)); \
  } while (0)
      if (d_keys) { LAUNCH_TILES(true, 8); LAUNCH_TILES(true, 16); }
      else { LAUNCH_TILES(false, 8); LAUNCH_TILES(false, 16); }
#undef LAUNCH_TILES
    }
    return odin_launch_status();
  }
  ODIN_CUDA(cudaFuncSetAttribute(onesweep_kernel<false, false, OS_INST_ITEMS, OS_INST_WINDOW, OS_THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)OS_SMEM));
  ODIN_CUDA(cudaFuncSetAttribute(onesweep_kernel<false, true, OS_INST_ITEMS, OS_INST_WINDOW, OS_THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)OS_SMEM));
  uint32_t* tile_diff = reinterpret_cast<uint32_t*>(base + L.tile_diff);
  uint32_t* inst_states = reinterpret_cast<uint32_t*>(base + L.inst_states);
  uint32_t* inst_keys[2] = {reinterpret_cast<uint32_t*>(base + L.inst_keys[0]), reinterpret_cast<uint32_t*>(base + L.inst_keys[1])};
  uint32_t* inst_vals[2] = {d_vals, reinterpret_cast<uint32_t*>(base + L.alt_vals)};
  uint32_t* chunk_row = reinterpret_cast<uint32_t*>(base + L.chunk_row);
  // ---- instances in depth order
  uint32_t* tile_dbase = dbase + ROW_BINS;
  const uint64_t chunks_cap = (capacity + DUP_CHUNK - 1) / DUP_CHUNK;
  {
    OdinKernelScope ks(ctx, K_ROW_OFFSETS, st);
    // shared-memory staging of the difference array for images of up to 40,000 tiles (e.g. 4096 x 2304)
    const uint32_t diff_words = n_tiles + 1 <= 40001u ? n_tiles + 1 : 0u;
    const size_t diff_smem = (size_t)diff_words * 4;
    ODIN_CUDA(cudaFuncSetAttribute(sorted_offsets_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 40001 * 4));
    ODIN_CUDA(odin_launch(ctx, true, sorted_offsets_kernel, dim3((proj->capacity + OFFSET_TILE - 1) / OFFSET_TILE),
                          dim3(RO_THREADS), diff_smem, st, sorted_row, rect, proj->num_rows, (uint32_t)capacity, TX,
                          sorted_off, chunk_row, (uint32_t)chunks_cap, tile_diff, diff_words, tickets + 8, scan_state,
                          ctx->d_status, ctx->spin_limit));
  }
  // the emission goes to the buffers from which `tile_passes` ping-pong steps end in d_vals
  int cur = tile_passes & 1;
  {
    OdinKernelScope ks(ctx, K_EMIT, st);
    const uint32_t grid = (uint32_t)(chunks_cap < (uint64_t)sms * 5 - 1 ? chunks_cap : (uint64_t)sms * 5 - 1) + 1;
    ODIN_CUDA(odin_launch(ctx, true, emit_instances_kernel, dim3(grid), dim3(DUP_THREADS), 0, st, sorted_off, sorted_row,
                          chunk_row, rect, proj->num_rows, proj->num_instances, capacity, TX, inst_keys[cur], inst_vals[cur],
                          ctx->d_status, tile_diff, n_tiles, tile_passes, d_tile_ranges, tile_dbase));
  }
  // ---- instances by tile id
  const uint32_t os_grid = L.tiles < sms * (OS_RESIDENT / OS_THREADS) ? L.tiles : sms * (OS_RESIDENT / OS_THREADS);
  for (int p = 0; p < tile_passes; ++p) {
    OdinKernelScope ks(ctx, K_ONESWEEP, st);
    uint32_t* states = inst_states + (size_t)p * L.tiles * SORT_RADIX;
    if (p + 1 < tile_passes)
      ODIN_CUDA(odin_launch(ctx, true, onesweep_kernel<false, false, OS_INST_ITEMS, OS_INST_WINDOW, OS_THREADS>, dim3(os_grid),
                            dim3(OS_THREADS), OS_SMEM, st, inst_keys[cur], inst_vals[cur], inst_keys[cur ^ 1],
                            inst_vals[cur ^ 1], nullptr, nullptr, nullptr, proj->num_instances, capacity,
                            p * (int)SORT_RADIX_BITS, tile_dbase + p * SORT_RADIX, states,
                            tickets + SORT_DEPTH_DIGITS + p, ctx->d_status, ctx->spin_limit, proj->capacity, RowPass{}));
    else  // the sorted tile ids themselves are not needed any more: the ranges came from the tile counts
      ODIN_CUDA(odin_launch(ctx, true, onesweep_kernel<false, true, OS_INST_ITEMS, OS_INST_WINDOW, OS_THREADS>, dim3(os_grid),
                            dim3(OS_THREADS), OS_SMEM, st, inst_keys[cur], inst_vals[cur], nullptr, inst_vals[cur ^ 1],
                            d_keys, depth_bits, nullptr, proj->num_instances, capacity, p * (int)SORT_RADIX_BITS,
                            tile_dbase + p * SORT_RADIX, states, tickets + SORT_DEPTH_DIGITS + p, ctx->d_status,
                            ctx->spin_limit, proj->capacity, RowPass{}));
    cur ^= 1;
  }
  return odin_launch_status();
}
