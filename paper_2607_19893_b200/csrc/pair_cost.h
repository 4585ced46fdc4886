// Which of the two kernels counts the pairs of odin_conflict_count: by their modelled costs (host code, no CUDA).
#pragma once
#include <stdint.h>

// How the masks of a call fill the sides of the matrix kernel: 2^side_log masks a side, blocks_m sides.
struct PairSides {
  int side_log;
  uint32_t blocks_m, block_pairs;
};
static inline PairSides pair_sides(uint32_t n_masks) {
  PairSides s;
  s.side_log = n_masks <= 32 ? 5 : (n_masks <= 64 ? 6 : 7);
  s.blocks_m = (n_masks + (1u << s.side_log) - 1) >> s.side_log;
  s.block_pairs = s.blocks_m * (s.blocks_m + 1) / 2;
  return s;
}

// Blocks per pair of the kernel that counts pair by pair, so that all together are about PAIR_RESIDENT per SM.
constexpr uint32_t PAIR_THREADS = 256, PAIR_RESIDENT = 8;
static inline uint32_t pair_grid(uint32_t words, uint32_t n_pairs, uint32_t sm_count) {
  const uint32_t fill = (words / 4 + PAIR_THREADS - 1) / PAIR_THREADS, cap = (sm_count * PAIR_RESIDENT + n_pairs - 1) / n_pairs;
  const uint32_t g = fill < cap ? fill : cap;
  return g ? g : 1u;
}

// Nanoseconds of the whole call, on 148 SMs.  Pair by pair: 5 us, and a block 0.5 ns per word of its share, in as many waves as the
// blocks need (a last wave that is not full counts half as such, half by its blocks), and 0.3 ns a pair.  The matrix kernel: 10 us, and
// for every two sides of 128 masks 0.17 ns per word on the diagonal (where one copy in shared memory is both operands) and 2.5 times as
// much off it, whatever the number of pairs.  Both kernels measured over 5 k to 20 M primitives, 4 to 512 masks and 4 to 65 k pairs: the
// cheaper one by this is more than a tenth slower than the other in 12 of 1,555 calls, at most by 23 %.  (Pairs per mask of a
// side beyond 3.5 or 7, which it was before, in 175, at most 2.4 times as slow: all pairs of a small pool, windows of a few
// neighbours of hundreds of masks.)
static inline double pair_cost_single(uint32_t words, uint32_t n_pairs, uint32_t sm_count) {
  const uint32_t grid = pair_grid(words, n_pairs, sm_count);
  const uint64_t blocks = (uint64_t)grid * n_pairs, resident = (uint64_t)sm_count * PAIR_RESIDENT;
  const double waves = 0.5 * ((double)((blocks + resident - 1) / resident) + (double)blocks / (double)resident);
  return 5000.0 + 0.5 * waves * words / grid + 0.3 * n_pairs;
}
static inline double pair_cost_matrix(uint32_t words, const PairSides& s, uint32_t sm_count) {
  const double sides = (double)s.blocks_m + 2.5 * (double)(s.block_pairs - s.blocks_m);
  return 10000.0 + 0.17 * words * sides * (double)(1u << s.side_log) / 128.0 * 148.0 / (double)sm_count;
}
static inline bool pair_by_matrix(uint32_t words, uint32_t n_masks, uint32_t n_pairs, uint32_t sm_count) {
  const PairSides s = pair_sides(n_masks);
  return s.blocks_m <= 256 && pair_cost_matrix(words, s, sm_count) < pair_cost_single(words, n_pairs, sm_count);
}
