// pair_rules.h -- the sizes that the coset-arithmetic product (pair.cu) takes: plain C++, so that
// the rules can be tested without a device.
#pragma once
#include <cstdint>

namespace pair_rules {

// Kernels count slots in 32 bits.  expand_kernel steps by its whole grid and enum_rows by 1024
// slots past the end of a class: a position beyond the last slot must still be one, or the loop
// starts again at the first slots and never ends.
constexpr uint32_t kExpandThreads = 256;
constexpr uint32_t kExpandMaxBlocks = 1u << 16;
constexpr uint64_t kMaxSlots = (1ull << 32) - (uint64_t)kExpandMaxBlocks * kExpandThreads;

inline uint32_t expand_blocks(uint64_t n_slots, uint32_t sm_count) {
  const uint64_t need = (n_slots + kExpandThreads - 1) / kExpandThreads, most = 16ull * sm_count;
  const uint64_t b = need < most ? need : most;
  return (uint32_t)(b < kExpandMaxBlocks ? b : kExpandMaxBlocks);
}

// How a product over `rows` rows (or the class expectations, over all of them) finds its terms.
enum Route {
  kSearch,     // the representative of every term by search: nothing to prepare
  kDirect,     // coset arithmetic; a term reads its slot's index, its weight and x
  kExpanded,   // coset arithmetic; x is first spread over all slots, then a term is one read
};

// Expanding costs a pass over the slots and a call to the memory pool, reading directly two more
// accesses per term.  Measured (us, search / direct / expanded; GB300):
//   3.2e7 states fp32, 16 rows 136 / 41 / 278, 2.6e5 rows 847 / 320 / 354, 1e6 2486 / 1272 / 655
//   7.1e6 states c64 (chain), 16 rows 23 / 16 / 62, 2.6e5 rows 117 / 63 / 83, 1e6 334 / 180 / 151
//   6.4e7 states c64, D/1024 rows 253 / 90 / 399, D/128 856 / 522 / 563, D/9 9712 / 11004 / 4084
//   810 states fp64, all rows 31 / 12 / 15; 9252 states 45 / 14 / 15
// so directly up to one term per four slots, and on sectors so small that the second launch
// outweighs the reads: up to 2^14 slots and some fifteen terms per row (497 states c64 45 / 14 / 16).
// Complex fp64 multiplies each by its weight in the fp64 pipe and gains on the smallest only (168
// states 25 / 12 / 14, 497 states 58 / 21 / 17; 66 states of 13 terms 195 / 21 / 21).
// One-block splits read a term's representative from a whole table.  Where that stays in L2 (up to
// 22 sites), small sectors of few terms are done sooner so in complex fp32, where coset arithmetic
// multiplies twice by a character: 20 sites, 9225 states 16.5 / 18 / 19 (fp32 17 / 12 / 15); 26
// sites, 8844 states 20 / 16 / 17.
// At 8.6e8 states every read is a DRAM sector and the search is as fast for narrow ranges
// (us, D/4096 rows 238 / 298 / 17384, D/9 82 / 145 / 77 ms).  Fewer rows than half a warp leave
// both kernels waiting for one memory access after the other (775 states c64, 8 rows 12 / 12 / 15).
constexpr int64_t kMaxDirectDim = (int64_t)1 << 27;

inline Route route(int64_t rows, int64_t dim, double terms_per_row, uint64_t n_slots, bool complex_fp64,
                   bool table_complex_fp32 = false) {
  if (rows < 16) return kSearch;
  if (table_complex_fp32 && n_slots <= 1u << 14 && terms_per_row <= 11.0) return kSearch;
  if (dim > kMaxDirectDim) return rows >= dim / 8 ? kExpanded : kSearch;
  if ((double)rows * terms_per_row <= 0.25 * (double)n_slots) return kDirect;
  if (n_slots > 1u << 14) return kExpanded;
  if (complex_fp64 ? terms_per_row <= 11.0 && (double)rows * terms_per_row <= 1500.0 : terms_per_row <= 15.0) return kDirect;
  return kExpanded;
}

// Device memory.  A plan is made where, beside it, there is still room for the vectors of a
// Lanczos run and its ground state: the tables (6 bytes per slot) and one call's xs, then the row
// order (10 bytes per state).  The pool of a basis keeps the xs of two calls in its widest type.
struct Plan { bool pair, rows; };
inline uint64_t xs_most(uint64_t n_slots, bool is_real) { return (is_real ? 8 : 16) * (n_slots + 1); }
inline uint64_t pool_keep(uint64_t n_slots, bool is_real) { return 2 * xs_most(n_slots, is_real) + (16ull << 20); }
inline Plan fits(uint64_t free_bytes, uint64_t dim, uint64_t n_slots, bool is_real) {
  const uint64_t vectors = 4 * (is_real ? 8 : 16) * dim, pair = 6 * n_slots + xs_most(n_slots, is_real);
  return {pair + vectors <= free_bytes, pair + 10 * dim + vectors <= free_bytes};
}
inline bool always_fits(uint64_t dim, uint64_t n_slots) { return 22 * n_slots + 10 * dim < (64ull << 20); }

}  // namespace pair_rules
