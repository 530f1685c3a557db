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

}  // namespace pair_rules
