// mlmc_pair.cuh -- what the multilevel kernel keeps of a pair between units, in
// one word: the fine steps taken and which of its walks are done.
#pragma once

#include <cstdint>

namespace pdd {

// Pairs are stored at the start of a unit only, so the word holds the number of
// units: with two steps or more to a unit that stays below 2^30 up to the largest
// step cap, 2^31 - 1 (the steps themselves would run into the two flags).
struct PairState {
  int32_t steps;
  bool fine_done, coarse_done;
};
constexpr uint32_t kPairUnits = (1u << 30) - 1u;
__host__ __device__ inline uint32_t pair_pack(int32_t steps, int32_t unit, bool fine_done,
                                              bool coarse_done) {
  return static_cast<uint32_t>(steps) / static_cast<uint32_t>(unit) | (fine_done ? 1u << 30 : 0u) |
         (coarse_done ? 1u << 31 : 0u);
}
__host__ __device__ inline PairState pair_unpack(uint32_t w, int32_t unit) {
  return {static_cast<int32_t>((w & kPairUnits) * static_cast<uint32_t>(unit)), ((w >> 30) & 1u) != 0,
          (w >> 31) != 0};
}

}  // namespace pdd
