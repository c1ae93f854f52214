// Work vectors of a product with several right-hand sides: what dev_batch_alloc allocates and what a lockstep
// solve counts when it decides how many systems fit (host logic, checked in tests/batch_bytes_check.cpp).
#pragma once
#include <cstddef>

namespace efie {

// entries for R right-hand sides (16 bytes: x, xs; 8 bytes: the others)
struct BatchSizes {
  std::size_t x, xs;        // unknowns, twice; superspace vectors, three times
  std::size_t xf;           // x* in FP32, R rounded up to 4 (8 x 8 blocks: hi + lo)
  std::size_t mom, src;     // moments and local expansions; sources and M2L results
  std::size_t bytes() const { return 16 * (2 * x + 3 * xs) + 8 * (xf + 2 * mom + 2 * src); }
};

inline BatchSizes batch_sizes(int R, std::size_t ndof, std::size_t nsup, std::size_t nodes, int nb) {
  const std::size_t r = (std::size_t)R;
  return {r * ndof, r * nsup, (r + 3) / 4 * 4 * nsup * (nb == 8 ? 2 : 1), r * nodes * 3, r * nodes * 4};
}

}  // namespace efie
