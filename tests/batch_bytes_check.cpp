// Host-only checks of the memory that a product with several right-hand sides is counted with (compiled and run by
// test_batch_bytes_cpu.py with the system C++ compiler).
#include <cstdio>

#include "../paper_1807_03097_gb300/csrc/batch_bytes.h"

static int failures = 0;
#define CHECK(cond)                                           \
  do {                                                        \
    if (!(cond)) {                                            \
      std::printf("FAILED line %d: %s\n", __LINE__, #cond);   \
      ++failures;                                             \
    }                                                         \
  } while (0)

int main() {
  using efie::batch_sizes;
  const std::size_t N = 1000, S = 4000, T = 3000;
  // per right-hand side: x, y (32 N); x*, y* and the near part (48 S); x* in FP32, 8 bytes an entry, 16 for 8 x 8 blocks,
  // which keep its rounding errors; moments, local expansions, sources and M2L results (112 T)
  CHECK(batch_sizes(4, N, S, T, 18).bytes() == 4 * (32 * N + 56 * S + 112 * T));
  CHECK(batch_sizes(4, N, S, T, 8).bytes() == 4 * (32 * N + 64 * S + 112 * T));
  // x* in FP32 in groups of four right-hand sides
  CHECK(batch_sizes(5, N, S, T, 8).bytes() == 5 * (32 * N + 48 * S + 112 * T) + 8 * 16 * S);
  CHECK(batch_sizes(64, N, S, T, 32).bytes() == 64 * (32 * N + 56 * S + 112 * T));
  // the largest problem's counts do not overflow 32 bits
  CHECK(batch_sizes(64, 1u << 24, 1u << 27, 1u << 28, 8).xs == (std::size_t)64 << 27);
  std::printf(failures ? "%d failures\n" : "ok\n", failures);
  return failures ? 1 : 0;
}
