// Host-only checks of the choice between the two forms of kept FP64 matrices (compiled and run by
// test_kept_matrices_cpu.py with the system C++ compiler).
#include <cstdio>

#include "../paper_1807_03097_gb300/csrc/kept_matrices.h"

static int failures = 0;
#define CHECK(cond)                                           \
  do {                                                        \
    if (!(cond)) {                                            \
      std::printf("FAILED line %d: %s\n", __LINE__, #cond);   \
      ++failures;                                             \
    }                                                         \
  } while (0)

int main() {
  using efie::keep_digits;
  CHECK(!keep_digits(1, 1, 0, 1000));  // always evaluate
  // always keep: whatever fits, with what belongs to it
  CHECK(keep_digits(2, 900, 100, 1000));
  CHECK(!keep_digits(2, 901, 100, 1000));  // the matrices alone would fit: the plain form runs
  CHECK(!keep_digits(2, 1000, 1, 1000));
  CHECK(!keep_digits(2, 0, 1001, 1000));
  // automatic: the matrices in at most half of the free memory
  CHECK(keep_digits(0, 500, 100, 1000));
  CHECK(!keep_digits(0, 501, 0, 1000));
  CHECK(!keep_digits(0, 500, 501, 1000));
  CHECK(keep_digits(0, 0, 0, 0));
  std::printf(failures ? "%d failures\n" : "ok\n", failures);
  return failures ? 1 : 0;
}
