// Host-only checks of the control flow that feeds the tensor-core M2L's ring of stages (compiled and
// run by test_tc_pipeline_cpu.py with the system C++ compiler): a wait that runs out at any stage.
#include <cstdio>
#include <vector>

#include "../paper_1807_03097_gb300/csrc/tc_pipeline.h"

static int failures = 0;
#define CHECK(cond)                                           \
  do {                                                        \
    if (!(cond)) {                                            \
      std::printf("FAILED line %d: %s\n", __LINE__, #cond);   \
      ++failures;                                             \
    }                                                         \
  } while (0)

// A ring whose consumer frees slots until stage `stall` (its slot's previous user is stuck), then nothing.
static void run(int T, int ring, int stall) {
  std::vector<int> in_flight(ring, -1);  // stage whose copies may still be writing the slot
  bool ran_out = false;
  int waits = 0;
  const int issued = efie::issue_stages(
      T,
      [&](int it) {
        if (it < ring) return true;
        ++waits;
        if (it >= stall) {
          ran_out = true;
          return false;
        }
        in_flight[it % ring] = -1;
        return true;
      },
      [&](int it) {
        CHECK(!ran_out);                    // nothing is issued after a wait has run out
        CHECK(in_flight[it % ring] == -1);  // nor into a slot still in use
        in_flight[it % ring] = it;
      });
  const int first = stall > ring ? stall : ring;  // the first `ring` stages need no wait
  CHECK(issued == (T < first ? T : first));
  CHECK(waits <= T);
  int drained = 0;
  efie::drain_stages(issued, ring, [&](int it) {
    CHECK(it >= 0 && it < issued && in_flight[it % ring] == it);  // the stage really in the slot
    in_flight[it % ring] = -1;
    ++drained;
  });
  CHECK(drained == (issued < ring ? issued : ring));
  for (int v : in_flight) CHECK(v == -1);  // nothing in flight at the end
}

int main() {
  for (int T = 0; T <= 13; ++T)
    for (int stall = 0; stall <= T + 1; ++stall) run(T, 4, stall);
  std::printf(failures ? "%d failures\n" : "ok\n", failures);
  return failures ? 1 : 0;
}
