// Control flow of a thread that feeds a ring of stages with asynchronous work (bulk copies, MMAs),
// apart from the instructions so that it is checked on the host: when a bounded wait runs out,
// nothing more may be issued into stages whose state is no longer known, and what is in
// flight has to be waited for before the block's shared or tensor memory goes to another use.
#pragma once

#ifdef __CUDACC__
#define EFIE_HD __host__ __device__ __forceinline__
#else
#define EFIE_HD inline
#endif

namespace efie {

// issue(it) for the stages it = 0 ... T - 1 in turn, each after ready(it); ready returns false when
// its wait ran out, which ends the sequence.  Returns the number of stages issued.
template <class Ready, class Issue>
EFIE_HD int issue_stages(int T, Ready ready, Issue issue) {
  int it = 0;
  for (; it < T; ++it) {
    if (!ready(it)) break;
    issue(it);
  }
  return it;
}

// wait(it) for the stages that may still be in flight after `issued` of them went into `ring` slots.
template <class Wait>
EFIE_HD void drain_stages(int issued, int ring, Wait wait) {
  for (int it = issued > ring ? issued - ring : 0; it < issued; ++it) wait(it);
}

}  // namespace efie
