// Host build of the cooperative solves' wait and publication rule (the header the CUDA kernels
// include), for the CPU tests in tests/test_waits.py: the blocks of a launch take their steps one
// after another, in the order the test gives.
#include "tg_wait.cuh"

extern "C" {

// One step of one block on the launch's two words and its status (0 running, 1 converged,
// 5 timed out).  what 0: arrive; 1: wait for round `round`, giving up after limit_ns (returns
// whether the wait ended, and marks the solve if not); 2: leave with the solve done.
int tgw_step(unsigned int* words, int* status, int what, unsigned int round, unsigned int blocks,
             unsigned long long limit_ns) {
  if (what == 0) {
    tg::wait_arrive(words);
    return 1;
  }
  if (what == 1) {
    const bool ok = tg::wait_for_arrivals(words, round, blocks, limit_ns);
    if (!ok) *status = 5;
    return ok;
  }
  const bool last = tg::leave_last(words, blocks);
  if (last) *status = 1;
  return last;
}

}  // extern "C"
