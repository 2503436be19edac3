// tg_wait.cuh -- the time-bounded grid-wide wait of the kernels that run a whole solve in one
// cooperative launch, and the rule by which such a launch publishes its result.  Usable on the
// device and, a block at a time, on the host (for the CPU tests).
//
// Two words, both zero before a launch and after one that ended well: words[0] counts arrivals
// at the waits (the round-th wait is over at round * blocks), words[1] the blocks that left with
// the solve done.  A block has arrived before it starts to wait, so one that gives up does not
// hold the others back: a late block may let them all pass the same wait and finish.  Hence the
// result is published by the block that leaves last and not by a fixed one.  A block that gave
// up never takes a leaving ticket, so the CG_TIMEOUT that it stored is then final, and both words
// stay as they are (the context refuses further work).
#pragma once

#include "tg_fpconv.cuh"

#if !defined(__CUDA_ARCH__)
#include <chrono>
#endif

namespace tg {

TG_HD unsigned long long wait_clock_ns() {
#if defined(__CUDA_ARCH__)
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
#else
  return (unsigned long long)std::chrono::duration_cast<std::chrono::nanoseconds>(
             std::chrono::steady_clock::now().time_since_epoch()).count();
#endif
}

// one acquire-release atomic: what the caller wrote is visible to whoever takes a later ticket
TG_HD unsigned int ticket_acq_rel(unsigned int* counter) {
#if defined(__CUDA_ARCH__)
  unsigned int t;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
  return t;
#else
  return (*counter)++;
#endif
}

TG_HD void wait_arrive(unsigned int* words) {
#if defined(__CUDA_ARCH__)
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(words) : "memory");
#else
  ++words[0];
#endif
}

// Waits for the round-th arrival of all blocks; false once limit_ns have passed.  The clock is
// read on the first four looks and then on every 256th.
TG_HD bool wait_for_arrivals(const unsigned int* words, unsigned int round, unsigned int blocks,
                             unsigned long long limit_ns) {
  const unsigned int want = round * blocks;
  unsigned long long t0 = 0;
  for (unsigned int spin = 0;; ++spin) {
    unsigned int seen;
#if defined(__CUDA_ARCH__)
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(words) : "memory");
#else
    seen = words[0];
#endif
    if ((int)(seen - want) >= 0) return true;   // rounds may wrap
    if (spin < 4u || (spin & 255u) == 0u) {
      const unsigned long long t = wait_clock_ns();
      if (spin == 0u) t0 = t;
      if (t - t0 > limit_ns) return false;
    }
  }
}

// A block leaves with the solve done: true in the last of the launch's blocks, which publishes
// the result; the words are then zero again.
TG_HD bool leave_last(unsigned int* words, unsigned int blocks) {
  if (ticket_acq_rel(words + 1) != blocks - 1) return false;
  words[0] = 0u;
  words[1] = 0u;
  return true;
}

}  // namespace tg
