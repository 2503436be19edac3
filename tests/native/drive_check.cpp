// Host build of the CG solves' host-side decisions (the header the library includes), exported
// for the CPU tests in tests/test_drive.py.
#include "tg_drive.h"

extern "C" {

int tgd_small_fits(long long nvox, int sms, int sharers) {
  return tg::cg_small_fits(nvox, sms, sharers) ? 1 : 0;
}

// a launch that returns `error`: the outcome, with *refused in and out and *launched counted up
int tgd_run_small(int fits, int* refused, int error, int* launched) {
  bool r = *refused != 0;
  const int out = tg::run_small(fits != 0, r, [&] {
    ++*launched;
    return error;
  });
  *refused = r;
  return out;
}

}  // extern "C"
