// Host build of the CG solves' host-side decisions (the header the library includes), exported
// for the CPU tests in tests/test_drive.py.
#include "tg_drive.h"

extern "C" {

int tgd_small_fits(long long nvox, int sms, int sharers) {
  return tg::cg_small_fits(nvox, sms, sharers) ? 1 : 0;
}

}  // extern "C"
