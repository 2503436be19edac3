// Host build of the CG solves' host-side decisions (the header the library includes), exported
// for the CPU tests in tests/test_drive.py.
#include "tg_drive.h"

extern "C" {

int tgd_small_fits(long long nvox, int sms, int sharers) {
  return tg::cg_small_fits(nvox, sms, sharers) ? 1 : 0;
}

long long tgd_flat_blocks(long long want, long long nblocks, int sms) {
  return tg::flat_blocks(want, nblocks, sms);
}

int tgd_op_planes(int zc, long long nblocks, int sms) { return tg::op_planes(zc, nblocks, sms); }

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

// Reads of the flags that a solve of `total` iterations takes whose residual falls evenly from
// rr0 to rtol^2 bb, the last such solve having taken `prev`.
int tgd_reads(int total, int prev, double bb, double rr0, double rtol) {
  struct Scal {
    double rr, bb, rtol;
    int it, status;
  } s = {rr0, bb, rtol, 0, 0}, seen = s;
  const double rate = std::log(rr0 / (rtol * rtol * bb)) / (total - 0.5);
  int chunk = tg::first_chunk(prev), grown = 2;
  for (int reads = 1;; ++reads) {
    s.it = std::min(total, s.it + chunk);
    s.rr = rr0 * std::exp(-rate * s.it);
    if (s.it == total) return reads;
    chunk = tg::next_chunk<Scal>(&s, reads > 1 ? &seen : nullptr, 1, 0, grown);
    if (reads == 1) seen = s;
    grown = std::min(grown * 2, 32);
  }
}

}  // extern "C"
