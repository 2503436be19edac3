// Host build of the CG solves' scalar helpers (the header the CUDA kernels include), exported
// for the CPU tests in tests/test_reductions.py.
#include "tg_fpconv.cuh"

extern "C" {

void tgr_pow2_inv_root(const double* x, double* out, long n) {
  for (long q = 0; q < n; ++q) out[q] = tg::pow2_inv_root(x[q]);
}

void tgr_norm_met(const double* rr, const double* rtol, const double* bb, int* out, long n) {
  for (long q = 0; q < n; ++q) out[q] = tg::cg_norm_met(rr[q], rtol[q], bb[q]) ? 1 : 0;
}

void tgr_pow2_recip(const double* x, double* out, long n) {
  for (long q = 0; q < n; ++q) out[q] = tg::pow2_recip(x[q]);
}

}  // extern "C"
