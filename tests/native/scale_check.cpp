// Host build of the FP64 z pass's scale (the header the CUDA kernels include), exported for the
// CPU test in tests/test_spectral_units.py.
#include "tg_fpconv.cuh"

extern "C" void tgs_pow2_scale(const double* x, double* out, long n) {
  for (long q = 0; q < n; ++q) out[q] = tg::pow2_scale(x[q]);
}
