// Host build of the larger radices of the CUDA path's line transforms (fft_radix.cuh), for the CPU
// test against a direct DFT.
#include "fft_radix.cuh"

namespace {
template <int R, bool INV>
void run(double* v) {
  double2 c[R];
  for (int k = 0; k < R; ++k) c[k] = make_double2(v[2 * k], v[2 * k + 1]);
  xfft::fast::Dft<double2, R, INV>::run(c);
  for (int k = 0; k < R; ++k) {
    v[2 * k] = c[k].x;
    v[2 * k + 1] = c[k].y;
  }
}
}  // namespace

// v: R complex values (interleaved re, im), transformed in place; returns 0 for an unknown radix
extern "C" int host_radix(int R, int inv, double* v) {
  switch (R) {
#define X(n) \
  case n: inv ? run<n, true>(v) : run<n, false>(v); return 1;
    X(9) X(10) X(12) X(15)
#undef X
    default: return 0;
  }
}
