// Line passes of the preconditioner, FP32 instantiation (kernels in fft_lines.cuh).
#include "fft_lines_launch.cuh"

namespace xfft {
XFFT_LINES_INST(float)
}  // namespace xfft
