// fftfx_lg8.cu -- the fixed-point passes for transforms of 256 points.
#include "fftfx.cuh"

namespace sg {
FxKernels fx_kernels_lg8() { return make_fx_kernels<8>(); }
}  // namespace sg
