// fftfx_lg12.cu -- the fixed-point passes for transforms of 4096 points.
#include "fftfx.cuh"

namespace sg {
FxKernels fx_kernels_lg12() { return make_fx_kernels<12>(); }
}  // namespace sg
