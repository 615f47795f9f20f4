// fftfx_lg9.cu -- the fixed-point passes for transforms of 512 points.
#include "fftfx.cuh"

namespace sg {
FxKernels fx_kernels_lg9() { return make_fx_kernels<9>(); }
}  // namespace sg
