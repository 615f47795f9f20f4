// fftconv_lg6.cu -- the FP32 column passes for transforms of 64 points with
// the length fixed at compile time (see FixedPassKernels in fftconv.cu).
#define SG_FFTCONV_KERNELS_ONLY
#include "fftconv.cu"

namespace sg {
FixedPassKernels fixed_pass_kernels_lg6() { return make_fixed_pass_kernels<6>(); }
}  // namespace sg
