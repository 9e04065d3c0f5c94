// The residual kernels of fftm_stencil.cuh instantiated for FP32 fields.
#include "fftm_stencil.cuh"

namespace fftm {

template cudaError_t launch_residual<float>(const ResParams<float>&, int, bool, cudaStream_t, int*);
template int residual_blocks<float>(const ResParams<float>&, int);
template bool residual_one_pass<float>(const ResParams<float>&);

}  // namespace fftm
