// The residual kernels of fftm_stencil.cuh instantiated for FP64 fields.
#include "fftm_stencil.cuh"

namespace fftm {

template cudaError_t launch_residual<double>(const ResParams<double>&, int, bool, cudaStream_t, int*);
template int residual_blocks<double>(const ResParams<double>&, int);
template bool residual_one_pass<double>(const ResParams<double>&);

}  // namespace fftm
