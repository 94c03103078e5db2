// FP32 instances of the axial kernels at J = 4 (see k_axial.cu).
#include "k_axial.cuh"

namespace isam {

template cudaError_t launch_ax_J<float, 4>(const AxArgs<float>&, int, cudaStream_t, int);

}  // namespace isam
