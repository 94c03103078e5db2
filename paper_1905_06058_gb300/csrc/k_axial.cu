// FP32 instances of the axial Stolt-mapped NUFFT kernels (k_axial.cuh): J = 6 and
// the dispatch; J = 4 and 8 are units of their own, compiled in parallel.
#include "k_axial.cuh"

namespace isam {

extern template cudaError_t launch_ax_J<float, 4>(const AxArgs<float>&, int, cudaStream_t, int);
extern template cudaError_t launch_ax_J<float, 8>(const AxArgs<float>&, int, cudaStream_t, int);
template cudaError_t launch_stolt_table<float>(const AxArgs<float>&, int4*, cudaStream_t);
template size_t ax_smem_bytes<float>(int);
template cudaError_t launch_ax_fwd<float>(const AxArgs<float>&, int, cudaStream_t);
template cudaError_t launch_ax_adj<float>(const AxArgs<float>&, int, cudaStream_t);
template cudaError_t launch_ax_fused<float>(const AxArgs<float>&, int, cudaStream_t);

}  // namespace isam
