// Instances of the axial Stolt-mapped NUFFT kernels (k_axial.cuh) for the
// FP64 plans; the two precisions compile as separate units, in parallel.
#include "k_axial.cuh"

namespace isam {

template cudaError_t launch_stolt_table<double>(const AxArgs<double>&, int4*, cudaStream_t);
template size_t ax_smem_bytes<double>(int);
template cudaError_t launch_ax_fwd<double>(const AxArgs<double>&, int, cudaStream_t);
template cudaError_t launch_ax_adj<double>(const AxArgs<double>&, int, cudaStream_t);
template cudaError_t launch_ax_fused<double>(const AxArgs<double>&, int, cudaStream_t);

cudaError_t launch_coef_table(const AxArgs<double>& a, double2* out, cudaStream_t s) {
  const int rows = (a.sc.ny / 2 + 1) * (a.sc.nx / 2 + 1);
  const dim3 grid((a.sc.nk / NRES + 127) / 128, rows);
  switch (a.sc.J) {
    case 4: k_coef_table<4><<<grid, 128, 0, s>>>(a, out); break;
    case 6: k_coef_table<6><<<grid, 128, 0, s>>>(a, out); break;
    case 8: k_coef_table<8><<<grid, 128, 0, s>>>(a, out); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace isam
