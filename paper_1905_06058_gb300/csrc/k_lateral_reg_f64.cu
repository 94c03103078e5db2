// FP64 instances of the lateral passes with the tile in registers.
#include "k_lateral_reg.cuh"

namespace isam {

template <> bool lat_reg_takes<double>(int L, int TZ) {
  return TZ == 2 && (L == 64 || L == 128 || L == 256 || L == 512);
}

template <> cudaError_t launch_lat_reg<double>(int mode, const LatArgs<double>& a,
                                               cudaStream_t s) {
  switch (a.L) {
    case 512: return launch_lat_reg_length<double, 512>(mode, a, s);
    case 256: return launch_lat_reg_length<double, 256>(mode, a, s);
    case 128: return launch_lat_reg_length<double, 128>(mode, a, s);
    case 64: return launch_lat_reg_length<double, 64>(mode, a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace isam
