// FP32 instances of the lateral passes with the tile in registers.
#include "k_lateral_reg.cuh"

namespace isam {

template <> bool lat_reg_takes<float>(int L, int TZ) {
  switch (L) {
    case 1024: case 768: return TZ == 4;
    case 512: case 384: case 256: case 192: case 128: case 64: return TZ == 8;
  }
  return false;
}

template <> cudaError_t launch_lat_reg<float>(int mode, const LatArgs<float>& a, cudaStream_t s) {
  switch (a.L) {
    case 1024: return launch_lat_reg_length<float, 1024>(mode, a, s);
    case 768: return launch_lat_reg_length<float, 768>(mode, a, s);
    case 512: return launch_lat_reg_length<float, 512>(mode, a, s);
    case 384: return launch_lat_reg_length<float, 384>(mode, a, s);
    case 256: return launch_lat_reg_length<float, 256>(mode, a, s);
    case 192: return launch_lat_reg_length<float, 192>(mode, a, s);
    case 128: return launch_lat_reg_length<float, 128>(mode, a, s);
    case 64: return launch_lat_reg_length<float, 64>(mode, a, s);
  }
  return cudaErrorInvalidValue;
}

bool lat_half_takes(int L, int M) {
  return lat_reg_takes<float>(L, L >= 768 ? 4 : 8) && M % (L >= 768 ? 16 : 32) == 0;
}

cudaError_t launch_lat_half(int mode, const LatArgs<float>& a, cudaStream_t s) {
  switch (a.L) {
    case 1024: return launch_lat_half_length<1024>(mode, a, s);
    case 768: return launch_lat_half_length<768>(mode, a, s);
    case 512: return launch_lat_half_length<512>(mode, a, s);
    case 384: return launch_lat_half_length<384>(mode, a, s);
    case 256: return launch_lat_half_length<256>(mode, a, s);
    case 192: return launch_lat_half_length<192>(mode, a, s);
    case 128: return launch_lat_half_length<128>(mode, a, s);
    case 64: return launch_lat_half_length<64>(mode, a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace isam
