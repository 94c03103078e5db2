// Dispersion-compensated inverse FFT of every A-scan (Eq. 9): the direct,
// non-iterative reconstruction on the full-range depth grid,
//   out(x, n) = (1/sqrt(nz)) sum_j s(x, k_j) e^{-j phi(k_j)} e^{-j 2 k_j z_n}.
// With k_j = k_min + j dk and z_n = (n - nz/2) dz, dz = pi/(nz dk):
//   2 k_j z_n = 2 pi (kappa_0 + j)(n - nz/2)/nz,  kappa_0 = k_min/dk, so
//   out(x, n) = post_n sum_j [(-1)^j s_j e^{-j phi_j}] e^{-2 pi i j n / nz},
//   post_n = e^{-2 pi i kappa_0 (n - nz/2)/nz} / sqrt(nz)   (tabulated in FP64),
// an nz-point DFT of the zero-padded, modulated samples (nk <= nz).
#include "fft_smem.cuh"
#include "internal.cuh"
#include "lat_reg.cuh"

namespace isam {

template <typename T>
__global__ void k_dc_ifft(const T* s, cplx<T>* out, const cplx<T>* disp, const cplx<T>* post,
                          const cplx<T>* roots, int nk, int nz, int lognz) {
  extern __shared__ __align__(16) unsigned char raw[];
  cplx<T>* buf = reinterpret_cast<cplx<T>*>(raw);
  const size_t a = blockIdx.x;
  const T* x = s + a * nk;
  const cplx<T>* tw = build_twiddles<T>(buf + padded_rows(nz), roots, nz, lognz);
  for (int j = threadIdx.x; j < nz; j += blockDim.x) {
    cplx<T> v = mk<T>(0, 0);
    if (j < nk) {
      const T sj = (j & 1) ? -x[j] : x[j];
      const cplx<T> d = __ldg(disp + j);
      v = mk<T>(sj * d.x, -sj * d.y);
    }
    buf[prow(j)] = v;
  }
  __syncthreads();
  const int nb = nz >= 8 ? nz / 8 : 1;
  fft_smem<-1, false, T>(buf, 1, 0, threadIdx.x, nz, lognz, tw, threadIdx.x < nb);
  cplx<T>* o = out + a * nz;
  for (int n = threadIdx.x; n < nz; n += blockDim.x) o[n] = cmul(buf[prow(n)], __ldg(post + n));
}

// FP32, nz = 256 .. 2048: the register transform of lat_reg.cuh on A-scans (columns
// of contiguous rows, so W = 1), 128 threads a block.  The shared-memory form's 256
// threads an A-scan moved it ten times through shared memory between barriers that
// left 1,024 blocks' loads and stores uncovered; here 512 blocks of two A-scans are
// resident at once (1024 x 2048: 18.5 -> 12.0 us a call; 25 MB, so the loads' latency
// and the launch are what is left).
template <int L>
__global__ void __launch_bounds__(128, lreg::Plan<float, L>::P == 32 ? 4 : 6)
    k_dc_ifft_regs(const float* s, float2* out, const float2* disp, const float2* post, int nk,
                   int n_ascans) {
  constexpr int P = lreg::Plan<float, L>::P, TH = L / P, PER = 128 / TH;
  __shared__ float2 S[PER][lreg::smem_elements<float, L, 1>()];
  const int b = threadIdx.x % TH, sl = threadIdx.x / TH;
  const int scan = blockIdx.x * PER + sl;
  const bool in = scan < n_ascans;
  const lreg::Twiddles<float, L> tw(b, nullptr);
  cudaGridDependencySynchronize();
  const float* x = s + size_t(scan) * nk;
  float2 v[P];
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int j = b + i * TH;                          // parity of j: that of b
    float2 w = make_float2(0.0f, 0.0f);
    if (in && j < nk) {
      const float sj = (b & 1) ? -x[j] : x[j];
      const float2 d = __ldg(disp + j);
      w = make_float2(sj * d.x, -sj * d.y);
    }
    v[i] = w;
  }
  lreg::transform<-1, L, 1, 0, float>(v, S[sl], tw, b, 0, true, [] {});
  cudaTriggerProgrammaticLaunchCompletion();
  if (!in) return;
  float2* o = out + size_t(scan) * L;
#pragma unroll
  for (int i = 0; i < P; ++i) o[b + i * TH] = cmul(v[i], __ldg(post + b + i * TH));
}

template <int L>
static cudaError_t launch_dc_regs(const float* s, float2* out, const float2* disp,
                                  const float2* post, int nk, int n, cudaStream_t st) {
  constexpr int PER = 128 / (L / lreg::Plan<float, L>::P);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((n + PER - 1) / PER);
  cfg.blockDim = dim3(128);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_dc_ifft_regs<L>, s, out, disp, post, nk, n);
}

template <typename T> cudaError_t launch_dc_ifft(const T* s, cplx<T>* out, const cplx<T>* disp,
                                                 const cplx<T>* post, const cplx<T>* roots, int nk,
                                                 int nz, int lognz, int n_ascans, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    switch (nz) {
      case 2048: return launch_dc_regs<2048>(s, out, disp, post, nk, n_ascans, st);
      case 1024: return launch_dc_regs<1024>(s, out, disp, post, nk, n_ascans, st);
      case 512: return launch_dc_regs<512>(s, out, disp, post, nk, n_ascans, st);
      case 256: return launch_dc_regs<256>(s, out, disp, post, nk, n_ascans, st);
    }
  }
  const int threads = nz / 8 > 32 ? nz / 8 : 32;
  const size_t sm = size_t(padded_rows(nz) + twiddle_entries<T>(nz, lognz)) * sizeof(cplx<T>);
  allow_smem(k_dc_ifft<T>, sm);
  k_dc_ifft<T><<<n_ascans, threads, sm, st>>>(s, out, disp, post, roots, nk, nz, lognz);
  return cudaGetLastError();
}
template cudaError_t launch_dc_ifft<float>(const float*, float2*, const float2*, const float2*,
                                           const float2*, int, int, int, int, cudaStream_t);
template cudaError_t launch_dc_ifft<double>(const double*, double2*, const double2*,
                                            const double2*, const double2*, int, int, int, int,
                                            cudaStream_t);

}  // namespace isam
