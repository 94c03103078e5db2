// Kernels for calibrating the dispersion coefficients a_1..a_4 (Eq. 7) and
// the focal depth z0 by gradient descent through the model.
//
// A depends on theta = (a_1..a_4, z0) only through the spectral phase
// P(q, k) = e^{j phi(k)} e^{j (2k + beta) z0}, so with S_x = P . N(F x) (the
// lateral spectrum of K_hat x before the real part) and F y the unitary
// lateral FFT of real spectra y,
//   <dA/dtheta x, y> = sum_{q,k} D_theta(q, k) Re( j conj(F y) S_x ),
//   D_{a_i} = (k - k0)^i,   D_{z0} = 2k + beta = a / (2 kappa + p) dk,
// in plan grid units (kappa = k/dk, a = (q/dk)^2, p = sqrt(4 kappa^2 - a)).
//
// k_param_reduce forms these sums per column pair (q, -q).  Where the "data"
// spectrum is itself the real part of a model spectrum E, F y = (E(q) +
// conj E(-q))/2 is formed pointwise from the pair, exactly as the fused
// gradient kernel forms the residual.  Sums are FP64: the polynomial moments
// m_i = sum t^i v with t = j - (nk-1)/2 (then a_i gradient = dk^i m_i) and
// m_z = sum (a / (2 kappa + p)) v (then z0 gradient = dk m_z).
#include <math.h>

#include <type_traits>

#include "fft_smem.cuh"
#include "internal.cuh"

namespace isam {

// Programmatic dependent launch, of FP32 plans (as the axial and lateral kernels)
template <typename T, typename... P, typename... A>
static cudaError_t launch_dependent(void (*kern)(P...), unsigned blocks, unsigned threads,
                                    cudaStream_t s, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = sizeof(T) == 4;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename T>
__device__ __forceinline__ T im_part(cplx<T> F, cplx<T> S) {   // Re(j conj(F) S)
  return F.y * S.x - F.x * S.y;
}

template <typename T>
__device__ __forceinline__ cplx<T> real_part_spectrum(cplx<T> a, cplx<T> b) {
  return cscale(cadd(a, cconj(b)), T(0.5));   // F(Re v)(q) from F v(q), F v(-q)
}

// a + b for an exact b
__device__ __forceinline__ ff plus(ff a, float b) {
  const ff t = ff_two_sum(a.hi, b);
  return ff_quick(t.hi, __fadd_rn(t.lo, a.lo));
}

// What bounds k_param_reduce: the latency of its loads and the FP64 pipe (2 lanes a
// clock), for 40 bytes of each column sample.  A thread takes two neighbouring samples
// of both columns a load and has two such groups in flight; TPB is a quarter of nk up
// to 512, so that they cover nk = 2048.  FP32 plans keep the samples' arithmetic in
// float, the cancelling 4 kappa^2 - a from float pairs, and the threads'
// sums are added in double by one warp a moment.  512 x 2048: 24.7 -> 15.2 us (16.5 at
// one block a multiprocessor, 72 registers).
//
// FIT (FP32 calibrations with nz > nk, see FitOrder): sample j belongs to thread j mod
// TPB, whose terms are summed in that order, and 4 kappa^2 - a is formed in double.
template <typename T> struct ParamSamples {
  cpair<T> S1, S2, E1, E2, f1, f2;
};

template <typename T, int TPB, bool FIT = false>
__global__ void __launch_bounds__(TPB, sizeof(T) == 4 && TPB == 512 ? 2 : 1)
    k_param_reduce(const __grid_constant__ ParamArgs<T> A) {
  using C = cplx<T>;
  const int2 pr = A.pairs[blockIdx.x];
  const int c1 = pr.x, c2 = pr.y;
  const bool two = c1 != c2;
  const int nk = A.sc.nk, nx = A.sc.nx;
  const int mx = c1 % nx <= (nx - 1) / 2 ? c1 % nx : c1 % nx - nx;
  const int ny = A.sc.ny, iy = c1 / nx;
  const int my = iy <= (ny - 1) / 2 ? iy : iy - ny;
  const double a = A.sc.Qx * double(mx) * mx + A.sc.Qy * double(my) * my;
  const double tc = 0.5 * double(nk - 1);
  // FP32: 2 kappa_0 - sqrt(a), 2 kappa_0 + sqrt(a) and 2 kappa_0 as float pairs, and a
  __shared__ float cut_s[7];
  __shared__ T part[5][TPB];
  ff lo = {}, hi = {}, mid = {};
  float af = 0.0f;
  if constexpr (std::is_same<T, float>::value && !FIT) {
    if (threadIdx.x == 0) {
      const double sa = sqrt(a), v[3] = {2.0 * A.sc.kap - sa, 2.0 * A.sc.kap + sa, 2.0 * A.sc.kap};
      for (int i = 0; i < 3; ++i) {
        cut_s[2 * i] = float(v[i]);
        cut_s[2 * i + 1] = float(v[i] - double(float(v[i])));
      }
      cut_s[6] = float(a);
    }
  }
  C* s1 = A.su + size_t(c1) * nk;
  C* s2 = A.su + size_t(c2) * nk;
  const C* e1 = A.se ? A.se + size_t(c1) * nk : nullptr;
  const C* e2 = A.se ? A.se + size_t(c2) * nk : nullptr;
  const C* f1 = A.fd ? A.fd + size_t(c1) * nk : nullptr;
  const C* f2 = A.fd ? A.fd + size_t(c2) * nk : nullptr;
  T m[5] = {};
  cudaGridDependencySynchronize();
  auto load = [&](int j) {
    ParamSamples<T> x{};
    if (j < nk) {
      x.S1 = load_two<T>(s1 + j);
      x.S2 = load_two<T>(s2 + j);
      if (e1) {
        x.E1 = load_two<T>(e1 + j);
        x.E2 = load_two<T>(e2 + j);
      }
      if (f1) {
        x.f1 = load_two<T>(f1 + j);
        x.f2 = load_two<T>(f2 + j);
      }
    }
    return x;
  };
  // v of sample j; Fa1, Fa2: the spectra of the real part of S
  auto point = [&](int j, C S1, C S2, C E1, C E2, C d1, C d2, C& Fa1, C& Fa2) {
    const C F1 = cadd(real_part_spectrum<T>(E1, E2), cscale(d1, A.fd_sign));
    const C F2 = cadd(real_part_spectrum<T>(E2, E1), cscale(d2, A.fd_sign));
    Fa1 = real_part_spectrum<T>(S1, S2);
    Fa2 = real_part_spectrum<T>(S2, S1);
    T v = im_part<T>(F1, S1);
    if (two) v += im_part<T>(F2, S2);
    if (e1) {
      v += im_part<T>(Fa1, E1);
      if (two) v += im_part<T>(Fa2, E2);
    }
    if constexpr (std::is_same<T, float>::value) {
      // weights (k_j - k0)^i (t = j - (nk-1)/2 is exact) and a / (2 kappa +
      // sqrt(4 kappa^2 - a)); a thread's few terms summed in float
      const float t = float(j) - float(tc);
      float tp = t;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        m[i] = fmaf(tp, v, m[i]);
        tp *= t;
      }
      if constexpr (FIT) {
        const double kap = A.sc.kap + double(j), x = fma(4.0 * kap, kap, -a);
        if (x > 0.0)
          m[4] = fmaf(float(a) / (2.0f * float(kap) + sqrtf(float(x))), v, m[4]);
        return;
      }
      // 4 kappa^2 - a as the product of its factors, each a float pair (44 bits): as
      // near as the difference in double, rounded to float
      const float j2 = float(2 * j);
      const ff dm = plus(lo, j2), dp = plus(hi, j2), k2 = plus(mid, j2);
      const float x = fmaf(dm.hi, dp.hi, fmaf(dm.hi, dp.lo, dm.lo * dp.hi));
      if (dm.hi > 0.0f) m[4] = fmaf(af / (k2.hi + sqrtf(x)), v, m[4]);
    } else {
      const double dv = double(v);
      const double t = double(j) - tc;
      double tp = t;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        m[i] = fma(tp, dv, m[i]);
        tp *= t;
      }
      const double kap = A.sc.kap + double(j);
      const double x = 4.0 * kap * kap - a;
      if (x > 0.0) m[4] = fma(a / (2.0 * kap + sqrt(x)), dv, m[4]);
    }
  };
  auto use = [&](int j, const ParamSamples<T>& x) {
    if (j >= nk) return;
    cpair<T> a1, a2;
    point(j, x.S1.a, x.S2.a, x.E1.a, x.E2.a, x.f1.a, x.f2.a, a1.a, a2.a);
    point(j + 1, x.S1.b, x.S2.b, x.E1.b, x.E2.b, x.f1.b, x.f2.b, a1.b, a2.b);
    if (A.write_fa) {
      store_two<T>(s1 + j, a1.a, a1.b);
      if (two) store_two<T>(s2 + j, a2.a, a2.b);
    }
  };
  if constexpr (FIT) {
    const C zero = mk<T>(0, 0);
    for (int j = threadIdx.x; j < nk; j += TPB) {
      C Fa1, Fa2;
      point(j, s1[j], s2[j], e1 ? e1[j] : zero, e1 ? e2[j] : zero, f1 ? f1[j] : zero,
            f1 ? f2[j] : zero, Fa1, Fa2);
      if (A.write_fa) {
        s1[j] = Fa1;
        if (two) s2[j] = Fa2;
      }
    }
  } else {
    for (int j = 2 * threadIdx.x; j < nk || j == 2 * threadIdx.x; j += 4 * TPB) {
      const ParamSamples<T> x = load(j), y = load(j + 2 * TPB);
      if (j == 2 * threadIdx.x) {
        __syncthreads();
        lo = {cut_s[0], cut_s[1]};
        hi = {cut_s[2], cut_s[3]};
        mid = {cut_s[4], cut_s[5]};
        af = cut_s[6];
      }
      use(j, x);
      use(j + 2 * TPB, y);
    }
  }
  cudaTriggerProgrammaticLaunchCompletion();
#pragma unroll
  for (int i = 0; i < 5; ++i) part[i][threadIdx.x] = m[i];
  __syncthreads();
  for (int i = threadIdx.x >> 5; i < 5; i += TPB / 32) {
    double s = 0.0;
    for (int k = threadIdx.x & 31; k < TPB; k += 32) s += double(part[i][k]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) A.partial[size_t(blockIdx.x) * 5 + i] += s;
  }
}

template <typename T> cudaError_t launch_param_reduce(const ParamArgs<T>& a, int npairs,
                                                      cudaStream_t s) {
  if constexpr (sizeof(T) == 4)
    if (a.fit) return launch_dependent<T>(k_param_reduce<T, 256, true>, npairs, 256, s, a);
  if (a.sc.nk > 1024) return launch_dependent<T>(k_param_reduce<T, 512>, npairs, 512, s, a);
  if (a.sc.nk > 256) return launch_dependent<T>(k_param_reduce<T, 256>, npairs, 256, s, a);
  return launch_dependent<T>(k_param_reduce<T, 64>, npairs, 64, s, a);
}
template cudaError_t launch_param_reduce<float>(const ParamArgs<float>&, int, cudaStream_t);
template cudaError_t launch_param_reduce<double>(const ParamArgs<double>&, int, cudaStream_t);

// ubar = J_T(u)^T zbar for z = T_tau(u) (Eq. 14), tau = lambda w_n / L:
// where the threshold passes u (the same test as the forward update),
// ubar = zbar - tau (zbar/|u| - u Re(conj(u) zbar)/|u|^3); else 0.
__device__ __forceinline__ float2 st_vjp(float2 u, float2 zb, float tau) {
  const float m2 = fmaf(u.x, u.x, u.y * u.y);
  const float inv = m2 > 0.0f ? rsqrtf(m2) : 0.0f;
  if (!(1.0f - tau * inv > 0.0f)) return make_float2(0.0f, 0.0f);
  const float rz = fmaf(u.x, zb.x, u.y * zb.y) * inv * inv * inv;
  return make_float2(zb.x - tau * (zb.x * inv - u.x * rz), zb.y - tau * (zb.y * inv - u.y * rz));
}
__device__ __forceinline__ double2 st_vjp(double2 u, double2 zb, double tau) {
  const double m2 = fma(u.x, u.x, u.y * u.y);
  const double am = sqrt(m2);
  if (!(m2 > 0.0) || !(1.0 - tau / am > 0.0)) return make_double2(0.0, 0.0);
  const double inv = 1.0 / am;
  const double rz = fma(u.x, zb.x, u.y * zb.y) * inv * inv * inv;
  return make_double2(zb.x - tau * (zb.x * inv - u.x * rz), zb.y - tau * (zb.y * inv - u.y * rz));
}

// The pointwise kernels move 24 and 40 bytes an element (48, and 8 to clear zbar^{k-3},
// when zbar^{k-2} was added to); a thread takes two pairs of neighbours, half a grid
// apart, all of its loads in flight at once.  512 x 2048, cold caches: 7.3 -> 7.5 and
// 10.0 -> 9.0 us; dependent launch hides their ramps (7.15 -> 6.8 ms a calibration
// case of 120 such launches).
constexpr int POINT_THREADS = 256;
inline unsigned point_blocks(size_t n) {
  return unsigned((n + 4 * POINT_THREADS - 1) / (4 * POINT_THREADS));
}

template <typename T>
__global__ void __launch_bounds__(POINT_THREADS)
    k_st_vjp(const cplx<T>* u, const cplx<T>* zbar, const T* w, T lam_over_L, int nz,
             cplx<T>* out, size_t n) {
  const size_t half = size_t(gridDim.x) * (2 * POINT_THREADS);
  const size_t i = 2 * (size_t(blockIdx.x) * POINT_THREADS + threadIdx.x);
  cpair<T> x[2] = {}, y[2] = {};
  cudaGridDependencySynchronize();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const size_t g = i + h * half;
    if (g >= n) continue;
    x[h] = load_two<T>(u + g);
    y[h] = load_two<T>(zbar + g);
  }
  cudaTriggerProgrammaticLaunchCompletion();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const size_t g = i + h * half;
    if (g >= n) continue;
    const T t0 = w ? lam_over_L * w[g & size_t(nz - 1)] : lam_over_L;
    const T t1 = w ? lam_over_L * w[(g + 1) & size_t(nz - 1)] : lam_over_L;
    store_two<T>(out + g, st_vjp(x[h].a, y[h].a, t0), st_vjp(x[h].b, y[h].b, t1));
  }
}
template <typename T> cudaError_t launch_st_vjp(const cplx<T>* u, const cplx<T>* zbar, const T* w,
                                                T lam_over_L, int nz, cplx<T>* out, size_t n,
                                                cudaStream_t s) {
  return launch_dependent<T>(k_st_vjp<T>, point_blocks(n), POINT_THREADS, s, u, zbar, w,
                             lam_over_L, nz, out, n);
}
template cudaError_t launch_st_vjp<float>(const float2*, const float2*, const float*, float, int,
                                          float2*, size_t, cudaStream_t);
template cudaError_t launch_st_vjp<double>(const double2*, const double2*, const double*, double,
                                           int, double2*, size_t, cudaStream_t);

// etabar = ubar - b / L;  zb1 += (1 + mu) etabar;  zb2 = -mu etabar  (zb2 may be null)
template <typename T>
__global__ void __launch_bounds__(POINT_THREADS)
    k_bwd_combine(const cplx<T>* ubar, const cplx<T>* b, T inv_L, T mu, cplx<T>* zb1, cplx<T>* zb2,
                  size_t n) {
  const size_t half = size_t(gridDim.x) * (2 * POINT_THREADS);
  const size_t i = 2 * (size_t(blockIdx.x) * POINT_THREADS + threadIdx.x);
  cpair<T> x[2] = {}, y[2] = {}, z[2] = {};
  cudaGridDependencySynchronize();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const size_t g = i + h * half;
    if (g >= n) continue;
    x[h] = load_two<T>(ubar + g);
    y[h] = load_two<T>(b + g);
    z[h] = load_two<T>(zb1 + g);
  }
  cudaTriggerProgrammaticLaunchCompletion();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const size_t g = i + h * half;
    if (g >= n) continue;
    const cplx<T> e0 = csub(x[h].a, cscale(y[h].a, inv_L)), e1 = csub(x[h].b, cscale(y[h].b, inv_L));
    store_two<T>(zb1 + g, cadd(z[h].a, cscale(e0, T(1) + mu)), cadd(z[h].b, cscale(e1, T(1) + mu)));
    if (zb2) store_two<T>(zb2 + g, cscale(e0, -mu), cscale(e1, -mu));
  }
}
template <typename T> cudaError_t launch_bwd_combine(const cplx<T>* ubar, const cplx<T>* b,
                                                     T inv_L, T mu, cplx<T>* zb1, cplx<T>* zb2,
                                                     size_t n, cudaStream_t s) {
  return launch_dependent<T>(k_bwd_combine<T>, point_blocks(n), POINT_THREADS, s, ubar, b, inv_L,
                             mu, zb1, zb2, n);
}
template cudaError_t launch_bwd_combine<float>(const float2*, const float2*, float, float, float2*,
                                               float2*, size_t, cudaStream_t);
template cudaError_t launch_bwd_combine<double>(const double2*, const double2*, double, double,
                                                double2*, double2*, size_t, cudaStream_t);

}  // namespace isam
