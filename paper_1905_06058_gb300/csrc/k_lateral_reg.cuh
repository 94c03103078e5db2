// k_lat's modes with the tile in registers (lat_reg.cuh); instances in
// k_lateral_reg.cu (FP32) and k_lateral_reg_f64.cu.
//
// What bounds the FP32 form: the update's four global streams (u_hat, z^{k-1} in; z^k,
// eta_hat^{k+1} out), 67 MB at 1024 x 2048 out of the L2.  256 blocks of 256
// threads, two on a multiprocessor (128 registers: 32 points of data, 8 of
// z^{k-1} in flight).  The iterates are loaded in batches of eight, the first
// before the last exchange's barrier so that its latency covers the exchange
// (one by one as the points are used up: 4 us a launch more).  LAT_UPDATE_U at 1024 x
// 2048: 25.6 -> 16.5 us; along y of a 128 x 128 x 2048 volume 209 -> 158 us, 6.8 TB/s.
#pragma once

#include <type_traits>

#include "lat_point.cuh"
#include "lat_reg.cuh"

namespace isam {

template <typename T, int L> __host__ __device__ constexpr int lat_reg_threads() {
  return lreg::threads_per_column<T, L>() * lreg::columns<T, L>();
}
template <typename T, int L> __host__ __device__ constexpr int lat_reg_min_blocks() {
  constexpr int P = lreg::Plan<T, L>::P;
  constexpr int regs = sizeof(T) == 8 ? 128 : P == 32 ? 128 : P == 24 ? 112 : 80;
  constexpr int n = 65536 / (regs * lat_reg_threads<T, L>());
  return n > 16 ? 16 : n;
}

// of a plain transform's grid (see k_lat_reg)
__device__ __forceinline__ bool trigger_at_once() {
  const unsigned blocks = gridDim.x * gridDim.y;
  return blocks <= 32 || blocks > unsigned(kMultiprocessors);
}

template <typename T, int MODE, int L>
__global__ void __launch_bounds__(lat_reg_threads<T, L>(), lat_reg_min_blocks<T, L>())
    k_lat_reg(const __grid_constant__ LatArgs<T> a) {
  using C = cplx<T>;
  constexpr int P = lreg::Plan<T, L>::P, TH = L / P, NT = lat_reg_threads<T, L>();
  constexpr int W = lreg::columns<T, L>();
  // iterates in flight: eight points of z^{k-1}, or four of z^{k-1} and z^{k-2}
  constexpr int BATCH = MODE == LAT_UPDATE ? 4 : 8;
  static_assert(P % BATCH == 0, "the iterates are loaded in whole batches");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* S = reinterpret_cast<C*>(smem_raw);
  const int tid = threadIdx.x, c = tid % W, b = tid / W;
  // programmatic dependent launch: build the twiddles, then wait for the previous
  // kernel's results.  The next kernel may start its prologue before the last
  // transform or stores of a solve's pass (see k_ax_fused).  The plain transforms of
  // 33 to kMultiprocessors blocks, which leave multiprocessors free for the next grid's
  // blocks to crowd, allow it before their stores, the others at once: more blocks
  // leave none free (1024 x 2048: 69 us, 71 if late), and up to 32 are over before the
  // next launch comes, which is then what takes the time.  A + A^H, GPU time at once
  // and late: 4 blocks (128 x 64) 13.4 and 16.2 us, 32 (128 x 512) 13.5 and 15.8, (512 x
  // 512) 23.9 and 25.9, 64 (192 x 1024) 22.5 and 20.5, (256 x 1024) 22.2 and 20.5,
  // 128 (1024 x 1024) 40.0 and 39.2.
  constexpr bool PLAIN = MODE == LAT_C2C_FWD || MODE == LAT_C2C_INV || MODE == LAT_R2C_FWD ||
                         MODE == LAT_INV_REAL;
  const bool early = PLAIN && trigger_at_once();
  if (early) cudaTriggerProgrammaticLaunchCompletion();
  const lreg::Twiddles<T, L> tw(b, a.roots);
  cudaGridDependencySynchronize();
  // the solve's stop flag (written by an earlier kernel, so visible after the
  // wait): loaded here, tested before the first global write
  const bool stopped = a.stop != nullptr && __ldcg(a.stop) != 0;
  const size_t M = size_t(a.M), step = M * TH;         // rows b + i TH of the thread
  const size_t g0 = size_t(blockIdx.y) * L * M + size_t(b) * M + size_t(blockIdx.x) * W + c;
  const T nrm = a.norm;
  auto nothing = [] {};

  C v[P];
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const size_t g = g0 + i * step;
    if constexpr (MODE == LAT_R2C_FWD) {
      v[i] = mk<T>(static_cast<const T*>(a.in)[g], T(0));
    } else if constexpr (MODE == LAT_EXTRAP_FWD) {
      const C z1 = a.z1[g];
      v[i] = cadd(z1, cscale(csub(z1, a.z2[g]), a.mu));
    } else {
      v[i] = static_cast<const C*>(a.in)[g];
    }
  }
  constexpr bool UPDATE = MODE == LAT_UPDATE || MODE == LAT_UPDATE_U;
  constexpr bool FROM_U = MODE == LAT_UPDATE_U;
  constexpr bool EARLY = FROM_U || MODE == LAT_GRAD_STEP;   // first batch before the barrier
  C z1v[BATCH], z2v[BATCH];
  auto load_iterates = [&](int h) {
#pragma unroll
    for (int i = 0; i < BATCH; ++i) {
      z1v[i] = a.z1[g0 + (h + i) * step];
      if constexpr (!FROM_U) z2v[i] = a.z2[g0 + (h + i) * step];
    }
  };
  if constexpr (MODE == LAT_C2C_FWD || MODE == LAT_R2C_FWD || MODE == LAT_EXTRAP_FWD)
    lreg::transform<-1, L, W, 0, T>(v, S, tw, b, c, true, nothing);
  else if constexpr (EARLY)
    lreg::transform<+1, L, W, 0, T>(v, S, tw, b, c, true, [&] { load_iterates(0); });
  else
    lreg::transform<+1, L, W, 0, T>(v, S, tw, b, c, true, nothing);
  if (!UPDATE && !early) cudaTriggerProgrammaticLaunchCompletion();
  if (stopped) return;   // an earlier check stopped the solve: write nothing

  if constexpr (MODE == LAT_INV_REAL) {
    T* out = static_cast<T*>(a.out);
#pragma unroll
    for (int i = 0; i < P; ++i) out[g0 + i * step] = v[i].x * nrm;
  }
  C* out = static_cast<C*>(a.out);
  if constexpr (MODE == LAT_GRAD_STEP) {
    // u = eta^k - g/L with eta^k = z1 + mu_prev (z1 - z2), written to out
    const T sg = nrm * a.inv_L;
    bool bad = false;
#pragma unroll
    for (int h = 0; h < P; h += BATCH) {
      if (h || !EARLY) load_iterates(h);
#pragma unroll
      for (int i = 0; i < BATCH; ++i) {
        const C eta = cadd(z1v[i], cscale(csub(z1v[i], z2v[i]), a.mu_prev));
        const C u = csub(eta, cscale(v[h + i], sg));
        out[g0 + (h + i) * step] = u;
        bad |= !(isfinite(u.x) && isfinite(u.y));
      }
    }
    if (bad) atomicOr(a.flag, 1);
  }
  if constexpr (UPDATE) {
    // the FISTA step of k_lat: LAT_UPDATE forms u = eta^k - g/L from the gradient,
    // LAT_UPDATE_U transformed u itself; norm partials as there (at most 16 points of a
    // thread, so 32 squares, in the plan's precision, then in double)
    T acc0 = T(0), acc1 = T(0), acc2 = T(0), first0 = T(0), first1 = T(0), first2 = T(0);
    bool bad = false;
    const T sg = nrm * a.inv_L;
    T tau = a.lam_dev ? T(a.lam_scale * *a.lam_dev) : a.lam_over_L;
    if (a.w) tau *= a.w[(size_t(blockIdx.x) * W + c) & size_t(a.nz - 1)];
#pragma unroll
    for (int h = 0; h < P; h += BATCH) {
      if (h || !EARLY) load_iterates(h);
      if (!FROM_U && P > 16 && h == P / 2) {
        first0 = acc0; first1 = acc1; first2 = acc2;
        acc0 = acc1 = acc2 = T(0);
      }
#pragma unroll
      for (int i = 0; i < BATCH; ++i) {
        const size_t g = g0 + (h + i) * step;
        const C z1 = z1v[i];
        C gr, eta, u;
        if constexpr (FROM_U) {
          u = cscale(v[h + i], nrm);
        } else {
          gr = cscale(v[h + i], sg);                       // g^k = (1/L) A^H(A eta - s)
          eta = cadd(z1, cscale(csub(z1, z2v[i]), a.mu_prev));
          u = csub(eta, gr);
        }
        if (a.uout) a.uout[g] = u;
        const C z = soft_threshold(u, tau);
        a.zout[g] = z;
        v[h + i] = cadd(z, cscale(csub(z, z1), a.mu));
        // (whether or not they are asked for: a test here made the 1024-point form
        // spill 0.5 KB a thread instead of 0.15; a check iteration 87 -> 82 us)
        if constexpr (!FROM_U) {
          const C d = csub(z, eta);
          const C dg = cadd(d, gr);
          acc0 += d.x * d.x + d.y * d.y;
          acc1 += gr.x * gr.x + gr.y * gr.y;
          acc2 += dg.x * dg.x + dg.y * dg.y;
        }
        bad |= !(isfinite(z.x) && isfinite(z.y));
      }
    }
    if (bad) atomicOr(a.flag, 1);
    cudaTriggerProgrammaticLaunchCompletion();
    lreg::transform<-1, L, W, 0, T>(v, S, tw, b, c, false, nothing);
    if constexpr (!FROM_U) {
      if (a.partial != nullptr) {
        __shared__ double red[3][NT / 32];
        const int wid = tid >> 5, lane = tid & 31;
        const double w0 = warp_sum_lanes(double(acc0) + double(first0), 32);
        const double w1 = warp_sum_lanes(double(acc1) + double(first1), 32);
        const double w2 = warp_sum_lanes(double(acc2) + double(first2), 32);
        if (lane == 0) { red[0][wid] = w0; red[1][wid] = w1; red[2][wid] = w2; }
        __syncthreads();
        if (tid < 3) {
          double s = 0.0;
          for (int w = 0; w < NT / 32; ++w) s += red[tid][w];
          a.partial[3 * (size_t(blockIdx.y) * gridDim.x + blockIdx.x) + tid] = s;
        }
      }
    }
  }
  if constexpr (MODE != LAT_INV_REAL && MODE != LAT_GRAD_STEP) {
#pragma unroll
    for (int i = 0; i < P; ++i) out[g0 + i * step] = cscale(v[i], nrm);
  }
}

template <typename T, int MODE, int L>
static cudaError_t launch_lat_reg_mode(const LatArgs<T>& a, cudaStream_t s) {
  auto* kern = k_lat_reg<T, MODE, L>;
  constexpr size_t sm = lreg::smem_elements<T, L, lreg::columns<T, L>()>() * sizeof(cplx<T>);
  allow_smem(kern, sm);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.M / lreg::columns<T, L>(), a.B);
  cfg.blockDim = dim3(lat_reg_threads<T, L>());
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = sizeof(T) == 4;   // as the axial kernels
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

// Real transforms of the half spectrum: a thread's complex column is two neighbouring
// real ones, z = x_m + i x_{m+1}, so a real array takes half the transforms and its
// spectrum half the memory.  FWD: H_m = (Z(q) + conj Z(-q)) / 2 and H_{m+1} = -i (Z(q) -
// conj Z(-q)) / 2 of rows q <= L/2 after one more exchange; else Z(q) = H_m(q) + i
// H_{m+1}(q), with H(-q) = conj H(q), as the rows are loaded.  M: real columns.
template <bool FWD, int L>
__global__ void __launch_bounds__(lat_reg_threads<float, L>(), lat_reg_min_blocks<float, L>())
    k_lat_half(const __grid_constant__ LatArgs<float> a) {
  constexpr int P = lreg::Plan<float, L>::P, TH = L / P, W = lreg::columns<float, L>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* S = reinterpret_cast<float2*>(smem_raw);
  const int tid = threadIdx.x, c = tid % W, b = tid / W;
  // dependent launch as the plain passes of k_lat_reg
  const bool early = trigger_at_once();
  if (early) cudaTriggerProgrammaticLaunchCompletion();
  const lreg::Twiddles<float, L> tw(b, nullptr);
  cudaGridDependencySynchronize();
  const size_t M = size_t(a.M), m = size_t(blockIdx.x) * (2 * W) + 2 * c;
  const size_t real0 = size_t(blockIdx.y) * L * M + m, half0 = size_t(blockIdx.y) * (L / 2 + 1) * M + m;
  float2 v[P];
  if constexpr (FWD) {
    const float* in = static_cast<const float*>(a.in) + real0;
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = *reinterpret_cast<const float2*>(in + (b + i * TH) * M);
    lreg::transform<-1, L, W, 0, float>(v, S, tw, b, c, true, [] {});
    __syncthreads();
#pragma unroll
    for (int i = 0; i < P; ++i) S[lreg::slot<float, L, W>(b + i * TH, c)] = v[i];
    __syncthreads();
    if (!early) cudaTriggerProgrammaticLaunchCompletion();
    float2* out = static_cast<float2*>(a.out) + half0;
    const float f = 0.5f * a.norm;
#pragma unroll
    for (int i = 0; i <= P / 2; ++i) {
      const int q = b + i * TH;
      if (q > L / 2) break;
      const float2 z = v[i], y = S[lreg::slot<float, L, W>(q ? L - q : 0, c)];
      const float4 h = make_float4(f * (z.x + y.x), f * (z.y - y.y), f * (z.y + y.y), f * (y.x - z.x));
      *reinterpret_cast<float4*>(out + q * M) = h;
    }
  } else {
    const float2* in = static_cast<const float2*>(a.in) + half0;
#pragma unroll
    for (int i = 0; i < P; ++i) {
      const int q = b + i * TH;
      const bool upper = q > L / 2;
      const float4 h = *reinterpret_cast<const float4*>(in + (upper ? L - q : q) * M);
      const float s = upper ? -1.0f : 1.0f;             // conj
      v[i] = make_float2(h.x - s * h.w, s * h.y + h.z);
    }
    lreg::transform<+1, L, W, 0, float>(v, S, tw, b, c, true, [] {});
    if (!early) cudaTriggerProgrammaticLaunchCompletion();
    float* out = static_cast<float*>(a.out) + real0;
#pragma unroll
    for (int i = 0; i < P; ++i)
      *reinterpret_cast<float2*>(out + (b + i * TH) * M) = cscale(v[i], a.norm);
  }
}

template <int L> static cudaError_t launch_lat_half_length(int mode, const LatArgs<float>& a,
                                                           cudaStream_t s) {
  constexpr int W = lreg::columns<float, L>();
  constexpr size_t sm = lreg::smem_elements<float, L, W>() * sizeof(float2);
  auto* kern = mode == LAT_R2C_HALF ? k_lat_half<true, L> : k_lat_half<false, L>;
  allow_smem(kern, sm);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.M / (2 * W), a.B);
  cfg.blockDim = dim3(lat_reg_threads<float, L>());
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <typename T, int L>
static cudaError_t launch_lat_reg_length(int mode, const LatArgs<T>& a, cudaStream_t s) {
  switch (mode) {
    case LAT_C2C_FWD: return launch_lat_reg_mode<T, LAT_C2C_FWD, L>(a, s);
    case LAT_C2C_INV: return launch_lat_reg_mode<T, LAT_C2C_INV, L>(a, s);
    case LAT_R2C_FWD: return launch_lat_reg_mode<T, LAT_R2C_FWD, L>(a, s);
    case LAT_INV_REAL: return launch_lat_reg_mode<T, LAT_INV_REAL, L>(a, s);
    case LAT_UPDATE: return launch_lat_reg_mode<T, LAT_UPDATE, L>(a, s);
    case LAT_GRAD_STEP: return launch_lat_reg_mode<T, LAT_GRAD_STEP, L>(a, s);
    case LAT_EXTRAP_FWD: return launch_lat_reg_mode<T, LAT_EXTRAP_FWD, L>(a, s);
    case LAT_UPDATE_U: return launch_lat_reg_mode<T, LAT_UPDATE_U, L>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace isam
