// The other priors' proxes.
//
// Total-variation prior (§3.1 names TV among the convex priors Eq. 12 extends
// to): isotropic TV over (x, z) of each B-scan slice of the image
// [ny][nx][nz], with forward differences that are zero at the far edge.  Its
// prox z = argmin 1/2 ||z - u||^2 + tau TV(z) is found on the dual,
// z = u - tau grad^H p with |p| <= 1 per pixel, by fast gradient projection
// (Beck & Teboulle): steps of 1/(8 tau) (||grad||^2 <= 8), projection, and
// momentum beta_k from the host.
//
// FP32 runs several dual steps per launch on tiles in registers (k_tv_tile);
// FP64, whose arithmetic the tiles' halos would repeat at the FP64 pipe's rate, and
// FP32 plans without room for the tiles' images run two kernels a step, each writing
// only its own pixel.
#include <math.h>

#include "internal.cuh"
#include "lat_point.cuh"

namespace isam {

template <typename T>
__device__ __forceinline__ T tv_tau(T tau, const double* lam_dev, double lam_scale) {
  return lam_dev ? T(lam_scale * *lam_dev) : tau;
}

// w = u - tau grad^H r,  (grad^H r)(x, z) = r_x(x-1, z) - r_x(x, z) + r_z(x, z-1) - r_z(x, z)
// with r_x(x, .) = 0 for x = -1 or x = nx - 1 and r_z(., z) = 0 for z = -1 or z = nz - 1
template <typename T>
__global__ void k_tv_primal(const cplx<T>* u, const cplx<T>* rx, const cplx<T>* rz, T tau0,
                            const double* lam_dev, double lam_scale, cplx<T>* w, int nx, int nz,
                            size_t n) {
  const T tau = tv_tau(tau0, lam_dev, lam_scale);
  for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += size_t(gridDim.x) * blockDim.x) {
    const int z = int(i & size_t(nz - 1));
    const int x = int((i / size_t(nz)) % size_t(nx));
    cplx<T> a = mk<T>(0, 0);
    if (x < nx - 1) a = csub(a, rx[i]);
    if (x > 0) a = cadd(a, rx[i - nz]);
    if (z < nz - 1) a = csub(a, rz[i]);
    if (z > 0) a = cadd(a, rz[i - 1]);
    w[i] = tau > T(0) ? csub(u[i], cscale(a, tau)) : u[i];
  }
}

// q = r + grad(w) / (8 tau), p_new = q / max(1, |q|), r = p_new + beta (p_new - p), p = p_new
template <typename T>
__global__ void k_tv_dual(const cplx<T>* w, cplx<T>* px, cplx<T>* pz, cplx<T>* rx, cplx<T>* rz,
                          T tau0, const double* lam_dev, double lam_scale, T beta, int nx, int nz,
                          size_t n) {
  const T tau = tv_tau(tau0, lam_dev, lam_scale);
  for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += size_t(gridDim.x) * blockDim.x) {
    if (!(tau > T(0))) {                       // tau = 0: z = u
      px[i] = pz[i] = rx[i] = rz[i] = mk<T>(0, 0);
      continue;
    }
    const int z = int(i & size_t(nz - 1));
    const int x = int((i / size_t(nz)) % size_t(nx));
    const cplx<T> wi = w[i];
    const cplx<T> gx = x < nx - 1 ? csub(w[i + nz], wi) : mk<T>(0, 0);
    const cplx<T> gz = z < nz - 1 ? csub(w[i + 1], wi) : mk<T>(0, 0);
    const T s = T(1) / (T(8) * tau);
    const cplx<T> qx = cadd(rx[i], cscale(gx, s));
    const cplx<T> qz = cadd(rz[i], cscale(gz, s));
    const T m2 = qx.x * qx.x + qx.y * qx.y + qz.x * qz.x + qz.y * qz.y;
    const T f = m2 > T(1) ? T(1) / sqrt(m2) : T(1);
    const cplx<T> nxv = cscale(qx, f), nzv = cscale(qz, f);
    rx[i] = cadd(nxv, cscale(csub(nxv, px[i]), beta));
    rz[i] = cadd(nzv, cscale(csub(nzv, pz[i]), beta));
    px[i] = nxv;
    pz[i] = nzv;
  }
}

// Several dual steps of one tile.  A dual step at a pixel reaches one pixel to
// each side, so a tile of 64 x 64 pixels loaded with a halo of `steps` pixels is
// right inside the halo after `steps` steps (one more for the last launch, which
// also forms z = u - tau grad^H p).  512 threads: thread (g, c) holds column
// z = c of rows 8 g .. 8 g + 7, with u, p, r and w in registers; the neighbours in
// z and across row groups go through shared memory.
//
// One step as two kernels moved 10 images through the L2; a launch of five steps
// reads 5 images and writes 4, with 1.2 to 1.4 times the arithmetic, and its time
// is the steps' arithmetic, barriers and shared-memory neighbours.  20 steps at
// 384 x 1024: 41 launches in 250 us before, 4 in 70 us now.  At 128 registers it spills 128
// bytes a thread.
constexpr int TV_TILE = 64, TV_ROWS = 8;

struct TvTile {
  const float2 *u, *px, *pz, *rx, *rz;   // rx null: r = p (the first launch)
  float2 *px_out, *pz_out, *rx_out, *rz_out, *z;   // z: last launch (then no r)
  float tau;
  const double* lam_dev;
  double lam_scale;
  int nx, nz, steps, halo;
  float beta[TV_STEPS];
};

// 1 / sqrt(x) of a finite x >= 1: one Newton step on the approximation.  Over all floats of
// [1, 4) off by 7.4e-8 at most and 2.9e-8 rms (1.0f / sqrtf(x): 8.9e-8 and 3.6e-8), and
// the TV solve at 384 x 1024 takes 1,105 us (1,256 with that).
__device__ __forceinline__ float rsqrt_newton(float x) {
  const float y = rsqrtf(x);
  return fmaf(0.5f * y, fmaf(-x * y, y, 1.0f), y);
}

__global__ void __launch_bounds__(512, 1) k_tv_tile(const __grid_constant__ TvTile A) {
  extern __shared__ __align__(16) unsigned char raw[];
  float2(*RZ)[TV_TILE] = reinterpret_cast<float2(*)[TV_TILE]>(raw);            // r_z
  float2(*W)[TV_TILE] = RZ + TV_TILE;                                          // w
  float2(*RX)[TV_TILE] = W + TV_TILE;                                          // r_x of row 8 g + 7
  const int c = threadIdx.x & (TV_TILE - 1), g = threadIdx.x / TV_TILE, row0 = TV_ROWS * g;
  const int inner = TV_TILE - 2 * A.halo;
  const int gz = blockIdx.x * inner - A.halo + c, gx0 = blockIdx.y * inner - A.halo + row0;
  const int nx = A.nx, nz = A.nz;
  const size_t at = (size_t(blockIdx.z) * nx + gx0) * nz + gz;    // of row 0; used where valid
  // programmatic dependent launch, as the other kernels of an iteration
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  const float tau = tv_tau(A.tau, A.lam_dev, A.lam_scale);
  const bool col = gz >= 0 && gz < nz;
  const float2 zero = make_float2(0.0f, 0.0f);
  float2 u[TV_ROWS], px[TV_ROWS], pz[TV_ROWS], rx[TV_ROWS], rz[TV_ROWS], w[TV_ROWS];
#pragma unroll
  for (int i = 0; i < TV_ROWS; ++i) {
    const bool in = col && gx0 + i >= 0 && gx0 + i < nx;
    const size_t k = at + size_t(i) * nz;
    u[i] = in ? A.u[k] : zero;
    px[i] = in ? A.px[k] : zero;
    pz[i] = in ? A.pz[k] : zero;
    rx[i] = in && A.rx ? A.rx[k] : px[i];
    rz[i] = in && A.rx ? A.rz[k] : pz[i];
  }
  const bool live = tau > 0.0f;                          // tau = 0: p = r = 0, z = u
  const float s = live ? 1.0f / (8.0f * tau) : 0.0f;
  // u - tau grad^H r at the thread's pixels (k_tv_primal's form); a barrier before
  // its reads
  auto primal = [&](const float2* ax, const float2* az) {
#pragma unroll
    for (int i = 0; i < TV_ROWS; ++i) RZ[row0 + i][c] = az[i];
    RX[g][c] = ax[TV_ROWS - 1];
    __syncthreads();
    const float2 above = g ? RX[g - 1][c] : zero;
#pragma unroll
    for (int i = 0; i < TV_ROWS; ++i) {
      const int x = gx0 + i;
      float2 a = zero;
      if (x < nx - 1) a = csub(a, ax[i]);
      if (x > 0) a = cadd(a, i ? ax[i - 1] : above);
      if (gz < nz - 1) a = csub(a, az[i]);
      if (gz > 0) a = cadd(a, c ? RZ[row0 + i][c - 1] : zero);
      w[i] = csub(u[i], cscale(a, tau));
    }
  };
  if (live) {
    for (int k = 0; k < A.steps; ++k) {
      const float beta = A.beta[k];
      primal(rx, rz);
#pragma unroll
      for (int i = 0; i < TV_ROWS; ++i) W[row0 + i][c] = w[i];
      __syncthreads();
      const float2 below = g < TV_TILE / TV_ROWS - 1 ? W[row0 + TV_ROWS][c] : zero;
#pragma unroll
      for (int i = 0; i < TV_ROWS; ++i) {
        const float2 gxv = gx0 + i < nx - 1 ? csub(i < TV_ROWS - 1 ? w[i + 1] : below, w[i]) : zero;
        const float2 gzv = gz < nz - 1 && c < TV_TILE - 1 ? csub(W[row0 + i][c + 1], w[i]) : zero;
        const float2 qx = cadd(rx[i], cscale(gxv, s)), qz = cadd(rz[i], cscale(gzv, s));
        const float m2 = qx.x * qx.x + qx.y * qx.y + qz.x * qz.x + qz.y * qz.y;
        // (|q|^2 overflows at a very small tau: then tau p is 0 to rounding, so p = 0)
        const float f = m2 > 1.0f ? (m2 < INFINITY ? rsqrt_newton(m2) : 0.0f) : 1.0f;
        const float2 nxv = cscale(qx, f), nzv = cscale(qz, f);
        rx[i] = cadd(nxv, cscale(csub(nxv, px[i]), beta));
        rz[i] = cadd(nzv, cscale(csub(nzv, pz[i]), beta));
        px[i] = nxv;
        pz[i] = nzv;
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < TV_ROWS; ++i) px[i] = pz[i] = rx[i] = rz[i] = zero;
  }
  if (A.z) {
    // after a barrier of every step's readers of RZ (the one before the dual update)
    if (live) primal(px, pz);
    else {
#pragma unroll
      for (int i = 0; i < TV_ROWS; ++i) w[i] = u[i];
    }
  }
#pragma unroll
  for (int i = 0; i < TV_ROWS; ++i) {
    const int r = row0 + i;
    if (!col || gx0 + i >= nx || r < A.halo || r >= TV_TILE - A.halo || c < A.halo ||
        c >= TV_TILE - A.halo)
      continue;
    const size_t k = at + size_t(i) * nz;
    A.px_out[k] = px[i];
    A.pz_out[k] = pz[i];
    if (A.z) {
      A.z[k] = w[i];
    } else {
      A.rx_out[k] = rx[i];
      A.rz_out[k] = rz[i];
    }
  }
}

cudaError_t launch_tv_tile(const TvLaunch& l, cudaStream_t s) {
  TvTile a{};
  a.u = l.u;
  a.px = l.in[0]; a.pz = l.in[1]; a.rx = l.in[2]; a.rz = l.in[3];
  a.px_out = l.out[0]; a.pz_out = l.out[1]; a.rx_out = l.out[2]; a.rz_out = l.out[3];
  a.z = l.z;
  a.tau = l.tau; a.lam_dev = l.lam_dev; a.lam_scale = l.lam_scale;
  a.nx = l.nx; a.nz = l.nz;
  a.steps = l.steps;
  a.halo = l.steps + (l.z ? 1 : 0);
  for (int i = 0; i < l.steps; ++i) a.beta[i] = l.beta[i];
  const int inner = TV_TILE - 2 * a.halo;
  const dim3 grid((l.nz + inner - 1) / inner, (l.nx + inner - 1) / inner, l.ny);
  const size_t sm = (2 * TV_TILE + TV_TILE / TV_ROWS) * TV_TILE * sizeof(float2);
  allow_smem(k_tv_tile, sm);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_tv_tile, a);
}

template <typename T> cudaError_t launch_tv_primal(const cplx<T>* u, const cplx<T>* rx,
                                                   const cplx<T>* rz, T tau, const double* lam_dev,
                                                   double lam_scale, cplx<T>* w, int nx, int nz,
                                                   size_t n, cudaStream_t s) {
  k_tv_primal<T><<<1024, 256, 0, s>>>(u, rx, rz, tau, lam_dev, lam_scale, w, nx, nz, n);
  return cudaGetLastError();
}
template <typename T> cudaError_t launch_tv_dual(const cplx<T>* w, cplx<T>* px, cplx<T>* pz,
                                                 cplx<T>* rx, cplx<T>* rz, T tau,
                                                 const double* lam_dev, double lam_scale, T beta,
                                                 int nx, int nz, size_t n, cudaStream_t s) {
  k_tv_dual<T><<<1024, 256, 0, s>>>(w, px, pz, rx, rz, tau, lam_dev, lam_scale, beta, nx, nz, n);
  return cudaGetLastError();
}
template cudaError_t launch_tv_primal<float>(const float2*, const float2*, const float2*,
                                              float, const double*, double, float2*, int, int,
                                              size_t, cudaStream_t);
template cudaError_t launch_tv_primal<double>(const double2*, const double2*, const double2*,
                                              double, const double*, double, double2*, int, int,
                                              size_t, cudaStream_t);
template cudaError_t launch_tv_dual<float>(const float2*, float2*, float2*, float2*, float2*,
                                            float, const double*, double, float, int, int, size_t,
                                            cudaStream_t);
template cudaError_t launch_tv_dual<double>(const double2*, double2*, double2*, double2*, double2*,
                                            double, const double*, double, double, int, int, size_t,
                                            cudaStream_t);

// ---------------------------------------------------------------------------
// Haar prior
// ---------------------------------------------------------------------------
// prox of tau ||details(W u)||_1 per A-scan (nz contiguous samples), W the
// orthonormal Haar transform along depth: in-place lifting levels with
// stride h = 1, 2, .., nz/2 (pair (i, i + h), i a multiple of 2h, becomes
// ((x_i + x_{i+h})/sqrt 2, (x_i - x_{i+h})/sqrt 2)), the complex soft
// threshold on every coefficient but the approximation (index 0), and the
// same butterflies in reverse order, which invert them.
template <typename T>
__global__ void k_haar_prox(const cplx<T>* u, cplx<T>* z, int nz, T tau, const double* lam_dev,
                            double lam_scale) {
  extern __shared__ __align__(16) unsigned char raw[];
  cplx<T>* x = reinterpret_cast<cplx<T>*>(raw);
  const size_t col = blockIdx.x;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int i = tid; i < nz; i += nt) x[i] = u[col * nz + i];
  __syncthreads();
  const T r = T(0.70710678118654752440);
  for (int h = 1; h < nz; h <<= 1) {
    for (int p = tid; p < nz / (2 * h); p += nt) {
      const int i = p * 2 * h;
      const cplx<T> a0 = x[i], a1 = x[i + h];
      x[i] = cscale(cadd(a0, a1), r);
      x[i + h] = cscale(csub(a0, a1), r);
    }
    __syncthreads();
  }
  const T t = lam_dev ? T(lam_scale * *lam_dev) : tau;
  for (int i = tid; i < nz; i += nt)
    if (i) x[i] = soft_threshold(x[i], t);
  __syncthreads();
  for (int h = nz >> 1; h >= 1; h >>= 1) {
    for (int p = tid; p < nz / (2 * h); p += nt) {
      const int i = p * 2 * h;
      const cplx<T> a0 = x[i], a1 = x[i + h];
      x[i] = cscale(cadd(a0, a1), r);
      x[i + h] = cscale(csub(a0, a1), r);
    }
    __syncthreads();
  }
  for (int i = tid; i < nz; i += nt) z[col * nz + i] = x[i];
}

// The same for nz = 256 .. 2048, with the A-scan in registers: a lane holds 8
// consecutive samples (three levels), a warp 256 (five more by shuffles), and the
// A-scan's nz / 256 warps combine their approximations through shared memory; 8
// warps, so 2048 / nz A-scans, a block.  Loads and stores are transposed within
// the warp so that global rows stay contiguous.  The levels through shared memory
// took 22 barriers, the last of them for one pair: 17.5 us at 512 x 2048, whose
// 16.8 MB it now moves at the L2's rate.
template <typename T> __device__ __forceinline__ cplx<T> shfl_xor_c(cplx<T> a, int m) {
  return mk<T>(__shfl_xor_sync(0xffffffffu, a.x, m), __shfl_xor_sync(0xffffffffu, a.y, m));
}
template <typename T>
__global__ void __launch_bounds__(256) k_haar_regs(const cplx<T>* u, cplx<T>* z, int nz, size_t n,
                                                   T tau, const double* lam_dev,
                                                   double lam_scale) {
  using C = cplx<T>;
  __shared__ C buf[8][288];                            // a warp's 256 samples, padded
  __shared__ C approx[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = nz / 256, first = warp / G * G, part = warp - first;
  const size_t scan = size_t(blockIdx.x) * (8 / G) + warp / G;
  const bool in = scan < n;
  const size_t base = scan * nz + size_t(part) * 256;
  const T r = T(0.70710678118654752440);
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  const T t = lam_dev ? T(lam_scale * *lam_dev) : tau;
  C x[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int e = 32 * k + lane;
    buf[warp][e + (e >> 3)] = in ? u[base + e] : mk<T>(0, 0);
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 8; ++k) x[k] = buf[warp][9 * lane + k];
#pragma unroll
  for (int h = 1; h < 8; h <<= 1)
#pragma unroll
    for (int i = 0; i < 8; i += 2 * h) {
      const C a0 = x[i], a1 = x[i + h];
      x[i] = cscale(cadd(a0, a1), r);
      x[i + h] = soft_threshold(cscale(csub(a0, a1), r), t);
    }
  // one level between lanes h apart: sums on the lanes of even multiples of h, and
  // on those of odd ones the differences, thresholded on the way up
  auto level = [&](C a, int h, bool up) {
    const C v = shfl_xor_c<T>(a, h);
    const int m = lane & (2 * h - 1);
    if (m == 0) return cscale(cadd(a, v), r);
    if (m != h) return a;
    const C d = cscale(csub(v, a), r);
    return up ? soft_threshold(d, t) : d;
  };
  C a = x[0];
#pragma unroll
  for (int h = 1; h < 32; h <<= 1) a = level(a, h, true);
  if (lane == 0) approx[warp] = a;
  __syncthreads();
  C y = approx[first + (lane & (G - 1))];
  for (int h = 1; h < G; h <<= 1) y = level(y, h, true);
  for (int h = G >> 1; h >= 1; h >>= 1) y = level(y, h, false);
  y = mk<T>(__shfl_sync(0xffffffffu, y.x, part), __shfl_sync(0xffffffffu, y.y, part));
  if (lane == 0) a = y;
#pragma unroll
  for (int h = 16; h >= 1; h >>= 1) a = level(a, h, false);
  x[0] = a;
#pragma unroll
  for (int h = 4; h >= 1; h >>= 1)
#pragma unroll
    for (int i = 0; i < 8; i += 2 * h) {
      const C a0 = x[i], a1 = x[i + h];
      x[i] = cscale(cadd(a0, a1), r);
      x[i + h] = cscale(csub(a0, a1), r);
    }
#pragma unroll
  for (int k = 0; k < 8; ++k) buf[warp][9 * lane + k] = x[k];
  __syncwarp();
  if (!in) return;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int e = 32 * k + lane;
    z[base + e] = buf[warp][e + (e >> 3)];
  }
}

template <typename T> cudaError_t launch_haar_prox(const cplx<T>* u, cplx<T>* z, int nz,
                                                   size_t n_ascans, T tau, const double* lam_dev,
                                                   double lam_scale, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  if (nz >= 256) {
    const size_t per_block = 2048 / nz;
    cfg.gridDim = dim3(unsigned((n_ascans + per_block - 1) / per_block));
    cfg.blockDim = dim3(256);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = sizeof(T) == 4;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_haar_regs<T>, u, z, nz, n_ascans, tau, lam_dev, lam_scale);
  }
  cfg.gridDim = dim3(unsigned(n_ascans));
  cfg.blockDim = dim3(nz / 2 >= 32 ? nz / 2 : 32);
  cfg.dynamicSmemBytes = size_t(nz) * sizeof(cplx<T>);
  return cudaLaunchKernelEx(&cfg, k_haar_prox<T>, u, z, nz, tau, lam_dev, lam_scale);
}
template cudaError_t launch_haar_prox<float>(const float2*, float2*, int, size_t, float,
                                             const double*, double, cudaStream_t);
template cudaError_t launch_haar_prox<double>(const double2*, double2*, int, size_t, double,
                                              const double*, double, cudaStream_t);

}  // namespace isam
