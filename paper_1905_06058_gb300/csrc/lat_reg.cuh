// Lateral passes of FP32 plans with the tile held in registers.
//
// A block takes W consecutive columns m of one batch of data viewed as [B][L][M];
// each of its threads owns P points of one column, rows b + i T (T = L / P, thread
// b of the column, i < P).  A Stockham pass of radix R | P whose span divides T
// reads exactly those rows, and the last pass leaves its results in them, so a
// transform loads from global memory straight into its first pass, meets shared
// memory only in the exchange between passes, and ends in registers: the FISTA
// step and the forward transform after it start there, and the last pass stores
// to global memory.  1024 = 32 x 32, 512 = 16 x 32 and 256 = 16 x 16 take one
// exchange a transform.
//
// The tile in shared memory with 16 points a thread, three passes and a load, an
// update and a store phase moved it 16 times through shared memory at 166
// instructions a point of the update; this form moves it 4 times.
#pragma once

#include "fft_col16.cuh"
#include "internal.cuh"

namespace isam {
namespace lreg {

// cos and sin of 2 pi k / n at compile time (Taylor series, |angle| <= pi / 4
// after the octant symmetries)
constexpr double kPi = 3.14159265358979323846;
__host__ __device__ constexpr double series_cos(double x) {
  double t = 1.0, s = 1.0;
  for (int i = 1; i < 14; ++i) { t *= -x * x / ((2 * i - 1) * (2 * i)); s += t; }
  return s;
}
__host__ __device__ constexpr double series_sin(double x) {
  double t = x, s = x;
  for (int i = 1; i < 14; ++i) { t *= -x * x / ((2 * i) * (2 * i + 1)); s += t; }
  return s;
}
__host__ __device__ constexpr double cos_turn(int k, int n) {            // cos(2 pi k / n)
  k %= n;
  if (k < 0) k += n;
  if (2 * k > n) k = n - k;                           // cos even
  if (4 * k > n) return -cos_turn(n - 2 * k, 2 * n);  // cos(pi - x) = -cos x
  if (8 * k > n) return series_sin(2.0 * kPi * (double(n) / 4 - k) / n);
  return series_cos(2.0 * kPi * k / n);
}
__host__ __device__ constexpr double sin_turn(int k, int n) { return cos_turn(4 * k - n, 4 * n); }  // cos(x - pi/2)

// o times e^{SIGN 2 pi i k / N}
template <int SIGN, int N, int K> __device__ __forceinline__ float2 mul_root(float2 o) {
  constexpr int k = K % N;
  if constexpr (k == 0) return o;
  else if constexpr (4 * k == N) return cmul_i<SIGN>(o);
  else if constexpr (2 * k == N) return make_float2(-o.x, -o.y);
  else if constexpr (4 * k == 3 * N) return cmul_i<-SIGN>(o);
  else if constexpr (8 * k == N) return ew8_1<SIGN>(o);
  else if constexpr (8 * k == 3 * N) return ew8_3<SIGN>(o);
  else {
    constexpr float c = float(cos_turn(k, N)), s = float(SIGN * sin_turn(k, N));
    return make_float2(o.x * c - o.y * s, o.y * c + o.x * s);
  }
}

template <int SIGN> __device__ __forceinline__ void dft3(float2& a0, float2& a1, float2& a2) {
  const float h = 0.86602540378443864676f;            // sqrt(3)/2
  const float2 t1 = cadd(a1, a2), d = cscale(csub(a1, a2), h);
  const float2 t2 = csub(a0, cscale(t1, 0.5f));
  a0 = cadd(a0, t1);
  a1 = add_rot<SIGN>(t2, d);
  a2 = sub_rot<SIGN>(t2, d);
}

// W_N^{n2 k1} on column n2 of the first stage's outputs, k1 = 1 .. N1-1
template <int SIGN, int N, int N1, int N2, int n2, int k1 = 1>
__device__ __forceinline__ void root_column(float2 (&b)[N2][N1]) {
  if constexpr (k1 < N1) {
    b[n2][k1] = mul_root<SIGN, N, n2 * k1>(b[n2][k1]);
    root_column<SIGN, N, N1, N2, n2, k1 + 1>(b);
  }
}
template <int SIGN, int N, int N1, int N2, int n2 = 1>
__device__ __forceinline__ void root_columns(float2 (&b)[N2][N1]) {
  if constexpr (n2 < N2) {
    root_column<SIGN, N, N1, N2, n2>(b);
    root_columns<SIGN, N, N1, N2, n2 + 1>(b);
  }
}

// 8 N1-point DFT (N1 = 3 or 4) in place, natural order in and out:
// X[k1 + N1 k2] = sum_{n2 < 8} W8^{n2 k2} W_N^{n2 k1} sum_{n1} x[n2 + 8 n1] W_N1^{n1 k1}
template <int SIGN, int N1> __device__ __forceinline__ void dft_8x(float2* a) {
  constexpr int N = 8 * N1;
  float2 b[8][N1];
#pragma unroll
  for (int n2 = 0; n2 < 8; ++n2) {
    if constexpr (N1 == 4) {
      float2 x0 = a[n2], x1 = a[n2 + 8], x2 = a[n2 + 16], x3 = a[n2 + 24];
      dft4<SIGN>(x0, x1, x2, x3);
      b[n2][0] = x0; b[n2][1] = x1; b[n2][2] = x2; b[n2][3] = x3;
    } else {
      float2 x0 = a[n2], x1 = a[n2 + 8], x2 = a[n2 + 16];
      dft3<SIGN>(x0, x1, x2);
      b[n2][0] = x0; b[n2][1] = x1; b[n2][2] = x2;
    }
  }
  root_columns<SIGN, N, N1, 8>(b);
#pragma unroll
  for (int k1 = 0; k1 < N1; ++k1) {
    float2 y[8];
#pragma unroll
    for (int n2 = 0; n2 < 8; ++n2) y[n2] = b[n2][k1];
    dft8<SIGN>(y);
#pragma unroll
    for (int k2 = 0; k2 < 8; ++k2) a[k1 + N1 * k2] = y[k2];
  }
}

template <int SIGN, int R> __device__ __forceinline__ void dft(float2* a) {
  if constexpr (R == 32) dft_8x<SIGN, 4>(a);
  else if constexpr (R == 24) dft_8x<SIGN, 3>(a);
  else c16::dft_r<SIGN, R>(a);
}

// The radices of a length: P points a thread, N passes of radices R0, R1, R2, each of
// the span of those before it.  Every span divides T = L / P, so a thread's butterflies of a
// pass share one twiddle base.
template <int L> struct Plan;
template <> struct Plan<1024> { static constexpr int P = 32, N = 2, R0 = 32, R1 = 32, R2 = 1; };
template <> struct Plan<512> { static constexpr int P = 32, N = 2, R0 = 16, R1 = 32, R2 = 1; };
template <> struct Plan<256> { static constexpr int P = 16, N = 2, R0 = 16, R1 = 16, R2 = 1; };
template <> struct Plan<128> { static constexpr int P = 16, N = 2, R0 = 8, R1 = 16, R2 = 1; };
template <> struct Plan<64> { static constexpr int P = 8, N = 2, R0 = 8, R1 = 8, R2 = 1; };
template <> struct Plan<768> { static constexpr int P = 24, N = 3, R0 = 4, R1 = 8, R2 = 24; };
template <> struct Plan<384> { static constexpr int P = 24, N = 3, R0 = 4, R1 = 4, R2 = 24; };
template <> struct Plan<192> { static constexpr int P = 24, N = 2, R0 = 8, R1 = 24, R2 = 1; };

template <int L> __host__ __device__ constexpr int threads_per_column() { return L / Plan<L>::P; }
template <int L> __host__ __device__ constexpr int radix(int pass) {
  return pass == 0 ? Plan<L>::R0 : pass == 1 ? Plan<L>::R1 : Plan<L>::R2;
}
template <int L> __host__ __device__ constexpr int span(int pass) {
  return pass == 0 ? 1 : pass == 1 ? Plan<L>::R0 : Plan<L>::R0 * Plan<L>::R1;
}
// A padding row after every R0 rows where two rows share a half warp (W = 8):
// the first pass's writes to rows R0 b + r of neighbouring b then fall in
// different halves of the banks.  At W = 16 a half warp is one row.
template <int L, int W> __device__ __forceinline__ int slot(int row, int c) {
  if constexpr (W >= 16) return row * W + c;
  else return (row + row / Plan<L>::R0) * W + c;
}
template <int L, int W> __host__ __device__ constexpr size_t smem_bytes() {
  return size_t(W >= 16 ? L : L + L / Plan<L>::R0) * W * sizeof(float2);
}

// w^1, w^4, w^16 of a pass, w = e^{-2 pi i k / (span R)}, k = b mod span
struct Roots { float2 w1, w4, w16; };
__device__ __forceinline__ float2 root(int k, int n) {
  float s, c;
  sincospif(float(2 * k) / float(n), &s, &c);
  return make_float2(c, -s);
}
template <int L> struct Twiddles {
  Roots p[Plan<L>::N - 1];
  __device__ __forceinline__ explicit Twiddles(int b) {
#pragma unroll
    for (int i = 1; i < Plan<L>::N; ++i) {
      const int ns = span<L>(i), R = radix<L>(i), n = ns * R, k = b % ns;
      p[i - 1].w1 = root(k, n);
      if (R > 4) p[i - 1].w4 = root(4 * k, n);
      if (R > 16) p[i - 1].w16 = root(16 * k, n);
    }
  }
};

// a[r] *= w^r (conjugated for SIGN > 0)
template <int SIGN, int R> __device__ __forceinline__ void twiddle(float2* a, const Roots& t) {
  float2 w1 = t.w1, w4 = t.w4, w16 = t.w16;
  if (SIGN > 0) { w1.y = -w1.y; w4.y = -w4.y; w16.y = -w16.y; }
  const float2 w2 = cmul(w1, w1), w3 = cmul(w2, w1);
  float2 q = w4;                                      // w^(4 s)
#pragma unroll
  for (int s = 0; s < (R + 3) / 4; ++s) {
    if (s == 2) q = cmul(w4, w4);
    else if (s == 4) q = w16;
    else if (s > 2) q = cmul(q, w4);
    if (s) a[4 * s] = cmul(a[4 * s], q);
    a[4 * s + 1] = cmul(a[4 * s + 1], s ? cmul(q, w1) : w1);
    a[4 * s + 2] = cmul(a[4 * s + 2], s ? cmul(q, w2) : w2);
    a[4 * s + 3] = cmul(a[4 * s + 3], s ? cmul(q, w3) : w3);
  }
}

// Unnormalised transform of the thread's column in registers (SIGN -1: e^{-}).
// `first`: no thread of the block may still be reading S.  before(): called once,
// after the last exchange's writes, before its barrier.
template <int SIGN, int L, int W, int PASS = 0, typename Before>
__device__ __forceinline__ void transform(float2* v, float2* S, const Twiddles<L>& tw, int b, int c,
                                          bool first, Before before) {
  constexpr int P = Plan<L>::P, T = L / P, R = radix<L>(PASS), NB = P / R, NS = span<L>(PASS);
  constexpr bool last = PASS == Plan<L>::N - 1;
  static_assert(T % NS == 0 && P % R == 0, "a pass reads the rows its threads own");
  float2 a[NB][R];
#pragma unroll
  for (int u = 0; u < NB; ++u) {
#pragma unroll
    for (int r = 0; r < R; ++r) a[u][r] = v[u + r * NB];
    if constexpr (PASS > 0) twiddle<SIGN, R>(a[u], tw.p[PASS - 1]);
    dft<SIGN, R>(a[u]);
  }
  if constexpr (last) {
#pragma unroll
    for (int u = 0; u < NB; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) v[u + r * NB] = a[u][r];
  } else {
    if (!(PASS == 0 && first)) __syncthreads();
    const int k = b % NS;
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int base = (b + u * T - k) * R + k;
#pragma unroll
      for (int r = 0; r < R; ++r) S[slot<L, W>(base + r * NS, c)] = a[u][r];
    }
    if constexpr (PASS == Plan<L>::N - 2) before();
    __syncthreads();
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = S[slot<L, W>(b + i * T, c)];
    transform<SIGN, L, W, PASS + 1>(v, S, tw, b, c, false, before);
  }
}

}  // namespace lreg
}  // namespace isam
