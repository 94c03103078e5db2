// Lateral passes with the tile held in registers.
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
//
// FP64 takes eight points a thread (lengths to 512) and single columns where the
// shared-memory form took pairs of them: twice to four times the warps for the
// FP64 pipe, whose latency and not its rate bounds the small sizes; its twiddles
// are all loaded (see fft_smem.cuh).
#pragma once

#include "fft_smem.cuh"
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
template <int SIGN, int N, int K, typename C> __device__ __forceinline__ C mul_root(C o) {
  using T = decltype(o.x);
  constexpr int k = K % N;
  if constexpr (k == 0) return o;
  else if constexpr (4 * k == N) return cmul_i<SIGN>(o);
  else if constexpr (2 * k == N) return mk<T>(-o.x, -o.y);
  else if constexpr (4 * k == 3 * N) return cmul_i<-SIGN>(o);
  else if constexpr (8 * k == N) return ew8_1<SIGN>(o);
  else if constexpr (8 * k == 3 * N) return ew8_3<SIGN>(o);
  else {
    constexpr T c = T(cos_turn(k, N)), s = T(SIGN * sin_turn(k, N));
    return mk<T>(o.x * c - o.y * s, o.y * c + o.x * s);
  }
}

template <int SIGN, typename C> __device__ __forceinline__ void dft3(C& a0, C& a1, C& a2) {
  using T = decltype(a0.x);
  const T h = T(0.86602540378443864676);              // sqrt(3)/2
  const C t1 = cadd(a1, a2), d = cscale(csub(a1, a2), h);
  const C t2 = csub(a0, cscale(t1, T(0.5)));
  a0 = cadd(a0, t1);
  a1 = add_rot<SIGN>(t2, d);
  a2 = sub_rot<SIGN>(t2, d);
}

// W_N^{n2 k1} on column n2 of the first stage's outputs, k1 = 1 .. N1-1
template <int SIGN, int N, int N1, int N2, int n2, int k1 = 1, typename C>
__device__ __forceinline__ void root_column(C (&b)[N2][N1]) {
  if constexpr (k1 < N1) {
    b[n2][k1] = mul_root<SIGN, N, n2 * k1>(b[n2][k1]);
    root_column<SIGN, N, N1, N2, n2, k1 + 1>(b);
  }
}
template <int SIGN, int N, int N1, int N2, int n2 = 1, typename C>
__device__ __forceinline__ void root_columns(C (&b)[N2][N1]) {
  if constexpr (n2 < N2) {
    root_column<SIGN, N, N1, N2, n2>(b);
    root_columns<SIGN, N, N1, N2, n2 + 1>(b);
  }
}

// N2 N1-point DFT (N1 = 3 or 4, N2 = 4 or 8) in place, natural order in and out:
// X[k1 + N1 k2] = sum_{n2} W_N2^{n2 k2} W_N^{n2 k1} sum_{n1} x[n2 + N2 n1] W_N1^{n1 k1}
template <int SIGN, int N1, int N2, typename C> __device__ __forceinline__ void dft_2d(C* a) {
  constexpr int N = N2 * N1;
  C b[N2][N1];
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) {
    if constexpr (N1 == 4) {
      C x0 = a[n2], x1 = a[n2 + N2], x2 = a[n2 + 2 * N2], x3 = a[n2 + 3 * N2];
      dft4<SIGN>(x0, x1, x2, x3);
      b[n2][0] = x0; b[n2][1] = x1; b[n2][2] = x2; b[n2][3] = x3;
    } else {
      C x0 = a[n2], x1 = a[n2 + N2], x2 = a[n2 + 2 * N2];
      dft3<SIGN>(x0, x1, x2);
      b[n2][0] = x0; b[n2][1] = x1; b[n2][2] = x2;
    }
  }
  root_columns<SIGN, N, N1, N2>(b);
#pragma unroll
  for (int k1 = 0; k1 < N1; ++k1) {
    C y[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) y[n2] = b[n2][k1];
    if constexpr (N2 == 8) dft8<SIGN>(y);
    else dft4<SIGN>(y[0], y[1], y[2], y[3]);
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) a[k1 + N1 * k2] = y[k2];
  }
}

template <int SIGN, int R, typename C> __device__ __forceinline__ void dft(C* a) {
  if constexpr (R == 32) dft_2d<SIGN, 4, 8>(a);
  else if constexpr (R == 24) dft_2d<SIGN, 3, 8>(a);
  else if constexpr (R == 16) dft_2d<SIGN, 4, 4>(a);
  else if constexpr (R == 8) dft8<SIGN>(a);
  else if constexpr (R == 4) dft4<SIGN>(a[0], a[1], a[2], a[3]);
  else dft2<SIGN>(a[0], a[1]);
}

// The radices of a length: P points a thread, N passes of radices R0, R1, R2, each of
// the span of those before it.  Every span divides T = L / P, so a thread's butterflies of a
// pass share one twiddle base.
template <typename T, int L> struct Plan;
template <> struct Plan<float, 2048> { static constexpr int P = 32, N = 3, R0 = 8, R1 = 8, R2 = 32; };
template <> struct Plan<float, 1024> { static constexpr int P = 32, N = 2, R0 = 32, R1 = 32, R2 = 1; };
template <> struct Plan<float, 512> { static constexpr int P = 32, N = 2, R0 = 16, R1 = 32, R2 = 1; };
template <> struct Plan<float, 256> { static constexpr int P = 16, N = 2, R0 = 16, R1 = 16, R2 = 1; };
template <> struct Plan<float, 128> { static constexpr int P = 16, N = 2, R0 = 8, R1 = 16, R2 = 1; };
template <> struct Plan<float, 64> { static constexpr int P = 8, N = 2, R0 = 8, R1 = 8, R2 = 1; };
template <> struct Plan<float, 768> { static constexpr int P = 24, N = 3, R0 = 4, R1 = 8, R2 = 24; };
template <> struct Plan<float, 384> { static constexpr int P = 24, N = 3, R0 = 4, R1 = 4, R2 = 24; };
template <> struct Plan<float, 192> { static constexpr int P = 24, N = 2, R0 = 8, R1 = 24, R2 = 1; };

template <> struct Plan<double, 512> { static constexpr int P = 8, N = 3, R0 = 8, R1 = 8, R2 = 8; };
template <> struct Plan<double, 256> { static constexpr int P = 8, N = 3, R0 = 4, R1 = 8, R2 = 8; };
template <> struct Plan<double, 128> { static constexpr int P = 8, N = 3, R0 = 2, R1 = 8, R2 = 8; };
template <> struct Plan<double, 64> { static constexpr int P = 8, N = 2, R0 = 8, R1 = 8, R2 = 1; };

template <typename T, int L> __host__ __device__ constexpr int threads_per_column() {
  return L / Plan<T, L>::P;
}
template <typename T, int L> __host__ __device__ constexpr int radix(int pass) {
  return pass == 0 ? Plan<T, L>::R0 : pass == 1 ? Plan<T, L>::R1 : Plan<T, L>::R2;
}
template <typename T, int L> __host__ __device__ constexpr int span(int pass) {
  return pass == 0 ? 1 : pass == 1 ? Plan<T, L>::R0 : Plan<T, L>::R0 * Plan<T, L>::R1;
}
// Columns a block takes: FP32: 8 at 1024 and 768 (64-byte rows), 16 at the
// others; FP64: 4.
template <typename T, int L> __host__ __device__ constexpr int columns() {
  return sizeof(T) == 8 ? 4 : L >= 768 ? 8 : 16;
}
// Rows of W columns.  Rows shorter than 128 bytes get a padding row after every R0:
// the first pass's writes to rows R0 b + r of neighbouring b then fall in different
// banks.  Rows of 128 bytes need none.
template <typename T, int W> __host__ __device__ constexpr bool padded() {
  return W * sizeof(cplx<T>) < 128;
}
template <typename T, int L, int W> __device__ __forceinline__ int slot(int row, int c) {
  if constexpr (padded<T, W>()) return (row + row / Plan<T, L>::R0) * W + c;
  else return row * W + c;
}
// ... of (row + STEP r, c) less that of (row, c), for a STEP that is a multiple of
// the padding period or r < R0 rows from a multiple of it: a constant
template <typename T, int L, int W, int STEP>
__device__ __forceinline__ constexpr int slot_step(int r) {
  constexpr int R0 = Plan<T, L>::R0;
  static_assert(!padded<T, W>() || STEP == 1 || STEP % R0 == 0, "a constant distance");
  return (padded<T, W>() && STEP % R0 == 0 ? r * (STEP + STEP / R0) : r * STEP) * W;
}
template <typename T, int L, int W> __host__ __device__ constexpr size_t smem_elements() {
  return size_t(padded<T, W>() ? L + L / Plan<T, L>::R0 : L) * W;
}

// w^1, w^4, w^16 of a pass, w = e^{-2 pi i k / (span R)}, k = b mod span
struct Roots { float2 w1, w4, w16; };
__device__ __forceinline__ float2 root(int k, int n) {
  float s, c;
  sincospif(float(2 * k) / float(n), &s, &c);
  return make_float2(c, -s);
}
template <typename T, int L> struct Twiddles;
template <int L> struct Twiddles<float, L> {
  Roots p[Plan<float, L>::N - 1];
  __device__ __forceinline__ Twiddles(int b, const float2*) {
#pragma unroll
    for (int i = 1; i < Plan<float, L>::N; ++i) {
      const int ns = span<float, L>(i), R = radix<float, L>(i), n = ns * R, k = b % ns;
      p[i - 1].w1 = root(k, n);
      if (R > 4) p[i - 1].w4 = root(4 * k, n);
      if (R > 16) p[i - 1].w16 = root(16 * k, n);
    }
  }
  // a[r] *= w^r of pass PASS (conjugated for SIGN > 0)
  template <int SIGN, int PASS> __device__ __forceinline__ void apply(float2* a) const {
    constexpr int R = radix<float, L>(PASS);
    float2 w1 = p[PASS - 1].w1, w4 = p[PASS - 1].w4, w16 = p[PASS - 1].w16;
    if (SIGN > 0) { w1.y = -w1.y; w4.y = -w4.y; w16.y = -w16.y; }
    const float2 w2 = cmul(w1, w1), w3 = cmul(w2, w1);
    float2 q = w4;                                    // w^(4 s)
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
};
template <int L> struct Twiddles<double, L> {
  const double2* roots;                               // e^{-2 pi i m / L}
  int b;
  __device__ __forceinline__ Twiddles(int b_, const double2* r) : roots(r), b(b_) {}
  template <int SIGN, int PASS> __device__ __forceinline__ void apply(double2* a) const {
    constexpr int ns = span<double, L>(PASS), R = radix<double, L>(PASS);
    twiddle_powers<SIGN, R, double>(a, roots, b % ns, L / (ns * R));
  }
};

// Unnormalised transform of the thread's column in registers (SIGN -1: e^{-}).
// `first`: no thread of the block may still be reading S.  before(): called once,
// after the last exchange's writes, before its barrier.
template <int SIGN, int L, int W, int PASS = 0, typename T, typename Before>
__device__ __forceinline__ void transform(cplx<T>* v, cplx<T>* S, const Twiddles<T, L>& tw, int b,
                                          int c, bool first, Before before) {
  using Pl = Plan<T, L>;
  constexpr int P = Pl::P, TH = L / P, R = radix<T, L>(PASS), NB = P / R, NS = span<T, L>(PASS);
  constexpr bool last = PASS == Pl::N - 1;
  static_assert(TH % NS == 0 && P % R == 0, "a pass reads the rows its threads own");
  cplx<T> a[NB][R];
#pragma unroll
  for (int u = 0; u < NB; ++u) {
#pragma unroll
    for (int r = 0; r < R; ++r) a[u][r] = v[u + r * NB];
    if constexpr (PASS > 0) tw.template apply<SIGN, PASS>(a[u]);
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
      cplx<T>* out = S + slot<T, L, W>((b + u * TH - k) * R + k, c);
#pragma unroll
      for (int r = 0; r < R; ++r) out[slot_step<T, L, W, NS>(r)] = a[u][r];
    }
    if constexpr (PASS == Pl::N - 2) before();
    __syncthreads();
    const cplx<T>* in = S + slot<T, L, W>(b, c);
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = in[slot_step<T, L, W, TH>(i)];
    transform<SIGN, L, W, PASS + 1, T>(v, S, tw, b, c, false, before);
  }
}

}  // namespace lreg
}  // namespace isam
