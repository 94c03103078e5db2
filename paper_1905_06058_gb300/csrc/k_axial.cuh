// Axial Stolt-mapped NUFFT kernels.  One thread block per pair of lateral-
// frequency columns (q, -q): both share the Stolt map beta(|q|, k), so the
// positions, phases and interpolation coefficients are computed once and
// applied to two columns whose FFTs run in lock step (16- or 32-byte
// shared-memory elements).
//
//   k_ax_fwd  (§3.2, Eq. 3, 13, 16; min-max NUFFT of Fessler & Sutton):
//     S(q, k_j) = e^{j phi(k_j)} e^{j (2 k_j + beta) z0}
//                 sum_l c_l(f_j) Y[(m0_j + l) mod K],
//     Y = K-point e^{+} DFT of the scaled, zero-padded column
//         s(n - nz/2) eta_hat(q, z_n) / sqrt(nz) placed at (n - nz/2) mod K.
//   k_ax_adj  (Eq. 17, the exact adjoint of k_ax_fwd): every sample adds
//     c_l(f_j) conj(phase_j) R_hat(q, k_j) to bins m0_j + l, race-free without
//     atomics (see scatter_samples), then the K-point e^{-} DFT, truncation
//     and scaling.
//   k_ax_fused  both, with the data residual formed in between.
//
// Stolt positions are evaluated per sample from per-plan constants in
// float-float arithmetic (FP32 path) or double (FP64 path): the grid
// coordinate reaches ~5e4 bins while its fractional part must be right to
// ~1e-7.  Interpolation coefficients are evaluated from their even/odd
// polynomial form (see Poly), held in kernel parameters.
#pragma once

#include <limits.h>

#include <algorithm>

#include "fft_col16.cuh"
#include "fft_smem.cuh"
#include "internal.cuh"
#include "tmem.cuh"

namespace isam {

__device__ __forceinline__ int signed_freq(int i, int n) { return i <= (n - 1) / 2 ? i : i - n; }
static inline int ilog2_dev(int v) { int r = 0; while ((1 << r) < v) ++r; return r; }

template <typename T> struct StoltPos;

// p_j = sqrt(4 kappa_j^2 - a), a = (q/dk)^2, in float-float; the unwrapped
// grid index is p_j - B with B = 2 kappa_0 - c0 (a multiple of K).
template <> struct StoltPos<float> {
  ff a;
  __device__ StoltPos(const StoltConst& c, int mx, int my) {
    a = ff_add(ff_mul_f({c.qx_hi, c.qx_lo}, float(mx * mx)),
               ff_mul_f({c.qy_hi, c.qy_lo}, float(my * my)));
  }
  __device__ __forceinline__ bool at(const StoltConst& c, int j, int& mfl, float& frac,
                                     float& turn) const {
    ff kap = ff_two_sum(c.kap_hi, float(j));            // j is an exact integer
    kap = ff_quick(kap.hi, kap.lo + c.kap_lo);
    ff k2 = ff_mul(kap, kap);
    k2.hi *= 4.0f; k2.lo *= 4.0f;                       // exact
    const ff x = ff_sub(k2, a);
    if (!(x.hi > 0.0f)) return false;
    const ff p = ff_sqrt_fast(x);
    ff t = ff_two_sum(p.hi, -c.B);
    t.lo += p.lo;
    float fl = floorf(t.hi);
    float fr = __fadd_rn(__fsub_rn(t.hi, fl), t.lo);
    if (fr < 0.0f) { fr += 1.0f; fl -= 1.0f; }
    else if (fr >= 1.0f) { fr -= 1.0f; fl += 1.0f; }
    mfl = int(fl);
    frac = fr;
    turn = 0.0f;
    if (c.focus) {                                      // (2 kappa - p) zeta, in turns
      const ff d = ff_sub({2.0f * kap.hi, 2.0f * kap.lo}, p);
      const ff r = ff_mul(d, {c.zeta_hi, c.zeta_lo});
      const float n = rintf(r.hi);
      turn = __fadd_rn(__fsub_rn(r.hi, n), r.lo);
    }
    return true;
  }
};

template <> struct StoltPos<double> {
  double a;
  __device__ StoltPos(const StoltConst& c, int mx, int my) {
    a = c.Qx * double(mx) * double(mx) + c.Qy * double(my) * double(my);
  }
  __device__ __forceinline__ bool at(const StoltConst& c, int j, int& mfl, double& frac,
                                     double& turn) const {
    const double kap = c.kap + double(j);
    const double x = 4.0 * kap * kap - a;
    if (!(x > 0.0)) return false;
    const double p = sqrt(x);
    const double d = a / (2.0 * kap + p);               // 2 kappa - p without cancellation
    const double t = (c.c0d + 2.0 * double(j)) - d;     // = p - B
    const double fl = floor(t);
    frac = t - fl;                                      // exact, in [0, 1)
    mfl = int(fl);
    turn = 0.0;
    if (c.focus) {
      const double r = d * c.zeta;
      turn = r - rint(r);
    }
    return true;
  }
};

__device__ __forceinline__ void sincos_turn(float t, float* s, float* c) { sincospif(2.0f * t, s, c); }
__device__ __forceinline__ void sincos_turn(double t, double* s, double* c) { sincospi(2.0 * t, s, c); }

template <typename T>
__device__ __forceinline__ cplx<T> spectral_phase(const StoltConst& sc, const cplx<T>* disp, int j,
                                                  T turn) {
  cplx<T> ph = __ldg(disp + j);
  if (sc.focus) {
    T s, c;
    sincos_turn(turn, &s, &c);
    ph = cmul(ph, mk<T>(c, s));
  }
  return ph;
}

// Row of the Stolt table (and of the filter table) for lateral frequency
// (mx, my): rows by |mx|, |my|.
__device__ __forceinline__ int stolt_class(const StoltConst& sc, int mx, int my) {
  return abs(my) * (sc.nx / 2 + 1) + abs(mx);
}

// consecutive samples a thread of the adjoint interpolation owns (see
// scatter_samples)
constexpr int NRES = 4;

template <typename T, typename V> struct Sample {
  V val;          // conj(phase) R of the block's column or columns
  T frac;         // fractional Stolt offset
  int mfl;        // unwrapped floor of the Stolt position; INT_MIN: no contribution
                  // (evanescent, or past nk)
};

// Stolt positions and spectral phases of a quad of samples 4 q .. 4 q + 3 of one
// column pair, from the plan's table when present, else evaluated (float-float /
// double).
template <typename T> struct Positions {
  StoltPos<T> sp;
  const int4* row;           // the class's planes, nq vectors each
  const cplx<T>* frow;       // filter B of this column's |q| class (evaluated path)
  int nq, cls;
  __device__ Positions(const AxArgs<T>& A, int mx, int my) : sp(A.sc, mx, my) {
    cls = stolt_class(A.sc, mx, my);
    nq = A.sc.nk / NRES;
    row = A.tab.stab ? A.tab.stab + size_t(cls) * (size_t(StoltTable<T>::planes) * nq) : nullptr;
    frow = A.tab.filt ? A.tab.filt + size_t(cls) * A.sc.nk : nullptr;
  }
  // floors and fractions of the quad; an evaluated position also leaves its focus
  // turn in val.a.x, for phases()
  template <typename V>
  __device__ __forceinline__ void quad(const AxArgs<T>& A, int q, Sample<T, V>* sm) const {
    if (row) {
      const int4 m = __ldg(row + q);
      sm[0].mfl = m.x; sm[1].mfl = m.y; sm[2].mfl = m.z; sm[3].mfl = m.w;
      if constexpr (sizeof(T) == 4) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(row + nq + q));
        sm[0].frac = f.x; sm[1].frac = f.y; sm[2].frac = f.z; sm[3].frac = f.w;
      } else {
        const double2 f0 = __ldg(reinterpret_cast<const double2*>(row + nq + q));
        const double2 f1 = __ldg(reinterpret_cast<const double2*>(row + 2 * nq + q));
        sm[0].frac = f0.x; sm[1].frac = f0.y; sm[2].frac = f1.x; sm[3].frac = f1.y;
      }
      return;
    }
#pragma unroll
    for (int rho = 0; rho < NRES; ++rho) {
      sm[rho].frac = T(0);
      if (!sp.at(A.sc, NRES * q + rho, sm[rho].mfl, sm[rho].frac, sm[rho].val.a.x))
        sm[rho].mfl = INT_MIN;
    }
  }
  // phases of samples 2 h and 2 h + 1 of the quad (0 where evanescent)
  template <typename V>
  __device__ __forceinline__ cpair<T> phases(const AxArgs<T>& A, int q, int h,
                                             const Sample<T, V>* sm) const {
    cpair<T> p;
    if (row) {
      if constexpr (sizeof(T) == 4) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(row + (2 + h) * nq + q));
        p.a = make_float2(v.x, v.y);
        p.b = make_float2(v.z, v.w);
      } else {
        p.a = __ldg(reinterpret_cast<const double2*>(row + (3 + 2 * h) * nq + q));
        p.b = __ldg(reinterpret_cast<const double2*>(row + (4 + 2 * h) * nq + q));
      }
      return p;
    }
    p.a = evaluated(A, NRES * q + 2 * h, sm[2 * h].mfl, sm[2 * h].val.a.x);
    p.b = evaluated(A, NRES * q + 2 * h + 1, sm[2 * h + 1].mfl, sm[2 * h + 1].val.a.x);
    return p;
  }
  __device__ __forceinline__ cplx<T> evaluated(const AxArgs<T>& A, int j, int mfl, T turn) const {
    if (mfl == INT_MIN) return mk<T>(0, 0);
    cplx<T> ph = spectral_phase<T>(A.sc, A.tab.disp, j, turn);
    if (frow) ph = cmul(ph, __ldg(frow + j));
    return ph;
  }
};

// all J coefficients c_l(f)
template <typename T, int J>
__device__ __forceinline__ void coefficients(const Poly<T>& P, T frac, T* c) {
  constexpr int DE = PolyDeg<T>::DE, DO = PolyDeg<T>::DO;
  const T x = frac - T(0.5);
  const T y = T(4) * x * x;
#pragma unroll
  for (int p = 0; p < J / 2; ++p) {
    T e = P.e[p][DE];
#pragma unroll
    for (int k = DE - 1; k >= 0; --k) e = fma(e, y, P.e[p][k]);
    T o = P.o[p][DO];
#pragma unroll
    for (int k = DO - 1; k >= 0; --k) o = fma(o, y, P.o[p][k]);
    c[p] = fma(x, o, e);
    c[J - 1 - p] = fma(-x, o, e);
  }
}

// The coefficients of a quad's samples.  FP64 plans tabulate them next to the Stolt
// table (the polynomials took 42 of an FP64 sample's 56 FMAs): 2 J planes of one
// double2 per quad of the class, (c_{2i}, c_{2i+1}) of sample rho in plane
// rho J/2 + i.
template <typename T, int J> struct Coefficients {
  const Poly<T>& poly;
  const cplx<T>* tab;        // the quad's first plane, or null: evaluate
  int nq;
  __device__ __forceinline__ Coefficients(const AxArgs<T>& A, const Positions<T>& pos, int q)
      : poly(A.poly), tab(nullptr), nq(pos.nq) {
    if (sizeof(T) == 8 && A.tab.coef) tab = A.tab.coef + size_t(pos.cls) * (2 * J) * nq + q;
  }
  __device__ __forceinline__ void operator()(int rho, T frac, T* c) const {
    if constexpr (sizeof(T) == 8) {
      if (tab) {
#pragma unroll
        for (int i = 0; i < J / 2; ++i) {
          const cplx<T> v = __ldg(tab + (rho * (J / 2) + i) * nq);
          c[2 * i] = v.x;
          c[2 * i + 1] = v.y;
        }
        return;
      }
    }
    coefficients<T, J>(poly, frac, c);
  }
};

// The block's columns: a pair (q, -q), or with ONE the column blockIdx.x (c1; c2 is
// the column of -q).
template <typename T, bool ONE = false>
__device__ __forceinline__ void pair_columns(const AxArgs<T>& A, int& c1, int& c2, int& mx,
                                             int& my) {
  if (ONE) {
    const int nx = A.sc.nx, ny = A.sc.ny, ix = blockIdx.x % nx, iy = blockIdx.x / nx;
    c1 = blockIdx.x;
    c2 = (iy ? ny - iy : 0) * nx + (ix ? nx - ix : 0);
  } else {
    const int2 pr = A.pairs[blockIdx.x];
    c1 = pr.x;
    c2 = pr.y;
  }
  mx = signed_freq(c1 % A.sc.nx, A.sc.nx);
  my = signed_freq(c1 / A.sc.nx, A.sc.ny);
}

// Column c of the spectra arrays (of the half spectrum, for x <= nx/2)
template <typename T>
__device__ __forceinline__ int spectrum_column(const AxArgs<T>& A, int c, bool half) {
  return half ? c - c / A.sc.nx * (A.sc.nx - A.sc.nx / 2 - 1) : c;
}

// Shared memory of the axial kernels: the FFT buffer Y (padded rows of
// column pairs) followed by the K-point twiddle table.
template <typename T>
__device__ __forceinline__ cplx<T>* twiddle_table(unsigned char* raw, int K) {
  return reinterpret_cast<cplx<T>*>(raw + size_t(padded_rows(K)) * sizeof(cpair<T>));
}
// the element of Y: a pair's two columns, or one column
template <typename T, bool ONE> using column_t = std::conditional_t<ONE, cone<T>, cpair<T>>;

// The forward K-point transform of the block's column pair: the
// compile-time-length Stockham form when LOGK > 0 (K = 2^LOGK, the sizes the
// kernels are instantiated for), else the runtime-length one.  Ends with a
// barrier.  (The inverse is in inverse_and_store.)
template <int LOGK, typename T, typename V>
__device__ __forceinline__ void axial_fft_fwd(V* Y, int K, int logK, const cplx<T>* tw) {
  if constexpr (LOGK > 0) fft_smem_ct<+1, true, LOGK, T>(Y, threadIdx.x, tw);
  else fft_smem<+1, true, T>(Y, 1, 0, threadIdx.x, K, logK, tw, true);
}

// K and the block size K/8, as compile-time constants when LOGK > 0
template <int LOGK> __device__ __forceinline__ int axial_K(const StoltConst& sc) {
  return LOGK > 0 ? (1 << LOGK) : sc.K;
}
template <int LOGK> __device__ __forceinline__ int axial_threads() {
  return LOGK > 0 ? (1 << LOGK) / 8 : int(blockDim.x);
}

// Y (padded rows) = scaled columns c1 (a) and c2 (b), zero-padded to K, then
// the K-point e^{+} DFT.  The padding rows [nz/2, K - nz/2) are never stored:
// the first FFT pass knows them to be zero.  Ends with a barrier.
template <typename T, int LOGK, typename V>
__device__ __forceinline__ void load_and_fft(const AxArgs<T>& A, V* Y, const cplx<T>* tw,
                                             int c1, int c2, bool two) {
  using C = cplx<T>;
  constexpr bool ONE = sizeof(V) == sizeof(C);
  const StoltConst& sc = A.sc;
  const int K = axial_K<LOGK>(sc), nz = K / 2;
  const int tid = threadIdx.x, nt = axial_threads<LOGK>();
  const C* x1 = A.in + size_t(c1) * nz;
  const C* x2 = A.in + size_t(c2) * nz;
  // nz = 4 * blockDim: four samples per thread, loads issued before use
  V v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int n = tid + i * nt;
    v[i].a = x1[n];
    if constexpr (!ONE) v[i].b = two ? x2[n] : mk<T>(0, 0);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int n = tid + i * nt;
    int p = n - nz / 2;
    if (p < 0) p += K;
    Y[prow(p)] = escale(v[i], __ldg(A.tab.scale + n));
  }
  __syncthreads();
  axial_fft_fwd<LOGK, T, V>(Y, K, sc.logK, tw);
}

// forward interpolation of the columns at one sample (before the phase)
template <typename T, int J, typename V>
__device__ __forceinline__ V interp_sample(const V* Y, int K, int mfl, const T* c) {
  const int m0 = mfl - J / 2 + 1;
  V s{};
#pragma unroll
  for (int l = 0; l < J; ++l) s = efma_r(c[l], Y[prow((m0 + l) & (K - 1))], s);
  return s;
}

// Adjoint interpolation in scatter form.  Thread t owns samples
// j = NRES t + rho (rho < NRES; nk <= K/2 = NRES * blockDim).  Stolt
// positions rise by at least two bins per sample (dp/dj = 4 kappa / p >= 2),
// so samples of one residue class rho lie >= 2 NRES >= J bins apart and
// their J-bin neighbourhoods are disjoint: in phase rho every thread adds
// its sample's J contributions to Y without atomics.  Phases are further
// split into chunks of K/2 unwrapped bins (chunk = floor(mfl / (K/2))) so
// that the wrap mod K never folds two neighbourhoods of one phase together.
// Each bin receives at most ceil(J/2) + 1 contributions per chunk, summed in
// a fixed order with fused multiply-adds.
// Zero Y, find the block's range of Stolt positions (shared atomics on
// *lo, *hi, initialised by the caller before an earlier barrier) and assign
// every sample to a chunk of width K - J of unwrapped positions: within a
// chunk the J-bin neighbourhoods span fewer than K bins, so they never meet
// again after the wrap mod K.  Returns the number of chunks.
//
// warp_tail: there are two chunks and every chunk-1 sample belongs to the
// block's last warp.  Stolt positions rise with j (samples below the
// evanescent cut-off come first) and warp w owns samples
// [32 NRES w, 32 NRES (w + 1)), so this holds when the last sample of the
// warp before it, j* = NRES (nt - 32) - 1 (thread nt - 33), exists (j* < nk)
// and is in chunk 0 or evanescent.  Its position goes through *tail
// (INT_MAX: j* >= nk, INT_MIN: evanescent).
template <typename T, int J, typename V>
__device__ __forceinline__ int prepare_scatter(V* Y, int K, int nt, int nk,
                                               const Sample<T, V>* sm, int* chunk, int* lo,
                                               int* hi, int* tail, bool& warp_tail) {
  const V zero{};
  for (int i = threadIdx.x; i < K; i += nt) Y[prow(i)] = zero;
  int l = INT_MAX, h = INT_MIN;
#pragma unroll
  for (int rho = 0; rho < NRES; ++rho)
    if (sm[rho].mfl != INT_MIN) {
      l = min(l, sm[rho].mfl);
      h = max(h, sm[rho].mfl);
    }
  if (l != INT_MAX) {
    atomicMin(lo, l);
    atomicMax(hi, h);
  }
  if (int(threadIdx.x) == nt - 33)
    *tail = NRES * (nt - 32) - 1 >= nk ? INT_MAX
            : sm[NRES - 1].mfl;
  __syncthreads();
  const int base = *lo, width = K - J;
  warp_tail = false;
  if (base == INT_MAX) return 0;
#pragma unroll
  for (int rho = 0; rho < NRES; ++rho) {
    chunk[rho] = INT_MIN;
    if (sm[rho].mfl != INT_MIN) {
      int c = 0, d = sm[rho].mfl - base;
      while (d >= width) { d -= width; ++c; }
      chunk[rho] = c;
    }
  }
  int n = 1;
  for (int d = *hi - base; d >= width; d -= width) ++n;
  const int t = *tail;
  warp_tail = n == 2 && nt >= 64 && t != INT_MAX && (t == INT_MIN || t - base < width);
  return n;
}

// the J contributions of one sample
template <typename T, int J, typename V>
__device__ __forceinline__ void add_sample(const Coefficients<T, J>& co, V* Y, int K, int rho,
                                           const Sample<T, V>& sm) {
  T c[J];
  co(rho, sm.frac, c);
  const int m0 = sm.mfl - J / 2 + 1;
#pragma unroll
  for (int l = 0; l < J; ++l) {
    const int bi = prow((m0 + l) & (K - 1));
    Y[bi] = efma_r(c[l], sm.val, Y[bi]);
  }
}

// Y must be zero; every thread adds its samples' J contributions, residue
// class by residue class and chunk by chunk (see the comment above NRES),
// each phase closed by a block barrier.  With warp_tail the last chunk's
// phases involve the last warp only and are closed by warp barriers, then one
// block barrier: the same phases in the same order, so the same sums.
template <typename T, int J, typename V>
__device__ __forceinline__ void scatter_samples(const Coefficients<T, J>& co, V* Y, int K, int nt,
                                                const Sample<T, V>* sm, const int* chunk,
                                                int nchunks, bool warp_tail) {
  const int block_chunks = warp_tail ? 1 : nchunks;
  for (int ch = 0; ch < block_chunks; ++ch) {
#pragma unroll
    for (int rho = 0; rho < NRES; ++rho) {
      if (chunk[rho] == ch) add_sample<T, J, V>(co, Y, K, rho, sm[rho]);
      __syncthreads();
    }
  }
  if (warp_tail) {
    if ((int(threadIdx.x) >> 5) == (nt >> 5) - 1) {
#pragma unroll
      for (int rho = 0; rho < NRES; ++rho) {
        if (chunk[rho] == 1) add_sample<T, J, V>(co, Y, K, rho, sm[rho]);
        __syncwarp();
      }
    }
    __syncthreads();
  }
}

// WINDOW form of the interpolation's and the scatter's shared-memory traffic.
//
// A thread's four samples lie 2 to 2.3 bins apart (StoltConst::window), so
// their J-bin neighbourhoods overlap: together they touch WS = J + 7 bins, not
// 4 J.  Sample rho sits at cumulative offset 2 rho or 2 rho + 1 from the
// thread's first sample; with its J coefficients shifted by that 0 or 1 into
// J + 1 taps (window_taps) every register index is a constant.  The gather
// reads each of the WS bins once.  The scatter sums the four samples in
// registers and touches shared memory once per bin: the bins before the next
// thread's window belong to this thread alone and are stored (no zeroing pass,
// no read), the J - 1 or so after it are added after a barrier, where they are
// disjoint again (at least seven bins separate the windows of neighbours).
// Bins a window reaches past one period of K are added in a second pass of the
// same two phases, taken only by the last warps' threads and only when a column
// spans more than K.
//
// What bounded the kernels was the load/store data path: the residue-class
// scatter took 56 shared-memory accesses a thread (8 to zero, 24 reads, 24
// writes) in 8 barrier phases, the per-sample gather 24; the windows take 23
// and 13 (J = 6).  k_ax_fused, 1024 x 2048 B-scan: 51.5 -> 47.6 us, 256 x 256 x
// 2048 volume: 2,414 -> 2,117 us; k_ax_adj 36.8 -> 30.7 us and 1,598 -> 1,300 us
// (40.2, 1,817 and 1,096 us with what followed: the quad-major table, constant
// shared-memory distances, tensor memory, half spectra).
//
// The bound of 2.3 bins keeps four samples and the next thread's first within
// the offsets the kernels hold as constants (three steps below 7 bins, four
// below 10); the acquisitions in use reach 2.06 (B-scan, NA 0.15) to 2.23
// (volume corner, NA 0.2).
//
// Positions of q = 0 columns can round to an offset outside {0, 1} when their
// common fraction is within rounding of an integer; then the block takes the
// residue-class scatter, as do all blocks of evanescent or steeper geometries.
template <int J> __host__ __device__ constexpr int window_slots() { return J + 2 * NRES - 1; }

// sample rho's offset from bin 2 rho of the thread's window (0 or 1 where it fits)
template <typename S> __device__ __forceinline__ unsigned window_offset(const S* sm, int rho) {
  return unsigned(sm[rho].mfl) - unsigned(sm[0].mfl) - 2u * unsigned(rho);
}

// J coefficients as J + 1 taps, shifted up by one when `shift`
template <typename T, int J>
__device__ __forceinline__ void window_taps(const Coefficients<T, J>& co, int rho, T frac,
                                            bool shift, T* e) {
  T c[J];
  co(rho, frac, c);
  e[0] = shift ? T(0) : c[0];
#pragma unroll
  for (int l = 1; l < J; ++l) e[l] = shift ? c[l - 1] : c[l];
  e[J] = shift ? c[J - 1] : T(0);
}

// One thread's window: sums its samples, of taps (rho, e), slot by slot and hands
// each finished slot (l, value) to put.
template <typename T, int J, typename V, typename Taps, typename Put>
__device__ __forceinline__ void window_sums(const Sample<T, V>* sm, Taps taps, Put put) {
  constexpr int WS = window_slots<J>();
  V w[WS];
#pragma unroll
  for (int rho = 0; rho < NRES; ++rho) {
    T e[J + 1];
    taps(rho, e);
#pragma unroll
    for (int l = 0; l <= J; ++l) {
      V& x = w[2 * rho + l];
      if (rho == 0 || l > J - 2) x = escale(sm[rho].val, e[l]);
      else x = efma_r(e[l], sm[rho].val, x);
    }
    if (rho < NRES - 1) {
      put(2 * rho, w[2 * rho]);
      put(2 * rho + 1, w[2 * rho + 1]);
    }
  }
#pragma unroll
  for (int l = 2 * (NRES - 1); l < WS; ++l) put(l, w[l]);
}

// Y = the scatter of all samples (every bin written; ends with a barrier).
// Every read of Y must be done and heads complete (a barrier before).  WARP: taps is
// called by whole warps.
template <typename T, int J, bool WARP, typename V, typename Taps>
__device__ __forceinline__ void window_scatter(V* Y, int K, int nt, int nk,
                                               const Sample<T, V>* sm, V* past,
                                               const int* heads, Taps taps) {
  constexpr int WS = window_slots<J>(), W_MIN = 2 * NRES - 1;
  const int tid = threadIdx.x, nact = nk / NRES;
  const bool active = tid < nact;
  const int off = 1 - J / 2;                          // first bin of a window - its head
  const int base = heads[0] + off, end = heads[nact - 1] + off + WS;
  const int m0 = active ? heads[tid] + off : 0;
  // bins before the next thread's window (all of them for the last thread)
  const int own = tid < nact - 1 ? heads[tid + 1] + off - m0 : WS;
  const int limit = base + K - m0;                    // slots from here on lie past one period
  for (int i = end + tid; i < base + K; i += nt)
    Y[prow(i & (K - 1))] = V{};
  auto row = [&](int l) -> V& {
    return l < limit ? Y[prow((m0 + l) & (K - 1))] : past[l - limit];
  };
  V tail[WS - W_MIN];
  if (WARP ? (tid & ~31) < nact : active)
    window_sums<T, J, V>(sm, taps, [&](int l, const V& v) {
      if (l >= W_MIN) tail[l - W_MIN] = v;
      if ((!WARP || active) && (l < W_MIN || l < own)) row(l) = v;
    });
  __syncthreads();
  if (active)
#pragma unroll
    for (int l = W_MIN; l < WS; ++l)
      if (l >= own) {
        V& y = row(l);
        y = eadd(y, tail[l - W_MIN]);
      }
  __syncthreads();
  if (end > base + K) {                               // the same for the whole block
    for (int i = tid; i < end - base - K; i += nt) {
      V& y = Y[prow((base + i) & (K - 1))];
      y = eadd(y, past[i]);
    }
    __syncthreads();
  }
}

// The bins past one period: A.sc.past elements after the twiddles.  The heads, the first
// sample's floor of every thread that has samples: a static array where K is a constant,
// else after the bins.
template <typename T, typename V>
__device__ __forceinline__ V* window_past(const AxArgs<T>& A, V* Y) {
  return reinterpret_cast<V*>(reinterpret_cast<unsigned char*>(Y) + A.past_offset);
}
template <int LOGK> __host__ __device__ constexpr int window_heads_fixed() {
  return LOGK > 0 ? (1 << LOGK) / 8 : 1;
}
template <typename T, typename V>
__device__ __forceinline__ int* window_heads(const AxArgs<T>& A, V* Y) {
  return reinterpret_cast<int*>(window_past<T, V>(A, Y) + A.sc.past);
}

// the thread's samples fit one window
template <typename T, typename V>
__device__ __forceinline__ bool quad_fits(const AxArgs<T>& A, const Sample<T, V>* sm) {
  bool ok = A.sc.window != 0;
#pragma unroll
  for (int rho = 0; rho < NRES; ++rho) ok &= window_offset(sm, rho) <= 1u;
  return ok;
}

// Y = the scatter of the block's samples, in the window form where every thread's
// samples fit one (fits; true where a thread has none; false in FitOrder's calls).  heads
// holds every such thread's first floor; taps gives the window's taps (see
// window_scatter), reload the samples' positions again for the residue-class form.
// Starts with a barrier (all reads of Y are done) and ends with one.
template <typename T, int J, bool WARP, typename V, typename Taps, typename Reload>
__device__ __forceinline__ void scatter(const AxArgs<T>& A, const Coefficients<T, J>& co, V* Y,
                                        int K, int nt, int nk, Sample<T, V>* sm, bool fits,
                                        int* lo, int* hi, int* ch_tail, const int* heads,
                                        Taps taps, Reload reload) {
  if (__syncthreads_and(fits)) {
    window_scatter<T, J, WARP, V>(Y, K, nt, nk, sm, window_past<T, V>(A, Y), heads, taps);
    return;
  }
  reload();
  bool warp_tail;
  int chunk[NRES];
  const int nch = prepare_scatter<T, J, V>(Y, K, nt, nk, sm, chunk, lo, hi, ch_tail, warp_tail);
  scatter_samples<T, J, V>(co, Y, K, nt, sm, chunk, nch, warp_tail);
}

// The forward interpolation of a thread's samples (before the phase): hands
// (rho, N(x) of the columns) to put, in order; evanescent samples give 0.  Where they
// fit a window, keep is given its taps (rho, e) too.
template <typename T, int J, typename V, typename Keep, typename Put>
__device__ __forceinline__ void interp_quad(const Coefficients<T, J>& co, const V* Y, int K,
                                            const Sample<T, V>* sm, bool fits, Keep keep, Put put) {
  if (fits) {
    constexpr int WS = window_slots<J>();
    const int m0 = sm[0].mfl - J / 2 + 1;
    V y[WS];
#pragma unroll
    for (int l = 0; l < J - 1; ++l) y[l] = Y[prow((m0 + l) & (K - 1))];
#pragma unroll
    for (int rho = 0; rho < NRES; ++rho) {
#pragma unroll
      for (int l = J - 1; l <= J; ++l)
        y[2 * rho + l] = Y[prow((m0 + 2 * rho + l) & (K - 1))];
      T e[J + 1];
      window_taps<T, J>(co, rho, sm[rho].frac, window_offset(sm, rho) != 0, e);
      keep(rho, e);
      V s = escale(y[2 * rho], e[0]);
#pragma unroll
      for (int l = 1; l <= J; ++l) s = efma_r(e[l], y[2 * rho + l], s);
      put(rho, s);
    }
    return;
  }
#pragma unroll
  for (int rho = 0; rho < NRES; ++rho) {
    V s{};
    if (sm[rho].mfl != INT_MIN) {
      T c[J];
      co(rho, sm[rho].frac, c);
      s = interp_sample<T, J, V>(Y, K, sm[rho].mfl, c);
    }
    put(rho, s);
  }
}

// Sample n of both output columns: G = s y, or, when the kernel writes the
// lateral spectrum of u = eta^k - g/L, u_hat = eta_hat - G/L with eta_hat = A.eta
// (the fused kernel's own input, re-read here).
template <typename T>
__device__ __forceinline__ void put_output(const AxArgs<T>& A, cplx<T>* o1, cplx<T>* o2, int n,
                                           const cpair<T>& y, T s, int c1, int c2, bool two) {
  const int nz = A.sc.nz;
  if (A.u_hat_scale != T(0)) {
    const T f = s * A.u_hat_scale;
    o1[n] = csub(A.eta[size_t(c1) * nz + n], cscale(y.a, f));
    if (two) o2[n] = csub(A.eta[size_t(c2) * nz + n], cscale(y.b, f));
  } else {
    o1[n] = cscale(y.a, s);
    if (two) o2[n] = cscale(y.b, s);
  }
}

// Sample n of one output column (column index col of the plan's layout): the
// single-column form of put_output.
template <typename T>
__device__ __forceinline__ void put_output1(const AxArgs<T>& A, cplx<T>* o, int col, int n,
                                            const cplx<T>& y, T s) {
  if (A.u_hat_scale != T(0))
    o[n] = csub(A.eta[size_t(col) * A.sc.nz + n], cscale(y, s * A.u_hat_scale));
  else
    o[n] = cscale(y, s);
}

template <typename T>
__device__ __forceinline__ void put_output(const AxArgs<T>& A, cplx<T>* o1, cplx<T>* o2, int n,
                                           const cone<T>& y, T s, int c1, int c2, bool two) {
  put_output1(A, o1, c1, n, y.a, s);
}

// Y (after the e^{-} DFT): truncate to the nz samples, scale, store columns.
template <typename T, int LOGK, typename V>
__device__ __forceinline__ void store_columns(const AxArgs<T>& A, const V* Y, int c1, int c2,
                                              bool two) {
  using C = cplx<T>;
  const int K = axial_K<LOGK>(A.sc), nz = K / 2, nt = axial_threads<LOGK>();
  C* o1 = A.out + size_t(c1) * nz;
  C* o2 = A.out + size_t(c2) * nz;
  for (int n = threadIdx.x; n < nz; n += nt) {
    int p = n - nz / 2;
    if (p < 0) p += K;
    const T s = __ldg(A.tab.scale + n);
    const V y = Y[prow(p)];
    put_output(A, o1, o2, n, y, s, c1, c2, two);
  }
}

// The inverse transform of Y and store_columns.  Compile-time K: the last
// pass runs in registers and writes the kept rows straight to the columns
// (the rows thread b's last-pass butterfly produces, b + i K/8, are rows it
// stores: natural row p goes to sample n = p + nz/2 for p < nz/2 and
// p - (K - nz/2) for p >= K - nz/2, nz = K/2; the others are dropped).
template <typename T, int LOGK, typename V>
__device__ __forceinline__ void inverse_and_store(const AxArgs<T>& A, V* Y, const cplx<T>* tw,
                                                  int c1, int c2, bool two) {
  if constexpr (LOGK > 0) {
    using C = cplx<T>;
    constexpr int K = 1 << LOGK, nz = K / 2, K8 = K / 8;
    const int b = threadIdx.x;
    fft_passes_ct<-1, false, K, 1, 1, T, true>(Y, 0, b, tw);
    C* o1 = A.out + size_t(c1) * nz;
    C* o2 = A.out + size_t(c2) * nz;
    last_pass_regs_ct<-1, LOGK, 1, T>(Y, 0, b, tw, [&](int i, const V& y) {
      const int p = b + i * K8;
      if (i * K8 >= K / 4 && (i + 1) * K8 <= 3 * K / 4) return;   // rows [K/4, 3K/4)
      const int n = p < K / 4 ? p + nz / 2 : p - (K - nz / 2);
      put_output(A, o1, o2, n, y, __ldg(A.tab.scale + n), c1, c2, two);
    });
  } else {
    fft_smem<-1, false, T>(Y, 1, 0, threadIdx.x, A.sc.K, A.sc.logK, tw, true);
    store_columns<T, LOGK, V>(A, Y, c1, c2, two);
  }
}

// FP32 plans at K = 1024 to 4096 can take the column-split radix-16
// transforms (fft_col16.cuh): three shared-memory passes per transform instead
// of four, the same threads and registers; the forward ends, and the inverse
// starts, in the layout of the interpolation and the scatter.  C16 selects
// them (the plan's choice, AxArgs::radix16); other instances ignore it.
template <typename T, int LOGK> __host__ __device__ constexpr bool ax_col16_exists() {
  return std::is_same<T, float>::value && LOGK >= 10;
}
template <typename T, int LOGK, bool C16> __host__ __device__ constexpr bool ax_col16() {
  return C16 && ax_col16_exists<T, LOGK>();
}

template <typename T, int LOGK, bool C16>
__device__ __forceinline__ const cplx<T>* ax_twiddles(const AxArgs<T>& A, unsigned char* smem) {
  const int K = axial_K<LOGK>(A.sc);
  cplx<T>* tw = twiddle_table<T>(smem, K);
  if constexpr (ax_col16<T, LOGK, C16>()) {
    c16::build_twiddles<LOGK>(reinterpret_cast<float4*>(tw));
    return tw;
  } else {
    return build_twiddles<T>(tw, A.tab.roots, K, A.sc.logK);
  }
}

// Y = the K-point e^{+} DFT of the pair's scaled, zero-padded columns
// (column-split form: loaded(v) as c16::forward)
template <typename T, int LOGK, bool C16, typename V, typename Loaded>
__device__ __forceinline__ void ax_forward(const AxArgs<T>& A, V* Y, const cplx<T>* tw,
                                           int c1, int c2, bool two, Loaded loaded) {
  if constexpr (ax_col16<T, LOGK, C16>()) {
    constexpr int nz = (1 << LOGK) / 2;
    const int c = threadIdx.x & 1;
    const cplx<T>* x = c == 0 ? A.in + size_t(c1) * nz : (two ? A.in + size_t(c2) * nz : nullptr);
    c16::forward<LOGK>(reinterpret_cast<float2*>(Y), reinterpret_cast<const float2*>(x),
                       reinterpret_cast<const float*>(A.tab.scale),
                       reinterpret_cast<const float4*>(tw), loaded);
  } else {
    load_and_fft<T, LOGK, V>(A, Y, tw, c1, c2, two);
  }
}

// The e^{-} DFT of Y, truncation to the nz kept rows, scaling, the columns'
// output (G, or u_hat = eta_hat - G/L).  STASH: eta_hat comes from stash(v), the
// eight samples forward's `loaded` was given, instead of memory.
template <typename T, int LOGK, bool C16, bool STASH, typename V, typename Stash>
__device__ __forceinline__ void ax_inverse(const AxArgs<T>& A, V* Y, const cplx<T>* tw,
                                           int c1, int c2, bool two, Stash stash) {
  if constexpr (ax_col16<T, LOGK, C16>()) {
    // rows j + i K/16 of this thread's column; rows [K/4, 3K/4) are dropped
    constexpr int K = 1 << LOGK, nz = K / 2, K16 = K / 16;
    const int c = threadIdx.x & 1, jb = threadIdx.x >> 1;
    const int col = c ? c2 : c1;
    cplx<T>* o = A.out + size_t(col) * nz;
    const bool keep = c == 0 || two;
    float2 v[8];
    const bool u_hat = A.u_hat_scale != T(0);
    c16::inverse<LOGK>(reinterpret_cast<float2*>(Y), reinterpret_cast<const float4*>(tw),
                       [&] { if (STASH) stash(v); },
                       [&](int i, const float2& y) {
                         if (!keep || (i >= 4 && i < 12)) return;
                         const int p = jb + i * K16;
                         const int n = i < 4 ? p + nz / 2 : p - (K - nz / 2);
                         const float s = __ldg(A.tab.scale + n);
                         if (STASH && u_hat)
                           o[n] = csub(v[i < 4 ? i + 4 : i - 12], cscale(y, s * A.u_hat_scale));
                         else
                           put_output1(A, o, col, n, reinterpret_cast<const cplx<T>&>(y), s);
                       });
  } else {
    inverse_and_store<T, LOGK, V>(A, Y, tw, c1, c2, two);
  }
}

// FP32: 64 registers a thread (two blocks of 512 threads on an SM).  FP64: the pair at
// K = 4096 fills an SM's shared memory by itself, so one (128 registers; at 64
// the adjoint half spilled 0.5 to 2 KB a thread).
// WIDE: the FP32 runtime lengths (K <= 1024, 128 threads at most) at 96 registers, for
// grids that one round of blocks holds at that width: latency is what they take, and the
// spills of 64 registers (up to 52 B) and their later trigger lie in it.  An iteration
// at 32 x 24 x 256 takes 25.8 us (29.2 with the residue-class scatter, 33.1 with windows
// and 64 registers), at 24 x 24 x 128 27.5 (28.5, 32.0), at 64 x 64 x 128 20.8 (47.7,
// 24.4).  Larger grids are quicker at 64: 128 x 128 x 256 93 us, 100 wide.
// FIT: FitOrder's operators (FP32): the scatter by residue classes, which product of the
// spectra and the phase rounds first, and at K = 4096 a trigger at the start (A + A^H at
// 512 x 1024 -> 2048: 53.3 us, 55.9 late; at 512 x 512 -> 1024 47.4, 38.5 late).  (As a
// flag of the other instances that cost 1.3 % of k_ax_fwd and k_ax_adj.)
enum AxVariant { PLAIN = 0, WIDE = 1, FIT = 2 };
template <typename T, int VAR> __host__ __device__ constexpr int ax_max_threads() {
  return VAR == WIDE ? 128 : 512;
}
template <typename T, int VAR> __host__ __device__ constexpr int ax_min_blocks() {
  return VAR == WIDE ? 5 : std::is_same<T, float>::value ? 2 : 1;
}

// ONE: a block per column instead of per pair (FP64, see
// launch_ax_JKC).
template <typename T, int J, int LOGK, bool C16, bool ONE, int VAR>
__global__ void __launch_bounds__(ax_max_threads<T, VAR>(), (ax_min_blocks<T, VAR>())) k_ax_fwd(const __grid_constant__ AxArgs<T> A) {
  using C = cplx<T>;
  using V = column_t<T, ONE>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const StoltConst& sc = A.sc;
  const int K = axial_K<LOGK>(sc), nk = sc.nk;
  V* Y = reinterpret_cast<V*>(smem_raw);
  int c1, c2, mx, my;
  pair_columns<T, ONE>(A, c1, c2, mx, my);
  const bool two = !ONE && c2 != c1;
  // programmatic dependent launch (as k_ax_fused): twiddles before the wait
  if (VAR == FIT && LOGK == 12) cudaTriggerProgrammaticLaunchCompletion();
  const C* tw = ax_twiddles<T, LOGK, C16>(A, smem_raw);
  cudaGridDependencySynchronize();
  ax_forward<T, LOGK, C16, V>(A, Y, tw, c1, c2, two, [](const float2*) {});

  cudaTriggerProgrammaticLaunchCompletion();   // as late as k_ax_fused, for its reason
  const Positions<T> pos(A, mx, my);
  const bool half = !ONE && A.half;
  C* o1 = A.out + size_t(spectrum_column(A, c1, half)) * nk;
  C* o2 = A.out + size_t(spectrum_column(A, c2, half)) * nk;
  // the half spectrum holds the pair's second column where both have x = 0 or nx/2
  const bool second = two && (!half || c1 % sc.nx == 0 || 2 * (c1 % sc.nx) == sc.nx);
  // nk <= K/2 = NRES blockDim: a quad of samples per thread
  const int q = threadIdx.x;
  if (NRES * q >= nk) return;
  Sample<T, V> sm[NRES];
  pos.quad(A, q, sm);
  cpair<T> ph;
  C a1, a2;
  interp_quad<T, J, V>(Coefficients<T, J>(A, pos, q), Y, K, sm, quad_fits<T, V>(A, sm),
                       [](int, const T*) {}, [&](int rho, V s) {
    const int j = NRES * q + rho;
    if (rho % 2 == 0) ph = pos.phases(A, q, rho / 2, sm);
    const C p = rho % 2 == 0 ? ph.a : ph.b;
    C s1 = cmul(s.a, p), s2 = s1;
    if constexpr (!ONE) {
      if (two) s2 = cmul(s.b, p);
      if (half) {
        s1 = cscale(cadd(s1, cconj(s2)), T(0.5));
        s2 = cconj(s1);
      }
    }
    if (rho % 2 == 0) {
      a1 = s1;
      a2 = s2;
    } else {
      store_two<T>(o1 + j - 1, a1, s1);
      if (second) store_two<T>(o2 + j - 1, a2, s2);
    }
  });
}

// a conj(b), by cmulc_ordered or as the kernel contracts it
template <bool ORDERED, typename C> __device__ __forceinline__ C conj_product(C a, C b) {
  if constexpr (ORDERED) return cmulc_ordered(a, b);
  else return cmulc(a, b);
}

// RES: the input holds the model spectra S and the kernel forms the residual
// spectrum R(q) = (S(q) + conj S(-q)) / 2 - F s_d(q) on load (ONE only; see
// k_ax_fused).
template <typename T, int J, int LOGK, bool C16, bool ONE, bool RES, int VAR>
__global__ void __launch_bounds__(ax_max_threads<T, VAR>(), (ax_min_blocks<T, VAR>())) k_ax_adj(const __grid_constant__ AxArgs<T> A) {
  static_assert(ONE || !RES, "the pair kernel with a residual is k_ax_fused");
  using C = cplx<T>;
  using V = column_t<T, ONE>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const StoltConst& sc = A.sc;
  const int K = axial_K<LOGK>(sc), nk = sc.nk;
  V* Y = reinterpret_cast<V*>(smem_raw);
  __shared__ int ch_lo, ch_hi, ch_tail;
  __shared__ int heads_fixed[window_heads_fixed<LOGK>()];
  int* heads = LOGK > 0 ? heads_fixed : window_heads<T, V>(A, Y);
  const int tid = threadIdx.x, nt = axial_threads<LOGK>();
  int c1, c2, mx, my;
  pair_columns<T, ONE>(A, c1, c2, mx, my);
  const bool two = !ONE && c2 != c1;
  if (tid == 0) { ch_lo = INT_MAX; ch_hi = INT_MIN; }
  // programmatic dependent launch (as k_ax_fused): twiddles before the wait
  if (VAR == FIT && LOGK == 12) cudaTriggerProgrammaticLaunchCompletion();
  const C* tw = ax_twiddles<T, LOGK, C16>(A, smem_raw);
  cudaGridDependencySynchronize();
  const bool stopped = RES && A.stop != nullptr && __ldcg(A.stop) != 0;
  const Positions<T> pos(A, mx, my);
  const bool half = !ONE && A.half;
  const C* r1 = A.in + size_t(spectrum_column(A, c1, half)) * nk;
  const C* r2 = A.in + size_t(c2) * nk;
  Sample<T, V> sm[NRES];
#pragma unroll
  for (int rho = 0; rho < NRES; ++rho) sm[rho].mfl = INT_MIN;
  if (NRES * tid < nk) {
    pos.quad(A, tid, sm);
#pragma unroll
    for (int h = 0; h < NRES / 2; ++h) {
      const int j = NRES * tid + 2 * h;
      const cpair<T> ph = pos.phases(A, tid, h, sm);
      cpair<T> x = load_two<T>(r1 + j);
      if constexpr (RES) {
        const cpair<T> y = load_two<T>(r2 + j), d = load_two<T>(A.sdh + size_t(c1) * nk + j);
        x.a = csub(cscale(cadd(x.a, cconj(y.a)), T(0.5)), d.a);
        x.b = csub(cscale(cadd(x.b, cconj(y.b)), T(0.5)), d.b);
      }
      sm[2 * h].val.a = conj_product<VAR == FIT>(x.a, ph.a);
      sm[2 * h + 1].val.a = conj_product<VAR == FIT>(x.b, ph.b);
      if constexpr (!ONE) {
        cpair<T> y{};
        if (two) y = half ? cpair<T>{cconj(x.a), cconj(x.b)} : load_two<T>(r2 + j);
        sm[2 * h].val.b = conj_product<VAR == FIT>(y.a, ph.a);
        sm[2 * h + 1].val.b = conj_product<VAR == FIT>(y.b, ph.b);
      }
    }
  }
  if (stopped) return;   // an earlier check stopped the solve: write nothing
  const Coefficients<T, J> co(A, pos, tid);
  bool fits = A.sc.window != 0;
  if (NRES * tid < nk) {
    heads[tid] = sm[0].mfl;
    fits = quad_fits<T, V>(A, sm);
  }
  scatter<T, J, false, V>(A, co, Y, K, nt, nk, sm, fits && VAR != FIT, &ch_lo, &ch_hi, &ch_tail, heads,
                          [&](int rho, T* e) {
                            window_taps<T, J>(co, rho, sm[rho].frac, window_offset(sm, rho) != 0, e);
                          }, [] {});
  cudaTriggerProgrammaticLaunchCompletion();
  ax_inverse<T, LOGK, C16, false, V>(A, Y, tw, c1, c2, two, [](float2*) {});
}

// Forward model, data residual and adjoint of one column pair in one pass
// (Alg. 1 gradient):  S = phase . N(eta_hat);  the lateral spectrum of the
// real residual Re(F^{-1} S) - s_d is, column by column,
//   R(q) = (S(q) + conj(S(-q))) / 2 - F s_d (q),
// because F(Re v)(q) = (F v(q) + conj(F v(-q))) / 2 and q, -q are the two
// columns of the pair; then G = N'(conj(phase) R), written as is or, when
// u_hat_scale = 1/L, as u_hat = eta_hat - G/L (put_output).  F s_d is
// Hermitian, so only its c1 column is read.
//
// What bounds it: two blocks a multiprocessor (64 registers a thread) with some 2,300
// instructions a warp between ten barriers.  On a 128 x 128 x 2048 volume (464 us, 27
// waves) 53 % of the issue slots and 64 % of the load/store data path are taken, half
// of the latter by the transforms' exchanges; DRAM 21 %.  A 1024 x 2048 B-scan (513
// blocks, 40.2 us) leaves the second of its 1.7 waves two thirds full.
// At 64 registers the column-split form spills 8 bytes a thread at J = 6 (44 with WS), 60
// (112) at J = 8, whose four samples share 15 slots.  conj(phase) R goes by the packed
// ordered product (1024 x 2048 solve 9.99 -> 9.89 ms), with WS, where that spilled more,
// by the compiler's, which rounds alike.
// WS: also write the model spectra S to A.s_out.
template <typename T, int J, int LOGK, bool WS, bool C16, int VAR>
__global__ void __launch_bounds__(ax_max_threads<T, VAR>(), (ax_min_blocks<T, VAR>())) k_ax_fused(const __grid_constant__ AxArgs<T> A) {
  using C = cplx<T>;
  using V = cpair<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const StoltConst& sc = A.sc;
  const int K = axial_K<LOGK>(sc), nk = sc.nk;
  V* Y = reinterpret_cast<V*>(smem_raw);
  __shared__ int ch_lo, ch_hi, ch_tail;
  __shared__ int heads_fixed[window_heads_fixed<LOGK>()];
  int* heads = LOGK > 0 ? heads_fixed : window_heads<T, V>(A, Y);
  // The column-split form keeps in tensor memory (tmem.cuh) what its 64 registers a
  // thread do not hold from the forward half to the adjoint: the samples' taps,
  // which it evaluated twice, and its eight samples of eta_hat, which it read twice
  // (1024 x 2048 solve 10.34 -> 10.17 ms, 768 x 1024 2.65 -> 2.42 ms; of either alone
  // the taps gain nothing and eta_hat half).
  constexpr bool TM = ax_col16<T, LOGK, C16>();
  constexpr int TAPS = tmem::kTapWords<J>, ETA = NRES * TAPS;
  static_assert(ETA + 16 <= tmem::kWords, "a thread's words");
  __shared__ uint32_t tm_slot;
  const int tid = threadIdx.x, nt = axial_threads<LOGK>();
  int c1, c2, mx, my;
  pair_columns(A, c1, c2, mx, my);
  const bool two = c2 != c1;
  if (tid == 0) { ch_lo = INT_MAX; ch_hi = INT_MIN; }
  // Programmatic dependent launch: this grid builds its twiddles, then waits for
  // the previous kernel before touching global data; the next kernel may start
  // once every block here is in its inverse transform (below).
  if (TM && tid < 32) tmem::allocate(&tm_slot, nt);
  const C* tw = ax_twiddles<T, LOGK, C16>(A, smem_raw);   // ends with a barrier
  const uint32_t tm = TM ? tmem::base(tm_slot) : 0;
  cudaGridDependencySynchronize();
  // the solve's stop flag (written by an earlier kernel, so visible after the
  // wait): loaded here, tested after the forward transform (before the first
  // global write), so its latency overlaps the transform
  const bool stopped = A.stop != nullptr && __ldcg(A.stop) != 0;
  const C* d1 = A.sdh + size_t(c1) * nk;
  ax_forward<T, LOGK, C16, V>(A, Y, tw, c1, c2, two, [&](const float2* v) {
    tmem::put16(tm + ETA, &v[0].x);
  });
  auto finish = [&] {                    // every warp's accesses to tensor memory done
    if (TM) {
      tmem::wait_stores();
      tmem::before_barrier();
      __syncthreads();
      if (tid < 32) tmem::release(tm_slot, nt);
    }
  };
  if (stopped) {         // an earlier check stopped the solve: write nothing
    finish();
    return;
  }
  const Positions<T> pos(A, mx, my);
  Sample<T, V> sm[NRES];
#pragma unroll
  for (int rho = 0; rho < NRES; ++rho) sm[rho].mfl = INT_MIN;
  bool fits = A.sc.window != 0;
  // tensor memory takes whole warps: lanes without samples follow the last ones
  const bool active = NRES * tid < nk;
  if (TM ? NRES * (tid & ~31) < nk : active) {
    const int q = TM ? min(tid, nk / NRES - 1) : tid;
    pos.quad(A, q, sm);
    fits = quad_fits<T, V>(A, sm);
    if (TM) fits = __all_sync(0xffffffffu, fits);
    if (active) heads[tid] = sm[0].mfl;
    V php, dq, w1, w2;                   // of two samples: phases, F s_d, model spectra
    interp_quad<T, J, V>(Coefficients<T, J>(A, pos, q), Y, K, sm, fits, [&](int rho, const T* e) {
      if constexpr (TM) tmem::put_taps<J>(tm + rho * TAPS, e);
    }, [&](int rho, V n) {
      const int j = NRES * q + rho;
      if (rho % 2 == 0) {
        php = pos.phases(A, q, rho / 2, sm);
        dq = load_two<T>(d1 + j);
      }
      const C ph = rho % 2 == 0 ? php.a : php.b;
      const C s1 = cmul(n.a, ph), s2 = two ? cmul(n.b, ph) : s1;
      if (WS) {
        if (rho % 2 == 0) {
          w1.a = s1;
          w2.a = s2;
        } else if (active) {
          store_two<T>(A.s_out + size_t(c1) * nk + j - 1, w1.a, s1);
          if (two) store_two<T>(A.s_out + size_t(c2) * nk + j - 1, w2.a, s2);
        }
      }
      // R(-q) = conj R(q): the residual is real
      const C R = csub(cscale(cadd(s1, cconj(s2)), T(0.5)), rho % 2 == 0 ? dq.a : dq.b);
      sm[rho].val.a = conj_product<!WS>(R, ph);
      sm[rho].val.b = two ? conj_product<!WS>(cconj(R), ph) : mk<T>(0, 0);
    });
  }
  if (TM) tmem::wait_stores();
  const Coefficients<T, J> co(A, pos, tid);
  scatter<T, J, TM, V>(A, co, Y, K, nt, nk, sm, fits && !A.fit, &ch_lo, &ch_hi, &ch_tail, heads,
                       [&](int rho, T* e) {
                         if constexpr (TM) tmem::get_taps<J>(tm + rho * TAPS, e);
                         else window_taps<T, J>(co, rho, sm[rho].frac,
                                                window_offset(sm, rho) != 0, e);
                       }, [&] {
                         // (positions are not kept in registers for this)
                         if (!TM) return;
                         Sample<T, V> again[NRES];
                         if (active) pos.quad(A, tid, again);
#pragma unroll
                         for (int rho = 0; rho < NRES; ++rho) {
                           sm[rho].mfl = active ? again[rho].mfl : INT_MIN;
                           sm[rho].frac = again[rho].frac;
                         }
                       });
  // Not earlier: the next kernel's waiting blocks take the first slots that fall
  // free, several to a multiprocessor, and stay there (1024 x 2048 solve 11.4 ms
  // with the trigger at the start of this kernel and of the update, 10.9 ms so)
  cudaTriggerProgrammaticLaunchCompletion();
  ax_inverse<T, LOGK, C16, TM, V>(A, Y, tw, c1, c2, two, [&](float2* v) {
    tmem::get16(tm + ETA, &v[0].x);
  });
  finish();
}

// One thread per (|q| class, quad): the same evaluation the kernels do on the fly.
template <typename T>
__global__ void k_stolt_table(const __grid_constant__ AxArgs<T> A, int4* out) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  const int cls = blockIdx.y;
  const int nq = A.sc.nk / NRES;
  if (q >= nq) return;
  const int ncx = A.sc.nx / 2 + 1;
  const int mx = cls % ncx, my = cls / ncx;
  const Positions<T> pos(A, mx, my);
  Sample<T, cone<T>> sm[NRES];
  pos.quad(A, q, sm);
  const cpair<T> p0 = pos.phases(A, q, 0, sm), p1 = pos.phases(A, q, 1, sm);
  int4* row = out + size_t(cls) * (size_t(StoltTable<T>::planes) * nq) + q;
  row[0] = make_int4(sm[0].mfl, sm[1].mfl, sm[2].mfl, sm[3].mfl);
  if constexpr (sizeof(T) == 4) {
    float4* f = reinterpret_cast<float4*>(row);
    f[nq] = make_float4(sm[0].frac, sm[1].frac, sm[2].frac, sm[3].frac);
    f[2 * nq] = make_float4(p0.a.x, p0.a.y, p0.b.x, p0.b.y);
    f[3 * nq] = make_float4(p1.a.x, p1.a.y, p1.b.x, p1.b.y);
  } else {
    double2* f = reinterpret_cast<double2*>(row);
    f[nq] = make_double2(sm[0].frac, sm[1].frac);
    f[2 * nq] = make_double2(sm[2].frac, sm[3].frac);
    f[3 * nq] = p0.a;
    f[4 * nq] = p0.b;
    f[5 * nq] = p1.a;
    f[6 * nq] = p1.b;
  }
}

// The FP64 coefficient table, from the Stolt table's fractions.
template <int J>
__global__ void k_coef_table(const __grid_constant__ AxArgs<double> A, double2* out) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x, nq = A.sc.nk / NRES;
  if (q >= nq) return;
  const int ncx = A.sc.nx / 2 + 1, cls = blockIdx.y;
  const Positions<double> pos(A, cls % ncx, cls / ncx);
  Sample<double, cone<double>> sm[NRES];
  pos.quad(A, q, sm);
  double2* o = out + size_t(cls) * (2 * J) * nq + q;
  for (int rho = 0; rho < NRES; ++rho) {
    double c[J];
    coefficients<double, J>(A.poly, sm[rho].mfl == INT_MIN ? 0.0 : sm[rho].frac, c);
    for (int i = 0; i < J / 2; ++i)
      o[(rho * (J / 2) + i) * nq] = make_double2(c[2 * i], c[2 * i + 1]);
  }
}

template <typename T> cudaError_t launch_stolt_table(const AxArgs<T>& a, int4* out,
                                                     cudaStream_t s) {
  const int rows = (a.sc.ny / 2 + 1) * (a.sc.nx / 2 + 1);
  dim3 grid((a.sc.nk / NRES + 127) / 128, rows);
  AxArgs<T> b = a;
  b.tab.stab = nullptr;
  k_stolt_table<T><<<grid, 128, 0, s>>>(b, out);
  return cudaGetLastError();
}

// shared memory of a pair's block (ONE: of a column's): Y and the twiddles
template <typename T, bool ONE> static size_t ax_smem(int K) {
  using V = column_t<T, ONE>;
  const size_t b = size_t(padded_rows(K)) * sizeof(V) +
                   size_t(twiddle_entries<T>(K, ilog2_dev(K))) * sizeof(cplx<T>);
  return (b + sizeof(V) - 1) / sizeof(V) * sizeof(V);
}
template <typename T> size_t ax_smem_bytes(int K) { return ax_smem<T, false>(K); }

// AX_ADJ_RES: the adjoint of the residual of model spectra (one column a block)
enum { AX_FWD = 0, AX_ADJ = 1, AX_FUSED = 2, AX_ADJ_RES = 3 };

// FP64 runs one column per block: no shared kernel, so the pair's fused form is
// compiled for FP32 only
template <typename T> constexpr bool ax_one() { return sizeof(T) == 8; }

template <typename T, int J, int LOGK, bool C16, int VAR = PLAIN>
static cudaError_t launch_ax_JKC(const AxArgs<T>& a, int npairs, cudaStream_t s, int kind) {
  constexpr bool ONE = ax_one<T>();
  using V = column_t<T, ONE>;
  const int K = a.sc.K;
  const int threads = K / 8;
  size_t sm = ax_smem<T, ONE>(K);
  AxArgs<T> b = a;
  b.past_offset = unsigned(sm);
  if (kind != AX_FWD) {
    sm += size_t(a.sc.past) * sizeof(V);
    if (LOGK == 0) sm += a.sc.nk / NRES * sizeof(int);
  }
  void (*kern)(AxArgs<T>) = nullptr;
  if (kind == AX_ADJ) kern = k_ax_adj<T, J, LOGK, C16, ONE, false, VAR>;
  else if (kind == AX_FWD) kern = k_ax_fwd<T, J, LOGK, C16, ONE, VAR>;
  else if constexpr (ONE) kern = k_ax_adj<T, J, LOGK, C16, ONE, true, VAR>;
  else if constexpr (VAR == FIT) return cudaErrorInvalidValue;
  else kern = a.s_out ? k_ax_fused<T, J, LOGK, true, C16, VAR> : k_ax_fused<T, J, LOGK, false, C16, VAR>;
  allow_smem(kern, sm);
  // programmatic dependent launch: each axial kernel builds its twiddles while
  // the previous kernel finishes, then waits for it (cudaGridDependencySynchronize)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ONE ? a.sc.nx * a.sc.ny : npairs);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  // not FP64: its blocks' time is the FP64 pipe's, so two of the next grid waiting
  // on one multiprocessor double that grid's time (128 x 512 solve: 28 ms against 10)
  at[0].val.programmaticStreamSerializationAllowed = sizeof(T) == 4;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, b);
}

// the plan's radix choice (a.radix16) where both forms exist
template <typename T, int J, int LOGK>
static cudaError_t launch_ax_JK(const AxArgs<T>& a, int npairs, cudaStream_t s, int kind) {
  if constexpr (ax_col16_exists<T, LOGK>()) {
    if (a.radix16) return launch_ax_JKC<T, J, LOGK, true>(a, npairs, s, kind);
  }
  return launch_ax_JKC<T, J, LOGK, false>(a, npairs, s, kind);
}

// K = 4096 and 2048 (nz = 2048, 1024) run the compile-time-length instances, and
// K = 1024 the FP32 column-split form (A + A^H at 128 x 256 -> 512: 14.4 us, 16.1 in
// runtime-length radix-8 passes; at K = 512, where it saves no pass, those stay
// ahead: a 128 x 128 x 256 volume's iteration takes 98 us, 102 split)
template <typename T, int J>
cudaError_t launch_ax_J(const AxArgs<T>& a, int npairs, cudaStream_t s, int kind) {
  if constexpr (sizeof(T) == 4) {
    if (a.fit && kind != AX_FUSED) {
      if (a.radix16 && a.sc.K == 4096) return launch_ax_JKC<T, J, 12, true, FIT>(a, npairs, s, kind);
      if (a.radix16 && a.sc.K == 2048) return launch_ax_JKC<T, J, 11, true, FIT>(a, npairs, s, kind);
      return launch_ax_JKC<T, J, 0, false, FIT>(a, npairs, s, kind);
    }
  }
  switch (a.sc.K) {
    case 4096: return launch_ax_JK<T, J, 12>(a, npairs, s, kind);
    case 2048: return launch_ax_JK<T, J, 11>(a, npairs, s, kind);
  }
  if constexpr (sizeof(T) == 4) {
    if (a.radix16 && a.sc.K == 1024) return launch_ax_JKC<T, J, 10, true>(a, npairs, s, kind);
  }
  if constexpr (sizeof(T) == 4) {
    // one round of blocks of whole warps at 96 registers
    const int threads = std::max(32, a.sc.K / 8), resident = kMultiprocessors * (65536 / 96);
    if (size_t(npairs) * threads <= size_t(resident))
      return launch_ax_JKC<T, J, 0, false, WIDE>(a, npairs, s, kind);
  }
  return launch_ax_JK<T, J, 0>(a, npairs, s, kind);
}

template <typename T>
static cudaError_t launch_ax(const AxArgs<T>& a, int npairs, cudaStream_t s, int kind) {
  switch (a.sc.J) {
    case 4: return launch_ax_J<T, 4>(a, npairs, s, kind);
    case 6: return launch_ax_J<T, 6>(a, npairs, s, kind);
    case 8: return launch_ax_J<T, 8>(a, npairs, s, kind);
  }
  return cudaErrorInvalidValue;
}

template <typename T> cudaError_t launch_ax_fwd(const AxArgs<T>& a, int npairs, cudaStream_t s) {
  return launch_ax<T>(a, npairs, s, AX_FWD);
}
template <typename T> cudaError_t launch_ax_adj(const AxArgs<T>& a, int npairs, cudaStream_t s) {
  return launch_ax<T>(a, npairs, s, AX_ADJ);
}
template <typename T> cudaError_t launch_ax_fused(const AxArgs<T>& a, int npairs,
                                                  cudaStream_t s) {
  if constexpr (ax_one<T>()) {
    // forward into the spectra workspace (or s_out), then the residual's adjoint
    AxArgs<T> f = a;
    f.out = a.s_out ? a.s_out : a.spec;
    const cudaError_t e = launch_ax<T>(f, npairs, s, AX_FWD);
    if (e != cudaSuccess) return e;
    f.in = f.out;
    f.out = a.out;
    return launch_ax<T>(f, npairs, s, AX_ADJ_RES);
  } else {
    return launch_ax<T>(a, npairs, s, AX_FUSED);
  }
}

}  // namespace isam
