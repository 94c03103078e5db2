// Tensor memory as a per-thread stash.  An SM's tensor memory (128 lanes of 512
// 32-bit columns) is reached beside the load/store path that bounds the axial
// kernels: a warp writes and reads registers against the 32 lanes of its quarter
// (warp id mod 4), a column a register.  A block takes one column per two threads, so
// the 1,024 threads that fit an SM at 64 registers share all 512, 64 words each.
//
// Every call is warp-wide: all 32 lanes (put_taps, get_taps, put16 and get16 bring
// them together first).
#pragma once

#include <stdint.h>

namespace isam {
namespace tmem {

constexpr int kWords = 64;      // of a thread

// threads: of the block, a multiple of 128
__host__ __device__ constexpr int columns(int threads) { return threads / 128 * kWords; }

// Warp 0 of the block: allocates and writes the base address to *slot (shared); a
// barrier, then base().  Waits while other blocks of the SM hold the columns.
__device__ __forceinline__ void allocate(uint32_t* slot, int threads) {
  const uint32_t s = uint32_t(__cvta_generic_to_shared(slot));
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s),
               "r"(columns(threads))
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
// Warp 0, after a barrier that follows every warp's last access.
__device__ __forceinline__ void release(uint32_t allocated, int threads) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(allocated),
               "r"(columns(threads))
               : "memory");
}
// this thread's word 0
__device__ __forceinline__ uint32_t base(uint32_t allocated) {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t warp = threadIdx.x >> 5;
  return allocated + ((warp & 3) << 21) + (warp >> 2) * kWords;   // lane 32 (warp mod 4)
}
__device__ __forceinline__ void before_barrier() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void wait_stores() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void put8(uint32_t a, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(a),
               "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]),
               "f"(v[7])
               : "memory");
}
__device__ __forceinline__ void put4(uint32_t a, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(a), "f"(v[0]),
               "f"(v[1]), "f"(v[2]), "f"(v[3])
               : "memory");
}
__device__ __forceinline__ void put1(uint32_t a, float v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(a), "f"(v) : "memory");
}
// the loads wait for their registers
__device__ __forceinline__ void get8(uint32_t a, float* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
        "=f"(v[7])
      : "r"(a)
      : "memory");
}
__device__ __forceinline__ void get4_1(uint32_t a, float* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%5];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x1.b32 {%4}, [%6];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4])
      : "r"(a), "r"(a + 4)
      : "memory");
}
__device__ __forceinline__ void get8_1(uint32_t a, float* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%9];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x1.b32 {%8}, [%10];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
        "=f"(v[7]), "=f"(v[8])
      : "r"(a), "r"(a + 8)
      : "memory");
}

// J + 1 taps of a sample, TAP_WORDS<J> apart
template <int J> constexpr int kTapWords = J == 6 ? 8 : J + 1;
template <int J> __device__ __forceinline__ void put_taps(uint32_t a, const float* e) {
  __syncwarp();
  if constexpr (J == 4) {
    put4(a, e);
    put1(a + 4, e[4]);
  } else if constexpr (J == 6) {
    const float v[8] = {e[0], e[1], e[2], e[3], e[4], e[5], e[6], 0.0f};
    put8(a, v);
  } else {
    put8(a, e);
    put1(a + 8, e[8]);
  }
}
template <int J> __device__ __forceinline__ void get_taps(uint32_t a, float* e) {
  __syncwarp();
  if constexpr (J == 4) get4_1(a, e);
  else if constexpr (J == 8) get8_1(a, e);
  else {
    float v[8];
    get8(a, v);
#pragma unroll
    for (int l = 0; l <= J; ++l) e[l] = v[l];
  }
}

__device__ __forceinline__ void put16(uint32_t a, const float* v) {
  __syncwarp();
  put8(a, v);
  put8(a + 8, v + 8);
}
__device__ __forceinline__ void get16(uint32_t a, float* v) {
  __syncwarp();
  get8(a, v);
  get8(a + 8, v + 8);
}

}  // namespace tmem
}  // namespace isam
