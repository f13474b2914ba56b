// Tensor memory as a place to park registers.
//
// An SM has 256 KB of tensor memory (128 lanes x 512 columns of 32 bits) beside its registers and
// shared memory.  A transform that is needed twice (phi in the z pass, the strip of B in the
// inverse y passes) is parked there between its uses: each thread writes its own words and reads
// them back, a warp in its quarter of the lanes, in about 100 cycles per 32 words for both ways
// (measured), instead of a round trip through L2 or a second exchange buffer in shared memory.
#pragma once
#include <cstdint>

#include "tma.cuh"

namespace cola {

// columns a block of `threads` threads needs for `words` words per thread: the warps beyond the
// first four share their lane quarters; an allocation is a power of two of at least 32 columns
__host__ __device__ constexpr int tmem_columns(int threads, int words) {
  const int want = (threads + 127) / 128 * words;
  int c = 32;
  while (c < want) c *= 2;
  return c;
}

#define COLA_R16(r, o) "r"(r[o]), "r"(r[o + 1]), "r"(r[o + 2]), "r"(r[o + 3]), "r"(r[o + 4]), "r"(r[o + 5]), \
      "r"(r[o + 6]), "r"(r[o + 7]), "r"(r[o + 8]), "r"(r[o + 9]), "r"(r[o + 10]), "r"(r[o + 11]), "r"(r[o + 12]), \
      "r"(r[o + 13]), "r"(r[o + 14]), "r"(r[o + 15])
#define COLA_W16(r, o) "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), \
      "=r"(r[o + 6]), "=r"(r[o + 7]), "=r"(r[o + 8]), "=r"(r[o + 9]), "=r"(r[o + 10]), "=r"(r[o + 11]), \
      "=r"(r[o + 12]), "=r"(r[o + 13]), "=r"(r[o + 14]), "=r"(r[o + 15])

// One block's allocation.  The constructor and close() are called by every thread of the block;
// store and load by whole warps.  Every instruction on tensor memory is .sync.aligned: the lanes of
// a warp must reach it together, so each function brings them together first, whatever branch the
// caller took per lane (a column beyond the last one, the mode k = 0) just before.
template <int THREADS, int WORDS>
struct TmemPark {
  static constexpr int COLS = tmem_columns(THREADS, WORDS);
  static_assert(COLS <= 512, "more words than the tensor memory holds");
  static_assert(WORDS % 16 == 0, "whole 16-word chunks");
  uint32_t base, addr;  // the block's allocation, this thread's warp in it

  // (slot: 4 bytes of shared memory; contains a block barrier)
  __device__ __forceinline__ explicit TmemPark(uint32_t* slot) {
    const int warp = threadIdx.x >> 5;
    __syncwarp();
    if (warp == 0) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)), "n"(COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    base = *slot;
    addr = base + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * WORDS;  // lane 32 (warp mod 4)
  }

  // (N <= WORDS words of this thread)
  template <int N>
  __device__ __forceinline__ void store(const uint32_t (&r)[N]) const {
    static_assert(N <= WORDS && N % 16 == 0, "whole chunks of this thread's words");
    __syncwarp();
#pragma unroll
    for (int o = 0; o < N; o += 16)
      asm volatile(
          "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
              addr + o),
          COLA_R16(r, o)
          : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  // (the wait is part of each load's statement: its results may be used right after it)
  template <int N>
  __device__ __forceinline__ void load(uint32_t (&r)[N]) const {
    static_assert(N <= WORDS && N % 16 == 0, "whole chunks of this thread's words");
    __syncwarp();
    if constexpr (N % 32 == 0) {
#pragma unroll
      for (int o = 0; o < N; o += 32)
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
            "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\ttcgen05.wait::ld.sync.aligned;"
            : COLA_W16(r, o), COLA_W16(r, o + 16)
            : "r"(addr + o)
            : "memory");
    } else {
#pragma unroll
      for (int o = 0; o < N; o += 16)
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
            "[%16];\n\ttcgen05.wait::ld.sync.aligned;"
            : COLA_W16(r, o)
            : "r"(addr + o)
            : "memory");
    }
  }

  // words o .. o + 15 of this thread (o a multiple of 16)
  __device__ __forceinline__ void load16(int o, uint32_t (&r)[16]) const {
    __syncwarp();
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
        "[%16];\n\ttcgen05.wait::ld.sync.aligned;"
        : COLA_W16(r, 0)
        : "r"(addr + o)
        : "memory");
  }

  // gives the columns back (contains a block barrier: every warp's accesses are done)
  __device__ __forceinline__ void close() const {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (threadIdx.x < 32)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "n"(COLS) : "memory");
  }
};
// The same in the thread's own registers, for transforms short enough to leave room for a copy.
template <int MAX>
struct RegPark {
  mutable uint32_t kept[MAX];
  __device__ __forceinline__ explicit RegPark(uint32_t*) { __syncthreads(); }
  template <int N>
  __device__ __forceinline__ void store(const uint32_t (&r)[N]) const {
    static_assert(N <= MAX, "this thread's words");
#pragma unroll
    for (int i = 0; i < N; ++i) kept[i] = r[i];
  }
  template <int N>
  __device__ __forceinline__ void load(uint32_t (&r)[N]) const {
#pragma unroll
    for (int i = 0; i < N; ++i) r[i] = kept[i];
  }
  __device__ __forceinline__ void load16(int o, uint32_t (&r)[16]) const {
#pragma unroll
    for (int i = 0; i < 16; ++i) r[i] = kept[o + i];
  }
  __device__ __forceinline__ void close() const {}
};
// for a kernel that parks nothing
struct NoPark {
  __device__ __forceinline__ explicit NoPark(uint32_t*) {}
  __device__ __forceinline__ void close() const {}
};
#undef COLA_R16
#undef COLA_W16

}  // namespace cola
