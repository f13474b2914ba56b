// Host side of the column passes (pm_bodies.cuh): shared memory and grid.
#pragma once
#include <algorithm>

#include "pm_bodies.cuh"

namespace cola {

// shared memory of a block: the groups' exchange buffers, the stage twiddle table and
// `sinc` floats
template <class Cfg>
constexpr size_t cols_smem(int sinc) {
  constexpr size_t bytes = sizeof(float2) * (Cfg::TABLE + stw_size<typename Cfg::C>());
  static_assert(bytes + sizeof(float) * Cfg::N_ <= 227 * 1024, "column pass: too much shared memory");
  return bytes + sizeof(float) * sinc;
}

// Blocks of a launch of kernel FN over `strips` strips: for a persistent shape the resident ones
// (found once per device), or as many as there are strips.
template <class Cfg, auto* FN>
int cols_grid(size_t smem, int64_t strips, unsigned* grid) {
  static std::atomic<int> resident[64] = {};
  int dev = 0;
  COLA_CUDA_CHECK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(COLA_EUNSUPPORTED, "device index above 63");
  int cap = resident[dev].load(std::memory_order_acquire);
  if (!cap) {
    int occ = 0, sms = 0;
    COLA_CUDA_CHECK(cudaFuncSetAttribute(FN, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    COLA_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, FN, Cfg::THREADS, smem));
    COLA_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (occ < 1) return fail(COLA_EUNSUPPORTED, "column pass does not fit on an SM");
    cap = std::min(occ, Cfg::MIN_BLOCKS) * sms;
    resident[dev].store(cap, std::memory_order_release);
  }
  *grid = (unsigned)(Cfg::RESIDENT ? std::min<int64_t>(strips, cap) : (strips + Cfg::G - 1) / Cfg::G);
  return COLA_OK;
}

}  // namespace cola
