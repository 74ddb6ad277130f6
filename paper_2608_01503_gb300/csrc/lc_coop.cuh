// lc_coop.cuh — barrier of the cooperative kernels: one kernel whose blocks
// are all resident (cudaLaunchCooperativeKernel) and meet between phases.
#pragma once

#include "lc_internal.cuh"

namespace lc {

constexpr int kCoopThreads = 1024;
constexpr int kCoopBlocks = 152;  // at most one block per SM

// int32 entries of a call's scratch for the blocks' counts: the bins' count
// kBins per block, the new-cluster ids one 64-bit word.
constexpr int64_t kCoopScratch = (int64_t)kBins * kCoopBlocks;

// Polls before a wait gives up (about 0.6 us each): the launch then sets the
// error flag and every block returns, so the call ends with LC_ERR_DEVICE.
constexpr unsigned kCoopPolls = 1u << 24;

// Arrivals are counted monotonically within a launch; the last block to
// leave zeroes both counters for the next one.  1.2 us per barrier over 152
// blocks, measured; a block of its own only synchronises its threads.
struct GridBarrier {
  Scalars *sc;
  unsigned target = 0;
  __device__ explicit GridBarrier(Scalars *s) : sc(s) {}

  // Every thread of every block; false once a wait ran out (uniform over the
  // block): the caller returns.
  __device__ bool sync() {
    __shared__ int ok;
    const unsigned nb = gridDim.x;
    __syncthreads();
    if (nb == 1) return true;
    target += nb;
    if (threadIdx.x == 0) {
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&sc->bar_arrived) : "memory");
      unsigned seen = 0, polls = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&sc->bar_arrived) : "memory");
      } while (seen < target && ++polls < kCoopPolls);
      ok = seen >= target;
      if (!ok) sc->error = 1;
    }
    __syncthreads();
    return ok != 0;
  }

  // Once per block after its last sync().
  __device__ void leave() {
    if (gridDim.x == 1) return;
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&sc->bar_left, 1u) == gridDim.x - 1) {
      sc->bar_arrived = 0;
      sc->bar_left = 0;
      __threadfence();
    }
  }
};

// Blocks a cooperative launch of one block per SM may have on this device, of
// at most `limit` (a call's share of the SMs while others run beside it).
inline int coop_blocks(int limit) {
  int dev = 0, sms = 1;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 1;
  if (sms > kCoopBlocks) sms = kCoopBlocks;
  return limit < 1 ? 1 : limit < sms ? limit : sms;
}

}  // namespace lc
