// lc_coop.cuh — barrier of the cooperative kernels: one kernel whose blocks
// are all resident (cudaLaunchCooperativeKernel) and meet between phases.
#pragma once

#include "lc_internal.cuh"

namespace lc {

constexpr int kCoopThreads = 1024;
constexpr int kCoopBlocks = 152;  // at most one block per SM

// Blocks of the passes' and a level end's launches for n vertices and nnz
// stored edges: one per 64 vertices or 1,024 edges, at most one per SM.
inline int64_t level_grid(int64_t n, int64_t nnz) {
  const int64_t b = n / 64 > nnz / 1024 ? n / 64 : nnz / 1024;
  return b < 1 ? 1 : b > kCoopBlocks ? kCoopBlocks : b;
}
// The most blocks any cooperative launch of a call on such a graph has (the
// bins take one per kCoopThreads vertices, new-cluster ids fewer); its scratch
// is sized by it, so that a graph of a few vertices takes little.
inline int64_t coop_most(int64_t n, int64_t nnz) {
  const int64_t b = level_grid(n, nnz), bins = (n + kCoopThreads - 1) / kCoopThreads;
  return bins > kCoopBlocks ? kCoopBlocks : b > bins ? b : bins;
}
// int32 entries for the blocks' counts: kBins a block for the bins, one 64-bit
// word for the new-cluster ids.
inline int64_t coop_scratch(int64_t n, int64_t nnz) { return (int64_t)kBins * coop_most(n, nnz); }

// Polls before a wait gives up (about 0.6 us each): the call then ends with
// LC_ERR_DEVICE (see GridBarrier).
constexpr unsigned kCoopPolls = 1u << 24;

// Set in bar_arrived, above every count, when a wait ran out.
constexpr unsigned kBarDead = 1u << 31;

// Arrivals are counted monotonically within a launch; the last block to
// leave zeroes both counters for the next one.  1.2 us per barrier over 152
// blocks, measured; a block of its own only synchronises its threads.
//
// A wait that ran out marks the counter, which no block zeroes then: the other
// blocks' waits end at once, and so does the first sync() of every later
// cooperative kernel of the call.  No phase behind a barrier starts unless all
// blocks have arrived at it, so what is lost is the kernel's result, and the
// kernels see to it that what may be followed before the host looks is in
// range: the bins and a level's end say that they are complete (leave), the
// passes leave singleton labels, new-cluster ids leave no vertex unlabelled.
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
    if (nb == 1) {
      if (target != 0) return true;
      target = 1;
      if (threadIdx.x == 0) ok = (*(volatile unsigned *)&sc->bar_arrived & kBarDead) == 0;
      __syncthreads();
      return ok != 0;
    }
    target += nb;
    if (threadIdx.x == 0) {
#if LC_DEBUG
      const unsigned most = sc->dbg_skip ? sc->dbg_polls : kCoopPolls;
      const bool skip = sc->dbg_skip && blockIdx.x == nb - 1 && ++sc->dbg_syncs == sc->dbg_skip;
#else
      constexpr unsigned most = kCoopPolls;
      constexpr bool skip = false;
#endif
      unsigned seen = 0, polls = 0;
      if (!skip) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&sc->bar_arrived) : "memory");
        do {
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&sc->bar_arrived) : "memory");
        } while (seen < target && ++polls < most);
      }
      ok = seen >= target && seen < kBarDead;
      if (!ok) {
        sc->error = 1;
        if (!skip && seen < kBarDead) atomicOr(&sc->bar_arrived, kBarDead);
      }
    }
    __syncthreads();
    return ok != 0;
  }

  // Once per block after its last sync(); done: null, or set to 1 once every
  // block has got here.
  __device__ void leave(int32_t *done = nullptr) {
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (gridDim.x > 1) {
      if (atomicAdd(&sc->bar_left, 1u) != gridDim.x - 1) return;
      sc->bar_arrived = 0;
      sc->bar_left = 0;
    }
    if (done) *done = 1;
    __threadfence();
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
