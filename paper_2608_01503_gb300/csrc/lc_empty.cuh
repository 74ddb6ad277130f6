// lc_empty.cuh — ids for the movers to new empty clusters, as phases of a
// cooperative kernel (all blocks, T threads each).
#pragma once

#include "lc_coop.cuh"
#include "lc_pass.cuh"

namespace lc {

// Exclusive scan over the block of packed counts; `total` is the block's sum.
// red: T / 32 entries of shared memory.
template <int T>
__device__ __forceinline__ unsigned long long coop_scan(unsigned long long x, unsigned long long *red,
                                                        unsigned long long &total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += y;
  }
  __syncthreads();  // the last call's reads of red are done
  if (lane == 31) red[wid] = incl;
  __syncthreads();
  unsigned long long before = 0;
  total = 0;
  for (int w = 0; w < T / 32; ++w) {
    const unsigned long long t = red[w];
    before += w < wid ? t : 0;
    total += t;
  }
  return before + incl - x;
}

// Labels the `total` > 0 vertices with C[v] = kEmpty.  Free ids and movers
// are counted and listed together: packed as free << 32 | movers (both below
// 2^31).  marked: w.used already marks the ids in use.  False if a barrier
// ran out.
template <int T>
__device__ __forceinline__ bool assign_empty(const PassArgs &a, const EmptyScratch &w, int total, bool marked,
                                             GridBarrier &bar) {
  __shared__ unsigned long long red[T / 32];
  const int64_t n = a.g.n;
  const int64_t tid = (int64_t)blockIdx.x * T + threadIdx.x;
  const int64_t nt = (int64_t)gridDim.x * T;
  if (!marked) {
    for (int64_t x = tid; x < n; x += nt) w.used[x] = 0;
    if (!bar.sync()) return false;
    for (int64_t v = tid; v < n; v += nt) {
      const int32_t x = a.C[v];
      if (x >= 0) w.used[x] = 1;
    }
    if (!bar.sync()) return false;
  }
  // each block its own run of ids
  const int64_t per = ((n + gridDim.x - 1) / gridDim.x + T - 1) / T * T;
  const int64_t lo = (int64_t)blockIdx.x * per, hi = lo + per < n ? lo + per : n;
  auto flags = [&](int64_t x) {
    if (x >= hi) return 0ull;
    return (w.used[x] == 0 ? 1ull << 32 : 0ull) | (a.C[x] == kEmpty ? 1ull : 0ull);
  };
  unsigned long long mine = 0, sum;
  for (int64_t x = lo + threadIdx.x; x < hi; x += T) mine += flags(x);
  coop_scan<T>(mine, red, sum);
  if (threadIdx.x == 0) w.blocks[blockIdx.x] = sum;
  if (!bar.sync()) return false;
  unsigned long long before = 0;
  coop_scan<T>((int)threadIdx.x < (int)blockIdx.x ? w.blocks[threadIdx.x] : 0ull, red, before);
  for (int64_t base = lo; base < hi; base += T) {
    const int64_t x = base + threadIdx.x;
    const unsigned long long f = flags(x);
    const unsigned long long at = before + coop_scan<T>(f, red, sum);
    before += sum;
    if (x < hi) {
      const int32_t pf = (int32_t)(at >> 32), pm = (int32_t)(uint32_t)at;
      if (f >> 32) w.freelist[pf] = (int32_t)x;
      if (f & 1ull) w.movers[pm] = (int32_t)x;
      const int g = a.gid ? a.gid[x] : 0;
      if (a.gp[g].vbase == x) {
        w.gfree[g] = pf;
        w.gmover[g] = pm;
      }
    }
  }
  if (!bar.sync()) return false;
  for (int64_t i = tid; i < total; i += nt) {
    const int32_t v = w.movers[i];
    const int g = a.gid ? a.gid[v] : 0;
    const int64_t idx = (int64_t)w.gfree[g] + (i - w.gmover[g]);
    const int32_t x = (idx >= 0 && idx < n) ? w.freelist[idx] : -1;
    // there are always at least as many free ids in a graph as movers; an
    // id outside the graph would be a bound violation, reported, not used
    if (x < 0 || x >= n || (a.gid ? a.gid[x] : 0) != g) {
      a.sc->error = 1;
      a.C[v] = v;
      continue;
    }
    a.C[v] = x;
    a.W[x] = a.g.vw[v];
  }
  return true;
}

}  // namespace lc
