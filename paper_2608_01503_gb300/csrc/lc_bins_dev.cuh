// lc_bins_dev.cuh — the two phases of the degree bins (both in lc_bins.cu; the
// second in lc_level.cu for a level built on the device).
#pragma once

#include <type_traits>

#include "lc_bin_rule.cuh"
#include "lc_bins.cuh"
#include "lc_coop.cuh"

namespace lc {

// What the bins are built from and into.
struct BinWork {
  int32_t max_deg[kBins - 1];
  int32_t hub_chunk;
  VRec *recs;
  int32_t *lists;
  int32_t *counts;  // [kBins][blocks of the launch]
};

inline BinWork bin_work(const BinPlan &plan, const Bins &b, int32_t *counts) {
  BinWork w{};
  for (int k = 0; k < kBins - 1; ++k) w.max_deg[k] = (int32_t)plan.max_deg[k];
  w.hub_chunk = (int32_t)plan.hub_chunk;
  w.recs = b.recs;
  w.lists = b.lists;
  w.counts = counts;
  return w;
}

// Every block takes a run of vertices of its own.
struct BinRun {
  int64_t lo, hi;
};
template <int T>
__device__ __forceinline__ BinRun bin_run(int64_t n) {
  const int64_t per = ((n + gridDim.x - 1) / gridDim.x + T - 1) / T * T;
  const int64_t lo = (int64_t)blockIdx.x * per;
  return BinRun{lo, lo + per < n ? lo + per : n};
}

// Phase 1 (T threads): the bins of the block's run into w.counts; the hub
// figures are summed in *out.  A grid barrier follows.  deg_of: the row_degree
// that the records of phase 2 hold.
template <int T, typename Deg>
__device__ __forceinline__ void bins_count(const BinWork &w, int64_t n, BinOut *out, Deg deg_of) {
  __shared__ int32_t s_cnt[kBins];
  __shared__ long long s_chunks;
  __shared__ int32_t s_max;
  static_assert(std::is_same<decltype(deg_of(int64_t())), int32_t>::value, "the degree as phase 2 bins it");
  const int lane = threadIdx.x & 31;
  const BinRun run = bin_run<T>(n);
  if (threadIdx.x < kBins) s_cnt[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    s_chunks = 0;
    s_max = 0;
  }
  __syncthreads();
  int cnt[kBins] = {};
  long long chunks = 0;
  int32_t longest = 0;
  for (int64_t v = run.lo + threadIdx.x; v < run.hi; v += T) {
    const int32_t deg = deg_of(v);
    const int b = bin_of(w.max_deg, deg);
#pragma unroll
    for (int k = 0; k < kBins; ++k) cnt[k] += b == k;
    if (b == kHubBin) {
      chunks += ((int64_t)deg + w.hub_chunk - 1) / w.hub_chunk;
      longest = deg > longest ? deg : longest;
    }
  }
#pragma unroll
  for (int k = 0; k < kBins; ++k) {
    const int t = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)cnt[k]);
    if (lane == 0 && t) atomicAdd(&s_cnt[k], t);
  }
  if (longest > 0) {
    atomicAdd((unsigned long long *)&s_chunks, (unsigned long long)chunks);
    atomicMax(&s_max, longest);
  }
  __syncthreads();
  if (threadIdx.x < kBins) w.counts[threadIdx.x * gridDim.x + blockIdx.x] = s_cnt[threadIdx.x];
  if (threadIdx.x == 0 && s_max > 0) {
    atomicAdd((unsigned long long *)&out->chunks, (unsigned long long)s_chunks);
    atomicMax(&out->max_deg, s_max);
  }
}

// Phase 2, by as many blocks: the vertices of the run that the block of this
// number counted in phase 1 into the lists and records, ascending in each bin;
// out: null, or where block 0 leaves the bins' starts.  A place past the
// arrays (row_ptr written to between the phases) is not taken.
template <int T, typename Rec>
__device__ __forceinline__ void bins_place(const BinWork &w, int64_t n, const BinRun run, int blocks, BinOut *out,
                                           Rec rec_of) {
  constexpr int W = T / 32;
  static_assert(W >= kBins && W <= 32, "a warp per bin, a lane per warp");
  __shared__ int32_t s_cnt[kBins], s_run[kBins];
  __shared__ int32_t s_w[W][kBins + 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // a bin per warp: its total and what the blocks before this one hold
  if (wid < kBins) {
    int total = 0, before = 0;
    for (int b = lane; b < blocks; b += 32) {
      const int c = w.counts[wid * blocks + b];
      total += c;
      before += b < (int)blockIdx.x ? c : 0;
    }
    total = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)total);
    before = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)before);
    if (lane == 0) {
      s_cnt[wid] = total;
      s_run[wid] = before;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const bool tell = out && blockIdx.x == 0;
    int at = 0;
    for (int k = 0; k < kBins; ++k) {
      s_run[k] += at;
      if (tell) out->offs[k] = at;
      at += s_cnt[k];
    }
    if (tell) out->offs[kBins] = at;
  }
  __syncthreads();
  for (int64_t base = run.lo; base < run.hi; base += T) {
    const int64_t v = base + threadIdx.x;
    VRec r{};
    int b = kBins;
    if (v < run.hi) {
      r = rec_of(v);
      b = bin_of(w.max_deg, r.deg);
    }
    // rank within the tile: in the warp by ballots, then over the warps
    int rank = 0, mine = 0;
#pragma unroll
    for (int k = 0; k < kBins; ++k) {
      const unsigned m = __ballot_sync(0xFFFFFFFFu, b == k);
      if (b == k) rank = __popc(m & ((1u << lane) - 1u));
      if (lane == k) mine = __popc(m);
    }
    if (lane < kBins) s_w[wid][lane] = mine;
    __syncthreads();
    if (wid < kBins) {
      const int c = lane < W ? s_w[lane][wid] : 0;
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
      }
      const int start = s_run[wid];
      if (lane < W) s_w[lane][wid] = start + incl - c;
      __syncwarp();
      if (lane == 31) s_run[wid] = start + incl;
    }
    __syncthreads();
    if (b < kBins) {
      const int at = s_w[wid][b] + rank;
      if (at < n) {
        w.lists[at] = r.v;
        w.recs[at] = r;
      }
    }
    __syncthreads();
  }
}

}  // namespace lc
