// lc_bins.cu — the degree bins of a level (Section IV-C-2's buckets): the
// vertices of each bin in ascending order with their records, and the chunk
// plan of the hub bin.
#include "lc_bins.cuh"
#include "lc_coop.cuh"

namespace lc {

namespace {

constexpr int kT = kCoopThreads, kW = kT / 32;

struct BinArgs {
  LevelGraph g;
  const int32_t *gid;         // graph of each vertex (nullptr: one graph)
  int32_t max_deg[kBins - 1];
  int32_t hub_chunk;
  VRec *recs;
  int32_t *lists;
  BinOut *out;
  int32_t *counts;            // [kBins][kCoopBlocks]
  Scalars *sc;
};

__device__ __forceinline__ int bin_of(const BinArgs &a, int64_t deg) {
  int b = 0;
#pragma unroll
  for (int k = 0; k < kBins - 1; ++k) b += deg > a.max_deg[k] ? 1 : 0;
  return b;
}

// One cooperative launch: every block counts the bins of its run of vertices,
// and once all have met, places them.  Bound by the records it writes: 52
// bytes a vertex, 16 of them read twice.  Ten scans of three launches and a
// separate pass for the records took 0.35 ms at 912,673 vertices and 70 us,
// all launches, on 10,000; this takes 30 us and 8 us.
__global__ void __launch_bounds__(kT, 1) k_bins(const __grid_constant__ BinArgs a) {
  __shared__ int32_t s_cnt[kBins], s_run[kBins];
  __shared__ int32_t s_w[kW][kBins + 1];
  __shared__ long long s_chunks;
  __shared__ int32_t s_max;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t n = a.g.n;
  const int64_t per = ((n + gridDim.x - 1) / gridDim.x + kT - 1) / kT * kT;
  const int64_t lo = (int64_t)blockIdx.x * per, hi = lo + per < n ? lo + per : n;
  GridBarrier bar(a.sc);
  if (threadIdx.x < kBins) s_cnt[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    s_chunks = 0;
    s_max = 0;
  }
  __syncthreads();
  {
    int cnt[kBins] = {};
    long long chunks = 0;
    int32_t longest = 0;
    for (int64_t v = lo + threadIdx.x; v < hi; v += kT) {
      const int64_t deg = a.g.rp[v + 1] - a.g.rp[v];
      const int b = bin_of(a, deg);
#pragma unroll
      for (int k = 0; k < kBins; ++k) cnt[k] += b == k;
      if (b == kHubBin) {
        chunks += (deg + a.hub_chunk - 1) / a.hub_chunk;
        longest = deg > longest ? (int32_t)deg : longest;
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
  }
  __syncthreads();
  if (threadIdx.x < kBins) a.counts[threadIdx.x * kCoopBlocks + blockIdx.x] = s_cnt[threadIdx.x];
  if (threadIdx.x == 0 && s_max > 0) {
    atomicAdd((unsigned long long *)&a.out->chunks, (unsigned long long)s_chunks);
    atomicMax(&a.out->max_deg, s_max);
  }
  if (!bar.sync()) return;
  // a bin per warp: its total and what the blocks before this one hold
  if (wid < kBins) {
    int total = 0, before = 0;
    for (int b = lane; b < (int)gridDim.x; b += 32) {
      const int c = a.counts[wid * kCoopBlocks + b];
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
    int at = 0;
    for (int k = 0; k < kBins; ++k) {
      s_run[k] += at;
      if (blockIdx.x == 0) a.out->offs[k] = at;
      at += s_cnt[k];
    }
    if (blockIdx.x == 0) a.out->offs[kBins] = at;
  }
  __syncthreads();
  for (int64_t base = lo; base < hi; base += kT) {
    const int64_t v = base + threadIdx.x;
    VRec r{};
    int b = kBins;
    if (v < hi) {
      r.v = (int32_t)v;
      r.beg = a.g.rp[v];
      const int64_t deg = a.g.rp[v + 1] - r.beg;
      r.deg = (int32_t)deg;
      r.g = a.gid ? a.gid[v] : 0;
      r.w = a.g.vw[v];
      b = bin_of(a, deg);
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
      const int c = s_w[lane][wid];  // kW == 32 warps
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
      }
      const int run = s_run[wid];
      s_w[lane][wid] = run + incl - c;
      __syncwarp();
      if (lane == 31) s_run[wid] = run + incl;
    }
    __syncthreads();
    if (b < kBins) {
      const int at = s_w[wid][b] + rank;
      a.lists[at] = r.v;
      a.recs[at] = r;
    }
    __syncthreads();
  }
  bar.leave();
}
static_assert(kW == 32, "one lane per warp in the tile scan");

// Cuts the hub rows into chunks of hub_chunk edges: c0[h] = the first chunk
// of hub h, and each chunk's hub and edges.  One block.
__global__ void __launch_bounds__(kT, 1)
    k_hub_plan(const VRec *__restrict__ hubs, int H, int32_t hub_chunk, int32_t *c0, int32_t *hub_of, int64_t *e0,
               int64_t *e1, long long *acc, int32_t *done) {
  __shared__ int32_t s_w[kW];
  __shared__ int32_t s_run;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_run = 0;
  for (int base = 0; base < H; base += kT) {
    const int h = base + threadIdx.x;
    const int c = h < H ? (hubs[h].deg + hub_chunk - 1) / hub_chunk : 0;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += y;
    }
    __syncthreads();
    if (lane == 31) s_w[wid] = incl;
    __syncthreads();
    int before = s_run, total = 0;
    for (int w = 0; w < kW; ++w) {
      before += w < wid ? s_w[w] : 0;
      total += s_w[w];
    }
    if (h < H) {
      c0[h] = before + incl - c;
      acc[h] = 0;
      done[h] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) s_run += total;
  }
  __syncthreads();
  if (threadIdx.x == 0) c0[H] = s_run;
  for (int h = wid; h < H; h += kW) {  // a hub's chunks by a warp
    const VRec r = hubs[h];
    const int first = c0[h];
    const int64_t end = r.beg + r.deg;
    for (int k = lane; r.beg + (int64_t)k * hub_chunk < end; k += 32) {
      const int64_t b = r.beg + (int64_t)k * hub_chunk;
      hub_of[first + k] = h;
      e0[first + k] = b;
      e1[first + k] = b + hub_chunk < end ? b + hub_chunk : end;
    }
  }
}

}  // namespace

void launch_bins(const LevelGraph &g, const int32_t *gid, const BinPlan &plan, const Bins &b, BinOut *out,
                 int32_t *counts, Scalars *sc, int coop, cudaStream_t s) {
  cudaMemsetAsync(out, 0, sizeof(BinOut), s);
  if (g.n <= 0) return;
  BinArgs a{};
  a.g = g;
  a.gid = gid;
  for (int k = 0; k < kBins - 1; ++k) a.max_deg[k] = (int32_t)plan.max_deg[k];
  a.hub_chunk = (int32_t)plan.hub_chunk;
  a.recs = b.recs;
  a.lists = b.lists;
  a.out = out;
  a.counts = counts;
  a.sc = sc;
  int64_t blocks = (g.n + kT - 1) / kT;
  if (blocks > coop_blocks(coop)) blocks = coop_blocks(coop);
  void *args[] = {&a};
  cudaLaunchCooperativeKernel((const void *)k_bins, dim3((unsigned)blocks), dim3(kT), args, 0, s);
}

void finish_bins(Bins &b, const BinOut &out) {
  for (int k = 0; k < kBins; ++k) {
    b.list[k] = b.lists + out.offs[k];
    b.rec[k] = b.recs + out.offs[k];
    b.count[k] = out.offs[k + 1] - out.offs[k];
  }
}

void launch_hub_plan(const Bins &b, const BinPlan &plan, const Hubs &hub, cudaStream_t s) {
  k_hub_plan<<<1, kT, 0, s>>>(b.rec[kHubBin], hub.H, (int32_t)plan.hub_chunk, const_cast<int32_t *>(hub.c0),
                             const_cast<int32_t *>(hub.hub_of), const_cast<int64_t *>(hub.e0),
                             const_cast<int64_t *>(hub.e1), hub.acc, hub.done);
}

}  // namespace lc
