// lc_bins.cu — the degree bins of a level (Section IV-C-2's buckets): the
// vertices of each bin in ascending order with their records, and the chunk
// plan of the hub bin.
#include "lc_bins_dev.cuh"

namespace lc {

namespace {

constexpr int kT = kCoopThreads, kW = kT / 32;

struct BinArgs {
  LevelGraph g;
  const int32_t *gid;  // graph of each vertex (nullptr: one graph)
  BinWork w;
  BinOut *out;
  Scalars *sc;
};

// One cooperative launch: every block counts the bins of its run of vertices,
// and once all have met, places them.  Bound by the records it writes: 52
// bytes a vertex, 16 of them read twice.  Ten scans of three launches and a
// separate pass for the records took 0.35 ms at 912,673 vertices and 70 us,
// all launches, on 10,000; this takes 30 us and 8 us.
__global__ void __launch_bounds__(kT, 1) k_bins(const __grid_constant__ BinArgs a) {
  const int64_t *__restrict__ rp = a.g.rp;
  GridBarrier bar(a.sc);
  bins_count<kT>(a.w, a.g.n, a.out, [&](int64_t v) { return row_degree(rp[v], rp[v + 1]); });
  if (!bar.sync()) return;
  bins_place<kT>(a.w, a.g.n, bin_run<kT>(a.g.n), gridDim.x, a.out, [&](int64_t v) {
    VRec r{};
    r.v = (int32_t)v;
    r.beg = rp[v];
    r.deg = row_degree(r.beg, rp[v + 1]);
    r.g = a.gid ? a.gid[v] : 0;
    r.w = a.g.vw[v];
    return r;
  });
  bar.leave(&a.out->done);
}

// The chunks of hub h, by `lanes` threads of rank `lane`.
__device__ __forceinline__ void cut_hub(const VRec &r, int h, int first, int32_t hub_chunk, int32_t *hub_of, int64_t *e0,
                                        int64_t *e1, int lane, int lanes) {
  const int64_t end = r.beg + r.deg;
  for (int k = lane; r.beg + (int64_t)k * hub_chunk < end; k += lanes) {
    const int64_t b = r.beg + (int64_t)k * hub_chunk;
    hub_of[first + k] = h;
    e0[first + k] = b;
    e1[first + k] = b + hub_chunk < end ? b + hub_chunk : end;
  }
}

// Cuts the hub rows into chunks of hub_chunk edges: c0[h] = the first chunk
// of hub h, and each chunk's hub and edges (up to kPlanHubs hubs; more are cut
// by k_hub_chunks, a thread each: with 100,000 hubs the one block took 0.48 ms).
// One block.
constexpr int kPlanHubs = 8192;
__global__ void __launch_bounds__(kT, 1)
    k_hub_plan(const VRec *__restrict__ hubs, int H, int32_t hub_chunk, int32_t *c0, int32_t *hub_of, int64_t *e0,
               int64_t *e1, long long *acc, int32_t *done) {
  __shared__ int32_t s_w[kW];
  __shared__ int32_t s_run;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_run = 0;
  for (int base = 0; base < H; base += kT) {
    const int h = base + threadIdx.x;
    const int c = h < H ? (int)(((int64_t)hubs[h].deg + hub_chunk - 1) / hub_chunk) : 0;
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
  if (H > kPlanHubs) return;
  for (int h = wid; h < H; h += kW) cut_hub(hubs[h], h, c0[h], hub_chunk, hub_of, e0, e1, lane, 32);  // by a warp
}
__global__ void __launch_bounds__(256) k_hub_chunks(const VRec *__restrict__ hubs, int H, int32_t hub_chunk,
                                                    const int32_t *__restrict__ c0, int32_t *hub_of, int64_t *e0,
                                                    int64_t *e1) {
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  if (h < H) cut_hub(hubs[h], h, c0[h], hub_chunk, hub_of, e0, e1, 0, 1);
}

}  // namespace

void launch_bins(const LevelGraph &g, const int32_t *gid, const BinPlan &plan, const Bins &b, BinOut *out,
                 int32_t *counts, Scalars *sc, int coop, cudaStream_t s) {
  cudaMemsetAsync(out, 0, sizeof(BinOut), s);
  if (g.n <= 0) return;
  BinArgs a{};
  a.g = g;
  a.gid = gid;
  a.w = bin_work(plan, b, counts);
  a.out = out;
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

int launch_hub_plan(const Bins &b, const BinPlan &plan, const Hubs &hub, cudaStream_t s) {
  const VRec *hubs = b.rec[kHubBin];
  const int32_t chunk = (int32_t)plan.hub_chunk;
  int32_t *c0 = const_cast<int32_t *>(hub.c0), *hub_of = const_cast<int32_t *>(hub.hub_of);
  int64_t *e0 = const_cast<int64_t *>(hub.e0), *e1 = const_cast<int64_t *>(hub.e1);
  k_hub_plan<<<1, kT, 0, s>>>(hubs, hub.H, chunk, c0, hub_of, e0, e1, hub.acc, hub.done);
  if (hub.H <= kPlanHubs) return 1;
  k_hub_chunks<<<(unsigned)((hub.H + 255) / 256), 256, 0, s>>>(hubs, hub.H, chunk, c0, hub_of, e0, e1);
  return 2;
}

}  // namespace lc
