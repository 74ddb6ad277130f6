// lc_level.cu — the end of a small coarsening level in a cooperative kernel and
// a plain one: label compaction and Algorithm 4's contraction (and the bins of the
// next level), which as separate launches (marks, three scans of three
// launches each, bounds, six insert kernels, a compaction, two read-backs)
// took 28 launches of 2-4 us and two more waits of the host, whatever the
// level's size: a call on an SBM of 10,000 vertices, four such level ends,
// went from 2.14 to 1.60 ms, and with the bins, one scan by label and two
// barriers less from 1.48 to 1.40.  Bound by seven grid barriers on small
// levels, by the inserts' probes on the largest.  The method is
// lc_contract.cu's: coarse vertex x owns 2 bound[x] slots of the global hash
// scratch, every fine edge that leaves its cluster is inserted there, and
// the occupied slots in order are the coarse rows.
#include "lc_bins_dev.cuh"
#include "lc_compact_dev.cuh"
#include "lc_coop.cuh"
#include "lc_group.cuh"
#include "lc_level.cuh"
#include "lc_move.cuh"

namespace lc {

namespace {

constexpr int kT = 512, kW = kT / 32;
static_assert(kLevelWarps == kW, "one count per warp");

struct EndArgs {
  LevelGraph g;
  const int32_t *gid;
  const GraphParam *gp;
  int32_t G;
  const VRec *rec;
  int64_t off[kBins + 1];
  Hubs hub;
  int32_t max_deg[kBins - 1];
  int32_t hub_chunk;
  const int32_t *C;
  int32_t *Cd;
  LevelScratch w;
  LevelOut *out;
  int32_t *bin_counts;  // [kBins][blocks]
  Scalars *sc;
};

// Exclusive scan over the grid of in(i), i < n: out(i, prefix, value); the
// total to every thread.  Each warp takes a run of its own, a block's warps
// one after the other.  False if a barrier ran out.
__device__ __forceinline__ int64_t warp_run(int64_t n, int blocks) {
  const int nw = blocks * kW;
  return ((n + nw - 1) / nw + 31) / 32 * 32;
}
template <typename In, typename Out>
__device__ __forceinline__ bool grid_scan(int64_t n, long long *counts, GridBarrier &bar, In in, Out out,
                                          long long &total) {
  __shared__ long long red[kW], red_all[kW];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = gridDim.x * kW, me = blockIdx.x * kW + wid;
  const int64_t per = warp_run(n, gridDim.x);
  const int64_t lo = (int64_t)me * per, hi = lo + per < n ? lo + per : n;
  long long mine = 0;
  for (int64_t i = lo + lane; i < hi; i += 32) mine += in(i);
  mine = warp_sum(mine);
  if (lane == 0) counts[me] = mine;
  if (!bar.sync()) return false;
  long long before = 0, all = 0;
  for (int k = threadIdx.x; k < nw; k += kT) {
    const long long c = counts[k];
    all += c;
    before += k < blockIdx.x * kW ? c : 0;
  }
  before = warp_sum(before);
  all = warp_sum(all);
  if (lane == 0) {
    red[wid] = before;
    red_all[wid] = all;
  }
  __syncthreads();
  before = all = 0;
  for (int k = 0; k < kW; ++k) {
    before += red[k];
    all += red_all[k];
  }
  for (int k = 0; k < wid; ++k) before += counts[blockIdx.x * kW + k];
  total = all;
  __syncthreads();
  for (int64_t base = lo; base < hi; base += 32) {
    const int64_t i = base + lane;
    const long long x = i < hi ? in(i) : 0;
    long long incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += y;
    }
    if (i < hi) out(i, before + incl - x, x);
    before += __shfl_sync(0xFFFFFFFFu, incl, 31);
  }
  return true;
}

// Inserts edges [beg + r, end) (stride GS) of a vertex of coarse id x;
// returns the slots claimed.
template <int GS>
__device__ __forceinline__ int insert_row(const EndArgs &a, int32_t x, int64_t beg, int64_t end, int r, bool &ok) {
  constexpr int U = 4;
  const int64_t o0 = a.w.off[x];
  const uint32_t cap = (uint32_t)(2 * (a.w.off[x + 1] - o0));
  unsigned long long *tab = a.w.tab + 2 * o0;
  int fresh_n = 0;
  for (int64_t base = beg + r; base < end; base += (int64_t)GS * U) {
    int32_t u[U], w[U], y[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int64_t e = base + (int64_t)k * GS;
      u[k] = -1;
      w[k] = 0;
      if (e < end) {
        u[k] = LC_IDX(__ldg(a.g.col + e), a.g.n, kDbgColumn);
        w[k] = __ldg(a.g.ew + e);
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) y[k] = u[k] >= 0 ? LC_IDX(a.Cd[u[k]], a.g.n, kDbgCoarse) : x;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (y[k] == x) continue;
      bool fresh = false;
      ok &= table_add(tab, cap, y[k], w[k], fresh);
      fresh_n += fresh;
    }
  }
  return fresh_n;
}

// The rows of records [lo, hi) by GS lanes each.
template <int GS>
__device__ __forceinline__ void insert_group(const EndArgs &a, int64_t lo, int64_t hi, bool &ok) {
  constexpr int V = 32 / GS;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, sub = lane & (GS - 1);
  const int64_t nw = (int64_t)gridDim.x * kW;
  for (int64_t i0 = lo + ((int64_t)wid * gridDim.x + blockIdx.x) * V; i0 < hi; i0 += nw * V) {
    const int64_t i = i0 + lane / GS;
    int32_t x = -1;
    int f = 0;
    if (i < hi) {
      const VRec vr = a.rec[i];
      x = a.Cd[vr.v];
      if (x >= 0) f = insert_row<GS>(a, x, vr.beg, vr.beg + vr.deg, sub, ok);
    }
    __syncwarp();
    f = group_sum<GS>(f);
    if (sub == 0 && f) atomicAdd(&a.w.cnt[x], f);
  }
}

__global__ void __launch_bounds__(kT, 1) k_level_end(const __grid_constant__ EndArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t n = a.g.n;
  const int64_t tid = (int64_t)blockIdx.x * kT + threadIdx.x, nt = (int64_t)gridDim.x * kT;
  const int64_t wbase = tid - lane;
  GridBarrier bar(a.sc);
  for (int64_t x = tid; x < n; x += nt) {
    a.w.used[x] = 0;
    a.w.cnt[x] = 0;
    a.w.bound[x] = 0;
    a.w.label_w[x] = 0;
  }
  for (int64_t g = tid; g < a.G; g += nt) a.w.nc[g] = 0;
  if (!bar.sync()) return;
  // labels in use, their edge bounds and weights
  for (int64_t v0 = wbase; v0 < n; v0 += nt) {
    const int64_t v = v0 + lane;
    const bool on = v < n;
    const int32_t X = on ? LC_IDX(a.C[v], n, kDbgLabel) : 0;
    if (on) a.w.used[X] = 1;
    add_weights(a.w.bound, on, X, on ? a.g.rp[v + 1] - a.g.rp[v] : 0);
    add_weights(a.w.label_w, on, X, on ? a.g.vw[v] : 0);
  }
  if (!bar.sync()) return;
  if (a.gid) {  // labels in use per graph, which tell the graphs that go on
    for (int64_t x0 = wbase; x0 < n; x0 += nt) {
      const int64_t x = x0 + lane;
      const int g = x < n && a.w.used[x] ? a.gid[x] : -1;
      const unsigned on = __ballot_sync(0xFFFFFFFFu, g >= 0);
      if (!on) continue;
      const int g0 = __shfl_sync(0xFFFFFFFFu, g, __ffs(on) - 1);
      if (__all_sync(0xFFFFFFFFu, g < 0 || g == g0)) {
        if (lane == 0) atomicAdd(&a.w.nc[g0], __popc(on));
      } else if (g >= 0) {
        atomicAdd(&a.w.nc[g], 1);
      }
    }
    if (!bar.sync()) return;
  }
  // dense ids, ascending, of the labels of the graphs that go on, and where
  // their slots start: one scan of (edge bound, 1), both below 2^31 here
  auto goes_on = [&](int64_t x) {
    const int g = a.gid ? a.gid[x] : 0;
    return !a.gid || a.w.nc[g] < a.gp[g].nv;
  };
  long long all = 0;
  if (!grid_scan(
          n, a.w.counts, bar,
          [&](int64_t x) -> long long { return a.w.used[x] && goes_on(x) ? (a.w.bound[x] << 32) | 1 : 0; },
          [&](int64_t x, long long at, long long here) {
            if (!here) return;
            const int32_t id = (int32_t)at;
            a.w.newid[x] = id;
            a.w.off[id] = at >> 32;
            a.w.vw[id] = a.w.label_w[x];
            if (a.gid) a.w.gid[id] = a.gid[x];  // a label is a vertex of its graph
          },
          all))
    return;
  long long n_c = all & 0xFFFFFFFFll;
  if (!a.gid && n_c == n) n_c = 0;  // nothing merges
  if (tid == 0) {
    a.out->n_c = n_c;
    a.w.off[n_c] = all >> 32;
  }
  if (n_c == 0) {  // uniform: the host reads no more than this
    bar.leave(&a.out->bins.done);
    return;
  }
  if (!bar.sync()) return;
  for (int64_t v = tid; v < n; v += nt) a.Cd[v] = goes_on(v) ? a.w.newid[a.C[v]] : -1;
  if (!bar.sync()) return;
  // insert: the chunks of bin 9 and the rows of bins 7-8 by a block, 3-6 by a warp, 1-2 by eight lanes, bin 0 by a thread
  bool ok = true;
  {
    __shared__ int s_fresh;
    // hub rows by their chunks: with all blocks at one row after the other, the
    // rows of a few thousand edges kept two of them busy
    for (int c = blockIdx.x; c < a.hub.Q; c += gridDim.x) {
      const int32_t x = a.Cd[a.hub.vtx[a.hub.hub_of[c]]];
      if (x < 0) continue;
      int f = insert_row<kT>(a, x, a.hub.e0[c], a.hub.e1[c], threadIdx.x, ok);
      f = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)f);
      if (lane == 0 && f) atomicAdd(&a.w.cnt[x], f);
    }
    for (int64_t i = a.off[7] + blockIdx.x; i < a.off[kHubBin]; i += gridDim.x) {
      const VRec vr = a.rec[i];
      const int32_t x = a.Cd[vr.v];
      if (x < 0) continue;  // block-uniform
      __syncthreads();
      if (threadIdx.x == 0) s_fresh = 0;
      __syncthreads();
      const int f = (int)__reduce_add_sync(
          0xFFFFFFFFu, (unsigned)insert_row<kT>(a, x, vr.beg, vr.beg + vr.deg, threadIdx.x, ok));
      if (lane == 0 && f) atomicAdd(&s_fresh, f);
      __syncthreads();
      if (threadIdx.x == 0 && s_fresh) atomicAdd(&a.w.cnt[x], s_fresh);
    }
    // short rows by eight lanes, four edges each in flight: the walk is bound
    // by the latency of its gathers and probes
    insert_group<32>(a, a.off[3], a.off[7], ok);
    insert_group<8>(a, a.off[1], a.off[3], ok);
    for (int64_t i = a.off[0] + tid; i < a.off[1]; i += nt) {
      const VRec vr = a.rec[i];
      const int32_t x = a.Cd[vr.v];
      if (x < 0) continue;
      const int f = insert_row<1>(a, x, vr.beg, vr.beg + vr.deg, 0, ok);
      if (f) atomicAdd(&a.w.cnt[x], f);
    }
  }
  if (!ok) a.sc->error = 1;
  if (!bar.sync()) return;
  // coarse row offsets, and the sizes of the coarse bins
  __shared__ int s_bin[kBins], s_max;
  __shared__ long long s_chunks;
  if (threadIdx.x < kBins) s_bin[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    s_max = 0;
    s_chunks = 0;
  }
  __syncthreads();
  long long nnz_c = 0;
  if (!grid_scan(
          n_c, a.w.counts, bar, [&](int64_t x) -> long long { return a.w.cnt[x]; },
          [&](int64_t x, long long at, long long deg) {
            a.w.rp[x] = at;
            const int b = bin_of(a.max_deg, (int32_t)deg);
            atomicAdd(&s_bin[b], 1);
            if (b == kHubBin) {
              atomicMax(&s_max, (int)deg);
              atomicAdd((unsigned long long *)&s_chunks,
                        (unsigned long long)((deg + a.hub_chunk - 1) / a.hub_chunk));
            }
          },
          nnz_c))
    return;
  __syncthreads();
  // the block's run for k_level_build; offs[k + 1] counts bin k here, the host sums
  if (threadIdx.x < kBins) a.bin_counts[threadIdx.x * gridDim.x + blockIdx.x] = s_bin[threadIdx.x];
  if (threadIdx.x < kBins && s_bin[threadIdx.x]) atomicAdd(&a.out->bins.offs[threadIdx.x + 1], s_bin[threadIdx.x]);
  if (threadIdx.x == 0 && s_max > 0) {
    atomicMax(&a.out->bins.max_deg, s_max);
    atomicAdd((unsigned long long *)&a.out->bins.chunks, (unsigned long long)s_chunks);
  }
  if (tid == 0) {
    a.out->nnz_c = nnz_c;
    a.w.rp[n_c] = nnz_c;
  }
  bar.leave(&a.out->bins.done);
}

struct BuildArgs {
  CompactArgs slots;
  LevelScratch w;
  int64_t *rp_c, *vw_c;
  int32_t *gid_c;
  BinWork bins;
};

// The coarse graph into its own arrays, and its bins (counted by k_level_end
// over runs of half as many blocks): the first half of the blocks takes the
// vertices, the other the edges.  A plain kernel: what follows reads the
// coarse graph before the host looks at the error flag, so it may not stop
// half way, as a cooperative kernel's wait can.  All levels of an SBM of 10,000
// vertices: 51 us as one cooperative kernel with a scan over the slots, 65 us
// with all blocks at the edges and then the vertices, 31 us like this.
__global__ void __launch_bounds__(kT, 2) k_level_build(const __grid_constant__ BuildArgs a) {
  const int64_t n_c = a.slots.n_c;
  const int blocks = gridDim.x / 2, me = (int)blockIdx.x - blocks;
  if (me >= 0) {
    // short runs where there are warps for them: a run's 256 slots a step are a chain
    const int64_t used = 2 * a.w.off[n_c], nw = (int64_t)blocks * kW;
    int64_t run = (used + 256 * nw - 1) / (256 * nw) * 256;
    run = run > kCompactRun ? kCompactRun : run;
    for (int64_t s = ((int64_t)(threadIdx.x >> 5) * blocks + me) * run; s < used; s += nw * run)
      compact_run(a.slots, s, run, used);
    return;
  }
  for (int64_t x = (int64_t)blockIdx.x * kT + threadIdx.x; x <= n_c; x += (int64_t)blocks * kT) {
    a.rp_c[x] = a.w.rp[x];
    if (x == n_c) break;
    a.vw_c[x] = a.w.vw[x];
    if (a.gid_c) a.gid_c[x] = a.w.gid[x];
  }
  const int64_t per = warp_run(n_c, blocks) * kW, lo = blockIdx.x * per;
  bins_place<kT>(a.bins, n_c, BinRun{lo, lo + per < n_c ? lo + per : n_c}, blocks, nullptr, [&](int64_t x) {
    VRec r{};
    r.v = (int32_t)x;
    r.beg = a.w.rp[x];
    r.deg = row_degree(r.beg, a.w.rp[x + 1]);
    r.g = a.gid_c ? a.w.gid[x] : 0;
    r.w = a.w.vw[x];
    return r;
  });
}

unsigned level_blocks(int64_t n, int64_t nnz, int coop) {
  const int64_t blocks = level_grid(n, nnz), most = coop_blocks(coop);
  return (unsigned)(blocks < most ? blocks : most);
}

}  // namespace

void launch_level_end(const LevelGraph &g, const int32_t *gid, const GraphParam *gp, int G, const Bins &b,
                      const Hubs &hub, const BinPlan &plan, const int32_t *C, int32_t *Cd, const LevelScratch &w, LevelOut *out,
                      int32_t *bin_counts, Scalars *sc, int coop, cudaStream_t s) {
  cudaMemsetAsync(out, 0, sizeof(LevelOut), s);
  EndArgs a{};
  a.g = g;
  a.gid = gid;
  a.gp = gp;
  a.G = G;
  a.rec = b.recs;
  for (int k = 0; k < kBins; ++k) a.off[k] = b.list[k] - b.list[0];
  a.off[kBins] = g.n;
  a.hub = hub;
  for (int k = 0; k < kBins - 1; ++k) a.max_deg[k] = (int32_t)plan.max_deg[k];
  a.hub_chunk = (int32_t)plan.hub_chunk;
  a.C = C;
  a.Cd = Cd;
  a.w = w;
  a.out = out;
  a.bin_counts = bin_counts;
  a.sc = sc;
  void *args[] = {&a};
  cudaLaunchCooperativeKernel((const void *)k_level_end, dim3(level_blocks(g.n, g.nnz, coop)), dim3(kT), args, 0, s);
}

void launch_level_build(const LevelGraph &g, const LevelScratch &w, const LevelOut &out, int64_t *rp_c, int32_t *col_c,
                        int32_t *ew_c, int64_t *vw_c, int32_t *gid_c, const BinWork &bins, int coop, cudaStream_t s) {
  const CompactArgs slots{w.tab, w.off, w.rp, w.cnt, out.n_c, col_c, ew_c};
  k_level_build<<<2 * level_blocks(g.n, g.nnz, coop), kT, 0, s>>>(BuildArgs{slots, w, rp_c, vw_c, gid_c, bins});
}

}  // namespace lc
