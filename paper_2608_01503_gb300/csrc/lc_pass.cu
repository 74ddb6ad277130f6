// lc_pass.cu — kernels of one synchronous local-move pass (Algorithm 2 with
// the afterburner filter of Algorithm 3) and the per-level objective.
//
// Every vertex is handled by a thread group sized to its degree bin (see
// kBinMaxDeg in lc_internal.cuh).  The kernels are bound by the latency of
// dependent gathers (row offsets -> neighbours -> their clusters -> cluster
// weights), so each group issues its loads in batches before using them, and
// the bins keep many vertices in flight per SM.  Rows above 4096 entries
// ("hubs") are cut into chunks processed by independent blocks.
//
// All sums are integer (commutative atomics and shuffles), argmax ties go to
// the smallest cluster id and the afterburner order is a total order, so the
// results do not depend on scheduling.
#include <algorithm>
#include <climits>

#include "lc_coop.cuh"
#include "lc_empty.cuh"
#include "lc_group.cuh"
#include "lc_internal.cuh"
#include "lc_move.cuh"
#include "lc_pass.cuh"
#include "lc_scan.cuh"
#include "lc_step.cuh"

namespace lc {

// Kept tables: writes (X, S) into a table that only the calling thread
// touches (plain loads and stores; X is not in the table yet).  False if
// the table is full.
__device__ __forceinline__ bool tab_put(unsigned long long *t, uint32_t cap, int32_t X, long long S) {
  uint32_t s = slot_of(X, cap);
  for (uint32_t probe = 0; probe < cap; ++probe) {
    if (t[s] == kEmptySlot) {
      t[s] = ((unsigned long long)((uint32_t)X + 1u) << 32) | (uint32_t)S;
      return true;
    }
    s = (s + 1 == cap) ? 0 : s + 1;
  }
  return false;
}

// ------------------------------------------- move step, bins 0-8

// Chunks of vertices per warp: base = warp * chunk, one chunk each.
struct WarpChunk {
  int64_t base;
  int m;
};
__device__ __forceinline__ WarpChunk warp_chunk_of(int64_t count, int chunk) {
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t base = warp * chunk;
  const int64_t left = count - base;
  return WarpChunk{base, left <= 0 ? 0 : left < chunk ? (int)left : chunk};
}

// First pass, bins 0-4: a thread, 16 lanes or a warp per vertex.
template <int G>
__global__ void __launch_bounds__(256) k_first_pass(PassArgs a, const VRec *__restrict__ rec, int64_t count,
                                                    int chunk) {
  step_begin();
  __shared__ MoveStage st[8];
  MoveState ms = move_state(a);
  const WarpChunk c = warp_chunk_of(count, chunk);
  if (c.m > 0) first_chunk<G>(a, rec, c.base, c.m, st[threadIdx.x >> 5], ms);
  flush_block_sum(ms.cntL, &a.sc->count_L);
  step_end();
}

__global__ void __launch_bounds__(256) k_first_thread(PassArgs a, const VRec *__restrict__ rec, int64_t count) {
  step_begin();
  MoveState ms = move_state(a);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x)
    first_thread(a, rec, i, ms);
  flush_block_sum(ms.cntL, &a.sc->count_L);
  step_end();
}

__global__ void __launch_bounds__(256, 4) k_move_thread(PassArgs a, const VRec *__restrict__ rec, int64_t count) {
  step_begin();
  MoveState ms = move_state(a);
  // warp-uniform trip count: phi_add takes whole warps
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < count; base += (int64_t)gridDim.x * blockDim.x)
    move_thread(a, base + threadIdx.x < count, rec, base + threadIdx.x, ms);
  flush_move(a, ms);
  step_end();
}

template <int G>
__global__ void __launch_bounds__(256) k_move_lanes(PassArgs a, const VRec *__restrict__ rec, int64_t count,
                                                    int chunk) {
  step_begin();
  __shared__ MoveStage st[8];
  __shared__ LaneTags tags[8];
  MoveState ms = move_state(a);
  const WarpChunk c = warp_chunk_of(count, chunk);
  if (c.m > 0) lanes_chunk<G>(a, rec, c.base, c.m, st[threadIdx.x >> 5], tags[threadIdx.x >> 5], ms);
  flush_move(a, ms);
  step_end();
}

// Bins 3-4: one warp per vertex, a per-warp split shared table of kWarpSlots
// slots.
constexpr int kWarpSlots = 512;
__global__ void __launch_bounds__(kWarpBinWarps * 32, 4)
    k_move_warp(PassArgs a, const VRec *__restrict__ rec, int64_t count, int chunk) {
  step_begin();
  __shared__ uint32_t keys[kWarpBinWarps][kWarpSlots];
  __shared__ int32_t vals[kWarpBinWarps][kWarpSlots];
  __shared__ MoveStage st[kWarpBinWarps];
  MoveState ms = move_state(a);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const SplitTab tab{keys[wid], vals[wid]};
  const WarpChunk c = warp_chunk_of(count, chunk);
  if (c.m > 0) {
    for (int s = lane; s < kWarpSlots; s += 32) {
      tab.key[s] = 0u;
      tab.val[s] = 0;
    }
    __syncwarp();
    warp_chunk(a, rec, c.base, c.m, st[wid], tab, kWarpSlots, ms);
  }
  flush_move(a, ms);
  step_end();
}

// A block's chunk of vertices, staged and decided by its first warp.
struct BlockChunk {
  int64_t base;
  int m;
};
__device__ __forceinline__ BlockChunk block_chunk_of(int64_t count, int chunk) {
  const int64_t base = (int64_t)blockIdx.x * chunk;
  const int64_t left = count - base;
  return BlockChunk{base, left <= 0 ? 0 : left < chunk ? (int)left : chunk};
}

// First pass, bins 5-8: one block per vertex.
template <int GS>
__global__ void __launch_bounds__(GS) k_first_block(PassArgs a, const VRec *__restrict__ rec, int64_t count,
                                                    int chunk) {
  step_begin();
  __shared__ MoveStage st;
  __shared__ long long rg[GS / 32];
  __shared__ int32_t rx[GS / 32];
  MoveState ms = move_state(a);
  const BlockChunk b = block_chunk_of(count, chunk);
  ChunkLane c{};
  if (threadIdx.x < 32) c = stage_move(a, rec, b.base, b.m, threadIdx.x, true, st.ctx);
  __syncthreads();
  for (int k = 0; k < b.m; ++k) {
    const MoveCtx x = st.ctx[k];
    long long gb = LLONG_MIN;
    int32_t xb = kNone;
#pragma unroll 4
    for (int64_t e = x.beg + threadIdx.x; e < x.beg + x.deg; e += GS) first_edge(a, x.Lam, x.muw, e, gb, xb);
    Grp<GS>::argmax(gb, xb, rg, rx);
    if (threadIdx.x == 0) st.res[k] = MoveRes{gb, xb, 0};
  }
  __syncthreads();
  if (threadIdx.x < 32) settle_move(a, c, b.m, threadIdx.x, true, st.res, ms);
  flush_block_sum(ms.cntL, &a.sc->count_L);
  step_end();
}

// Bins 5-8: one block per vertex; dynamic shared memory holds the split
// table (SLOTS keys, then SLOTS values): bin 8 (deg <= 4096) has 6144 slots,
// a load factor of at most 2/3, so that four blocks fit in an SM's shared
// memory.  N: edges per thread of the bin's longest row.
// BUILD: the tables use the kept-table layout (tab_cap slots), are scanned,
// and copied out to each vertex's gtab region with S(v, C[v]) added.
template <int GS, int SLOTS, int N, bool BUILD>
__global__ void __launch_bounds__(GS) k_move_block(PassArgs a, const VRec *__restrict__ rec,
                                                   int64_t count, int chunk) {
  step_begin();
  extern __shared__ uint32_t smem_tab[];
  const SplitTab tab{smem_tab, reinterpret_cast<int32_t *>(smem_tab + SLOTS)};
  __shared__ MoveStage st;
  // per-warp partials, double-buffered by vertex parity: thread 0 combines
  // vertex k's while the other threads already insert vertex k + 1, and the
  // buffer is written again only after two more barriers (vertex k + 2)
  __shared__ long long rg[2][GS / 32];
  __shared__ int32_t rx[2][GS / 32], rs[2][GS / 32];
  int par = 0;
  MoveState ms = move_state(a);
  const BlockChunk b = block_chunk_of(count, chunk);
  ChunkLane c{};
  if (threadIdx.x < 32) c = stage_move(a, rec, b.base, b.m, threadIdx.x, false, st.ctx);
  for (int s = threadIdx.x; s < SLOTS; s += GS) {
    tab.key[s] = 0u;
    tab.val[s] = 0;
  }
  __syncthreads();
  for (int k = 0; k < b.m; ++k) {
    const MoveCtx x = st.ctx[k];
    const uint32_t cap = BUILD ? tab_cap(x.deg) : (uint32_t)SLOTS;
    bool ok = true;
    int32_t self, slot[N];
    if constexpr (BUILD)
      self = (int32_t)split_insert_row<GS, 4>(a, x.beg, x.beg + x.deg, x.Cv, tab, cap, threadIdx.x, ok);
    else
      self = claim_row<GS, N>(a, x.beg, x.deg, x.Cv, tab, cap, threadIdx.x, slot, ok);
    if (!ok) {
      a.sc->error = 1;
      LC_DBG_FAIL(kDbgProbe, b.base + k, a.g.n);
    }
    __syncthreads();
    long long gb = LLONG_MIN;
    int32_t xb = kNone;
    unsigned long long *gt = a.gtab + 2 * x.beg;
    if constexpr (BUILD)
      split_argmax<GS>(a, x.Lam, x.muw, tab, cap, threadIdx.x, gb, xb, gt, ms.nX);
    else
      claim_argmax<N>(a, x.Lam, x.muw, tab, slot, gb, xb, ms.nX);
    // one reduction of (best gain, cluster, S_self) for thread 0 only: warp
    // level, one barrier, thread 0 combines the warps
    warp_argmax(gb, xb);
    self = (int32_t)__reduce_add_sync(0xFFFFFFFFu, (unsigned)self);
    if ((threadIdx.x & 31) == 0) {
      rg[par][threadIdx.x >> 5] = gb;
      rx[par][threadIdx.x >> 5] = xb;
      rs[par][threadIdx.x >> 5] = self;
    }
    // the table is read and reset by every thread past this barrier, so the
    // next vertex may start inserting at once
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < GS / 32; ++w) {
        self += rs[par][w];
        if (better(rg[par][w], rx[par][w], gb, xb)) {
          gb = rg[par][w];
          xb = rx[par][w];
        }
      }
      // the barrier above made every thread's copied slots visible
      if (BUILD && self > 0 && !tab_put(gt, cap, x.Cv, self)) a.sc->error = 1;
      st.res[k] = MoveRes{gb, xb, self};
    }
    par ^= 1;
  }
  __syncthreads();
  if (threadIdx.x < 32) settle_move(a, c, b.m, threadIdx.x, false, st.res, ms);
  flush_move(a, ms);
  step_end();
}

// --------------------------------------------------------- hubs (bin 9)

// Block-wide argmax of (g, x) into the chunk partials.
__device__ __forceinline__ void hub_part_store(const PassArgs &a, int c, long long gb, int32_t xb) {
  __shared__ long long rg[kHubThreads / 32];
  __shared__ int32_t rx[kHubThreads / 32];
  Grp<kHubThreads>::argmax(gb, xb, rg, rx);
  if (threadIdx.x == 0) {
    a.hub.part_g[c] = gb;
    a.hub.part_x[c] = xb;
  }
}

__device__ __forceinline__ void hub_acc_add(const PassArgs &a, int h, long long x) {
  __shared__ long long rs[kHubThreads / 32];
  x = Grp<kHubThreads>::sum(x, rs);
  if (threadIdx.x == 0 && x != 0) atomicAdd((unsigned long long *)&a.hub.acc[h], (unsigned long long)x);
}

// Hubs of one chunk are settled by a lane each in a kernel after the step, if
// the bin plan can have any (hub_chunk above the longest row of bin 8): a block
// to itself, a short row's decision is a chain of loads that nothing hides
// (ms a call, SBM of 100,000 vertices with every row above 8 edges a hub, block
// / lane: 29.1 / 22.5, 2.4 of them by k_hub_chunks).  Longer hubs are decided by their last chunk.
__device__ __forceinline__ bool left_to_settle(const PassArgs &a, int h) {
  return a.hub.settle && a.hub.c0[h + 1] - a.hub.c0[h] == 1;
}

__global__ void __launch_bounds__(256) k_hub_settle(PassArgs a, int first) {
  MoveState ms = move_state(a);
  for (int base = blockIdx.x * blockDim.x; base < a.hub.H; base += gridDim.x * blockDim.x) {
    const int h = base + threadIdx.x;
    const bool on = h < a.hub.H && left_to_settle(a, h);
    int g = 0;
    long long gC = 0;
    if (on) {
      const int32_t v = a.hub.vtx[h], c = a.hub.c0[h];
      g = graph_of(a, v);
      const GraphParam P = a.gp[g];
      const int32_t Cv = a.C[v];
      if (!first) {
        gC = gain_self(P, a.hub.acc[h], a.g.vw[v], a.W[Cv]);
        a.hub.acc[h] = 0;
      }
      decide(a, P, v, Cv, gC, a.hub.part_x[c], a.hub.part_g[c], ms);
    }
    if (!first) phi_add(a, ms.acc, on, g, gC, ms.phi);
  }
  if (first)
    flush_block_sum(ms.cntL, &a.sc->count_L);
  else
    flush_move(a, ms);
}

// The update of the same hubs from their chunk's sum.
__global__ void __launch_bounds__(256) k_hub_settle_update(PassArgs a) {
  UpdateSums sum;
  for (int base = blockIdx.x * blockDim.x; base < a.hub.H; base += gridDim.x * blockDim.x) {
    const int h = base + threadIdx.x;
    const bool on = h < a.hub.H && left_to_settle(a, h);
    int32_t v = 0;
    AbRec r{0, kNone, 0};
    int64_t deg = 0;
    bool keep = false;
    if (on) {
      v = a.hub.vtx[h];
      r = a.ab[v];
      deg = a.g.rp[v + 1] - a.g.rp[v];
      if (r.D != kNone) {
        keep = a.delta[v] + a.hub.acc[h] >= 0;
        a.hub.acc[h] = 0;
      }
    }
    apply_lanes(a, on, v, deg, r, on ? a.g.vw[v] : 0, keep, sum);
  }
  flush_update(a, sum);
}

// Move, step 1: insert a chunk of a hub row into the hub's global table.
// Lanes of a warp holding the same cluster are combined first (lane_sums),
// so a popular cluster costs one global atomic per warp.
__global__ void __launch_bounds__(kHubThreads) k_hub_move_insert(PassArgs a) {
  step_begin();
  __shared__ LaneTags tags[kHubThreads / 32];
  const int c = blockIdx.x, h = a.hub.hub_of[c];
  const long long self =
      hub_insert<kHubThreads>(a, a.hub.vtx[h], a.hub.e0[c], a.hub.e1[c], tags[threadIdx.x >> 5]);
  hub_acc_add(a, h, self);
  step_end();
}

// Move, step 2: argmax over the chunk's share of the hub table (reset as
// read, or kept as the hub's kept table with a.tab_build).
__global__ void __launch_bounds__(kHubThreads) k_hub_move_scan(PassArgs a) {
  const int c = blockIdx.x;
  const int h = a.hub.hub_of[c];
  const int32_t v = a.hub.vtx[h];
  const int64_t beg = a.g.rp[v];
  const long long wv = a.g.vw[v];
  const GraphParam P = a.gp[graph_of(a, v)];
  MoveState ms = move_state(a);
  long long gb = LLONG_MIN;
  int32_t xb = kNone;
  range_argmax<kHubThreads>(a, P.Lam, P.mu * wv, a.gtab + 2 * beg, (uint32_t)(2 * (a.hub.e0[c] - beg)),
                            (uint32_t)(2 * (a.hub.e1[c] - beg)), threadIdx.x, gb, xb, ms.nX, a.tab_build != 0);
  hub_part_store(a, c, gb, xb);
  if (!left_to_settle(a, h) && last_of_hub(a, h) && threadIdx.x < 32) {
    const long long self = decide_hub(a, h, v, false, threadIdx.x, ms);
    // the hub's kept table gets its own cluster
    if (a.tab_build && self > 0 && !tab_put(a.gtab + 2 * beg, tab_cap(a.g.rp[v + 1] - beg), a.C[v], self))
      a.sc->error = 1;
  }
  flush_move(a, ms);
}

// First pass: argmax over a chunk of a hub row.
__global__ void __launch_bounds__(kHubThreads) k_hub_first(PassArgs a) {
  step_begin();
  const int c = blockIdx.x, h = a.hub.hub_of[c];
  const int32_t v = a.hub.vtx[h];
  const long long wv = a.g.vw[v];
  const GraphParam P = a.gp[graph_of(a, v)];
  MoveState ms = move_state(a);
  long long gb = LLONG_MIN;
  int32_t xb = kNone;
#pragma unroll 4
  for (int64_t e = a.hub.e0[c] + threadIdx.x; e < a.hub.e1[c]; e += kHubThreads)
    first_edge(a, P.Lam, P.mu * wv, e, gb, xb);
  hub_part_store(a, c, gb, xb);
  if (!left_to_settle(a, h) && last_of_hub(a, h) && threadIdx.x < 32) decide_hub(a, h, v, true, threadIdx.x, ms);
  flush_block_sum(ms.cntL, &a.sc->count_L);
  step_end();
}

// ------------------------------------------------ afterburner (Algorithm 3)

// Bin 0: a thread per vertex.
__global__ void __launch_bounds__(256, 4) k_ab_thread(PassArgs a, const VRec *__restrict__ rec, int64_t count) {
  step_begin();
  UpdateSums sum;
  // warp-uniform trip count: the update's lists are appended per warp
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < count; base += (int64_t)gridDim.x * blockDim.x)
    ab_thread<8>(a, base + threadIdx.x < count, rec, base + threadIdx.x, sum);
  flush_update(a, sum);
  step_end();
}

// 4, 8 or 16 lanes or a warp per candidate, a chunk of vertices per warp.
template <int G>
__global__ void __launch_bounds__(256, 4) k_ab_warp(PassArgs a, const VRec *__restrict__ rec, int64_t count,
                                                    int chunk) {
  step_begin();
  __shared__ AbStage st[8];
  UpdateSums sum;
  const WarpChunk c = warp_chunk_of(count, chunk);
  if (c.m > 0) ab_chunk<G>(a, rec, c.base, c.m, st[threadIdx.x >> 5], sum);
  flush_update(a, sum);
  step_end();
}

// A block per candidate, a chunk of vertices per block.  Every warp walks its
// part of all the chunk's candidates and leaves its sums, so the warps meet
// twice a chunk and not once a candidate (half of their time, before).
template <int GS>
__global__ void __launch_bounds__(GS, 2048 / GS / 2) k_ab_block(PassArgs a, const VRec *__restrict__ rec,
                                                                int64_t count, int chunk) {
  step_begin();
  __shared__ AbStage st;
  __shared__ long long rs[32][GS / 32];
  __shared__ int s_nc;
  UpdateSums sum;
  const BlockChunk b = block_chunk_of(count, chunk);
  VRec vr{};
  AbRec r{0, kNone, 0};
  long long delta = 0;
  int pos = 0;
  if (threadIdx.x < 32) {
    const int n = stage_ab(a, rec, b.base, b.m, threadIdx.x, st.ctx, vr, r, delta, pos);
    if (threadIdx.x == 0) s_nc = n;
  }
  __syncthreads();
  const int nc = s_nc;
  for (int k = 0; k < nc; ++k) {
    const AbCtx c = st.ctx[k];
    const long long acc = warp_sum(ab_edges<GS, 4>(a, c, c.beg, c.beg + c.deg, threadIdx.x));
    if ((threadIdx.x & 31) == 0) rs[k][threadIdx.x >> 5] = acc;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    long long t = delta;
    if (r.D != kNone)
      for (int w = 0; w < GS / 32; ++w) t += rs[pos][w];
    apply_lanes(a, (int)threadIdx.x < b.m, vr.v, vr.deg, r, vr.w, r.D != kNone && t >= 0, sum);
  }
  flush_update(a, sum);
  step_end();
}

__global__ void __launch_bounds__(kHubThreads) k_hub_afterburner(PassArgs a) {
  step_begin();
  const int c = blockIdx.x;
  const int h = a.hub.hub_of[c];
  const int32_t v = a.hub.vtx[h];
  const AbRec r = a.ab[v];
  UpdateSums sum;
  bool mine = c == a.hub.c0[h] && !left_to_settle(a, h);  // no candidate: its first chunk keeps it where it is
  long long t = -1;
  if (r.D != kNone) {  // block-uniform
    const AbCtx ctx = ab_ctx(a, v, r, a.gp[graph_of(a, v)], 0, 0, a.g.vw[v]);
    hub_acc_add(a, h, ab_edges<kHubThreads, 4>(a, ctx, a.hub.e0[c], a.hub.e1[c], threadIdx.x));
    mine = !left_to_settle(a, h) && last_of_hub(a, h);
    if (mine && threadIdx.x == 0) t = a.delta[v] + take_hub_acc(a, h);
  }
  if (mine && threadIdx.x < 32)
    apply_lanes(a, threadIdx.x == 0, v, a.g.rp[v + 1] - a.g.rp[v], r, a.g.vw[v], t >= 0, sum);
  flush_update(a, sum);
  step_end();
}

// ---------------------------------------------------- objective, S_self

// Phi(C) = sum over v of g(v, C[v]) (Eq. 1 regrouped per vertex): sweeps
// each row for neighbours in C[v].
template <int GS>
__global__ void __launch_bounds__(GS > 32 ? GS : 256)
    k_objective(PassArgs a, const int32_t *__restrict__ list, int64_t count) {
  step_begin();
  __shared__ long long rs[GS > 32 ? GS / 32 : 1];
  long long phi = 0;
  const int r = Grp<GS>::rank();
  for_each_vertex<GS>(count, [&](int64_t i, bool active) {
    const int32_t v = active ? list[i] : 0;
    long long self = 0;
    int32_t Cv = 0;
    if (active) {
      const int64_t beg = a.g.rp[v], end = a.g.rp[v + 1];
      Cv = a.C[v];
#pragma unroll 4
      for (int64_t e = beg + r; e < end; e += GS)
        if (a.C[LC_IDX(__ldg(a.g.col + e), a.g.n, kDbgColumn)] == Cv) self += __ldg(a.g.ew + e);
    }
    self = Grp<GS>::sum(self, rs);
    const bool owner = active && r == 0;
    const int g = owner ? graph_of(a, v) : 0;
    const long long gC = owner ? gain_self(a.gp[g], self, a.g.vw[v], a.W[Cv]) : 0;
    if constexpr (GS <= 32)
      phi_add(a, a.phi_acc, owner, g, gC, phi);
    else if (owner)
      phi_add_one(a, a.phi_acc, g, gC, phi);
  });
  flush_block_sum(phi, &a.phi_acc[0]);
  step_end();
}

__global__ void __launch_bounds__(kHubThreads) k_hub_objective(PassArgs a) {
  step_begin();
  const int c = blockIdx.x;
  const int h = a.hub.hub_of[c];
  const int32_t Cv = a.C[a.hub.vtx[h]];
  long long self = 0;
#pragma unroll 4
  for (int64_t e = a.hub.e0[c] + threadIdx.x; e < a.hub.e1[c]; e += kHubThreads)
    if (a.C[LC_IDX(__ldg(a.g.col + e), a.g.n, kDbgColumn)] == Cv) self += __ldg(a.g.ew + e);
  hub_acc_add(a, h, self);
  step_end();
}

__global__ void k_hub_obj_final(PassArgs a) {
  long long phi = 0;
  for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < a.hub.H; h += gridDim.x * blockDim.x) {
    const int32_t v = a.hub.vtx[h];
    const long long self = a.hub.acc[h];
    a.hub.acc[h] = 0;
    const int g = graph_of(a, v);
    phi_add_one(a, a.phi_acc, g, gain_self(a.gp[g], self, a.g.vw[v], a.W[a.C[v]]), phi);
  }
  flush_block_sum(phi, &a.phi_acc[0]);
}

// ------------------------------------------ kept tables (Section IV-A-3)
//
// Vertices of degree above kTabMinDeg (bins 5-9) may keep their S(v, .)
// across the passes of one LocalMovePasses call.  An aggregation pass with
// a.tab_build copies each block bin's shared table (own cluster included)
// to the vertex's gtab region in the layout of tab_cap, and leaves the hubs'
// global tables in place.  The next pass applies the previous pass's moves
// to those tables in place (Algorithm 2's update of the affected tables: a
// mover from X to Y takes w(u, v) from S(u, X) and adds it to S(u, Y) for
// each neighbour u that keeps a table), then reads the argmax of those
// vertices from their tables; vertices of lower degree aggregate from the
// CSR as in every other pass.  Keys are never removed: a sum that reaches
// 0 marks a cluster no longer adjacent and is skipped.  A table that runs
// out of slots is listed and rebuilt from the labels.

// Subtracts w from the sum of an existing key (nothing is inserted).
// Returns false when the key is absent, which only an overflowed table
// (rebuilt afterwards) can show.  Keys present before the kernel come
// before any empty slot of their probe sequence, so concurrent inserts of
// other keys cannot hide them.
__device__ __forceinline__ bool tab_sub(unsigned long long *t, uint32_t cap, int32_t key, int32_t w) {
  const unsigned long long tag = (unsigned long long)((uint32_t)key + 1u) << 32;
  uint32_t s = slot_of(key, cap);
  for (uint32_t probe = 0; probe < cap; ++probe) {
    const unsigned long long cur = t[s];
    if (cur == kEmptySlot) return false;
    if ((cur & 0xFFFFFFFF00000000ull) == tag) {
      atomicAdd(reinterpret_cast<unsigned int *>(&t[s]), (unsigned int)(-w));
      return true;
    }
    s = (s + 1 == cap) ? 0 : s + 1;
  }
  return false;
}

__device__ __forceinline__ void mark_dirty(const PassArgs &a, int32_t u) {
  if (atomicExch(&a.dirty[u], 1) == 0) a.dirty_list[atomicAdd(&a.sc->tab_dirty, 1)] = u;
}

// The move Xo -> Xn of one mover applied to the kept tables of its
// neighbours over edges [e0, e1) (strided by 32, loads batched U at a time).
__device__ __forceinline__ void tab_move_edges(const PassArgs &a, int64_t e0, int64_t e1, int lane,
                                               int32_t Xo, int32_t Xn) {
  constexpr int U = 4;
  for (int64_t base = e0 + lane; base < e1; base += 32 * U) {
    int32_t u[U], w[U];
    int64_t ub[U], ue[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int64_t e = base + 32 * k;
      u[k] = -1;
      w[k] = 0;
      if (e < e1) {
        u[k] = __ldg(a.g.col + e);
        w[k] = __ldg(a.g.ew + e);
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      ub[k] = u[k] >= 0 ? a.g.rp[u[k]] : 0;
      ue[k] = u[k] >= 0 ? a.g.rp[u[k] + 1] : 0;
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (u[k] < 0 || ue[k] - ub[k] <= kTabMinDeg) continue;  // no kept table
      unsigned long long *t = a.gtab + 2 * ub[k];
      const uint32_t cap = tab_cap(ue[k] - ub[k]);
      bool fresh;
      const bool ok = tab_sub(t, cap, Xo, w[k]);
      if (!(table_add(t, cap, Xn, w[k], fresh) && ok)) mark_dirty(a, u[k]);
    }
  }
}

// Update: one warp per chunk of a mover's row (the chunks were listed by
// the last pass's apply step).
__global__ void __launch_bounds__(256) k_tab_update(PassArgs a) {
  const int cnt = a.sc->upd_prev;
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  long long done = 0;  // edges applied (lane 0), for the profile's byte count
  for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < cnt; j += nw) {
    const int2 ch = a.upd_list[j];
    const int32_t v = ch.x;
    const int32_t Xo = a.ab[v].C, Xn = a.C[v];
    if (Xo == Xn) continue;  // a mover that got its own emptied id back
    const int64_t e0 = a.g.rp[v] + (int64_t)ch.y * kUpdChunk;
    const int64_t end = a.g.rp[v + 1];
    const int64_t e1 = e0 + kUpdChunk < end ? e0 + kUpdChunk : end;
    tab_move_edges(a, e0, e1, lane, Xo, Xn);
    if (lane == 0) done += e1 - e0;
  }
  flush_block_sum(done, &a.sc->tab_upd_edges);
}

// Rebuilds the listed overflowed tables from the current labels, one warp
// per table (rare: a table overflows only after more new clusters reached
// it than it has free slots).
__global__ void __launch_bounds__(256) k_tab_rebuild(PassArgs a) {
  const int cnt = a.sc->tab_dirty;
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  bool ok = true;
  for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < cnt; j += nw) {
    const int32_t v = a.dirty_list[j];
    const int64_t beg = a.g.rp[v], deg = a.g.rp[v + 1] - beg;
    unsigned long long *t = a.gtab + 2 * beg;
    const uint32_t cap = tab_cap(deg);
    for (int64_t s = lane; s < 2 * deg; s += 32) t[s] = kEmptySlot;
    __syncwarp();
    for (int64_t e = beg + lane; e < beg + deg; e += 32) {
      bool fresh;
      ok &= table_add(t, cap, LC_IDX(a.C[LC_IDX(__ldg(a.g.col + e), a.g.n, kDbgColumn)], a.g.n, kDbgLabel),
                      __ldg(a.g.ew + e), fresh);
    }
    __syncwarp();
    if (lane == 0) a.dirty[v] = 0;
  }
  if (!ok) {
    a.sc->error = 1;
    LC_DBG_FAIL(kDbgProbe, -1, a.g.n);  // the table of one of this thread's listed vertices
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && cnt > 0) a.sc->tab_rebuilt += cnt;
}

// Best (gain, cluster) over the slot pairs [p0, p1) of a kept table
// (16-byte loads, strided by GS, V pairs per thread at a time) and this
// thread's part of S(v, C[v]); with `reset` the slots are cleared as they
// are read (the last pass of a call leaves gtab clean).
template <int GS, int V>
__device__ __forceinline__ void tab_pairs_scan(const PassArgs &a, const GraphParam &P, ulonglong2 *t2,
                                               uint32_t p0, uint32_t p1, int32_t Cv, long long wv,
                                               bool reset, long long &self, long long &gb, int32_t &xb) {
  const long long Lam = P.Lam, muw = P.mu * wv;
  for (uint32_t base = p0 + threadIdx.x; base < p1; base += GS * V) {
    unsigned long long t[2 * V];
    long long WX[2 * V];
    bool use[2 * V];
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const uint32_t p = base + k * GS;
      ulonglong2 x = make_ulonglong2(kEmptySlot, kEmptySlot);
      if (p < p1) x = t2[p];
      if (reset && p < p1 && (x.x | x.y) != 0ull) t2[p] = make_ulonglong2(kEmptySlot, kEmptySlot);
      t[2 * k] = x.x;
      t[2 * k + 1] = x.y;
    }
#pragma unroll
    for (int k = 0; k < 2 * V; ++k) {
      const int32_t X = slot_key(t[k]), S = slot_val(t[k]);
      use[k] = t[k] != kEmptySlot && S > 0 && X != Cv;
      if (t[k] != kEmptySlot && X == Cv) self += S;
      WX[k] = use[k] ? a.W[X] : 0;
    }
#pragma unroll
    for (int k = 0; k < 2 * V; ++k) {
      if (!use[k]) continue;
      const int32_t X = slot_key(t[k]);
      const long long g = Lam * (long long)slot_val(t[k]) - muw * WX[k];
      if (better(g, X, gb, xb)) {
        gb = g;
        xb = X;
      }
    }
  }
}

// Argmax and candidate test of Algorithm 2 from the kept tables, one block
// per vertex of bins 5-8 (a single reduction to thread 0 per vertex; the
// partials alternate between two buffers, so one barrier per vertex).
template <int GS, int V>
__global__ void __launch_bounds__(GS) k_tab_scan(PassArgs a, const int32_t *__restrict__ list,
                                                 int64_t count) {
  __shared__ long long rs[2][GS / 32], rg[2][GS / 32];
  __shared__ int32_t rx[2][GS / 32];
  MoveState ms = move_state(a);
  int par = 0;
  for (int64_t i = blockIdx.x; i < count; i += gridDim.x) {
    const int32_t v = list[i];
    const int64_t beg = a.g.rp[v];
    const uint32_t cap = tab_cap(a.g.rp[v + 1] - beg);
    const int32_t Cv = a.C[v];
    const long long wv = a.g.vw[v];
    const GraphParam P = a.gp[graph_of(a, v)];
    long long self = 0, gb = LLONG_MIN;
    int32_t xb = kNone;
    tab_pairs_scan<GS, V>(a, P, reinterpret_cast<ulonglong2 *>(a.gtab + 2 * beg), 0, cap / 2, Cv, wv,
                          a.tab_reset != 0, self, gb, xb);
    group_argmax<32>(gb, xb);
    self = warp_sum(self);
    if ((threadIdx.x & 31) == 0) {
      rg[par][threadIdx.x >> 5] = gb;
      rx[par][threadIdx.x >> 5] = xb;
      rs[par][threadIdx.x >> 5] = self;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < GS / 32; ++w) {
        self += rs[par][w];
        if (better(rg[par][w], rx[par][w], gb, xb)) {
          gb = rg[par][w];
          xb = rx[par][w];
        }
      }
      const long long gC = gain_self(P, self, wv, a.W[Cv]);
      phi_add_one(a, ms.acc, graph_of(a, v), gC, ms.phi);
      decide(a, P, v, Cv, gC, xb, gb, ms);
    }
    par ^= 1;
  }
  flush_block_sum(ms.cntL, &a.sc->count_L);
  flush_block_sum(ms.phi, &ms.acc[0]);
}

// Hubs: each chunk scans its share of the hub's table; the last one combines
// the partials and the parts of S(v, C[v]).
__global__ void __launch_bounds__(kHubThreads) k_hub_tab_scan(PassArgs a) {
  const int c = blockIdx.x;
  const int h = a.hub.hub_of[c];
  const int32_t v = a.hub.vtx[h];
  const int64_t beg = a.g.rp[v];
  const GraphParam P = a.gp[graph_of(a, v)];
  MoveState ms = move_state(a);
  long long self = 0, gb = LLONG_MIN;
  int32_t xb = kNone;
  // a chunk of edges [e0, e1) owns the slot pairs [e0 - beg, e1 - beg)
  tab_pairs_scan<kHubThreads, 4>(a, P, reinterpret_cast<ulonglong2 *>(a.gtab + 2 * beg),
                                 (uint32_t)(a.hub.e0[c] - beg), (uint32_t)(a.hub.e1[c] - beg), a.C[v],
                                 a.g.vw[v], a.tab_reset != 0, self, gb, xb);
  hub_part_store(a, c, gb, xb);
  hub_acc_add(a, h, self);
  if (last_of_hub(a, h) && threadIdx.x < 32) decide_hub(a, h, v, false, threadIdx.x, ms);
  flush_move(a, ms);
}

// Takes over the objectives of the graphs that improved (k_bestof).
__device__ __forceinline__ void settle_bestof(const PassArgs &a) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < a.G; g += gridDim.x * blockDim.x) {
    const long long p = a.phi_acc[g];
    if (p > a.phi_out[g]) a.phi_out[g] = p;
    a.phi_acc[g] = 0;
  }
}
// ------------------------------------------------ ids of new clusters

// The movers to new empty clusters, ascending, take the ascending ids that
// are unused once every other move is applied, per graph.  Ids in use are
// marked from the labels (vertex weights may be zero, so W(x) == 0 does not
// mean x is empty).  Labels of a graph stay inside its own vertex range, so
// its free ids are consecutive in the ascending list of all free ids from
// gfree[g], its movers in the list of all movers from gmover[g].
//
// One cooperative launch whose blocks meet between the phases, in place of
// nine launches per pass that mostly found nothing to do (2 us each): it
// returns at once when the pass has no such mover.  It also settles the
// pass's best-of test, which as a launch of its own took 4 us a pass.
__global__ void __launch_bounds__(kCoopThreads) k_assign_empty(PassArgs a, EmptyScratch w) {
  settle_bestof(a);
  const int total = a.sc->empty_movers;  // nothing writes it during this launch
  if (total == 0) return;
  GridBarrier bar(a.sc);
  if (!assign_empty<kCoopThreads>(a, w, total, false, bar)) {
    // every block that gives up labels whatever is still without: the pass's
    // followers index by the labels, and the host looks later
    for (int64_t v = threadIdx.x; v < a.g.n; v += kCoopThreads)
      if (a.C[v] == kEmpty) a.C[v] = (int32_t)v;
    return;
  }
  bar.leave();
}

__global__ void k_destinations(const AbRec *__restrict__ ab, int32_t *__restrict__ D, int64_t n) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    D[v] = ab[v].D;
}

// ----------------------------------------------------------- best-of

__global__ void k_pass_begin(Scalars *sc, int advance) {
  if (advance) {
    const int i = sc->pass_idx++;
    sc->phi_live[0] = sc->phi_tab[i & 15][0];
    sc->phi_live[1] = sc->phi_tab[i & 15][1];
  }
  sc->count_L = 0;
  sc->count_M = 0;
  sc->empty_movers = 0;
  sc->tab_dirty = 0;
  sc->n_movers = 0;
  sc->upd_prev = sc->upd_count;
  sc->upd_count = 0;
}

// Algorithm 2's best-of test, per graph, on the objective accumulated in
// phi_acc (strict improvement keeps the earliest maximum): the labels of the
// graphs that improved are copied; settle_bestof, in a later kernel, takes the
// values over.  reset: the pass has no k_pass_begin (the update step counts
// from zero here).
__global__ void k_bestof(PassArgs a, int32_t *__restrict__ C_out, int reset) {
  if (reset && blockIdx.x == 0 && threadIdx.x == 0) {
    a.sc->empty_movers = 0;
    a.sc->n_movers = 0;
  }
  if (!a.gid && a.phi_acc[0] <= a.phi_out[0]) return;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < a.g.n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int g = graph_of(a, (int32_t)v);
    if (a.phi_acc[g] > a.phi_out[g]) C_out[v] = a.C[v];
  }
}

__global__ void k_bestof_settle(PassArgs a) { settle_bestof(a); }

// ------------------------------------------------------------ helpers

__global__ void k_iota(int32_t *C, int64_t n) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    C[v] = (int32_t)v;
}

__global__ void k_cluster_weights(const int32_t *__restrict__ C, const int64_t *__restrict__ vw,
                                  int64_t *W, int64_t n) {
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = base + threadIdx.x;
    add_weights(W, v < n, v < n ? C[v] : 0, v < n ? vw[v] : 0);
  }
}

// ================================================================ host

static inline unsigned blocks_for(int64_t items, int per_block) {
  int64_t b = (items + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > 152 * 64) b = 152 * 64;
  return (unsigned)b;
}

// a key and a sum per slot
static constexpr int block_table_bytes(int slots) { return slots * 8; }

void configure_kernels() {
  cudaFuncSetAttribute(k_move_block<64, 1024, 8, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       block_table_bytes(1024));
  cudaFuncSetAttribute(k_move_block<128, 2048, 8, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       block_table_bytes(2048));
  cudaFuncSetAttribute(k_move_block<256, 4096, 8, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       block_table_bytes(4096));
  cudaFuncSetAttribute(k_move_block<256, 6144, 16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       block_table_bytes(6144));
  cudaFuncSetAttribute(k_move_block<64, 1024, 8, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       block_table_bytes(1024));
  cudaFuncSetAttribute(k_move_block<128, 2048, 8, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       block_table_bytes(2048));
  cudaFuncSetAttribute(k_move_block<256, 4096, 8, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       block_table_bytes(4096));
  cudaFuncSetAttribute(k_move_block<256, 6144, 16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       block_table_bytes(6144));
}

// Vertices per warp of the chunked kernels: 32, so that one lane decides one
// vertex, unless that would leave SMs without warps (32 of theirs each).
static inline int warp_chunk_size(int64_t count) {
  const int64_t c = (count + 152 * 32 - 1) / (152 * 32);
  return c < 1 ? 1 : c > 32 ? 32 : (int)((c + 1) & ~1ll);  // even: two vertices per step in the half-warp kernels
}
static inline unsigned warp_chunk_blocks(int64_t count, int chunk) {
  return (unsigned)((count + (int64_t)chunk * 8 - 1) / ((int64_t)chunk * 8));
}
// Vertices per block: up to 32 once every SM has 64 blocks to run.
static inline int block_chunk_size(int64_t count) {
  const int64_t c = count / (152 * 64);
  return c < 1 ? 1 : c > 32 ? 32 : (int)c;
}

// The launches of one step of a pass.  Order: short rows first, long rows
// last.  Long rows first (so that short ones fill the last SMs) was slower:
// the block kernels' shared memory leaves the SMs a small L1 for whatever
// runs among them (ms, short / long rows first: R-MAT scale 22 65.1 / 73.1,
// 256^3 lattice 50.1 / 53.2, batch 59.5 / 62.8, R-MAT 20 level 6.09 / 6.50).
class PassStep : public Step {
 public:
  using Step::Step;
  // most: vertices per warp at most (fewer where rows are long: blocks that
  // end sooner even the SMs out)
  void warp_chunks(void (*k)(PassArgs, const VRec *, int64_t, int), const PassArgs &a, BinRange r, int most = 32) {
    if (r.count <= 0) return;
    const int chunk = std::min(warp_chunk_size(r.count), most);
    run(false, k, warp_chunk_blocks(r.count, chunk), 256, 0, a, r.rec, r.count, chunk);
  }
  void block_chunks(void (*k)(PassArgs, const VRec *, int64_t, int), int threads, size_t smem, const PassArgs &a,
                    BinRange r) {
    if (r.count <= 0) return;
    const int chunk = block_chunk_size(r.count);
    run(false, k, (unsigned)((r.count + chunk - 1) / chunk), threads, smem, a, r.rec, r.count, chunk);
  }
  void threads(void (*k)(PassArgs, const VRec *, int64_t), const PassArgs &a, BinRange r) {
    if (r.count > 0) run(false, k, blocks_for(r.count, 256), 256, 0, a, r.rec, r.count);
  }
};

static inline unsigned hub_final_blocks(int H) { return blocks_for(H, 256); }

// Kernels without tables take runs of bins: bin 0 -> 1 thread, 1 -> 16
// lanes, 2..4 -> one warp, 5..6 -> 128 threads, 7..8 -> 512 threads.
int launch_first_pass(const PassArgs &a, const Bins &b, cudaStream_t s) {
  PassStep st(s);
  st.threads(k_first_thread, a, bin_range(b, 0, 0));
  st.warp_chunks(k_first_pass<16>, a, bin_range(b, 1, 1));
  st.warp_chunks(k_first_pass<32>, a, bin_range(b, 2, 4));
  st.block_chunks(k_first_block<128>, 128, 0, a, bin_range(b, 5, 6));
  st.block_chunks(k_first_block<512>, 512, 0, a, bin_range(b, 7, 8));
  if (a.hub.H > 0) st.run(false, k_hub_first, a.hub.Q, kHubThreads, 0, a);
  if (a.hub.settle) st.run(true, k_hub_settle, blocks_for(a.hub.H, 256), 256, 0, a, 1);
  return st.launches;
}

// Bins 0-4 (degree <= 256) aggregate from the CSR in every pass; hubs: their
// inserts go among them.
static void move_low(PassStep &st, const PassArgs &a, const Bins &b, bool hubs) {
  st.threads(k_move_thread, a, bin_range(b, 0, 0));
  st.warp_chunks(k_move_lanes<16>, a, bin_range(b, 1, 1));
  st.warp_chunks(k_move_lanes<32>, a, bin_range(b, 2, 2));
  // after the block kernels these inserts cost R-MAT scale 22 5 ms in 65
  // (their shared memory leaves a small L1), before all others nothing
  if (hubs) st.run(false, k_hub_move_insert, a.hub.Q, kHubThreads, 0, a);
  st.warp_chunks(k_move_warp, a, bin_range(b, 3, 4), 16);
}

template <int GS, int SLOTS, int N>
static void move_block(PassStep &st, const PassArgs &a, BinRange r) {
  st.block_chunks(a.tab_build ? k_move_block<GS, SLOTS, N, true> : k_move_block<GS, SLOTS, N, false>, GS,
                  block_table_bytes(SLOTS), a, r);
}

int launch_move(const PassArgs &a, const Bins &b, cudaStream_t s) {
  PassStep st(s);
  move_low(st, a, b, a.hub.H > 0);
  move_block<64, 1024, 8>(st, a, bin_range(b, 5, 5));
  move_block<128, 2048, 8>(st, a, bin_range(b, 6, 6));
  move_block<256, 4096, 8>(st, a, bin_range(b, 7, 7));
  move_block<256, 6144, 16>(st, a, bin_range(b, 8, 8));
  if (a.hub.H > 0) st.run(true, k_hub_move_scan, a.hub.Q, kHubThreads, 0, a);
  if (a.hub.settle) st.run(true, k_hub_settle, blocks_for(a.hub.H, 256), 256, 0, a, 0);
  return st.launches;
}

int launch_table_pass(const PassArgs &a, const Bins &b, cudaStream_t s) {
  PassStep st(s);
  st.run(true, k_tab_update, 152 * 8, 256, 0, a);  // reads the last pass's records, before any is rewritten
  st.run(true, k_tab_rebuild, 152 * 4, 256, 0, a);
  // one 16-byte pair of slots per thread per batch of V: bin 5 has at most
  // 512 pairs, bin 6 1024, bin 7 2048, bin 8 3072
  const auto scan = [&](void (*k)(PassArgs, const int32_t *, int64_t), int threads, BinRange r) {
    if (r.count > 0) st.run(true, k, blocks_for(r.count, 1), threads, 0, a, r.list, r.count);
  };
  scan(k_tab_scan<128, 4>, 128, bin_range(b, 5, 5));
  scan(k_tab_scan<256, 4>, 256, bin_range(b, 6, 6));
  scan(k_tab_scan<512, 4>, 512, bin_range(b, 7, 8));
  if (a.hub.H > 0) st.run(true, k_hub_tab_scan, a.hub.Q, kHubThreads, 0, a);
  move_low(st, a, b, false);
  return st.launches;
}

// One of the afterburner's bin groups 2-4: 16 (group 2 only), 32, 128 or 512
// threads per candidate (BinPlan::ab_gs).  Bin 2 of group 2 (rows up to 32
// edges) always takes 8 lanes per candidate.
static void ab_group(PassStep &st, const PassArgs &a, const Bins &b, int g) {
  const BinRange r = bin_range(b, g == 2 ? 3 : kAbFirstBin[g], kAbFirstBin[g + 1] - 1);
  if (a.ab_gs[g] == 16)
    st.warp_chunks(k_ab_warp<16>, a, r, 16);
  else if (a.ab_gs[g] == 32)
    st.warp_chunks(k_ab_warp<32>, a, r, 16);
  else if (a.ab_gs[g] == 128)
    st.block_chunks(k_ab_block<128>, 128, 0, a, r);
  else
    st.block_chunks(k_ab_block<512>, 512, 0, a, r);
}

int launch_afterburner(const PassArgs &a, const Bins &b, cudaStream_t s) {
  PassStep st(s);
  st.threads(k_ab_thread, a, bin_range(b, 0, 0));
  st.warp_chunks(k_ab_warp<4>, a, bin_range(b, 1, 1));
  st.warp_chunks(k_ab_warp<8>, a, bin_range(b, 2, 2));
  for (int g = 2; g < kAbGroups; ++g) ab_group(st, a, b, g);
  if (a.hub.H > 0) st.run(false, k_hub_afterburner, a.hub.Q, kHubThreads, 0, a);
  if (a.hub.settle) st.run(true, k_hub_settle_update, blocks_for(a.hub.H, 256), 256, 0, a);
  return st.launches;
}

// ------------------------------------- symmetry-breaking ablations

__global__ void k_cluster_sizes(const int32_t *__restrict__ C, int32_t *__restrict__ size, int64_t n) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&size[C[v]], 1);
}

// Every candidate moves, except (mlh) a vertex alone in its cluster whose
// destination is another one-vertex cluster with a larger label.
__global__ void k_symmetry_ablation(PassArgs a, const int32_t *__restrict__ size, int mlh) {
  UpdateSums sum;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < a.g.n; base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = base + threadIdx.x;
    const bool on = v < a.g.n;
    AbRec r{0, kNone, 0};
    int64_t deg = 0;
    bool keep = false;
    if (on) {
      r = a.ab[v];
      deg = a.g.rp[v + 1] - a.g.rp[v];
      keep = r.D != kNone && !(mlh && size[r.C] == 1 && r.D >= 0 && size[r.D] == 1 && r.D > r.C);
    }
    apply_lanes(a, on, (int32_t)v, deg, r, on ? a.g.vw[v] : 0, keep, sum);
  }
  flush_update(a, sum);
}

int launch_symmetry_ablation(const PassArgs &a, bool mlh, int32_t *size, cudaStream_t s) {
  if (a.g.n == 0) return 0;
  int n = 1;
  if (mlh) {
    cudaMemsetAsync(size, 0, sizeof(int32_t) * (size_t)a.g.n, s);
    k_cluster_sizes<<<blocks_for(a.g.n, 256), 256, 0, s>>>(a.C, size, a.g.n);
    n++;
  }
  k_symmetry_ablation<<<blocks_for(a.g.n, 256), 256, 0, s>>>(a, size, mlh ? 1 : 0);
  return n;
}

int launch_objective(const PassArgs &a, const Bins &b, cudaStream_t s) {
  PassStep st(s);
  const auto rows = [&](void (*k)(PassArgs, const int32_t *, int64_t), int threads, int per_block, BinRange r) {
    if (r.count > 0) st.run(false, k, blocks_for(r.count, per_block), threads, 0, a, r.list, r.count);
  };
  rows(k_objective<1>, 256, 256, bin_range(b, 0, 0));
  rows(k_objective<16>, 256, 16, bin_range(b, 1, 1));
  rows(k_objective<32>, 256, 8, bin_range(b, 2, 4));
  rows(k_objective<128>, 128, 1, bin_range(b, 5, 6));
  rows(k_objective<512>, 512, 1, bin_range(b, 7, 8));
  if (a.hub.H > 0) {
    st.run(false, k_hub_objective, a.hub.Q, kHubThreads, 0, a);
    st.run(true, k_hub_obj_final, hub_final_blocks(a.hub.H), 256, 0, a);
  }
  return st.launches;
}

// ------------------------- objective after the last pass (one graph)
//
// Phi = Lam IN - mu Q (Eq. 1 regrouped): IN = sum_v S(v, C[v]) and
// Q = sum_X W(X)^2 - sum_v w(v)^2.  The last pass's move step sums Phi of
// the state entering it; its moves change IN only on the movers' edges, by
// ([C'[v] = C'[u]] - [C[v] = C[u]]) w(u, v) per direction, and Q follows
// from W before and after (an O(n) sweep each).  So the objective of the
// call's final state, which the best-of test of Algorithm 2 needs, costs a
// walk over the movers' rows instead of a sweep of the whole graph:
//   Phi' = Phi + Lam dIN - mu (Q' - Q).

// The per-graph accumulators of the objective update: a.obj holds
// [Phi entering | Q entering | Q after | dIN], G entries each.
__device__ __forceinline__ long long *obj_phi_enter(const PassArgs &a) { return a.obj; }
__device__ __forceinline__ long long *obj_q_enter(const PassArgs &a) { return a.obj + a.G; }
__device__ __forceinline__ long long *obj_q_final(const PassArgs &a) { return a.obj + 2 * a.G; }
__device__ __forceinline__ long long *obj_d_in(const PassArgs &a) { return a.obj + 3 * a.G; }

// dIN over the listed movers (not hubs), one warp each; a batch (BATCH)
// adds each mover's change to its own graph's sum.
template <bool BATCH>
__global__ void __launch_bounds__(256) k_delta_in(PassArgs a) {
  const int cnt = a.sc->n_movers;
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  long long d = 0, edges = 0;
  for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < cnt; j += nw) {
    const int32_t v = a.movers[j];
    if (a.C[v] == a.ab[v].C) continue;
    const int64_t beg = a.g.rp[v], end = a.g.rp[v + 1];
    const long long dv = delta_in_edges<32>(a, v, beg, end, lane);
    if constexpr (BATCH) {
      const long long t = warp_sum(dv);
      if (lane == 0 && t != 0) atomicAdd((unsigned long long *)&obj_d_in(a)[a.gid[v]], (unsigned long long)t);
    } else {
      d += dv;
    }
    if (lane == 0) edges += end - beg;
  }
  if (!BATCH) flush_block_sum(d, obj_d_in(a));
  flush_block_sum(edges, &a.sc->dphi_edges);
}

__global__ void __launch_bounds__(kHubThreads) k_hub_delta_in(PassArgs a) {
  __shared__ long long rs[kHubThreads / 32];
  const int c = blockIdx.x;
  const int32_t v = a.hub.vtx[a.hub.hub_of[c]];
  if (a.C[v] == a.ab[v].C) return;  // not a mover (block-uniform)
  const long long d =
      Grp<kHubThreads>::sum(delta_in_edges<kHubThreads>(a, v, a.hub.e0[c], a.hub.e1[c], threadIdx.x), rs);
  if (threadIdx.x == 0) {
    if (d != 0) atomicAdd((unsigned long long *)&obj_d_in(a)[graph_of(a, v)], (unsigned long long)d);
    atomicAdd((unsigned long long *)&a.sc->dphi_edges, (unsigned long long)(a.hub.e1[c] - a.hub.e0[c]));
  }
}

// Q = sum_x W(x)^2 - w(x)^2 over the level's ids x (W of an unused id is 0)
// into q[0] (zeroed by the caller).  Unsigned arithmetic: exact whenever Q
// fits (mu > 0 and the guard Lam T + mu V^2 < 2^60); with mu = 0 it is not
// used.
__global__ void k_q(PassArgs a, long long *q) {
  long long t = 0;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < a.g.n;
       x += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long W = (unsigned long long)a.W[x], w = (unsigned long long)a.g.vw[x];
    t += (long long)(W * W - w * w);
  }
  flush_block_sum(t, q);
}

// The same per graph of a batch, into q[g].  The labels of a graph lie in
// its own vertex range, so the lanes of a warp cover a few runs of one graph
// each; each run is summed by a segmented shuffle scan and added once.
__global__ void k_q_batch(PassArgs a, long long *q) {
  const int lane = threadIdx.x & 31;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < a.g.n; base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = base + threadIdx.x;
    long long t = 0;
    if (x < a.g.n) {
      const unsigned long long W = (unsigned long long)a.W[x], w = (unsigned long long)a.g.vw[x];
      t = (long long)(W * W - w * w);
    }
    const int g = x < a.g.n ? a.gid[x] : -1;
    // inclusive scan within runs of equal g
    const int gp = __shfl_up_sync(0xFFFFFFFFu, g, 1);
    const bool head = lane == 0 || gp != g;
    unsigned heads = __ballot_sync(0xFFFFFFFFu, head);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xFFFFFFFFu, t, o);
      // lanes o back are in the same run if no head lies in (lane - o, lane]
      const unsigned span = (lane >= o) ? (((1u << lane) << 1) - (1u << (lane - o + 1))) : 0u;
      if (lane >= o && (heads & span) == 0) t += y;
    }
    const int gn = __shfl_down_sync(0xFFFFFFFFu, g, 1);
    const bool tail = lane == 31 || gn != g;
    if (tail && g >= 0 && t != 0) atomicAdd((unsigned long long *)&q[g], (unsigned long long)t);
  }
}

static void launch_q(const PassArgs &a, long long *q, cudaStream_t s) {
  if (a.gid)
    k_q_batch<<<blocks_for(a.g.n, 256), 256, 0, s>>>(a, q);
  else
    k_q<<<blocks_for(a.g.n, 256), 256, 0, s>>>(a, q);
}

__global__ void k_save_phi_enter(PassArgs a) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < a.G; g += gridDim.x * blockDim.x)
    obj_phi_enter(a)[g] = a.phi_acc[g];
}

__global__ void k_final_phi(PassArgs a) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < a.G; g += gridDim.x * blockDim.x) {
    const GraphParam P = a.gp[g];
    const long long dq = obj_q_final(a)[g] - obj_q_enter(a)[g];
    a.phi_acc[g] = obj_phi_enter(a)[g] + P.Lam * obj_d_in(a)[g] - (P.mu != 0 ? P.mu * dq : 0);
  }
}

int launch_last_pass_enter(const PassArgs &a, cudaStream_t s) {
  cudaMemsetAsync(a.obj + a.G, 0, sizeof(long long) * (size_t)a.G, s);
  if (a.g.n > 0) launch_q(a, a.obj + a.G, s);
  return a.g.n > 0 ? 1 : 0;
}

int launch_save_phi_enter(const PassArgs &a, cudaStream_t s) {
  k_save_phi_enter<<<blocks_for(a.G, 256), 256, 0, s>>>(a);
  return 1;
}

int launch_final_objective(const PassArgs &a, cudaStream_t s) {
  cudaMemsetAsync(a.obj + 2 * a.G, 0, 2 * sizeof(long long) * (size_t)a.G, s);  // Q after, dIN
  if (a.gid)
    k_delta_in<true><<<152 * 8, 256, 0, s>>>(a);
  else
    k_delta_in<false><<<152 * 8, 256, 0, s>>>(a);
  int n = 1;
  if (a.hub.H > 0) {
    k_hub_delta_in<<<a.hub.Q, kHubThreads, 0, s>>>(a);
    n++;
  }
  if (a.g.n > 0) {
    launch_q(a, a.obj + 2 * a.G, s);
    n++;
  }
  k_final_phi<<<blocks_for(a.G, 256), 256, 0, s>>>(a);
  return n + 1;
}

int launch_assign_empty(const PassArgs &a, const EmptyScratch &w, cudaStream_t s) {
  if (a.g.n <= 0) return 0;
  int64_t blocks = (a.g.n + 4 * kCoopThreads - 1) / (4 * kCoopThreads);
  if (blocks > coop_blocks(a.coop)) blocks = coop_blocks(a.coop);
  PassArgs pa = a;
  EmptyScratch es = w;
  void *args[] = {&pa, &es};
  cudaLaunchCooperativeKernel((const void *)k_assign_empty, dim3((unsigned)blocks), dim3(kCoopThreads), args, 0, s);
  return 1;
}

void launch_destinations(const PassArgs &a, int32_t *D, cudaStream_t s) {
  if (a.g.n > 0) k_destinations<<<blocks_for(a.g.n, 256), 256, 0, s>>>(a.ab, D, a.g.n);
}

void launch_pass_begin(Scalars *sc, cudaStream_t s, int advance) { k_pass_begin<<<1, 1, 0, s>>>(sc, advance); }

// phi_final[g] = phi_out[g] for the graphs that ran in this call.
__global__ void k_keep_phi(const GraphParam *gp, const long long *phi_out, long long *phi_final, int G) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x)
    if (gp[g].active) phi_final[g] = phi_out[g];
}

int launch_keep_phi(const PassArgs &a, long long *phi_final, cudaStream_t s) {
  k_keep_phi<<<blocks_for(a.G, 256), 256, 0, s>>>(a.gp, a.phi_out, phi_final, a.G);
  return 1;
}

int launch_bestof(const PassArgs &a, int32_t *C_out, bool reset, cudaStream_t s) {
  k_bestof<<<blocks_for(a.g.n, 256), 256, 0, s>>>(a, C_out, reset ? 1 : 0);
  return 1;
}
int launch_final_bestof(const PassArgs &a, int32_t *C_out, cudaStream_t s) {
  k_bestof<<<blocks_for(a.g.n, 256), 256, 0, s>>>(a, C_out, 0);
  k_bestof_settle<<<blocks_for(a.G, 256), 256, 0, s>>>(a);
  return 2;
}

void launch_iota(int32_t *C, int64_t n, cudaStream_t s) {
  k_iota<<<blocks_for(n, 256), 256, 0, s>>>(C, n);
}

__global__ void k_fill(long long *a, long long value, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) a[i] = value;
}
void launch_fill(long long *a, long long value, int n, cudaStream_t s) {
  if (n > 0) k_fill<<<blocks_for(n, 256), 256, 0, s>>>(a, value, n);
}

void launch_cluster_weights(const int32_t *C, const int64_t *vw, int64_t *W, int64_t n,
                            cudaStream_t s) {
  cudaMemsetAsync(W, 0, sizeof(int64_t) * (size_t)(n > 0 ? n : 1), s);
  k_cluster_weights<<<blocks_for(n, 256), 256, 0, s>>>(C, vw, W, n);
}

}  // namespace lc
