// lc_fused.cu — one LocalMovePasses call (Algorithm 2) as one kernel.
//
// A level of a few thousand to about a million vertices keeps the chip busy
// for tens of microseconds per pass, while the separate kernels of a pass
// (up to nine move kernels, the best-of test and copy, up to seven
// afterburner kernels, the counters and the new-cluster ids) cost 2-4 us each
// whatever they find to do.  Here all passes of a call run in one cooperative
// launch of one 512-thread block per SM; the phases of a pass are separated
// by grid barriers (1.2 us over 152 blocks on their own, 2.2-2.6 us behind a
// phase's stores):
//
//   move:    gains, argmax, candidate test of every vertex; records written
//   barrier
//   update:  best-of test and copy (from the records), afterburner, moves
//   barrier  (then the new-cluster ids if the pass has such movers)
//
// The work inside a phase is the separate kernels' own device code
// (lc_move.cuh), so the results are identical.  Rows are taken by a thread
// (bin 0), 16 lanes, a warp (bins 2-4), four warps (bins 5-6) or the block
// (bins 7-8 and hubs of up to kRowSlots / 2 edges); longer hub rows go by
// chunks over the global table, with one more barrier per pass.
//
// What bounds it: on small levels the barrier and one chain of gathers per
// phase (4-10 us, also for a few thousand vertices), on the largest the
// gathers, a clock per lane and SM (an SBM of 100,000 vertices and 2 M stored
// edges: 35 us to move, 29 us to update).  Calls, ms, separate kernels / this
// when it was built: SBM of 10,000 vertices 5.1 / 3.8, R-MAT scale 16 21.9 /
// 13.5, SBM of 100,000 8.4 / 6.5; with later changes here and between the
// levels 1.45, 4.8 and 3.8.
#include "lc_coop.cuh"
#include "lc_empty.cuh"
#include "lc_fused.cuh"
#include "lc_move.cuh"

namespace lc {

namespace {

// 512 threads with 128 registers: 1,024 with 64 spilled 1.3 KB a thread and
// ran 15-18 % slower on SBM 10,000, R-MAT 16 and the 97^3 lattice, 768 with 80
// 5 % slower, in spite of more warps.
constexpr int kT = 512, kW = kT / 32;
constexpr int kWarpSlots = 1024;                // shared table of a warp (bins 3-4)
constexpr int kTeam = 128;                      // threads of a team (bins 5-6)
constexpr int kTeamSlots = kWarpSlots * kTeam / 32;
constexpr int kRowSlots = kWarpSlots * kW;      // the whole block's table
constexpr int64_t kRowMaxDeg = kRowSlots / 2;   // rows above go by chunks

// Per-warp staging; the move and update phases never hold theirs at once.
union Stage {
  struct {
    MoveStage st;
    LaneTags tags;
  } move;
  AbStage ab;
};
constexpr size_t kSmemBytes = sizeof(uint32_t) * 2 * kRowSlots + sizeof(Stage) * kW;

// Barrier of one team of kTeam threads (ids 1 .. kT / kTeam; 0 is the block's).
__device__ __forceinline__ void team_sync(int team) {
  asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(kTeam) : "memory");
}

// Work of a phase is handed out in order of cost: the first piece of a block,
// team or warp by its place in the grid (warps in turn over SMs, so a short
// list reaches every SM), every later piece from a counter, which evens out
// the blocks that had long rows.  Pieces are fetched one ahead.
enum { kNextRow = 0, kNextTeam = 1, kNextChunk = 2, kNextCount = 3 };

// The runs of bins that a phase's warps take in chunks, longest rows first:
// kept in shared memory, so that the loop over chunks holds no registers for
// them.
struct ChunkLists {
  unsigned end[5];  // chunks of the lists up to this one
  int c[5];         // vertices per chunk
  int lo[5];        // first bin
};
// Lists of bins lo .. hi, in chunks of at most `most` vertices: one per warp,
// but two (bin 2) or four (longer rows) where a warp has many, so that the
// last ones even out: half of the warps' time was spent at the phase's
// barrier on an SBM of 100,000 vertices (4.79 -> 4.50 ms a call), while finer
// chunks on short lists only add rounds (SBM of 10,000 vertices 1.60 -> 1.78).
// A thread per vertex (bin 0) takes 32.  Every thread of the block.
template <int N>
__device__ __forceinline__ void plan_chunks(const FusedArgs &f, ChunkLists &l, const int (&lo)[N], const int (&hi)[N],
                                            const int (&most)[N]) {
  __syncthreads();  // the last phase's lists are no longer read
  if (threadIdx.x == 0) {
    const int64_t nw = (int64_t)gridDim.x * kW;
    unsigned end = 0;
    for (int k = 0; k < N; ++k) {
      const int64_t count = f.off[hi[k] + 1] - f.off[lo[k]];
      int64_t c = (count + nw - 1) / nw;
      if (lo[k] >= 3 && c > 4) c = (c + 3) / 4;
      if (lo[k] == 2 && c > 8) c = (c / 2 + 3) & ~3ll;
      l.lo[k] = lo[k];
      l.c[k] = lo[k] == 0 ? 32 : c >= most[k] ? most[k] : c < 1 ? 1 : (int)c;
      end += (unsigned)((count + l.c[k] - 1) / l.c[k]);
      l.end[k] = end;
    }
  }
  __syncthreads();
}

// Calls body(list, rec, m) for the warp's chunks, rec its first record.
template <int N, typename Body>
__device__ __forceinline__ void for_chunks(const FusedArgs &f, const ChunkLists &l, const int (&hi)[N],
                                           unsigned *next, Body body) {
  const unsigned total = l.end[N - 1], nw = gridDim.x * kW;
  const int lane = threadIdx.x & 31;
  unsigned j = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  while (j < total) {
    unsigned after = 0;
    if (total > nw && lane == 0) after = nw + atomicAdd(next, 1u);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const unsigned start = k > 0 ? l.end[k > 0 ? k - 1 : 0] : 0u;
      if (j >= start && j < l.end[k]) {
        const int c = l.c[k];
        const int64_t from = f.off[l.lo[k]] + (int64_t)(j - start) * c, left = f.off[hi[k] + 1] - from;
        body(k, f.rec + from, (int)(left < c ? left : c));
      }
    }
    if (total <= nw) break;
    j = __shfl_sync(0xFFFFFFFFu, after, 0);
  }
}

// Rows for whole blocks, longest bins first: the hubs up to kRowMaxDeg edges
// and bins 8-7.  body must pass a block barrier.
template <typename Body>
__device__ __forceinline__ void block_rows(const FusedArgs &f, unsigned *next, Body body) {
  __shared__ unsigned s_next;
  const unsigned n = (unsigned)(f.off[kBins] - f.off[7]);
  const VRec *last = f.rec + f.off[kBins] - 1;
  for (unsigned i = blockIdx.x; i < n;) {
    __syncthreads();
    if (threadIdx.x == 0) s_next = n > gridDim.x ? gridDim.x + atomicAdd(next, 1u) : n;
    const VRec vr = last[-(int64_t)i];
    if (vr.deg <= kRowMaxDeg) body(vr);
    __syncthreads();
    i = s_next;
  }
}

// Rows for teams of kTeam threads (bins 6-5).
template <typename Body>
__device__ __forceinline__ void team_rows(const FusedArgs &f, unsigned *next, Body body) {
  constexpr int teams = kT / kTeam;
  __shared__ unsigned s_next[teams];
  const int team = threadIdx.x / kTeam;
  const unsigned n = (unsigned)(f.off[7] - f.off[5]);
  const VRec *last = f.rec + f.off[7] - 1;
  const unsigned nteams = gridDim.x * teams;
  for (unsigned i = team * gridDim.x + blockIdx.x; i < n;) {
    team_sync(team);
    if (threadIdx.x % kTeam == 0) s_next[team] = n > nteams ? nteams + atomicAdd(next, 1u) : n;
    body(last[-(int64_t)i]);
    team_sync(team);
    i = s_next[team];
  }
}

// Best (gain, cluster) and sum of S over `nw` warps' partials; every thread
// of them has called it, `first` combines.
struct RowPart {
  long long g[kW];
  int32_t x[kW], S[kW];
};

// Move step of one row of up to GS N edges by GS threads of rank r with
// `slots` table slots.
template <int GS, int N, typename Sync>
__device__ __forceinline__ void row_move(const PassArgs &a, const VRec &vr, SplitTab tab, uint32_t slots, int r,
                                         RowPart &part, Sync sync, MoveState &ms) {
  const int32_t v = vr.v;
  const int32_t Cv = LC_IDX(a.C[v], a.g.n, kDbgLabel);
  const GraphParam P = a.gp[vr.g];
  const long long muw = P.mu * vr.w;
  bool ok = true;
  int32_t slot[N];
  const int32_t self = claim_row<GS, N>(a, vr.beg, vr.deg, Cv, tab, slots, r, slot, ok);
  if (!ok) {
    a.sc->error = 1;
    LC_DBG_FAIL(kDbgProbe, v, a.g.n);
  }
  sync();
  long long gb = LLONG_MIN;
  int32_t xb = kNone;
  claim_argmax<N>(a, P.Lam, muw, tab, slot, gb, xb, ms.nX);
  warp_argmax(gb, xb);
  int32_t S = (int32_t)__reduce_add_sync(0xFFFFFFFFu, (unsigned)self);
  const int w0 = (threadIdx.x - r) >> 5;  // the row's first warp
  if ((threadIdx.x & 31) == 0) {
    part.g[threadIdx.x >> 5] = gb;
    part.x[threadIdx.x >> 5] = xb;
    part.S[threadIdx.x >> 5] = S;
  }
  sync();
  if (r == 0) {
    for (int w = 1; w < GS / 32; ++w) {
      S += part.S[w0 + w];
      if (better(part.g[w0 + w], part.x[w0 + w], gb, xb)) {
        gb = part.g[w0 + w];
        xb = part.x[w0 + w];
      }
    }
    const long long gC = gain_self(P, S, vr.w, a.W[Cv]);
    phi_add_one(a, ms.acc, vr.g, gC, ms.phi);
    decide(a, P, v, Cv, gC, xb, gb, ms);
  }
  // part is written again only after the next row's first sync
}

// First pass (singleton start) of one row by GS threads.
template <int GS, typename Sync>
__device__ __forceinline__ void row_first(const PassArgs &a, const VRec &vr, int r, RowPart &part, Sync sync,
                                          MoveState &ms) {
  const GraphParam P = a.gp[vr.g];
  const long long muw = P.mu * vr.w;
  long long gb = LLONG_MIN;
  int32_t xb = kNone;
#pragma unroll 4
  for (int64_t e = vr.beg + r; e < vr.beg + vr.deg; e += GS) first_edge(a, P.Lam, muw, e, gb, xb);
  warp_argmax(gb, xb);
  const int w0 = (threadIdx.x - r) >> 5;
  sync();  // the last row's partials have been read
  if ((threadIdx.x & 31) == 0) {
    part.g[threadIdx.x >> 5] = gb;
    part.x[threadIdx.x >> 5] = xb;
  }
  sync();
  if (r == 0) {
    for (int w = 1; w < GS / 32; ++w)
      if (better(part.g[w0 + w], part.x[w0 + w], gb, xb)) {
        gb = part.g[w0 + w];
        xb = part.x[w0 + w];
      }
    decide(a, P, vr.v, vr.v, 0, xb, gb, ms);
  }
}

// Sum of x over the block (every thread; the result in thread 0).
__device__ __forceinline__ long long block_total(long long x, long long *red) {
  x = warp_sum(x);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  if (threadIdx.x >= 32) return 0;
  return warp_sum(threadIdx.x < kW ? red[threadIdx.x] : 0ll);
}

// The chunks of the hubs above kRowMaxDeg edges.
template <typename Body>
__device__ __forceinline__ void big_chunks(const PassArgs &a, Body body) {
  for (int c = blockIdx.x; c < a.hub.Q; c += gridDim.x) {
    const int h = a.hub.hub_of[c];
    const int32_t v = a.hub.vtx[h];
    if (a.g.rp[v + 1] - a.g.rp[v] > kRowMaxDeg) body(c, h, v);
  }
}

// A barrier's wait ran out: labels that whatever follows may index with.  Not
// inlined at the barriers: that cost the passes 1 %.
__device__ __noinline__ void give_up(int32_t *C_out, int64_t n) {
  for (int64_t v = threadIdx.x; v < n; v += kT) C_out[v] = (int32_t)v;
}

__global__ void __launch_bounds__(kT, 1)
    k_passes(const __grid_constant__ PassArgs a, const __grid_constant__ FusedArgs f) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t *keys = reinterpret_cast<uint32_t *>(smem);
  int32_t *vals = reinterpret_cast<int32_t *>(keys + kRowSlots);
  Stage &stage = reinterpret_cast<Stage *>(vals + kRowSlots)[threadIdx.x >> 5];
  __shared__ RowPart part;
  __shared__ ChunkLists lists;
  __shared__ long long red[kW];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, team = threadIdx.x / kTeam;
  const SplitTab wtab{keys + wid * kWarpSlots, vals + wid * kWarpSlots};
  const SplitTab ttab{keys + team * kTeamSlots, vals + team * kTeamSlots};
  const SplitTab btab{keys, vals};
  auto bsync = [] { __syncthreads(); };
  auto tsync = [team] { team_sync(team); };
  const int64_t n = a.g.n;
  const int64_t tid = (int64_t)blockIdx.x * kT + threadIdx.x, nt = (int64_t)gridDim.x * kT;
  const int64_t wbase = tid - lane;  // whole-warp loops start here
  const int G = a.G;
  GridBarrier bar(a.sc);

  for (int s = threadIdx.x; s < kRowSlots; s += kT) {
    keys[s] = 0u;
    vals[s] = 0;
  }
  // clustering, cluster weights, accumulators of the call
  for (int64_t v = tid; v < n; v += nt) {
    if (f.singleton) {
      a.C[v] = (int32_t)v;
      f.C_out[v] = (int32_t)v;
      a.W[v] = a.g.vw[v];
    } else {
      a.W[v] = 0;
    }
  }
  for (int64_t g = tid; g < G; g += nt) {
    f.acc[g] = f.acc[G + g] = f.acc[2 * G + g] = 0;
    f.fin[g] = 0;
    f.best[g] = f.singleton ? 0 : LLONG_MIN;  // Phi(singletons) = 0
  }
  if (tid < 6) f.empties[tid] = 0;
  if (tid < 2 * kNextCount) f.next[tid] = 0;
  if (!bar.sync()) return give_up(f.C_out, n);
  if (!f.singleton) {
    for (int64_t v0 = wbase; v0 < n; v0 += nt) {
      const int64_t v = v0 + lane;
      add_weights(a.W, v < n, v < n ? a.C[v] : 0, v < n ? a.g.vw[v] : 0);
    }
    if (!bar.sync()) return give_up(f.C_out, n);
  }

  for (int i = 0; i < f.passes; ++i) {
    const bool first = f.singleton && i == 0, last = i + 1 == f.passes;
    long long *acc = f.acc + (int64_t)(i % 3) * G;       // Phi entering this pass
    const long long *best = f.best + (int64_t)(i & 1) * G;
    long long *best_next = f.best + (int64_t)((i & 1) ^ 1) * G;
    MoveState ms;
    ms.acc = acc;
    ms.num = f.phi[i][0];
    ms.den = f.phi[i][1];
    if (tid == 0) f.empties[(i + 1) % 3] = f.empties[3 + (i + 1) % 3] = 0;
    for (int64_t x = tid; x < n; x += nt) f.empty.used[x] = 0;

    // ------------------------------------------------------------ move
    unsigned *next = f.next + (i % 3) * 2 * kNextCount;
    if (tid < 2 * kNextCount) f.next[((i + 1) % 3) * 2 * kNextCount + tid] = 0;
    {
      if (first) {
        block_rows(f, next + kNextRow, [&](const VRec &vr) { row_first<kT>(a, vr, threadIdx.x, part, bsync, ms); });
        if (f.big)
          big_chunks(a, [&](int c, int h, int32_t v) {
            const GraphParam P = a.gp[graph_of(a, v)];
            const long long muw = P.mu * a.g.vw[v];
            long long gb = LLONG_MIN;
            int32_t xb = kNone;
            for (int64_t e = a.hub.e0[c] + threadIdx.x; e < a.hub.e1[c]; e += kT)
              first_edge(a, P.Lam, muw, e, gb, xb);
            Grp<kT>::argmax(gb, xb, part.g, part.x);
            if (threadIdx.x == 0) {
              a.hub.part_g[c] = gb;
              a.hub.part_x[c] = xb;
            }
            if (last_of_hub(a, h) && wid == 0) decide_hub(a, h, v, true, lane, ms);
          });
        constexpr int lo[4] = {5, 2, 1, 0}, hi[4] = {6, 4, 1, 0}, most[4] = {1, 8, 32, 32};
        plan_chunks(f, lists, lo, hi, most);
        for_chunks(f, lists, hi, next + kNextChunk, [&](int k, const VRec *rec, int m) {
          if (k <= 1)
            first_chunk<32>(a, rec, 0, m, stage.move.st, ms);
          else if (k == 2)
            first_chunk<16>(a, rec, 0, m, stage.move.st, ms);
          else if (lane < m)
            first_thread(a, rec, lane, ms);
        });
      } else {
        if (f.big) {
          // few chunks: a piece of one edge a thread each for the idle blocks,
          // whose table inserts would follow one another in a thread (R-MAT
          // scale 16, CPM 1/50: 6.19 / 5.71 ms a call; modularity on scales
          // 15 to 17 no difference)
          const int cut = gridDim.x >= 4u * (unsigned)a.hub.Q ? 4 : gridDim.x >= 2u * (unsigned)a.hub.Q ? 2 : 1;
          for (int j = blockIdx.x; j < a.hub.Q * cut; j += gridDim.x) {
            const int c = j / cut, h = a.hub.hub_of[c];
            const int32_t v = a.hub.vtx[h];
            if (a.g.rp[v + 1] - a.g.rp[v] <= kRowMaxDeg) continue;  // block-uniform
            const int64_t e0 = a.hub.e0[c], len = a.hub.e1[c] - e0, p = j % cut;
            const long long s =
                block_total(hub_insert<kT>(a, v, e0 + len * p / cut, e0 + len * (p + 1) / cut, stage.move.tags), red);
            if (threadIdx.x == 0 && s != 0) atomicAdd((unsigned long long *)&a.hub.acc[h], (unsigned long long)s);
          }
        }
        block_rows(f, next + kNextRow, [&](const VRec &vr) {
          row_move<kT, (int)(kRowMaxDeg / kT)>(a, vr, btab, kRowSlots, threadIdx.x, part, bsync, ms);
        });
        __syncthreads();
        team_rows(f, next + kNextTeam, [&](const VRec &vr) {
          row_move<kTeam, kTeamSlots / 2 / kTeam>(a, vr, ttab, kTeamSlots, threadIdx.x % kTeam, part, tsync, ms);
        });
        __syncthreads();  // the teams' tables are clean and their partials read
        constexpr int lo[4] = {3, 2, 1, 0}, hi[4] = {4, 2, 1, 0}, most[4] = {8, 32, 32, 32};
        plan_chunks(f, lists, lo, hi, most);
        for_chunks(f, lists, hi, next + kNextChunk, [&](int k, const VRec *rec, int m) {
          if (k == 0)
            warp_chunk(a, rec, 0, m, stage.move.st, wtab, kWarpSlots, ms);
          else if (k == 1)
            lanes_chunk<32, 4>(a, rec, 0, m, stage.move.st, stage.move.tags, ms);
          else if (k == 2)
            lanes_chunk<16, 4>(a, rec, 0, m, stage.move.st, stage.move.tags, ms);
          else
            move_thread(a, lane < m, rec, lane, ms);
        });
      }
      if (last)  // Q of W before the last update (see launch_final_objective)
        for (int64_t x0 = wbase; x0 < n; x0 += nt) {
          const int64_t x = x0 + lane;
          const int g = x < n ? graph_of(a, (int32_t)x) : -1;
          const unsigned long long W = x < n ? (unsigned long long)a.W[x] : 0ull;
          graph_add(f.fin, g, g >= 0 ? (long long)((unsigned long long)a.gp[g].mu * W * W) : 0ll);
        }
    }
    if (f.big && !first) {
      if (!bar.sync()) return give_up(f.C_out, n);
      big_chunks(a, [&](int c, int h, int32_t v) {
        const GraphParam P = a.gp[graph_of(a, v)];
        const int64_t beg = a.g.rp[v];
        long long gb = LLONG_MIN;
        int32_t xb = kNone;
        range_argmax<kT>(a, P.Lam, P.mu * a.g.vw[v], a.gtab + 2 * beg, (uint32_t)(2 * (a.hub.e0[c] - beg)),
                         (uint32_t)(2 * (a.hub.e1[c] - beg)), threadIdx.x, gb, xb, ms.nX);
        Grp<kT>::argmax(gb, xb, part.g, part.x);
        if (threadIdx.x == 0) {
          a.hub.part_g[c] = gb;
          a.hub.part_x[c] = xb;
        }
        if (last_of_hub(a, h) && wid == 0) decide_hub(a, h, v, false, lane, ms);
      });
    }
    {
      const int e = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)ms.empties);
      if (lane == 0 && e) atomicAdd(&f.empties[3 + i % 3], e);
    }
    if (!first && !a.gid) {
      const long long t = block_total(ms.phi, red);
      if (threadIdx.x == 0 && t != 0) atomicAdd((unsigned long long *)acc, (unsigned long long)t);
    }
    if (!bar.sync()) return give_up(f.C_out, n);

    // ---------------------------------------------------------- update
    // best-of test (Algorithm 2) on the state entering the pass: its labels
    // are in the records, which the moves below do not touch
    if (!first) {
      const bool all = !a.gid && acc[0] > best[0];
      if (a.gid || all)
        for (int64_t v = tid; v < n; v += nt) {
          const int g = graph_of(a, (int32_t)v);
          if (all || acc[g] > best[g]) f.C_out[v] = a.ab[v].C;
        }
    }
    for (int64_t g = tid; g < G; g += nt) {
      best_next[g] = !first && acc[g] > best[g] ? acc[g] : best[g];
      f.acc[(int64_t)((i + 1) % 3) * G + g] = 0;
    }
    UpdateSums us;
    // ids in use are marked if some candidate wants a new cluster (uniform)
    int32_t *used = f.empties[3 + i % 3] > 0 ? f.empty.used : nullptr;
    next += kNextCount;
    {
      if (f.big)
        big_chunks(a, [&](int c, int h, int32_t v) {
          const AbRec r = a.ab[v];
          const int64_t deg = a.g.rp[v + 1] - a.g.rp[v];
          if (r.D == kNone) {  // block-uniform
            if (wid == 0 && c == a.hub.c0[h]) apply_lanes(a, lane == 0, v, deg, r, a.g.vw[v], false, us, used);
            return;
          }
          const AbCtx ctx = ab_ctx(a, v, r, a.gp[graph_of(a, v)], 0, 0, a.g.vw[v]);
          const long long s = block_total(ab_edges<kT, 4>(a, ctx, a.hub.e0[c], a.hub.e1[c], threadIdx.x), red);
          if (threadIdx.x == 0 && s != 0)
            atomicAdd((unsigned long long *)&a.hub.acc[h], (unsigned long long)s);
          if (last_of_hub(a, h) && wid == 0) {
            long long t = 0;
            if (lane == 0) t = (long long)atomicExch((unsigned long long *)&a.hub.acc[h], 0ull);
            apply_lanes(a, lane == 0, v, deg, r, a.g.vw[v], lane == 0 && a.delta[v] + t >= 0, us, used);
          }
        });
      block_rows(f, next + kNextRow, [&](const VRec &vr) {
        const AbRec r = a.ab[vr.v];
        bool keep = false;
        if (r.D != kNone) {
          const AbCtx ctx = ab_ctx(a, vr.v, r, a.gp[vr.g], vr.beg, vr.deg, vr.w);
          const long long s = block_total(ab_edges<kT, 4>(a, ctx, vr.beg, vr.beg + vr.deg, threadIdx.x), red);
          keep = a.delta[vr.v] + s >= 0;  // thread 0's
        }
        if (wid == 0) apply_lanes(a, lane == 0, vr.v, vr.deg, r, vr.w, keep, us, used);
      });
      constexpr int lo[5] = {5, 3, 2, 1, 0}, hi[5] = {6, 4, 2, 1, 0}, most[5] = {1, 8, 32, 32, 32};
      plan_chunks(f, lists, lo, hi, most);
      for_chunks(f, lists, hi, next + kNextChunk, [&](int k, const VRec *rec, int m) {
        if (k <= 1)
          ab_chunk<32>(a, rec, 0, m, stage.ab, us, used);
        else if (k == 2)
          ab_chunk<8>(a, rec, 0, m, stage.ab, us, used);
        else if (k == 3)
          ab_chunk<4>(a, rec, 0, m, stage.ab, us, used);
        else
          ab_thread(a, lane < m, rec, lane, us, used);
      });
    }
    {
      const int e = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)us.empties);
      if (lane == 0 && e) atomicAdd(&f.empties[i % 3], e);
    }
    if (!bar.sync()) return give_up(f.C_out, n);
    const int total = f.empties[i % 3];
    if (total > 0) {  // uniform over the grid
      if (!assign_empty<kT>(a, f.empty, total, true, bar)) return give_up(f.C_out, n);
      if (!bar.sync()) return give_up(f.C_out, n);
    }
  }

  // ---------------------------------- objective of the final state
  // Phi' = Phi + Lam dIN - mu (Q' - Q), from the last pass's movers' rows
  // and W (lc_pass.cu, launch_final_objective); Q' - sum w^2 and Q - sum w^2
  // differ by the same constant, so W^2 alone is summed.
  const int p = f.passes;
  {
    long long dphi = 0;
    auto add = [&](int g, long long d) {  // one thread
      const long long x = a.gp[g].Lam * d;
      if (!a.gid)
        dphi += x;
      else if (x != 0)
        atomicAdd((unsigned long long *)&f.fin[g], (unsigned long long)x);
    };
    {
      const VRec *rec = f.rec + f.off[7];
      for (int64_t i = blockIdx.x; i < f.off[kBins] - f.off[7]; i += gridDim.x) {
        const VRec vr = rec[i];
        if (a.C[vr.v] == a.ab[vr.v].C) continue;  // not a mover
        const long long d = block_total(delta_in_edges<kT>(a, vr.v, vr.beg, vr.beg + vr.deg, threadIdx.x), red);
        if (threadIdx.x == 0) add(vr.g, d);
      }
    }
    constexpr int lo[3] = {5, 1, 0}, hi[3] = {6, 4, 0}, most[3] = {1, 8, 32};
    plan_chunks(f, lists, lo, hi, most);
    // the counters of the pass after the last were zeroed by it and not used
    for_chunks(f, lists, hi, f.next + (p % 3) * 2 * kNextCount, [&](int k, const VRec *rec, int m) {
      VRec vr{};
      bool mover = false;
      if (lane < m) {
        vr = rec[lane];
        mover = a.C[vr.v] != a.ab[vr.v].C;
      }
      if (k == 2) {
        if (mover) add(vr.g, delta_in_edges<1>(a, vr.v, vr.beg, vr.beg + vr.deg, 0));
        __syncwarp();
        return;
      }
      for (unsigned left = __ballot_sync(0xFFFFFFFFu, mover); left; left &= left - 1) {
        const int j = __ffs(left) - 1;
        const int32_t v = __shfl_sync(0xFFFFFFFFu, vr.v, j), deg = __shfl_sync(0xFFFFFFFFu, vr.deg, j);
        const int64_t beg = __shfl_sync(0xFFFFFFFFu, vr.beg, j);
        const long long d = warp_sum(delta_in_edges<32>(a, v, beg, beg + deg, lane));
        if (lane == j) add(vr.g, d);
      }
    });
    for (int64_t x0 = wbase; x0 < n; x0 += nt) {
      const int64_t x = x0 + lane;
      const int g = x < n ? graph_of(a, (int32_t)x) : -1;
      const unsigned long long W = x < n ? (unsigned long long)a.W[x] : 0ull;
      graph_add(f.fin, g, g >= 0 ? -(long long)((unsigned long long)a.gp[g].mu * W * W) : 0ll);
    }
    if (!a.gid) {
      const long long t = block_total(dphi, red);
      if (threadIdx.x == 0 && t != 0) atomicAdd((unsigned long long *)f.fin, (unsigned long long)t);
    }
  }
  if (!bar.sync()) return give_up(f.C_out, n);
  const long long *acc = f.acc + (int64_t)((p - 1) % 3) * G;
  const long long *best = f.best + (int64_t)(p & 1) * G;
  {
    const bool all = !a.gid && acc[0] + f.fin[0] > best[0];
    if (a.gid || all)
      for (int64_t v = tid; v < n; v += nt) {
        const int g = graph_of(a, (int32_t)v);
        if (all || acc[g] + f.fin[g] > best[g]) f.C_out[v] = a.C[v];
      }
  }
  for (int64_t g = tid; g < G; g += nt) {
    const long long now = acc[g] + f.fin[g];
    const long long out = now > best[g] ? now : best[g];
    a.phi_out[g] = out;
    if (a.gp[g].active) f.phi_final[g] = out;
  }
  bar.leave();
}

}  // namespace

void configure_fused() {
  cudaFuncSetAttribute(k_passes, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
}

int64_t fused_row_max() { return kRowMaxDeg; }

int launch_fused_passes(const PassArgs &a, const FusedArgs &f, cudaStream_t s) {
  int64_t blocks = level_grid(a.g.n, a.g.nnz);
  if (blocks > coop_blocks(a.coop)) blocks = coop_blocks(a.coop);
  PassArgs pa = a;
  FusedArgs fa = f;
  void *args[] = {&pa, &fa};
  cudaLaunchCooperativeKernel((const void *)k_passes, dim3((unsigned)blocks), dim3(kT), args, kSmemBytes, s);
  return 1;
}

}  // namespace lc
