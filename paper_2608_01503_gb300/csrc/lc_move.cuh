// lc_move.cuh — device code of a local-move pass (Algorithm 2 with the
// afterburner filter of Algorithm 3) below the kernels that launch it:
// gains of one vertex by a thread, a lane group, a warp or a block, the
// candidate test, the afterburner sum and the update.
//
// Warps and blocks work on chunks of up to 32 vertices of a degree bin: one
// lane loads each vertex (coalesced), the group then works through the
// chunk's rows, and at its end one lane per vertex decides it.  The
// per-vertex arithmetic (128-bit candidate test, 64-bit division of the
// epsilon bucket) thus runs on 32 lanes instead of one, and the vertices'
// loads are in flight together.
#pragma once

#include <climits>

#include "lc_group.cuh"
#include "lc_internal.cuh"
#include "lc_pass.cuh"

namespace lc {

// Graph of vertex v in a packed batch (one graph: 0).
__device__ __forceinline__ int graph_of(const PassArgs &a, int32_t v) { return a.gid ? a.gid[v] : 0; }

// Adds x to the objective of graph g (whole warps; lanes with on = false add
// nothing): one graph accumulates in a register that the kernel flushes once
// per block, a batch adds warp sums to the graph's accumulator.
__device__ __forceinline__ void phi_add(const PassArgs &a, long long *acc, bool on, int g, long long x,
                                        long long &phi) {
  if (!a.gid)
    phi += on ? x : 0;
  else
    graph_add(acc, on ? g : -1, x);
}
// The same from one thread of a block.
__device__ __forceinline__ void phi_add_one(const PassArgs &a, long long *acc, int g, long long x,
                                            long long &phi) {
  if (!a.gid)
    phi += x;
  else if (x != 0)
    atomicAdd((unsigned long long *)&acc[g], (unsigned long long)x);
}

// What a move step sums per thread, its temperature phi = num / den and the
// per-graph objective accumulator it adds to.
struct MoveState {
  long long *acc;
  int32_t num, den;
  long long cntL = 0, phi = 0, nX = 0;
  int empties = 0;  // candidates for a new empty cluster
};
__device__ __forceinline__ MoveState move_state(const PassArgs &a) {
  MoveState m;
  m.acc = a.phi_acc;
  m.num = a.phi_live ? a.phi_live[0] : a.phi_n;
  m.den = a.phi_live ? a.phi_live[1] : a.phi_d;
  return m;
}
__device__ __forceinline__ void flush_move(const PassArgs &a, const MoveState &m) {
  flush_block_sum(m.nX, &a.sc->distinct_x);
  flush_block_sum(m.cntL, &a.sc->count_L);
  flush_block_sum(m.phi, &m.acc[0]);
}

// ---------------------------------------------------- vertex decision

// Algorithm 2 for one vertex once g(v, C[v]) and the best other cluster
// (gbest, best) are known: the empty-cluster rule, the candidate test with
// temperature phi = phi_n / phi_d, delta_v and its epsilon bucket
// (Algorithm 3's priority).  Writes the record of every vertex.
__device__ __forceinline__ void decide(const PassArgs &a, const GraphParam &P, int32_t v, int32_t Cv,
                                       long long gC, int32_t best, long long gbest, MoveState &ms) {
  AbRec r;
  r.C = Cv;
  r.D = kNone;
  r.q = 0;
  if (P.active) {  // else: graph not moving at this level (finished coarsening earlier)
    if (gC < 0 && (best == kNone || gbest < 0)) {
      best = kEmpty;
      gbest = 0;
    }
    bool cand = best != kNone;
    if (gbest == (long long)(int32_t)gbest && gC == (long long)(int32_t)gC)  // the products fit 64 bits
      cand = cand && (long long)ms.den * (int32_t)gbest >= (long long)(ms.den - ms.num) * (int32_t)gC;
    else
      cand = cand && (__int128)ms.den * gbest >= (__int128)(ms.den - ms.num) * (__int128)gC;
    if (cand) {
      const long long delta = gbest - gC;
      r.D = best;
      r.q = eps_bucket(a.m, P.Lam, delta);
      a.delta[v] = delta;
      ms.cntL++;
      ms.empties += best == kEmpty;
    }
  }
  a.ab[v] = r;
}

// A chunk's vertices as the group that walks their rows needs them, and what
// it found: S(v, C[v]) and the best other cluster.
struct __align__(16) MoveCtx {
  int64_t beg;
  int32_t deg, Cv;
  long long Lam, muw;
};
struct __align__(16) MoveRes {
  long long g;
  int32_t x, S;  // S < 2^31: the exactness guard on the total edge weight
};
struct MoveStage {
  MoveCtx ctx[32];
  MoveRes res[32];
};

// One lane's vertex of a chunk.
struct ChunkLane {
  VRec vr;
  int32_t Cv;
  long long WC;
  GraphParam P;
};

// Loads vertex `lane` of the chunk and stages its context (full warp; first:
// the singleton start, where C[v] = v and W is not needed).
__device__ __forceinline__ ChunkLane stage_move(const PassArgs &a, const VRec *__restrict__ rec, int64_t base,
                                                int m, int lane, bool first, MoveCtx *ctx) {
  ChunkLane c{};
  if (lane < m) {
    c.vr = rec[base + lane];
    c.P = a.gp[c.vr.g];
    c.Cv = first ? c.vr.v : LC_IDX(a.C[c.vr.v], a.g.n, kDbgLabel);
    c.WC = first ? 0 : a.W[c.Cv];
    ctx[lane] = MoveCtx{c.vr.beg, c.vr.deg, c.Cv, c.P.Lam, c.P.mu * c.vr.w};
  }
  return c;
}

// Decides the chunk's vertices from the staged results (full warp).
__device__ __forceinline__ void settle_move(const PassArgs &a, const ChunkLane &c, int m, int lane, bool first,
                                            const MoveRes *res, MoveState &ms) {
  const bool on = lane < m;
  const MoveRes r = on ? res[lane] : MoveRes{0, kNone, 0};
  const long long gC = first ? 0 : gain_self(c.P, r.S, c.vr.w, c.WC);
  if (!first) phi_add(a, ms.acc, on, c.vr.g, gC, ms.phi);
  if (on) decide(a, c.P, c.vr.v, c.Cv, gC, r.x, r.g, ms);
}

// ------------------------------------------- first pass (Section IV-A-3)

// Singleton start: the adjacent clusters of v are its neighbours, so the
// gains are read straight from the CSR: g(v,{u}) = Lam*w(u,v) - mu*w(v)*w(u),
// and g(v, C[v]) = 0.
__device__ __forceinline__ void first_edge(const PassArgs &a, long long Lam, long long muw, int64_t e,
                                           long long &gb, int32_t &xb) {
  const int32_t u = LC_IDX(__ldg(a.g.col + e), a.g.n, kDbgColumn);
  const long long g = Lam * (long long)__ldg(a.g.ew + e) - muw * __ldg(a.g.vw + u);
  if (better(g, u, gb, xb)) {
    gb = g;
    xb = u;
  }
}

// Argmax over a lane group or a warp; every lane gets it.
template <int G>
__device__ __forceinline__ void lanes_argmax(long long &g, int32_t &x) {
  if constexpr (G == 32)
    warp_argmax(g, x);
  else
    group_argmax<G>(g, x);
}

template <int G>
__device__ __forceinline__ void first_chunk(const PassArgs &a, const VRec *__restrict__ rec, int64_t base, int m,
                                            MoveStage &st, MoveState &ms) {
  constexpr int V = 32 / G;
  const int lane = threadIdx.x & 31, grp = lane / G, sub = lane & (G - 1);
  const ChunkLane c = stage_move(a, rec, base, m, lane, true, st.ctx);
  __syncwarp();
  for (int k = 0; k < m; k += V) {
    const int idx = k + grp;
    long long gb = LLONG_MIN;
    int32_t xb = kNone;
    if (idx < m) {
      const MoveCtx x = st.ctx[idx];
#pragma unroll 4
      for (int64_t e = x.beg + sub; e < x.beg + x.deg; e += G) first_edge(a, x.Lam, x.muw, e, gb, xb);
    }
    __syncwarp();
    lanes_argmax<G>(gb, xb);
    if (idx < m && sub == 0) st.res[idx] = MoveRes{gb, xb, 0};
  }
  __syncwarp();
  settle_move(a, c, m, lane, true, st.res, ms);
  __syncwarp();
}

// ----------------------------------- aggregation + argmax, bin 0 (thread)

// One thread per vertex of degree <= 8: neighbour clusters and weights are
// held in registers; S(v, X) for each distinct X is an unrolled compare-sum.
// Returns S(v, C[v]).
__device__ __forceinline__ long long thread_gains(const PassArgs &a, const VRec &vr, int32_t Cv,
                                                  const GraphParam &P, long long &gb, int32_t &xb,
                                                  long long &nX) {
  constexpr int K = 8;
  const int64_t beg = vr.beg;
  const int deg = vr.deg;
  int32_t u[K], w[K], X[K];
#pragma unroll
  for (int j = 0; j < K; ++j) {
    u[j] = 0;
    w[j] = 0;
    if (j < deg) {
      u[j] = LC_IDX(__ldg(a.g.col + beg + j), a.g.n, kDbgColumn);
      w[j] = __ldg(a.g.ew + beg + j);
    }
  }
#pragma unroll
  for (int j = 0; j < K; ++j) X[j] = j < deg ? LC_IDX(a.C[u[j]], a.g.n, kDbgLabel) : -1;
  long long WX[K];
#pragma unroll
  for (int j = 0; j < K; ++j) WX[j] = (j < deg && X[j] != Cv) ? a.W[X[j]] : 0;
  long long self = 0;
  gb = LLONG_MIN;
  xb = kNone;
#pragma unroll
  for (int j = 0; j < K; ++j) {
    if (j >= deg) continue;
    if (X[j] == Cv) {
      self += w[j];
      continue;
    }
    bool first = true;
    int32_t S = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (X[k] == X[j]) {  // never past the row: -1 there
        S += w[k];
        if (k < j) first = false;
      }
    }
    if (first) {
      nX++;
      const long long g = gain_other(P, S, vr.w, WX[j]);
      if (better(g, X[j], gb, xb)) {
        gb = g;
        xb = X[j];
      }
    }
  }
  return self;
}

// Bin 0: one thread per vertex (full warp, lanes with on = false idle).
__device__ __forceinline__ void move_thread(const PassArgs &a, bool on, const VRec *__restrict__ rec, int64_t i,
                                            MoveState &ms) {
  VRec vr{};
  long long gC = 0;
  if (on) {
    vr = rec[i];
    const int32_t Cv = LC_IDX(a.C[vr.v], a.g.n, kDbgLabel);
    const GraphParam P = a.gp[vr.g];
    const long long WC = a.W[Cv];
    long long gb;
    int32_t xb;
    const long long self = thread_gains(a, vr, Cv, P, gb, xb, ms.nX);
    gC = gain_self(P, self, vr.w, WC);
    decide(a, P, vr.v, Cv, gC, xb, gb, ms);
  }
  phi_add(a, ms.acc, on, vr.g, gC, ms.phi);
}

__device__ __forceinline__ void first_thread(const PassArgs &a, const VRec *__restrict__ rec, int64_t i,
                                             MoveState &ms) {
  const VRec vr = rec[i];
  const GraphParam P = a.gp[vr.g];
  long long gb = LLONG_MIN;
  int32_t xb = kNone;
#pragma unroll 4
  for (int64_t e = vr.beg; e < vr.beg + vr.deg; ++e) first_edge(a, P.Lam, P.mu * vr.w, e, gb, xb);
  decide(a, P, vr.v, vr.v, 0, xb, gb, ms);
}

// ------------------------------------ aggregation + argmax, bins 1-2 (lanes)

// Shared scratch of a warp whose lanes hold one neighbour each: 1,024 byte
// tags and one sum per lane.
constexpr int kTagSlots = 1024;
struct LaneTags {
  uint8_t tag[kTagSlots];
  int32_t acc[32];
};

// Each lane holds one neighbour's cluster X.  The lanes of a group that hold
// the same X agree on a leader through the tag table: every undecided lane
// writes its number to the slot X hashes to and reads back whose survived; a
// lane whose X equals the survivor's has found its leader, the others hash
// again.  Equal X share the slot, so they are settled together, and a slot's
// survivor settles itself, so rounds end; the table is never cleared, since
// only slots written in the round are read.  This replaces __match_any_sync,
// which takes about two clocks per distinct value: 64 clocks per warp and SM
// for 32 distinct clusters against about 15 for the usual one or two rounds.
// Returns the sum of w over the lanes of the same X in its leader (leader ==
// lane); lanes with on = false have no part.
template <int G>
__device__ __forceinline__ int32_t lane_sums(LaneTags &t, int lane, bool on, int32_t X, int32_t w, int &leader) {
  constexpr unsigned full = 0xFFFFFFFFu;
  constexpr uint32_t slots = kTagSlots / (32 / G);  // a group's own part of the table
  const uint32_t off = (uint32_t)(lane / G) * slots;
  leader = lane;
  bool pend = on;
  uint32_t h = (uint32_t)X * 0x9E3779B1u;
  do {
    const uint32_t s = off + (h >> 16) % slots;
    if (pend) t.tag[s] = (uint8_t)lane;
    __syncwarp();
    const int who = pend ? (int)t.tag[s] : lane;
    const int32_t Xw = __shfl_sync(full, X, who);
    if (pend && Xw == X) {
      leader = who;
      pend = false;
    }
    h = (h ^ (h >> 15)) * 0x85EBCA6Bu;
    __syncwarp();  // every read of this round before the next round's writes
  } while (__any_sync(full, pend));
  const bool dup = on && leader != lane;
  if (!__any_sync(full, dup)) return w;
  t.acc[lane] = w;
  __syncwarp();
  if (dup) atomicAdd(&t.acc[leader], w);
  __syncwarp();
  const int32_t S = t.acc[lane];
  __syncwarp();
  return S;
}

// A step takes the rows of U (G = 32) or 2 U (G = 16) vertices: their label
// gathers are issued together, then their W gathers, while the next
// step's columns and weights are on their way.
template <int G, int U = 2>
__device__ __forceinline__ void lanes_chunk(const PassArgs &a, const VRec *__restrict__ rec, int64_t base, int m,
                                            MoveStage &st, LaneTags &tags, MoveState &ms) {
  constexpr int V = 32 / G;
  const int lane = threadIdx.x & 31, grp = lane / G, sub = lane & (G - 1);
  const ChunkLane c = stage_move(a, rec, base, m, lane, false, st.ctx);
  __syncwarp();
  auto load = [&](int idx, int32_t &u, int32_t &w) {
    u = -1;
    w = 0;
    if (idx < m && sub < st.ctx[idx].deg) {
      const int64_t e = st.ctx[idx].beg + sub;
      u = LC_IDX(__ldg(a.g.col + e), a.g.n, kDbgColumn);
      w = __ldg(a.g.ew + e);
    }
  };
  int32_t u[U], w[U];
#pragma unroll
  for (int j = 0; j < U; ++j) load(j * V + grp, u[j], w[j]);
  for (int k = 0; k < m; k += U * V) {
    int32_t X[U], wk[U];
    long long WX[U];
    bool other[U], self[U];
#pragma unroll
    for (int j = 0; j < U; ++j) X[j] = u[j] >= 0 ? LC_IDX(a.C[u[j]], a.g.n, kDbgLabel) : -1;
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int idx = k + j * V + grp;
      const int32_t Cv = idx < m ? st.ctx[idx].Cv : -2;
      self[j] = u[j] >= 0 && X[j] == Cv;
      other[j] = u[j] >= 0 && !self[j];
      wk[j] = w[j];
    }
#pragma unroll
    for (int j = 0; j < U; ++j) load(k + (U + j) * V + grp, u[j], w[j]);
#pragma unroll
    for (int j = 0; j < U; ++j) WX[j] = other[j] ? a.W[X[j]] : 0;
#pragma unroll
    for (int j = 0; j < U; ++j) {
      if (k + j * V >= m) break;  // uniform
      const int idx = k + j * V + grp;
      int32_t S_self;
      if constexpr (G == 32)
        S_self = (int32_t)__reduce_add_sync(0xFFFFFFFFu, (unsigned)(self[j] ? wk[j] : 0));
      else
        S_self = group_sum<G>(self[j] ? wk[j] : 0);
      int leader;
      const int32_t S = lane_sums<G>(tags, lane, other[j], X[j], wk[j], leader);
      long long g = LLONG_MIN;
      int32_t xb = kNone;
      if (other[j] && leader == lane) {
        g = st.ctx[idx].Lam * (long long)S - st.ctx[idx].muw * WX[j];
        xb = X[j];
        ms.nX++;
      }
      lanes_argmax<G>(g, xb);
      if (idx < m && sub == 0) st.res[idx] = MoveRes{g, xb, S_self};
    }
  }
  __syncwarp();
  settle_move(a, c, m, lane, false, st.res, ms);
  __syncwarp();
}

// ------------------------------------ shared-table aggregation, bins 3-5

// Shared tables stay clean between vertices: a vertex's argmax resets the
// slots it used.
// Best (gain, cluster) over slots [s0, s1) of a table (strided by GS),
// resetting the slots it reads unless `keep` (a kept table being built).
// g(v, X) = Lam S(v, X) - (mu w(v)) W(X), with mu w(v) formed once.
template <int GS>
__device__ __forceinline__ void range_argmax(const PassArgs &a, long long Lam, long long muw,
                                             unsigned long long *tab, uint32_t s0, uint32_t s1,
                                             int r, long long &gb, int32_t &xb,
                                             long long &nX, bool keep = false) {
  constexpr int U = 4;
  for (uint32_t base = s0 + r; base < s1; base += GS * U) {
    unsigned long long t[U];
    long long WX[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const uint32_t s = base + k * GS;
      t[k] = s < s1 ? tab[s] : kEmptySlot;
      if (t[k] != kEmptySlot && !keep) tab[s] = kEmptySlot;
    }
#pragma unroll
    for (int k = 0; k < U; ++k) WX[k] = t[k] != kEmptySlot ? a.W[LC_IDX(slot_key(t[k]), a.g.n, kDbgLabel)] : 0;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (t[k] == kEmptySlot) continue;
      nX++;
      const int32_t X = slot_key(t[k]);
      const long long g = Lam * (long long)slot_val(t[k]) - muw * WX[k];
      if (better(g, X, gb, xb)) {
        gb = g;
        xb = X;
      }
    }
  }
}

// ------------------------------ split shared tables (warp and block bins)

// A shared table kept as two 32-bit arrays: key[s] (0 = empty, else the
// cluster id + 1) and val[s] (the weight sum S(v, X)).  Claiming a slot is
// a 32-bit CAS on the key and every edge then adds its weight with a 32-bit
// atomic add, which shared memory executes far faster than 64-bit CAS.
struct SplitTab {
  uint32_t *key;
  int32_t *val;
};

// Sequential probing from slot s for cluster X (tag = X + 1).
__device__ __forceinline__ bool split_probe(SplitTab t, uint32_t cap, uint32_t tag, int32_t w,
                                            uint32_t s) {
  for (uint32_t probe = 0; probe < cap; ++probe) {
    uint32_t k = t.key[s];
    if (k == 0u) k = atomicCAS(&t.key[s], 0u, tag);
    if (k == 0u || k == tag) {
      atomicAdd(&t.val[s], w);
      return true;
    }
    s = (s + 1 == cap) ? 0 : s + 1;
  }
  return false;
}

// Adds (X[k], w[k]) for every k with todo[k]: the first probe of all U
// entries is read at once; a slot holding the key takes the weight, an
// empty one is claimed by CAS (a CAS that finds the key takes it too), and
// only a slot holding another key falls back to sequential probing.
template <int U>
__device__ __forceinline__ void split_add_batch(SplitTab t, uint32_t cap, const int32_t (&X)[U],
                                                const int32_t (&w)[U], const bool (&todo)[U],
                                                bool &ok) {
  uint32_t sl[U], cur[U];
#pragma unroll
  for (int k = 0; k < U; ++k) {
    sl[k] = todo[k] ? slot_of(X[k], cap) : 0;
    cur[k] = todo[k] ? t.key[sl[k]] : 0;
  }
#pragma unroll
  for (int k = 0; k < U; ++k)
    if (todo[k] && cur[k] == 0u) cur[k] = atomicCAS(&t.key[sl[k]], 0u, (uint32_t)X[k] + 1u);
#pragma unroll
  for (int k = 0; k < U; ++k) {
    if (!todo[k]) continue;
    const uint32_t tag = (uint32_t)X[k] + 1u;
    if (cur[k] == 0u || cur[k] == tag)
      atomicAdd(&t.val[sl[k]], w[k]);
    else
      ok &= split_probe(t, cap, tag, w[k], sl[k] + 1 == cap ? 0 : sl[k] + 1);
  }
}

// Inserts edges [beg, end) of v (strided by GS, U edges per thread at a
// time).  Returns this thread's part of S(v, C[v]).  Indices are
// row-relative 32-bit (a row has fewer than 2^31 entries).
template <int GS, int U>
__device__ __forceinline__ long long split_insert_row(const PassArgs &a, int64_t beg, int64_t end,
                                                      int32_t Cv, SplitTab t, uint32_t cap, int r,
                                                      bool &ok) {
  const int32_t *__restrict__ col = a.g.col + beg;
  const int32_t *__restrict__ ew = a.g.ew + beg;
  const int deg = (int)(end - beg);
  long long self = 0;
  for (int base = r; base < deg; base += GS * U) {
    int32_t u[U], w[U], X[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int e = base + k * GS;
      u[k] = -1;
      w[k] = 0;
      if (e < deg) {
        u[k] = LC_IDX(__ldg(col + e), a.g.n, kDbgColumn);
        w[k] = __ldg(ew + e);
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) X[k] = u[k] >= 0 ? LC_IDX(a.C[u[k]], a.g.n, kDbgLabel) : -1;
    bool todo[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      todo[k] = u[k] >= 0 && X[k] != Cv;
      if (u[k] >= 0 && X[k] == Cv) self += w[k];
    }
    split_add_batch<U>(t, cap, X, w, todo, ok);
  }
  return self;
}

// Best (gain, cluster) over slots [0, cap) (strided by GS), resetting the
// occupied ones.  g(v, X) = Lam S(v, X) - (mu w(v)) W(X).  Every slot is also
// copied to the kept table gt (same layout, empties included).
template <int GS>
__device__ __forceinline__ void split_argmax(const PassArgs &a, long long Lam, long long muw, SplitTab t,
                                             uint32_t cap, int r, long long &gb, int32_t &xb,
                                             unsigned long long *gt, long long &nX) {
  constexpr int U = 4;
  for (uint32_t base = r; base < cap; base += GS * U) {
    uint32_t key[U];
    int32_t S[U];
    long long WX[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const uint32_t s = base + k * GS;
      key[k] = s < cap ? t.key[s] : 0u;
      S[k] = 0;
      if (key[k] != 0u) {
        S[k] = t.val[s];
        t.key[s] = 0u;
        t.val[s] = 0;
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const uint32_t s = base + k * GS;
      if (s < cap) gt[s] = key[k] != 0u ? ((unsigned long long)key[k] << 32) | (uint32_t)S[k] : kEmptySlot;
    }
#pragma unroll
    for (int k = 0; k < U; ++k) WX[k] = key[k] != 0u ? a.W[LC_IDX(key[k] - 1u, a.g.n, kDbgLabel)] : 0;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (key[k] == 0u) continue;
      nX++;
      const int32_t X = (int32_t)(key[k] - 1u);
      const long long g = Lam * (long long)S[k] - muw * WX[k];
      if (better(g, X, gb, xb)) {
        gb = g;
        xb = X;
      }
    }
  }
}

// ------------------------------------------------- claimed slots
//
// A thread remembers the slots its own edges claimed, so the argmax reads
// and resets exactly the occupied slots and never scans the table: in passes
// from singletons it saves the walk over the empty half, in uncoarsening,
// where a row falls into a few clusters, nearly all of it, and the table may
// be as sparse as shared memory allows (fewer probes).  N: edges per thread
// at most, four at a time.
template <int GS, int N>
__device__ __forceinline__ int32_t claim_row(const PassArgs &a, int64_t beg, int deg, int32_t Cv, SplitTab t,
                                             uint32_t cap, int r, int32_t (&slot)[N], bool &ok) {
  constexpr int U = 4;
  const int32_t *__restrict__ col = a.g.col + beg;
  const int32_t *__restrict__ ew = a.g.ew + beg;
  int32_t self = 0;
#pragma unroll
  for (int b = 0; b < N; b += U) {
    int32_t u[U], w[U], X[U];
    uint32_t cur[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int e = r + (b + k) * GS;
      u[k] = -1;
      w[k] = 0;
      if (e < deg) {
        u[k] = LC_IDX(__ldg(col + e), a.g.n, kDbgColumn);
        w[k] = __ldg(ew + e);
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) X[k] = u[k] >= 0 ? LC_IDX(a.C[u[k]], a.g.n, kDbgLabel) : -1;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (u[k] >= 0 && X[k] == Cv) {
        self += w[k];
        X[k] = -1;
      }
      slot[b + k] = X[k] >= 0 ? (int32_t)slot_of(X[k], cap) : -1;
      cur[k] = X[k] >= 0 ? t.key[slot[b + k]] : 1u;
    }
#pragma unroll
    for (int k = 0; k < U; ++k)
      if (cur[k] == 0u) cur[k] = atomicCAS(&t.key[slot[b + k]], 0u, (uint32_t)X[k] + 1u);
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (X[k] < 0) continue;
      const uint32_t tag = (uint32_t)X[k] + 1u;
      uint32_t s = (uint32_t)slot[b + k];
      if (cur[k] != 0u && cur[k] != tag) {  // another key's slot: probe on
        uint32_t probe = 1;
        do {
          s = s + 1 == cap ? 0 : s + 1;
          cur[k] = t.key[s];
          if (cur[k] == 0u) cur[k] = atomicCAS(&t.key[s], 0u, tag);
        } while (cur[k] != 0u && cur[k] != tag && ++probe < cap);
        if (cur[k] != 0u && cur[k] != tag) {
          ok = false;
          slot[b + k] = -1;
          continue;
        }
      }
      atomicAdd(&t.val[s], w[k]);
      slot[b + k] = cur[k] == 0u ? (int32_t)s : -1;  // claimed by this edge, or not
    }
  }
  return self;
}

// Best (gain, cluster) over the thread's claimed slots, which it resets.
template <int N>
__device__ __forceinline__ void claim_argmax(const PassArgs &a, long long Lam, long long muw, SplitTab t,
                                             const int32_t (&slot)[N], long long &gb, int32_t &xb,
                                             long long &nX) {
  constexpr int U = 4;
#pragma unroll
  for (int b = 0; b < N; b += U) {
    int32_t X[U], S[U];
    long long WX[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      X[k] = -1;
      S[k] = 0;
      if (slot[b + k] >= 0) {
        X[k] = (int32_t)(t.key[slot[b + k]] - 1u);
        S[k] = t.val[slot[b + k]];
        t.key[slot[b + k]] = 0u;
        t.val[slot[b + k]] = 0;
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) WX[k] = X[k] >= 0 ? a.W[LC_IDX(X[k], a.g.n, kDbgLabel)] : 0;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (X[k] < 0) continue;
      nX++;
      const long long g = Lam * (long long)S[k] - muw * WX[k];
      if (better(g, X[k], gb, xb)) {
        gb = g;
        xb = X[k];
      }
    }
  }
}

// One row of up to 32 N edges by a warp.
template <int N>
__device__ __forceinline__ MoveRes warp_row(const PassArgs &a, const MoveCtx &x, int32_t v, SplitTab tab, uint32_t cap,
                                            int lane, MoveState &ms) {
  int32_t slot[N];
  bool ok = true;
  const int32_t self = claim_row<32, N>(a, x.beg, x.deg, x.Cv, tab, cap, lane, slot, ok);
  if (!ok) {
    a.sc->error = 1;
    LC_DBG_FAIL(kDbgProbe, v, a.g.n);
  }
  __syncwarp();
  long long gb = LLONG_MIN;
  int32_t xb = kNone;
  claim_argmax<N>(a, x.Lam, x.muw, tab, slot, gb, xb, ms.nX);
  warp_argmax(gb, xb);
  const int32_t S = (int32_t)__reduce_add_sync(0xFFFFFFFFu, (unsigned)self);
  return MoveRes{gb, xb, S};
}

// Bins 3-4: a warp's chunk, one row after the other in its own shared table
// of `cap` slots (at least 512).
__device__ __forceinline__ void warp_chunk(const PassArgs &a, const VRec *__restrict__ rec, int64_t base, int m,
                                           MoveStage &st, SplitTab tab, uint32_t cap, MoveState &ms) {
  const int lane = threadIdx.x & 31;
  const ChunkLane c = stage_move(a, rec, base, m, lane, false, st.ctx);
  __syncwarp();
  for (int k = 0; k < m; ++k) {
    const MoveCtx x = st.ctx[k];
    const MoveRes r = x.deg <= 128 ? warp_row<4>(a, x, (int32_t)(base + k), tab, cap, lane, ms)
                                   : warp_row<8>(a, x, (int32_t)(base + k), tab, cap, lane, ms);
    if (lane == 0) st.res[k] = r;
    __syncwarp();
  }
  settle_move(a, c, m, lane, false, st.res, ms);
  __syncwarp();
}

// Inserts edges [e0, e1) of hub v into its global table (GS threads, tg: this
// warp's tags); returns this thread's part of S(v, C[v]).
template <int GS>
__device__ __forceinline__ long long hub_insert(const PassArgs &a, int32_t v, int64_t e0, int64_t e1, LaneTags &tg) {
  constexpr int U = 4;
  const int64_t beg = a.g.rp[v], end = a.g.rp[v + 1];
  const int32_t Cv = LC_IDX(a.C[v], a.g.n, kDbgLabel);
  unsigned long long *tab = a.gtab + 2 * beg;
  const uint32_t cap = (uint32_t)(2 * (end - beg));
  const int lane = threadIdx.x & 31;
  long long self = 0;
  bool ok = true;
  for (int64_t base = e0; base < e1; base += GS * U) {
    int32_t u[U], w[U], X[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int64_t e = base + k * GS + threadIdx.x;
      u[k] = -1;
      w[k] = 0;
      if (e < e1) {
        u[k] = LC_IDX(__ldg(a.g.col + e), a.g.n, kDbgColumn);
        w[k] = __ldg(a.g.ew + e);
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) X[k] = u[k] >= 0 ? LC_IDX(a.C[u[k]], a.g.n, kDbgLabel) : -1;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (base + k * GS >= e1) break;  // uniform
      const bool other = u[k] >= 0 && X[k] != Cv;
      if (u[k] >= 0 && X[k] == Cv) self += w[k];
      int leader;
      const int32_t S = lane_sums<32>(tg, lane, other, X[k], w[k], leader);
      if (other && lane == leader) {
        bool fresh = false;
        ok &= table_add(tab, cap, X[k], S, fresh);
      }
    }
  }
  if (!ok) {
    a.sc->error = 1;
    LC_DBG_FAIL(kDbgProbe, v, a.g.n);
  }
  return self;
}

// Whether this block is the last of the chunks of hub h to get here (whole
// block; thread 0's earlier stores and atomics are then visible to the last
// one's L2 reads).  It leaves the counter at zero for the next use.
__device__ __forceinline__ bool last_of_hub(const PassArgs &a, int h) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    const int n = a.hub.c0[h + 1] - a.hub.c0[h];
    s_last = 1;  // of one chunk: what thread 0 stored, it reads itself
    if (n > 1) {
      __threadfence();
      s_last = atomicAdd(&a.hub.done[h], 1) == n - 1;
      if (s_last) {
        a.hub.done[h] = 0;
        __threadfence();
      }
    }
  }
  __syncthreads();
  return s_last != 0;
}

// Takes the sum of hub h's chunks and leaves zero.
__device__ __forceinline__ long long take_hub_acc(const PassArgs &a, int h) {
  return (long long)atomicExch((unsigned long long *)&a.hub.acc[h], 0ull);
}

// The decision for hub h from its chunks' partials (one warp of the last
// block of the hub; first: from singletons, S(v, C[v]) = 0).  Lane 0 returns
// S(v, C[v]).
__device__ __forceinline__ long long decide_hub(const PassArgs &a, int h, int32_t v, bool first, int lane,
                                                MoveState &ms) {
  long long gb = LLONG_MIN, gC = 0, self = 0;
  int32_t xb = kNone;
  for (int c = a.hub.c0[h] + lane; c < a.hub.c0[h + 1]; c += 32) {
    const long long pg = __ldcg(a.hub.part_g + c);
    const int32_t px = __ldcg(a.hub.part_x + c);
    if (better(pg, px, gb, xb)) {
      gb = pg;
      xb = px;
    }
  }
  warp_argmax(gb, xb);
  if (lane == 0) {
    const int g = graph_of(a, v);
    const GraphParam P = a.gp[g];
    const int32_t Cv = a.C[v];
    if (!first) {
      self = take_hub_acc(a, h);
      gC = gain_self(P, self, a.g.vw[v], a.W[Cv]);
      phi_add_one(a, ms.acc, g, gC, ms.phi);
    }
    decide(a, P, v, Cv, gC, xb, gb, ms);
  }
  return self;
}

// ------------------------------------------------ afterburner (Algorithm 3)

// What a candidate's row walk needs, staged per chunk.
struct __align__(16) AbCtx {
  int64_t beg;
  long long qv, muw, Lam;
  int32_t deg, v, Cv, Dv;
  int32_t vbase;
  uint32_t hv;  // the hash takes the id within the vertex's own graph
};

__device__ __forceinline__ AbCtx ab_ctx(const PassArgs &a, int32_t v, const AbRec &r, const GraphParam &P, int64_t beg,
                                        int32_t deg, long long wv) {
  AbCtx c;
  c.beg = beg;
  c.deg = deg;
  c.v = v;
  c.Cv = r.C;
  c.Dv = r.D;
  c.qv = r.q;
  c.muw = P.mu * wv;
  c.Lam = P.Lam;
  c.vbase = P.vbase;
  c.hv = fmix32((uint32_t)(v - P.vbase) ^ a.m.seed);
  return c;
}

// Sum over edges [e0, e1) (strided by GS, loads batched U at a time) of the
// change of v's two gains when an adjacent candidate u that precedes v moves
// from C[u] to D[u] (Algorithm 3's four rules).  A global gather costs one
// clock per lane and SM whatever its size (measured: 32 clocks per warp for
// 4, 8 and 16 bytes alike), so a neighbour's C and D come in one, and its q
// and w(u) follow only where u's move touches C[v] or D[v] (and, for w(u),
// precedes v).  q from the first gather would hold two more registers per
// edge in flight, which cost spills: 100,000-vertex SBM 4.41 / 3.94 ms with
// / without.
template <int GS, int U>
__device__ __forceinline__ long long ab_edges(const PassArgs &a, const AbCtx &c, int64_t e0, int64_t e1, int r) {
  long long d = 0;
  const int32_t *__restrict__ col = a.g.col + e0;
  const int32_t *__restrict__ ew = a.g.ew + e0;
  const int len = (int)(e1 - e0);
  const long long muw = c.muw;
  for (int base = r; base < len; base += GS * U) {
    int32_t u[U], w[U], s[U];
    int2 cd[U];  // the record's C and D; its q only where they matter
    long long q[U], wu[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int e = base + k * GS;
      u[k] = -1;
      w[k] = 0;
      if (e < len) {
        u[k] = LC_IDX(__ldg(col + e), a.g.n, kDbgColumn);
        w[k] = __ldg(ew + e);
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      cd[k] = make_int2(0, kNone);
      if (u[k] >= 0) cd[k] = *reinterpret_cast<const int2 *>(&a.ab[u[k]].C);
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int32_t Cu = cd[k].x, Du = cd[k].y;
      s[k] = 0;
      if (Du != kNone)
        s[k] = (c.Cv == Cu ? 1 : c.Dv == Cu ? -1 : 0) + (c.Cv == Du ? -1 : (c.Dv >= 0 && c.Dv == Du) ? 1 : 0);
      q[k] = s[k] != 0 ? a.ab[u[k]].q : 0;
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      wu[k] = 0;
      if (s[k] == 0) continue;
      if (!(q[k] != c.qv ? q[k] > c.qv
                         : earlier(q[k], fmix32((uint32_t)(u[k] - c.vbase) ^ a.m.seed), u[k], c.qv, c.hv, c.v)))
        s[k] = 0;
      if (s[k] != 0) wu[k] = a.g.vw[u[k]];
    }
#pragma unroll
    for (int k = 0; k < U; ++k) d += (long long)s[k] * (c.Lam * (long long)w[k] - muw * wu[k]);
  }
  return d;
}

// ----------------------------------------------------------- update

// What the update step sums per thread.
struct UpdateSums {
  long long moved = 0, cand = 0;
  int empties = 0;
};
__device__ __forceinline__ void flush_update(const PassArgs &a, const UpdateSums &u) {
  flush_block_sum(u.moved, &a.sc->count_M);
  flush_block_sum(u.cand, &a.sc->cand_edges);
  const int e = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)u.empties);
  if ((threadIdx.x & 31) == 0 && e) atomicAdd(&a.sc->empty_movers, e);
}

// W[X[lane]] += w[lane] over the lanes with on (full warp).  Many movers of
// a warp often join the same cluster (a hub's), and atomics on one address
// are served one after the other: the lanes that share the first two such
// clusters are summed first.
__device__ __forceinline__ void add_weights(int64_t *W, bool on, int32_t X, long long w) {
  constexpr unsigned full = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  unsigned todo = __ballot_sync(full, on);
#pragma unroll
  for (int round = 0; round < 2; ++round) {
    if (__popc(todo) < 4) break;  // uniform
    const int leader = __ffs(todo) - 1;
    const int32_t X0 = __shfl_sync(full, X, leader);
    const bool mine = ((todo >> lane) & 1u) && X == X0;
    const unsigned same = __ballot_sync(full, mine);
    if (same == (1u << leader)) break;
    // one instruction where the sum fits 32 bits
    const long long t = __all_sync(full, !mine || w == (long long)((int32_t)(w << 5) >> 5))
                            ? (long long)__reduce_add_sync(full, mine ? (int32_t)w : 0)
                            : warp_sum(mine ? w : 0ll);
    if (lane == leader) atomicAdd((unsigned long long *)&W[X0], (unsigned long long)t);
    todo &= ~same;
  }
  if ((todo >> lane) & 1u) atomicAdd((unsigned long long *)&W[X], (unsigned long long)w);
}

// Applies the pass to one vertex per lane (full warp): a survivor leaves its
// cluster for its destination (Algorithm 2, Update), or stays unlabelled
// (C[v] = kEmpty) until the new-cluster ids are given out.  The records
// still hold C and D, so other vertices' sums are not disturbed.  Lists the
// movers' row chunks (kept tables) and the movers that are not hubs (final
// objective) where those lists are kept, one append per warp.  used: null, or
// the ids in use, marked from every vertex's new label.
__device__ __forceinline__ void apply_lanes(const PassArgs &a, bool on, int32_t v, int64_t deg, const AbRec &r,
                                            long long wv, bool keep, UpdateSums &sum, int32_t *used = nullptr) {
  const int lane = threadIdx.x & 31;
  keep = keep && on;
  if (keep) {
    a.C[v] = r.D >= 0 ? LC_IDX(r.D, a.g.n, kDbgDest) : kEmpty;
    sum.empties += r.D < 0;
    sum.moved++;
  }
  add_weights(a.W, keep, r.C, -wv);
  add_weights(a.W, keep && r.D >= 0, LC_IDX(keep && r.D >= 0 ? r.D : 0, a.g.n, kDbgDest), wv);
  if (used && on && !(keep && r.D < 0)) used[keep ? r.D : r.C] = 1;
  if (on && r.D != kNone) sum.cand += deg;
  if (on && a.M) a.M[v] = keep;
  if (a.upd_list) {  // uniform over the launch
    const int nch = keep ? (int)((deg + kUpdChunk - 1) / kUpdChunk) : 0;
    int incl = nch;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    int first = 0;
    if (lane == 31 && total > 0) first = atomicAdd(&a.sc->upd_count, total);
    first = __shfl_sync(0xFFFFFFFFu, first, 31) + incl - nch;
    for (int k = 0; k < nch; ++k) a.upd_list[first + k] = make_int2(v, k);
  }
  if (a.movers) {  // uniform over the launch
    const bool listed = keep && deg <= a.hub_min;  // hubs: k_hub_delta_in
    const unsigned m = __ballot_sync(0xFFFFFFFFu, listed);
    int first = 0;
    if (lane == 0 && m) first = atomicAdd(&a.sc->n_movers, __popc(m));
    first = __shfl_sync(0xFFFFFFFFu, first, 0);
    if (listed) a.movers[first + __popc(m & ((1u << lane) - 1u))] = v;
  }
}

struct AbStage {
  AbCtx ctx[32];
  long long sum[32];
};

// A chunk's candidates staged at consecutive places (full warp): returns
// their number; `pos` is this lane's place.
__device__ __forceinline__ int stage_ab(const PassArgs &a, const VRec *__restrict__ rec, int64_t base, int m, int lane,
                                        AbCtx *ctx, VRec &vr, AbRec &r, long long &delta, int &pos) {
  bool cand = false;
  if (lane < m) {
    vr = rec[base + lane];
    r = a.ab[vr.v];
    cand = r.D != kNone;
  }
  const unsigned bal = __ballot_sync(0xFFFFFFFFu, cand);
  pos = __popc(bal & ((1u << lane) - 1u));
  if (cand) {
    delta = a.delta[vr.v];
    ctx[pos] = ab_ctx(a, vr.v, r, a.gp[vr.g], vr.beg, vr.deg, vr.w);
  }
  return __popc(bal);
}

// Afterburner and update of a chunk: for each candidate, delta_v adjusted by
// every adjacent candidate that precedes it; it survives iff the adjusted
// delta is >= 0.  G lanes per candidate, U edges each in flight, so that
// a row up to U G edges is one chain of gathers and a warp has 32 / G chains
// going: the walk is bound by their latency.
template <int G, int U = 4>
__device__ __forceinline__ void ab_chunk(const PassArgs &a, const VRec *__restrict__ rec, int64_t base, int m,
                                         AbStage &st, UpdateSums &sum, int32_t *used = nullptr) {
  constexpr int V = 32 / G;
  const int lane = threadIdx.x & 31, grp = lane / G, sub = lane & (G - 1);
  VRec vr{};
  AbRec r{0, kNone, 0};
  long long delta = 0;
  int pos;
  const int nc = stage_ab(a, rec, base, m, lane, st.ctx, vr, r, delta, pos);
  __syncwarp();
  for (int k = 0; k < nc; k += V) {
    long long acc = 0;
    if (k + grp < nc) {
      const AbCtx c = st.ctx[k + grp];
      acc = ab_edges<G, U>(a, c, c.beg, c.beg + c.deg, sub);
    }
    __syncwarp();
    if (__any_sync(0xFFFFFFFFu, acc != 0)) acc = group_sum<G>(acc);
    if (sub == 0 && k + grp < nc) st.sum[k + grp] = acc;
  }
  __syncwarp();
  const bool keep = r.D != kNone && delta + st.sum[r.D != kNone ? pos : 0] >= 0;
  apply_lanes(a, lane < m, vr.v, vr.deg, r, vr.w, keep, sum, used);
  __syncwarp();
}

// Bin 0: one thread per vertex (full warp, lanes with on = false idle).
template <int U = 4>
__device__ __forceinline__ void ab_thread(const PassArgs &a, bool on, const VRec *__restrict__ rec, int64_t i,
                                          UpdateSums &sum, int32_t *used = nullptr) {
  VRec vr{};
  AbRec r{0, kNone, 0};
  bool keep = false;
  if (on) {
    vr = rec[i];
    r = a.ab[vr.v];
    if (r.D != kNone) {
      const AbCtx c = ab_ctx(a, vr.v, r, a.gp[vr.g], vr.beg, vr.deg, vr.w);
      keep = a.delta[vr.v] + ab_edges<1, U>(a, c, c.beg, c.beg + c.deg, 0) >= 0;
    }
  }
  __syncwarp();
  apply_lanes(a, on, vr.v, vr.deg, r, vr.w, keep, sum, used);
}

// ------------------------------------------ objective after a pass

// Change of IN over edges [e0, e1) of mover v (strided by GS): an edge to
// a non-mover counts both directions, an edge between movers one (the
// other mover counts the other).  A mover that got its own emptied id back
// counts as a non-mover, from either end.
template <int GS>
__device__ __forceinline__ long long delta_in_edges(const PassArgs &a, int32_t v, int64_t e0, int64_t e1,
                                                    int r) {
  constexpr int U = 4;
  const int32_t Cvn = a.C[v], Cvo = a.ab[v].C;
  long long d = 0;
  for (int64_t base = e0 + r; base < e1; base += (int64_t)GS * U) {
    int32_t u[U], w[U], Cun[U], Cuo[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int64_t e = base + (int64_t)k * GS;
      u[k] = -1;
      w[k] = 0;
      if (e < e1) {
        u[k] = LC_IDX(__ldg(a.g.col + e), a.g.n, kDbgColumn);
        w[k] = __ldg(a.g.ew + e);
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      Cun[k] = u[k] >= 0 ? a.C[u[k]] : 0;
      Cuo[k] = u[k] >= 0 ? a.ab[u[k]].C : 0;
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (u[k] < 0) continue;
      const int s = (Cvn == Cun[k] ? 1 : 0) - (Cvo == Cuo[k] ? 1 : 0);
      d += (long long)(Cun[k] != Cuo[k] ? 1 : 2) * s * w[k];
    }
  }
  return d;
}

}  // namespace lc
