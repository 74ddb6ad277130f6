// lc_validate.cu — CSR precondition checks and the sums the exactness guards
// need (Section II: positive integer edge weights, undirected graph stored in
// both directions; vertex weights may also be zero, the weighted degree of an
// isolated vertex under modularity).  The edge checks are load-balanced over
// entries, so a single long row does not serialise them.
#include "lc_edge_print.cuh"
#include "lc_group.cuh"
#include "lc_internal.cuh"
#include "lc_move.cuh"
#include "lc_validate.cuh"

namespace lc {

__device__ __forceinline__ void report(GraphStats *st, int code, int64_t v) {
  const unsigned long long key = ((unsigned long long)code << 40) | (unsigned long long)(v & 0xFFFFFFFFFFll);
  atomicMin(&st->err_key, key);
}

// Per-vertex part: vertex-weight sums and checks, row-pointer sanity.
__global__ void __launch_bounds__(256) k_stats_vertices(LevelGraph g, int validate, GraphStats *st,
                                                        const int32_t *gid, long long *Vg,
                                                        long long *sw2g) {
  long long V = 0, sw2 = 0;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < g.n;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = base + threadIdx.x;
    long long w = 0;
    if (v < g.n) {
      w = g.vw[v];
      V += w;
      sw2 += w * w;
      if (validate && w < 0) report(st, LC_ERR_WEIGHT, v);
      const int64_t beg = g.rp[v], end = g.rp[v + 1];
      if (end < beg || beg < 0 || end > g.nnz) report(st, LC_ERR_ARG, v);
    }
    if (gid) {
      const int gg = v < g.n ? gid[v] : -1;
      graph_add(Vg, gg, w);
      graph_add(sw2g, gg, w * w);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->first = g.rp[0];
    st->last = g.rp[g.n];
  }
  flush_block_sum(V, &st->V);
  flush_block_sum(sw2, &st->sw2);
}

// Largest r in [0, n) with rp[r] <= e (rp[0] = 0; any r on a malformed
// row_ptr, which the vertex part reports), by a whole warp: each step tests
// 32 places of the remaining range.
__device__ __forceinline__ int64_t warp_find_row(const int64_t *__restrict__ rp, int64_t n, int64_t e, int lane) {
  int64_t lo = 0, hi = n;  // rp[lo] <= e, rp[hi] > e or hi == n
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) / 32;
    const int64_t at = lo + (lane + 1) * step;
    const bool le = at < hi && __ldg(rp + at) <= e;
    const int k = __popc(__ballot_sync(0xFFFFFFFFu, le));
    const int64_t nlo = lo + k * step;
    hi = nlo + step < hi ? nlo + step : hi;
    lo = nlo;
  }
  return lo;
}

// Per-edge part, load-balanced: a warp takes a run of consecutive entries,
// finds the row of its first by one search, and walks on 128 entries at a
// time, four consecutive ones per lane.  The rows that start inside the step
// mark their first entry in shared memory (of several rows at one place the
// last is the one with entries); a maximum scan over the marks gives every
// entry its row, and a mark says that an entry is its row's first.  Bound by
// instructions: the edge's two fingerprints are 40 of about 55 per entry.
// The former walk of 32 entries per thread spent 21 dependent loads per walk
// on finding its row: 0.80 ms at 62 M entries.
constexpr int kStatsThreads = 256;
constexpr int kStatsRun = 1024;  // entries per warp
constexpr int kStatsStep = 128;  // entries per step

struct Four {
  int32_t x[4];
};
// Entries e .. e + 3 (those below `end`; the others 0).  vec: p is 16-byte
// aligned and e a multiple of 4.
__device__ __forceinline__ Four load_four(const int32_t *__restrict__ p, int64_t e, int64_t end, bool vec) {
  Four r;
  if (vec && e + 3 < end) {
    const int4 t = __ldg(reinterpret_cast<const int4 *>(p + e));
    r.x[0] = t.x;
    r.x[1] = t.y;
    r.x[2] = t.z;
    r.x[3] = t.w;
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) r.x[k] = e + k < end ? __ldg(p + e + k) : 0;
  }
  return r;
}

// Marks row + 1 at the first entry of the rows r .. r + 32 K - 1 that start in
// the step (of `left` entries from `base`), and moves r past them; false if
// some row starts past the step.
template <int K>
__device__ __forceinline__ bool mark_rows(const LevelGraph &g, int64_t base, int left, int lane, int64_t &r,
                                          int32_t *mark) {
  int64_t d[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    d[k] = kStatsStep;
    if (r + 32 * k + lane < g.n) d[k] = __ldg(g.rp + r + 32 * k + lane) - base;
  }
  bool all = true;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const bool in = d[k] >= 0 && d[k] < left;
    if (in) atomicMax(&mark[d[k]], (int32_t)(r + 32 * k + lane) + 1);
    all = all && __all_sync(0xFFFFFFFFu, in);
  }
  r += 32 * K;
  return all;
}

// A faulty entry (row v, column x, weight w) of a row whose order it breaks
// (unsorted) or not.
__device__ __noinline__ void report_entry(GraphStats *st, int32_t v, int32_t x, int32_t n, bool unsorted, int32_t w) {
  if (x < 0 || x >= n) {
    report(st, LC_ERR_ARG, v);
    return;
  }
  if (x == v) report(st, LC_ERR_SELF_LOOP, v);
  if (unsorted) report(st, LC_ERR_DUPLICATE, v);
  if (w <= 0) report(st, LC_ERR_WEIGHT, v);
}

// INSIDE: also the weight inside the clusters of C (labels are compared, never
// followed).
template <bool VALIDATE, bool INSIDE>
__global__ void __launch_bounds__(kStatsThreads, 4) k_stats_edges(LevelGraph g, GraphStats *st,
                                                               const int32_t *__restrict__ gid,
                                                               const int64_t *__restrict__ gptr, long long *Tg,
                                                               const int32_t *__restrict__ C) {
  // col and ew are as long as row_ptr says, and the caller's nnz has not been
  // compared with it yet (uniform; the vertex part reports both ends)
  if (__ldg(g.rp) != 0 || __ldg(g.rp + g.n) != g.nnz) return;
  constexpr unsigned full = 0xFFFFFFFFu;
  __shared__ int4 s_mark[kStatsThreads / 32][kStatsStep / 4];
  const int lane = threadIdx.x & 31;
  int4 *mark4 = s_mark[threadIdx.x >> 5];
  int32_t *mark = reinterpret_cast<int32_t *>(mark4);
  const bool vec = ((reinterpret_cast<uintptr_t>(g.col) | reinterpret_cast<uintptr_t>(g.ew)) & 15) == 0;
  const int64_t runs = (g.nnz + kStatsRun - 1) / kStatsRun;
  const int64_t nwarps = (int64_t)gridDim.x * (kStatsThreads / 32);
  long long T = 0, inside = 0;
  unsigned long long f1 = 0, f2 = 0;
  unsigned minus = 0;  // edges subtracted: -h = ~h + 1, the ones added at the end
  mark4[lane] = make_int4(0, 0, 0, 0);
  __syncwarp();
  for (int64_t run = (int64_t)blockIdx.x * (kStatsThreads / 32) + (threadIdx.x >> 5); run < runs; run += nwarps) {
    const int64_t e0 = run * kStatsRun, e1 = e0 + kStatsRun < g.nnz ? e0 + kStatsRun : g.nnz;
    Four u = load_four(g.col, e0 + 4 * lane, e1, vec), w = load_four(g.ew, e0 + 4 * lane, e1, vec);
    int64_t r0 = 0;          // row of the entry before the step (of the run's first entry at its start)
    int32_t carry = -1;      // the column before the step
    if (VALIDATE || INSIDE || gid) {
      r0 = warp_find_row(g.rp, g.n, e0, lane);
      if (lane == 0 && __ldg(g.rp + r0) == e0) mark[0] = (int32_t)r0 + 1;
      if (e0 > 0) carry = __ldg(g.col + e0 - 1);
    }
    int cur_g = -1;  // graph of the weights summed into tg
    long long tg = 0;
    for (int64_t base = e0; base < e1; base += kStatsStep) {
      const int64_t en = base + kStatsStep + 4 * lane;
      const Four un = load_four(g.col, en, e1, vec), wn = load_four(g.ew, en, e1, vec);
      const int left = e1 - base < kStatsStep ? (int)(e1 - base) : kStatsStep;
#pragma unroll
      for (int k = 0; k < 4; ++k) T += w.x[k];  // 0 past the end
      if (!VALIDATE && !INSIDE && !gid) {
        u = un;
        w = wn;
        continue;
      }
      // marks: row + 1 at its first entry, for the rows after r0 that start
      // in the step
      int64_t r = r0 + 1;
      const bool more = mark_rows<1>(g, base, left, lane, r, mark) && mark_rows<4>(g, base, left, lane, r, mark);
      if (more && r < g.n) {
        // hundreds of rows start here, mostly empty ones (a skewed graph's
        // isolated vertices): each entry looks for its own row instead
        const int64_t hi = warp_find_row(g.rp, g.n, base + left - 1, lane) + 1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int64_t e = base + 4 * lane + k;
          int64_t lo = r - 1, up = hi;  // rp[lo] <= e once e is past row r - 1's start
          while (up - lo > 1) {
            const int64_t mid = (lo + up) >> 1;
            if (__ldg(g.rp + mid) <= e)
              lo = mid;
            else
              up = mid;
          }
          if (4 * lane + k < left && lo >= r && __ldg(g.rp + lo) == e) mark[4 * lane + k] = (int32_t)lo + 1;
        }
      }
      __syncwarp();
      const int4 m = mark4[lane];
      mark4[lane] = make_int4(0, 0, 0, 0);
      __syncwarp();
      // row + 1 of the last mark up to each entry
      const int32_t m0 = m.x, m1 = max(m0, m.y), m2 = max(m1, m.z), m3 = max(m2, m.w);
      int32_t scan = m3;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(full, scan, o);
        if (lane >= o) scan = max(scan, y);
      }
      int32_t prev = __shfl_up_sync(full, scan, 1);
      prev = max(lane > 0 ? prev : 0, (int32_t)r0 + 1);
      const int32_t row[4] = {max(prev, m0) - 1, max(prev, m1) - 1, max(prev, m2) - 1, max(prev, m3) - 1};
      const bool first[4] = {m.x != 0, m.y != 0, m.z != 0, m.w != 0};
      const int32_t up = __shfl_up_sync(full, u.x[3], 1);
      const int32_t before[4] = {lane > 0 ? up : carry, u.x[0], u.x[1], u.x[2]};
      if (INSIDE) {
        int32_t cu[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          cu[k] = 4 * lane + k < left && (uint32_t)u.x[k] < (uint32_t)g.n ? C[u.x[k]] : -1;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (cu[k] >= 0 && cu[k] == C[row[k]]) inside += w.x[k];
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const bool on = 4 * lane + k < left;
        const int32_t v = row[k], x = u.x[k];
        if (gid) {
          const int gv = on ? __ldg(gid + v) : -1;
          if (__all_sync(full, gv == cur_g || !on)) {
            tg += w.x[k];
          } else {  // the step reaches another graph
            if (cur_g >= 0) graph_add(Tg, cur_g, tg);
            graph_add(Tg, gv, w.x[k]);
            cur_g = __shfl_sync(full, gv, 31);
            tg = 0;
          }
          if (VALIDATE && on && x >= 0 && x < g.n && (x < __ldg(gptr + gv) || x >= __ldg(gptr + gv + 1)))
            report(st, LC_ERR_ARG, v);
        }
        if (!VALIDATE) continue;
        // one test for all of an entry's faults; telling them apart is rare
        if (on && ((uint32_t)x >= (uint32_t)g.n || x == v || (!first[k] && before[k] >= x) || w.x[k] <= 0))
          report_entry(st, v, x, (int32_t)g.n, !first[k] && before[k] >= x, w.x[k]);
        const uint32_t lo = (uint32_t)min(v, x), hi = (uint32_t)max(v, x);
        const EdgePrint h = edge_print(lo, hi, (uint32_t)w.x[k]);
        const unsigned long long neg = v < x ? 0ull : ~0ull;
        if (on) {
          f1 += h.a ^ neg;
          f2 += h.b ^ neg;
          minus += (unsigned)(neg & 1ull);
        }
      }
      carry = __shfl_sync(full, u.x[3], 31);
      r0 = max(__shfl_sync(full, scan, 31), (int32_t)r0 + 1) - 1;
      u = un;
      w = wn;
    }
    if (gid && cur_g >= 0) graph_add(Tg, cur_g, tg);
  }
  flush_block_sum(T, &st->T);
  if (INSIDE) flush_block_sum(inside, &st->inside);
  if (VALIDATE) {
    flush_block_sum((long long)(f1 + minus), (long long *)&st->fp1);
    flush_block_sum((long long)(f2 + minus), (long long *)&st->fp2);
  }
}

// Cluster weights and ids in use of the labels C, which are checked against
// [0, n) before they are followed.
__global__ void __launch_bounds__(256) k_label_sums(LevelGraph g, const int32_t *__restrict__ C, int64_t *W,
                                                    int32_t *__restrict__ used, GraphStats *st) {
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < g.n; base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = base + threadIdx.x;
    const int32_t x = v < g.n ? C[v] : 0;
    const bool ok = v < g.n && x >= 0 && x < g.n;
    if (v < g.n && !ok) atomicAdd(&st->bad_labels, 1ull);
    if (ok) used[x] = 1;
    add_weights(W, ok, ok ? x : 0, ok ? g.vw[v] : 0);
  }
}
// Q = sum_x W(x)^2 - w(x)^2 (unsigned arithmetic: exact whenever it fits) and
// the number of ids in use.
__global__ void __launch_bounds__(256) k_label_squares(LevelGraph g, const int64_t *__restrict__ W,
                                                       const int32_t *__restrict__ used, GraphStats *st) {
  long long q = 0, k = 0;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < g.n; x += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long a = (unsigned long long)W[x], b = (unsigned long long)g.vw[x];
    q += (long long)(a * a - b * b);
    k += used[x] != 0;
  }
  flush_block_sum(q, &st->q);
  flush_block_sum(k, &st->clusters);
}

void launch_label_stats(const LevelGraph &g, const int32_t *C, int64_t *W, int32_t *used, GraphStats *st,
                        cudaStream_t s) {
  if (g.n <= 0) return;
  int64_t b = (g.n + 255) / 256;
  if (b > 152 * 8) b = 152 * 8;
  cudaMemsetAsync(W, 0, sizeof(int64_t) * (size_t)g.n, s);
  cudaMemsetAsync(used, 0, sizeof(int32_t) * (size_t)g.n, s);
  k_label_sums<<<(unsigned)b, 256, 0, s>>>(g, C, W, used, st);
  k_label_squares<<<(unsigned)b, 256, 0, s>>>(g, W, used, st);
}

__global__ void k_labels_in_range(const int32_t *__restrict__ C, int64_t n, int64_t limit,
                                  GraphStats *st) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    if (C[v] < 0 || C[v] >= limit) st->bad_labels = 1;  // whoever comes last, the same value
}

void launch_stats(const LevelGraph &g, int validate, GraphStats *st, const int32_t *gid, const int64_t *gptr,
                  long long *Tg, long long *Vg, long long *sw2g, const int32_t *C, cudaStream_t s) {
  auto blocks = [](int64_t items) {
    int64_t b = (items + 255) / 256;
    if (b < 1) b = 1;
    if (b > 152 * 8) b = 152 * 8;
    return (unsigned)b;
  };
  k_stats_vertices<<<blocks(g.n), 256, 0, s>>>(g, validate, st, gid, Vg, sw2g);
  if (g.nnz > 0) {
    const int64_t runs = (g.nnz + kStatsRun - 1) / kStatsRun;
    // a run per warp: the block scheduler evens out what a loop over runs
    // would leave as a last, half-empty turn
    int64_t b = (runs + kStatsThreads / 32 - 1) / (kStatsThreads / 32);
    if (b > INT32_MAX) b = INT32_MAX;
    auto *k = C ? (validate ? k_stats_edges<true, true> : k_stats_edges<false, true>)
                : (validate ? k_stats_edges<true, false> : k_stats_edges<false, false>);
    k<<<(unsigned)b, kStatsThreads, 0, s>>>(g, st, gid, gptr, Tg, C);
  }
}

void launch_labels_in_range(const int32_t *C, int64_t n, int64_t limit, GraphStats *st,
                            cudaStream_t s) {
  int64_t blocks = (n + 255) / 256;
  if (blocks < 1) blocks = 1;
  if (blocks > 152 * 32) blocks = 152 * 32;
  k_labels_in_range<<<(unsigned)blocks, 256, 0, s>>>(C, n, limit, st);
}

}  // namespace lc
