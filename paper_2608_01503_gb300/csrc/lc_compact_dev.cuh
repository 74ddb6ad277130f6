// lc_compact_dev.cuh — the contraction table's occupied slots as coarse rows
// (lc_contract.cu, and lc_level.cu for a small level).
#pragma once

#include "lc_internal.cuh"

namespace lc {

// The largest x < n_c with 2 off[x] <= s, given 2 off[n_c] > s (full warp).
__device__ __forceinline__ int64_t row_of_slot(const int64_t *__restrict__ off, int64_t n_c, int64_t s, int lane) {
  int64_t lo = 0, hi = n_c;
  while (hi - lo > 1) {
    const int64_t step = (hi - lo + 31) / 32, p = lo + (lane + 1) * step;
    const unsigned le = __ballot_sync(0xFFFFFFFFu, p < hi && 2 * off[p] <= s);
    lo += __popc(le) * step;
    hi = lo + step < hi ? lo + step : hi;
  }
  return lo;
}

struct CompactArgs {
  unsigned long long *tab;
  const int64_t *off, *rp;  // of the coarse rows
  int32_t *cnt;             // entries of each row; a split row's entries left to place
  int64_t n_c;
  int32_t *col, *ew;
};

// The occupied slots [beg, end) of a run, in order, to position `at` on (full
// warp); row >= 0: to places taken from that row, 256 slots at a time.  Frees
// the slots.
__device__ __forceinline__ void emit_slots(const CompactArgs &a, int64_t beg, int64_t end, int64_t at, int64_t row,
                                           int lane) {
  constexpr int U = 4;
  constexpr unsigned full = 0xFFFFFFFFu;
  const unsigned below = (1u << lane) - 1u;
  for (int64_t base = beg; base < end; base += 64 * U) {
    ulonglong2 t[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int64_t s = base + 64 * k + 2 * lane;
      t[k] = make_ulonglong2(kEmptySlot, kEmptySlot);
      if (s < end) t[k] = *reinterpret_cast<const ulonglong2 *>(a.tab + s);
    }
    int n[U], total = 0;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const unsigned x = __ballot_sync(full, t[k].x != kEmptySlot), y = __ballot_sync(full, t[k].y != kEmptySlot);
      n[k] = total + __popc(x & below) + __popc(y & below);
      total += __popc(x) + __popc(y);
    }
    int64_t to = at;
    if (row >= 0) {
      int left = 0;
      if (lane == 0 && total > 0) left = atomicSub(&a.cnt[row], total);
      to = a.rp[row] + __shfl_sync(full, left, 0) - total;
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      int64_t p = to + n[k];
      if (t[k].x != kEmptySlot) {
        a.col[p] = slot_key(t[k].x);
        a.ew[p++] = slot_val(t[k].x);
      }
      if (t[k].y != kEmptySlot) {
        a.col[p] = slot_key(t[k].y);
        a.ew[p] = slot_val(t[k].y);
      }
      if (t[k].x != kEmptySlot || t[k].y != kEmptySlot)
        *reinterpret_cast<ulonglong2 *>(a.tab + base + 64 * k + 2 * lane) = make_ulonglong2(kEmptySlot, kEmptySlot);
    }
    at += total;
  }
}

// Slots [s0, s0 + run) of the `used` ones as coarse rows, and clean
// again, by a warp: one read of the table.  The rows that lie inside its
// run come out in slot order from the first one's offset; of a row that the
// run's edges cut, each piece takes places of that row as it comes (rows are
// unsorted).  Bound by reading 16 bytes per stored edge; a scan over the slots
// read the table twice and took three launches (ms per call, scan / this:
// R-MAT scale 20 level 5.66 / 5.50, R-MAT scale 22 64.3 / 62.9, 512-graph
// batch 59.2 / 57.9).  2,048 slots: the two row searches are 10 probes against
// 32 loads of 16 bytes per lane.
constexpr int kCompactRun = 2048;
__device__ __forceinline__ void compact_run(const CompactArgs &a, int64_t s0, int64_t run, int64_t used) {
  const int lane = threadIdx.x & 31;
  const int64_t s1 = s0 + run < used ? s0 + run : used;
  int64_t x = row_of_slot(a.off, a.n_c, s0, lane), beg = s0;
  if (2 * a.off[x] < s0) {  // began before the run
    const int64_t end = 2 * a.off[x + 1];
    beg = end < s1 ? end : s1;
    emit_slots(a, s0, beg, 0, x, lane);
    ++x;
  }
  if (beg >= s1) return;
  const int64_t last = row_of_slot(a.off, a.n_c, s1 - 1, lane);
  const int64_t cut = 2 * a.off[last + 1] > s1 ? 2 * a.off[last] : s1;  // the last row goes on after the run
  if (beg < cut) emit_slots(a, beg, cut, a.rp[x], -1, lane);
  if (cut < s1) emit_slots(a, cut, s1, 0, last, lane);
}

}  // namespace lc
