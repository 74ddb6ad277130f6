// lc_validate.cuh — launch interface of lc_validate.cu.
#pragma once

#include "lc_internal.cuh"

namespace lc {

struct GraphStats {
  long long T;    // sum of stored edge weights (2 m_w)
  long long V;    // sum of vertex weights
  long long sw2;  // sum of w(v)^2 (exact when the guards hold)
  unsigned long long fp1, fp2;  // symmetric-edge fingerprints, 0 when symmetric
  int64_t first, last;          // row_ptr[0], row_ptr[n]
  long long inside, q, clusters;  // of a given clustering: see launch_stats, launch_label_stats
  unsigned long long bad_labels;
  unsigned long long err_key;   // (code << 40 | vertex), min over violations; ~0 if none
};

// Sums T, V, sum w^2 (T and all else about the edges only if row_ptr runs from
// 0 to nnz); with validate: row structure, ranges, loops, weights,
// strictly increasing rows and the symmetry fingerprints.  *st must be
// zeroed with err_key = ~0 beforehand.
// With a packed batch (gid non-null, gptr its vertex ranges) also per-graph
// sums Tg, Vg, sw2g (zeroed beforehand) and a check that no edge crosses
// graphs.  C: null, or labels whose inside weight (the stored edges within a
// cluster) is wanted.
void launch_stats(const LevelGraph &g, int validate, GraphStats *st, const int32_t *gid, const int64_t *gptr,
                  long long *Tg, long long *Vg, long long *sw2g, const int32_t *C, cudaStream_t s);
// Of the clustering C: labels outside [0, n) (not followed), sum_x W(x)^2 - w(x)^2
// and the ids in use, with W and used (both [n]) as scratch.
void launch_label_stats(const LevelGraph &g, const int32_t *C, int64_t *W, int32_t *used, GraphStats *st,
                        cudaStream_t s);
// Sets bad_labels if any label lies outside [0, limit).
void launch_labels_in_range(const int32_t *C, int64_t n, int64_t limit, GraphStats *st,
                            cudaStream_t s);

}  // namespace lc
