// lc_level.cuh — launch interface of lc_level.cu.
#pragma once

#include "lc_bins_dev.cuh"

namespace lc {

// What the host reads back between the kernels of a level's end.
struct LevelOut {
  int64_t n_c, nnz_c;  // coarse vertices and stored edges
  BinOut bins;         // of the coarse graph (offs and hub figures only); done: of all of this
};

// Scratch of a level's end, all sized for the level (int32 [n] unless said).
struct LevelScratch {
  int32_t *used, *newid, *cnt;
  int64_t *bound, *label_w;   // [n] edge bound and weight by label
  int64_t *off;               // [n + 1] where a coarse vertex's slots start
  int64_t *vw, *rp;           // [n], [n + 1]: the coarse weights and row offsets
  unsigned long long *tab;    // [2 nnz] clean hash slots
  int32_t *nc;                // [G] labels in use per graph
  int32_t *gid;               // [n] graph of a coarse vertex (batches)
  long long *counts;          // [level_counts] per-warp counts
};
constexpr int kLevelWarps = 16;  // of a block
inline int64_t level_counts(int64_t n, int64_t nnz) { return kLevelWarps * level_grid(n, nnz); }

// The labels C (ids in [0, n)) of a level numbered densely per graph that
// merges something, the contraction's offsets, inserts and coarse row
// offsets, and the coarse bins' sizes: Cd, the scratch and *out.  A graph
// whose labels all differ is finished: its vertices get Cd = -1, and
// out->n_c = 0 when that is every graph.
void launch_level_end(const LevelGraph &g, const int32_t *gid, const GraphParam *gp, int G, const Bins &b,
                      const Hubs &hub, const BinPlan &plan, const int32_t *C, int32_t *Cd, const LevelScratch &w, LevelOut *out,
                      int32_t *bin_counts, Scalars *sc, int coop, cudaStream_t s);
// The coarse graph from the scratch into its own arrays (out as read back),
// its graph ids (null for one graph) and its bins; leaves the hash slots clean.
void launch_level_build(const LevelGraph &g, const LevelScratch &w, const LevelOut &out, int64_t *rp_c, int32_t *col_c,
                        int32_t *ew_c, int64_t *vw_c, int32_t *gid_c, const BinWork &bins, int coop, cudaStream_t s);

}  // namespace lc
