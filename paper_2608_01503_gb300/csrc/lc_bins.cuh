// lc_bins.cuh — launch interface of lc_bins.cu.
#pragma once

#include "lc_pass.cuh"

namespace lc {

// What the host reads back to size a level's launches.
struct BinOut {
  int32_t offs[kBins + 1];  // start of each bin in the lists
  int32_t max_deg;          // longest hub row (0: no hub)
  int64_t chunks;           // chunks of all hub rows
  int32_t done;             // 1: complete (no barrier's wait ran out)
};

// Fills b.lists and b.recs (ascending ids within each bin) and *out, all on
// the device; gid: graph of each vertex, or null for one graph.  counts:
// int32[coop_scratch] scratch; coop: blocks the launch may have.  The caller
// copies *out to the host and passes it to finish_bins.
void launch_bins(const LevelGraph &g, const int32_t *gid, const BinPlan &plan, const Bins &b, BinOut *out,
                 int32_t *counts, Scalars *sc, int coop, cudaStream_t s);
void finish_bins(Bins &b, const BinOut &out);
// Fills the arrays of a hub plan (H >= 1 hubs, Q chunks) and zeroes acc; returns
// the number of kernels launched.
int launch_hub_plan(const Bins &b, const BinPlan &plan, const Hubs &hub, cudaStream_t s);

}  // namespace lc
