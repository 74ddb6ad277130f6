// lc_fused.cuh — launch interface of lc_fused.cu.
#pragma once

#include "lc_pass.cuh"

namespace lc {

// One LocalMovePasses call beyond PassArgs.
struct FusedArgs {
  const VRec *rec;        // the level's vertex records, bin after bin
  int64_t off[kBins + 1]; // start of each bin in rec
  int32_t *C_out;
  long long *acc;         // [3 G] Phi entering a pass, by pass number modulo 3
  long long *best;        // [2 G] best Phi seen, by pass parity
  long long *fin;         // [G] change of Phi by the last pass
  long long *phi_final;   // [G] written for the graphs active in the call
  int *empties;           // [6] movers to new empty clusters, then candidates for one, each by
                          // pass number modulo 3
  unsigned *next;         // [18] work counters, by pass number modulo 3 and phase
  EmptyScratch empty;
  int32_t passes;         // >= 1
  int32_t singleton;      // start from singletons (else from a.C)
  int32_t big;            // some hub row is longer than fused_row_max()
  int32_t phi[16][2];     // temperatures
};

void configure_fused();
// Longest row a block aggregates in shared memory.
int64_t fused_row_max();
// All passes in one cooperative launch: C_out, phi_out and phi_final as the
// separate launches leave them (a.gp as uploaded; a.C, a.W, a.ab, a.delta
// are scratch).  Returns the number of kernels launched.
int launch_fused_passes(const PassArgs &a, const FusedArgs &f, cudaStream_t s);

}  // namespace lc
