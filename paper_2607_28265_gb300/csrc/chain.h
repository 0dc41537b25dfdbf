// Interface of the chain sampler (chain.cuh, chain.cu) to the host code.
#pragma once

#include "het.cuh"
#include "kernels.h"
#include "sampler.cuh"

namespace swig {

// What a CTA reads of an event.
struct ChainEvent {
  LikeConst L;
  SamplerConst S;
  FoldTables F;
  HetTables H;
  SamplerPtrs P;
};

enum ChainMode { CHAIN_FOLD = 0, CHAIN_HET = 1, CHAIN_HET_TM = 2 };

// Dynamic shared memory of a launch: fixed part (work, constants, inputs and
// sums of an evaluation), scratch (the boundary's sort buffers, between
// boundaries the anchors or the time pass's buffers), then, resident, the
// folded weights and tables.
struct ChainLayout {
  int scratch_off, scratch_bytes;
  int res_off;            // 0: weights and tables are read from global memory
  int base_off;           // folded: partial sums of the current point (0: none)
  int anc_off, panel;     // time marginalisation: HetTmLayout's, from scratch_off
  int n_ctas;
  long long spin_limit;
};

// Bytes before the scratch.
size_t chain_fixed_bytes(int n_det, int mode);
void* chain_kernel(int n_det, int mode);
constexpr int kChainBlock = 512;
constexpr size_t kChainSmemMax = 224 * 1024;

}  // namespace swig
