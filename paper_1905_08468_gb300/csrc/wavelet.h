// Arguments of one analysis level, shared by wavelet.cu and ana_cols.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace muffin {

struct AnaArgs {
  int n, M, L, K, last;
  int Lc;                       // bands per cube (per-cube scalars sc[l / Lc])
  const float *in;              // level >= 2: LL_{j-1}; level-1 operator: x
  const float *xt, *x;          // level-1 iteration inputs
  float *ll_out;                // LL_j scratch when !last
  float *u;
  const float *beta;
  const DevScalars *sc;
  uint32_t *masks;              // ana_cols: masks of the primal, a word an item of a tile
};

// One analysis level with h = M / 2 >= 16 (ana_cols.cu).  flip: the other tile
// height than the rule's (same results).
cudaError_t ana_cols(const AnaArgs &a, int chains, bool iterate, bool level1, int flip,
                     cudaStream_t st);
cudaError_t upload_cols_filters(const float2 hp[8][8], const float2 gp[8][8]);

}  // namespace muffin
