// Tensor-core GEMMs of the stateful Transducer form; see gemm_tc.cu.
#pragma once

#include <cuda.h>

#include "decoder.h"

namespace tsd {

enum GemmEpilogue { kEncProj = 0, kLstm = 1, kJointIn = 2 };

struct GemmArgs {
  int M;              // rows of A (and of the output) this launch covers
  int N;              // output columns (a multiple of 32; B's rows are padded to a multiple of 128)
  int K;              // inner size, a multiple of 64
  int ld;             // kEncProj: output row stride; kJointIn: P_enc row stride (floats)
  const float* bias;  // [N]
  float* out;         // kEncProj: [M][ld]
};

bool gemm_tc_maps(GemmMaps* m, int epi, const uint16_t* A, int a_rows, const uint16_t* B, int b_rows, int K);
cudaError_t gemm_tc_prepare();
void launch_gemm_tc(int epi, const DecView& d, const GemmArgs& g, const GemmMaps& m, cudaStream_t s, bool pdl);

}  // namespace tsd
