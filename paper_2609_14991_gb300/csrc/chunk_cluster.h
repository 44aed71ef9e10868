// The label loop of a chunk in one launch (chunk_cluster.cu): launch shapes
// and call arguments.
#pragma once

#include <vector>

#include "decoder.h"

namespace tsd {

constexpr int kChunkMaxRows = 384;  // rows one call passes by value (more than any shape's clusters hold)

struct ChunkArgs {
  const uint16_t* enc;  // as in Params
  int32_t* out_tok;
  int32_t* out_frame;
  float* out_score;
  int32_t* out_count;
  int32_t n, T;
  float lambda, beta;
  int32_t CS, nl, R;  // CTAs per cluster, most labels of a CTA, rows per cluster
  int32_t slots[kChunkMaxRows];
};

struct ChunkShape {
  int CS = 0;        // CTAs per cluster
  int RG = 0;        // row groups per CTA
  int NB = 0;        // 8-row blocks of the product
  int nl = 0;        // most labels of a CTA
  int smem = 0;      // bytes per CTA
  int clusters = 0;  // clusters the device runs at once
};

// The shapes whose shared memory holds W_out and the rows' scratch (none:
// the decoder takes the two-kernel step).
cudaError_t chunk_cluster_shapes(const DecView& d, std::vector<ChunkShape>& out);
// The shape for n rows, or nullptr if none holds them in one wave or the
// two-kernel step is faster.
const ChunkShape* chunk_cluster_pick(const std::vector<ChunkShape>& shapes, int n, int H);
// The stateful form's joint product with the same sums, for rows that a shape
// holds: softmax partials per row of N labels, launch.
int joint_rows_tiles(int N);
cudaError_t joint_rows_prepare();
void launch_joint_rows(const ChunkShape& s, const DecView& d, int n, int step, cudaStream_t st, bool pdl);
cudaError_t launch_chunk_cluster(const ChunkShape& s, const DecView& d, ChunkArgs& a, cudaStream_t st);

}  // namespace tsd
