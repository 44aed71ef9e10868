// The softmax partials of a row inside a cluster (chunk_cluster.cu): which of
// the owner's barriers counts a label step's, and which buffer holds them.
//
// A CTA sends a row's logits of step s and then, unordered against them, its
// partial of step s.  The row's next label needs every CTA's logits only, so a
// CTA's partial of step s may arrive after another one's of step s + 1: two
// barriers in turn, so that neither step counts the other's bytes.  Step s + 2
// cannot overtake: its partials follow every CTA's logits of step s + 1, and
// the owner sends its own (every CTA has labels) after it has waited for step
// s's partials.  It reads
// them only at the end of step s + 1, when those of s + 2 may arrive: three
// buffers.
#pragma once

#ifdef __CUDACC__
#define TSD_HD __host__ __device__
#else
#define TSD_HD
#endif

namespace tsd {

constexpr int kPartBars = 2, kPartBufs = 3;
TSD_HD constexpr int part_bar(int step) { return step % kPartBars; }
TSD_HD constexpr int part_parity(int step) { return step / kPartBars % 2; }
TSD_HD constexpr int part_buf(int step) { return step % kPartBufs; }

}  // namespace tsd
