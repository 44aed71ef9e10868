// The whole label loop of one decode_chunk call in one launch (greedy
// decoding, at most one n-gram LM, the streaming form of Eq. 1): a cluster of
// CS CTAs decodes R rows from the chunk's first frame to its last with W_out
// resident in its shared memory.
//
// What bounds the two-kernel label step (joint_greedy.cu, row_stream.cu) at
// few rows is not work but the chain of launches and round trips to L2: 9.4 us
// a step for one stream (V = 1024, H = 640), 10.4 us for 64, against well
// under 1 us of arithmetic.  Here a step has no launch, no grid-wide
// dependency and no logits in memory (13 frames of one stream: 614 -> 169 us,
// of 64 streams: 665 -> 243 us; 16 streams x 1 frame, H = 1024: 71 -> 29 us):
//   * CTA c of the cluster keeps its slice of W_out's labels in shared memory for
//     the whole chunk (read once per chunk, not once per step);
//   * warps 0-7 (GEMM) compute the slice's logits of all R rows: bf16
//     mma.sync 16 x 8 x 16 with labels as the 16-row operand and rows as the
//     8-column one, so one row costs one eighth of what a 128-row tcgen05 tile
//     does and the eight warps split H; their partials are summed in a fixed
//     order and sent to the row's owner CTA by st.async;
//   * row i is owned by CTA i mod CS, group i / CS: 128 threads (64 with three
//     groups) that keep the row's state in shared memory, take the argmax,
//     publish the label to every CTA (16 bytes each by st.async), and only
//     then advance the LM and trie chains and build the next state's deltas,
//     while the GEMM warps already load the embedding rows and multiply; the
//     arcs and trie children that the deltas need stay in the threads'
//     registers, so that the next label's search is a compare and one load;
//   * a cluster stops when its rows have finished their frames.
// Clusters never wait for one another.  Messages inside a cluster complete
// bytes on the receiver's mbarriers: `ybar` (every CTA: the R rows' labels of
// a step) and `lbar` (per owned row: its logits), one phase per step each.
// `sbar` (two per owned row, in turn: chunk_partials.h) does the same for the
// softmax partials that a score needs: GEMM warp q finishes row q's scores one
// step late, while it would wait.
// What is left of a step, in clocks, one stream: argmax 710, publishing 350,
// the label's records 1700, chains 770, deltas 1930 (three of these five wait
// for L2 once), beside labels to operands 1460, product 1430, sums and sending
// 700.
// Every wait is bounded (DecView::wait_ns); after an expired one the CTA
// records a code, leaves the loop, lets messages in flight land and meets the
// others at the cluster barrier that ends the kernel.
//
// The arithmetic is the streaming form's: fused + lse = (logit + D) + (c_r +
// lambda * delta), see row_stream.cu.  Level 0 of the LM chain comes from the
// unigram state's dense row (copied by cp.async while the label is searched),
// the levels above overwrite their labels' deltas.  The order of every sum
// depends on V and H only (the softmax partials are of units of labels that are
// the same for clusters of 8 and of 16), so a row's result does not depend
// on the other rows of the call, on R or on CS, as long as the call runs here.
#include <algorithm>

#include "row_common.cuh"
#include "chunk_cluster.h"
#include "chunk_partials.h"
#include "tc_common.cuh"

namespace tsd {

namespace {

using row::best_merge;
using row::checked;
using row::first_load;
using row::key_value;
using row::kNegInf;
using row::level_groups;
using row::lse_merge;
using row::order_key;
using row::warp_find_wide;
using tc::map_rank;

constexpr int kGemm = 256;     // GEMM threads (8 warps, each an eighth of H)
constexpr int kTiles = 5;      // 16-label tiles per accumulator block
constexpr int kMB = 16 * kTiles;
constexpr int kUnits = 4;      // 32-wide pieces of H per warp: H <= 1024
constexpr int kTrHeld = 3;     // trie chain nodes whose first children a thread requests together
constexpr int kWPad = 64;      // bytes after a W_out row: neighbouring rows start 16 banks apart

// Remote stores that complete their bytes on a barrier of the receiving CTA.
__device__ __forceinline__ void send16(uint32_t dst, float4 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst),
               "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void send8(uint32_t dst, int a, int b, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.s32 [%0], {%1, %2}, [%3];" ::"r"(dst), "r"(a),
               "r"(b), "r"(bar)
               : "memory");
}

// The phase of the given parity has completed (a look, without the wait that
// try_wait may spend in the hardware).
__device__ __forceinline__ bool test_cluster(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(tc::smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ bool try_cluster(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(tc::smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Waits for the phase of the given parity; false once limit_ns has passed or
// another warp of the CTA has given up.
__device__ __forceinline__ bool wait_cluster(uint64_t* b, uint32_t parity, unsigned long long limit_ns,
                                             volatile int* fail) {
  if (test_cluster(b, parity)) return true;
  if (limit_ns == 0) return false;  // no waiting allowed
  const unsigned long long t0 = tc::global_ns();
  while (!try_cluster(b, parity)) {
    if (*fail || tc::global_ns() - t0 > limit_ns) return false;
  }
  return true;
}

__device__ __forceinline__ void group_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
  __syncwarp();
}

// The same barrier with a vote: true if every thread's ok is (so that all of
// them leave a loop together, and none is left waiting at a later barrier).
__device__ __forceinline__ bool group_all(int id, int threads, bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(ok ? 1u : 0u), "r"(id), "r"(threads)
      : "memory");
  __syncwarp();
  return r != 0;
}

__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// bf16(ReLU(x + z)) of eight elements.  The bf16 add rounds the exact sum
// once; rounding it to fp32 first, as the row passes do, gives the same: the
// fp32 sum of two bf16 values is inexact only where the smaller one is below
// 2^-16 of the larger, far from the middle between two bf16 values.
__device__ __forceinline__ uint4 joint8(uint4 x, uint4 z) {
  uint4 o;
  const __nv_bfloat162* xa = reinterpret_cast<const __nv_bfloat162*>(&x);
  const __nv_bfloat162* za = reinterpret_cast<const __nv_bfloat162*>(&z);
  __nv_bfloat162* oa = reinterpret_cast<__nv_bfloat162*>(&o);
  const __nv_bfloat162 zero = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
  for (int q = 0; q < 4; ++q) oa[q] = __hmax2(__hadd2(xa[q], za[q]), zero);
  return o;
}

// A row's state and search results.
struct RowSm {
  int4 lmr[kLmChain + 1], trr[kTrChain];       // chain records, as in row_stream.cu
  int4 lm_hit[kLmChain + 1], tr_hit[kTrChain]; // records found for the emitted label
  int4 uni_hit, root_hit;
  int lm[kLmChain + 1], tr[kTrChain];
  int dd[kTrChain];                            // depth of the children of a found trie child
  int4 best[2][4];                             // the warps' bests (value, label, wait succeeded), by step parity
  int nl, nt;
};

// The labels of a CTA, and the softmax partials they make.  The labels are cut
// into eight slices and each slice into two units (u0 labels and the rest; of
// N = 1025: 132 = 68 + 64); a cluster of 8 gives a CTA a slice, a cluster of
// 16 a unit.  A unit makes a partial per kMB of its labels.
struct Slice {
  int start;           // its labels
  uint16_t len, first; // how many, and of those its first unit
  int part0, parts;    // its first partial among a row's, and a row's partials
};
__host__ __device__ inline int slice_labels(int N) { return (N + 31) / 32 * 4; }
__host__ __device__ inline Slice slice_of(int N, int CS, int rank) {
  const int nl = slice_labels(N), u0 = (nl + 7) / 8 * 4, u1 = nl - u0;
  const int p0 = (u0 + kMB - 1) / kMB, p1 = (u1 + kMB - 1) / kMB;
  Slice s;
  s.parts = 8 * (p0 + p1);
  if (CS == 8) {
    s.start = rank * nl, s.len = (uint16_t)nl, s.first = (uint16_t)u0, s.part0 = rank * (p0 + p1);
  } else {
    const int h = rank & 1;
    s.start = (rank >> 1) * nl + h * u0, s.len = s.first = (uint16_t)(h ? u1 : u0), s.part0 = (rank >> 1) * (p0 + p1) + h * p0;
  }
  return s;
}

// A block of a slice that the product takes at once: its end, and a lane's four
// labels in it (from its start; -1: none).  A slice of at most kMB labels is one
// block, its units on half a warp each; otherwise blocks end with their unit.
struct Block {
  int end;
  bool halves;
};
__device__ __forceinline__ Block block_at(const Slice& s, int m0) {
  if (s.len <= kMB) return {s.len, s.first < s.len};
  return {min(m0 + kMB, m0 < s.first ? s.first : s.len), false};
}
__device__ __forceinline__ int lane_labels(const Slice& s, const Block& b, int m0, int lane) {
  if (!b.halves) return 4 * lane < b.end - m0 ? 4 * lane : -1;
  const int o = (lane >> 4) * s.first + 4 * (lane & 15);
  return o < (lane < 16 ? s.first : s.len) ? o : -1;
}

// Shared-memory layout of a CTA (bytes from the 128-byte-aligned base).
struct Layout {
  int w, part, ps, dflt, uni, root, y, bars, rows, row_bytes, logits, lse, term, mark, list, total;
};
__host__ __device__ inline Layout layout(int N, int H, int V4, int nl, int CS, int NB, int RG) {
  Layout L;
  auto up = [](int x) { return (x + 15) & ~15; };
  int o = 0;
  L.bars = o, o += 128;                      // ybar, wbar, lbar[RG], sbar[RG][kPartBars], fail flag, slice
  L.y = o, o = up(o + 16 * CS * RG);         // every row's (previous label, frame or -1, fused value, output place or -1)
  L.w = o, o = up(o + nl * (2 * H + kWPad));
  // row stride of the partials, 4 mod 16: lanes (n = 2c, m = g) fall in different banks
  L.ps = ((nl < kMB ? nl : kMB) + 11) / 16 * 16 + 4;
  L.part = o, o = up(o + 8 * (8 * NB) * L.ps * 4);
  L.dflt = o, o = up(o + 4 * V4);            // the call's defaults D
  L.uni = o, o = up(o + 4 * V4);             // log p(v)
  L.root = o, o = up(o + (V4 + 31) / 32 * 4);
  L.rows = o;
  int r = up((int)sizeof(RowSm));
  L.logits = r, r = up(r + 4 * CS * nl);
  L.lse = r, r = up(r + kPartBufs * 8 * slice_of(N, CS, 0).parts);  // softmax partials
  L.term = r, r = up(r + 4 * V4);
  L.mark = r, r = up(r + 4 * V4);                               // levels and trie depths, 16 bits each
  L.list = RG < 3 ? r : -1;                  // level 0's labels
  if (RG < 3) r = up(r + 4 * V4 + 32);
  L.row_bytes = r;
  L.total = o + RG * r + 128;                // and the alignment of the base
  return L;
}

struct Ctx {
  unsigned char* sm;
  Layout L;
  uint64_t *ybar, *wbar, *lbar, *sbar;
  volatile int* fail;
  int4* y;
  const Slice* sl;  // in shared memory: the product's warps have few registers to spare
  int CS, rank, R, row0;
};

// ---------------------------------------------------------------- GEMM warps

// A lane's piece of a row's joint input operands: elements 32 un + 8 k4 ..
// of its encoder frame and of its previous label's embedding.
struct Piece {
  uint4 x[kUnits], z[kUnits];
};

// One block of HT half tiles of 8 labels from label m0 of the slice: this
// warp's part of H for 8 NB rows, written to the partials [warp][row][label].
// Labels past the slice read its last row again, and the upper half of an odd
// last tile its lower half: their sums are never sent.
// FU >= 0: every warp has FU pieces of H (H / 256) and some one more; -1: any number.
template <int HT, int NB, int FU>
__device__ __forceinline__ void tile_block(const unsigned char* W, int wstride, int nl, int m0, int U, int warp, int g, int k4,
                                           const uint4 (&b)[kUnits][NB], float* part, int ps) {
  constexpr int MT = (HT + 1) / 2;
  float acc[MT][NB][4];
  int off[HT];
#pragma unroll
  for (int t = 0; t < HT; ++t) off[t] = min(m0 + 8 * t + g, nl - 1) * wstride + k4 * 16;
#pragma unroll
  for (int t = 0; t < MT; ++t)
#pragma unroll
    for (int j = 0; j < NB; ++j)
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[t][j][x] = 0.f;
#pragma unroll
  for (int u = 0; u < kUnits; ++u) {
    const int un = warp + 8 * u;
    if (FU >= 0 && u > FU) break;
    if ((FU >= 0 && u < FU) || un < U) {
      uint4 a[HT];
#pragma unroll
      for (int t = 0; t < HT; ++t) a[t] = *reinterpret_cast<const uint4*>(W + off[t] + un * 64);
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int t = 0; t < MT; ++t)
#pragma unroll
          for (int j = 0; j < NB; ++j) {
            const uint4 lo = a[2 * t], hi = a[2 * t + 1 < HT ? 2 * t + 1 : 2 * t];
            if (h == 0) mma16816(acc[t][j], lo.x, hi.x, lo.y, hi.y, b[u][j].x, b[u][j].y);
            else mma16816(acc[t][j], lo.z, hi.z, lo.w, hi.w, b[u][j].z, b[u][j].w);
          }
    }
  }
#pragma unroll
  for (int t = 0; t < MT; ++t)
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      float* o = part + (warp * 8 * NB + 8 * j + 2 * k4) * ps + 16 * t + g;
      if (16 * t + g < ps) o[0] = acc[t][j][0], o[ps] = acc[t][j][1];
      if (2 * t + 1 < HT && 16 * t + 8 + g < ps) o[8] = acc[t][j][2], o[ps + 8] = acc[t][j][3];
    }
}

// Row n's logits of four labels of the block from o: the warps' partials in a fixed order.
template <int NB>
__device__ __forceinline__ float4 sum_parts(const float* part, int n, int ps, int o) {
  float4 s[8];
#pragma unroll
  for (int w = 0; w < 8; ++w) s[w] = *reinterpret_cast<const float4*>(part + (w * 8 * NB + n) * ps + o);
#pragma unroll
  for (int h = 1; h < 8; h *= 2)
#pragma unroll
    for (int w = 0; w < 8; w += 2 * h) {
      s[w].x += s[w + h].x;
      s[w].y += s[w + h].y;
      s[w].z += s[w + h].z;
      s[w].w += s[w + h].w;
    }
  return s[0];
}

// A unit's softmax partial (max, sum of exp(x - max)), by a warp whose lanes hold
// four logits each, nv of them labels.  halves: two units, of 16 lanes each
// (every lane gets its own unit's; the sums' order is that of a unit alone).
__device__ __forceinline__ float2 unit_softmax(float4 v, int nv, bool halves, int lane) {
  const float l[4] = {nv > 0 ? v.x : kNegInf, nv > 1 ? v.y : kNegInf, nv > 2 ? v.z : kNegInf, nv > 3 ? v.w : kNegInf};
  const int key = order_key(fmaxf(fmaxf(l[0], l[1]), fmaxf(l[2], l[3])));
  const int low = __reduce_max_sync(0xffffffffu, halves && lane >= 16 ? INT_MIN : key);
  const int high = __reduce_max_sync(0xffffffffu, halves && lane < 16 ? INT_MIN : key);
  const int top = lane < 16 ? low : high;
  const float m = key_value(top);
  const float m2 = m * tc::kLog2e;
  float z = 0.f;
  if (m != kNegInf)
    z = (tc::ex2_approx(fmaf(l[0], tc::kLog2e, -m2)) + tc::ex2_approx(fmaf(l[1], tc::kLog2e, -m2))) +
        (tc::ex2_approx(fmaf(l[2], tc::kLog2e, -m2)) + tc::ex2_approx(fmaf(l[3], tc::kLog2e, -m2)));
  const float other = __shfl_xor_sync(0xffffffffu, z, 16);
  z = halves ? z : z + other;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  return make_float2(m, z);
}

// Whether the product may take its rows in several passes of 8 NB.
__host__ __device__ constexpr bool several_passes(int NB, int RG) { return RG == 3 || (RG == 1 && NB == 1); }

template <int NB, int RG, int FU>
__device__ void gemm_loop(const DecView& d, const ChunkArgs& P, const Ctx& c) {
  constexpr bool kPasses = several_passes(NB, RG);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, k4 = lane & 3;
  const int U = d.H / 32, H = d.H, ps = c.L.ps;
  const int wstride = 2 * H + kWPad;
  const unsigned char* W = c.sm + c.L.w;
  float* part = reinterpret_cast<float*>(c.sm + c.L.part);
  const uint32_t sm0 = tc::smem_u32(c.sm);
  // Warp q < RG also finishes the scores of the CTA's row q: a step's softmax
  // partials are consumed one step later, while the warp would wait for the
  // next labels.
  const int own = warp * c.CS + c.rank;
  const bool mine = warp < RG && own < c.R;
  Slice sl;  // what the product needs of the slice stays in registers
  sl.start = c.sl->start, sl.len = c.sl->len, sl.first = c.sl->first;
  bool armed = false, ok = true;
  // this warp's operands of row i (zero for a finished row or none)
  auto load = [&](int i, Piece& q) {
    const int4 st = i < c.R ? c.y[i] : make_int4(0, -1, 0, -1);
    const uint4* e = reinterpret_cast<const uint4*>(P.enc + ((size_t)(c.row0 + i) * P.T + max(st.y, 0)) * H) + k4;
    const uint4* m = reinterpret_cast<const uint4*>(d.E + (size_t)st.x * H) + k4;
#pragma unroll
    for (int u = 0; u < kUnits; ++u) {
      const int un = warp + 8 * u;
      q.x[u] = q.z[u] = make_uint4(0u, 0u, 0u, 0u);
      if (un < U && st.y >= 0) {
        q.x[u] = __ldg(e + 4 * un);
        q.z[u] = __ldg(m + 4 * un);
      }
    }
  };
  for (int step = 0; ; ++step) {
    // the rows' labels (at first, W_out's slice as well)
    ok = wait_cluster(c.ybar, step & 1, d.wait_ns, c.fail) && ok;
    if (step == 0) ok = ok && wait_cluster(c.wbar, 0, d.wait_ns, c.fail);
    if (!group_all(1, kGemm, ok)) {
      if (tid == 0) atomicOr(d.err, 1);
      *c.fail = 1;
      return;
    }
    Piece q[NB];
    if (RG < 3) {  // (the first pass's: requested before the bookkeeping)
#pragma unroll
      for (int j = 0; j < NB; ++j) load(8 * j + g, q[j]);
    }
    int active = 0;  // rows still decoding: the next step's publishers
    for (int i = lane; i < c.R; i += 32) active += c.y[i].y >= 0 ? 1 : 0;
    active = __reduce_add_sync(0xffffffffu, active);
    if (tid == 0 && active) tc::mbar_expect_tx(c.ybar, 16u * (uint32_t)active);
    int4 said = make_int4(0, -1, 0, -1);  // the row's label of the step before
    bool score = false;
    if (mine) {
      said = c.y[own];
      if (armed) {  // the step before's partials are all in; before this CTA sends any logits of this step
        ok = __all_sync(0xffffffffu, wait_cluster(c.sbar + kPartBars * warp + part_bar(step - 1), part_parity(step - 1),
                                                  d.wait_ns, c.fail));
        score = ok && said.w >= 0;
      }
      armed = ok && said.y >= 0;
      if (armed && lane == 0)
        tc::mbar_expect_tx(c.sbar + kPartBars * warp + part_bar(step), 8u * (uint32_t)c.sl->parts);
    }
    auto write_score = [&]() {
      const float2* sp = reinterpret_cast<const float2*>(c.sm + c.L.rows + warp * c.L.row_bytes + c.L.lse) +
                         part_buf(step - 1) * c.sl->parts;
      float m = kNegInf, z = 0.f;
      for (int x = lane; x < c.sl->parts; x += 32) lse_merge(m, z, sp[x].x, sp[x].y);
      const float lse = row::warp_lse(m, z);
      if (lane == 0) P.out_score[(size_t)(c.row0 + own) * (P.T * d.max_sym) + said.w] = __int_as_float(said.z) - lse;
    };
    if (active == 0) {
      if (score) write_score();
      if (!ok) {
        if (lane == 0) atomicOr(d.err, 8);
        *c.fail = 1;
      }
      return;
    }
#pragma unroll 1
    for (int i0 = 0; i0 < (kPasses ? c.R : 1); i0 += 8 * NB) {
      // the joint inputs, bf16(ReLU(enc + E)); a lane's eight consecutive
      // elements feed two 16-deep MMAs (the same order of H in both operands)
      uint4 b[kUnits][NB];
      if (RG == 3 || (kPasses && i0 > 0)) {
#pragma unroll
        for (int j = 0; j < NB; ++j) load(i0 + 8 * j + g, q[j]);
      }
#pragma unroll
      for (int u = 0; u < kUnits; ++u)
#pragma unroll
        for (int j = 0; j < NB; ++j) b[u][j] = joint8(q[j].x[u], q[j].z[u]);
      __syncwarp();
      int p0 = 0;
      for (int m0 = 0; m0 < sl.len;) {
        const Block bl = block_at(sl, m0);
        const int left = bl.end - m0;
        if (left > 72) tile_block<10, NB, FU>(W, wstride, sl.len, m0, U, warp, g, k4, b, part, ps);
        else if (left > 64) tile_block<9, NB, FU>(W, wstride, sl.len, m0, U, warp, g, k4, b, part, ps);
        else if (left > 48) tile_block<8, NB, FU>(W, wstride, sl.len, m0, U, warp, g, k4, b, part, ps);
        else if (left > 32) tile_block<6, NB, FU>(W, wstride, sl.len, m0, U, warp, g, k4, b, part, ps);
        else if (left > 16) tile_block<4, NB, FU>(W, wstride, sl.len, m0, U, warp, g, k4, b, part, ps);
        else tile_block<2, NB, FU>(W, wstride, sl.len, m0, U, warp, g, k4, b, part, ps);
        const int lo = lane_labels(sl, bl, m0, lane), v0 = sl.start + m0 + lo;
        // the warps' partials summed in a fixed order and sent to the rows' owners
        group_sync(1, kGemm);
        float4 sum[NB];
        bool on[NB];  // read before the sends: a row's next label may follow its logits at once
#pragma unroll
        for (int j = 0; j < NB; ++j) on[j] = i0 + 8 * j + warp < c.R && c.y[i0 + 8 * j + warp].y >= 0;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          const int n = 8 * j + warp, i = i0 + n;
          if (!on[j] || lo < 0) continue;
          const int grp = i / c.CS, owner = i - grp * c.CS;
          sum[j] = sum_parts<NB>(part, n, ps, lo);
          const uint32_t dst = sm0 + c.L.rows + grp * c.L.row_bytes + c.L.logits + 4 * v0;
          send16(map_rank(dst, owner), sum[j], map_rank(tc::smem_u32(c.lbar + grp), owner));
        }
        // the units' softmax partials (max, sum of exp) follow: an emitted
        // label's score needs them, one step later
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          const int i = i0 + 8 * j + warp;
          __syncwarp();
          if (!on[j]) continue;  // the same for the warp's lanes
          const int grp = i / c.CS, owner = i - grp * c.CS;
          const float2 p = unit_softmax(sum[j], lo >= 0 ? d.N - v0 : 0, bl.halves, lane);
          if (lane == 0 || (bl.halves && lane == 16)) {
            const uint32_t dst = sm0 + c.L.rows + grp * c.L.row_bytes + c.L.lse +
                                 8 * (part_buf(step) * c.sl->parts + c.sl->part0 + p0 + (lane >> 4));
            send8(map_rank(dst, owner), __float_as_int(p.x), __float_as_int(p.y),
                  map_rank(tc::smem_u32(c.sbar + kPartBars * grp + part_bar(step)), owner));
          }
        }
        __syncwarp();
        group_sync(1, kGemm);
        m0 = bl.end;
        p0 += 1;
      }
    }
    if (score) write_score();
  }
}

// ---------------------------------------------------------------- row groups

template <int GT>
__device__ void row_loop(const DecView& d, const ChunkArgs& P, const Ctx& c, int grp) {
  constexpr int WG = GT / 32;  // warps of the group
  static_assert(WG >= 2 && WG <= 4, "the chains are assembled by two warps");
  const int tid = ((int)threadIdx.x - kGemm) % GT, lane = tid & 31, warp = tid >> 5;
  const int i = grp * c.CS + c.rank;  // the row's place in the cluster
  const int r = c.row0 + i;
  const int bar = 2 + grp;
  const int V = d.V, T = P.T, Q = d.V4 / 4;
  unsigned char* rs = c.sm + c.L.rows + grp * c.L.row_bytes;
  RowSm& s = *reinterpret_cast<RowSm*>(rs);
  const float* lg = reinterpret_cast<const float*>(rs + c.L.logits);
  float* term = reinterpret_cast<float*>(rs + c.L.term);          // every label's c_r + delta (while built: its LM delta / lambda)
  // per label: the LM chain levels above 0 with an arc for it (bit l), and its trie goto depth (0: none); apart,
  // because the first is set by 32-bit atomics (two labels each) while the second is stored
  uint16_t* lev = reinterpret_cast<uint16_t*>(rs + c.L.mark);
  uint16_t* dep = lev + d.V4;
  int* list = c.L.list >= 0 ? reinterpret_cast<int*>(rs + c.L.list) : nullptr;  // level 0's labels from its aligned first arc
  const float* dflt = reinterpret_cast<const float*>(c.sm + c.L.dflt);
  const float* uni = reinterpret_cast<const float*>(c.sm + c.L.uni);
  const uint32_t* root = reinterpret_cast<const uint32_t*>(c.sm + c.L.root);
  const bool lm2 = d.has_lm && d.lm.order >= 2;
  const float lam = P.lambda;
  const float bscale = P.beta * (d.has_tr ? d.tr.bonus : 0.f);
  const uint32_t y_addr = tc::smem_u32(c.y + i), y_bar = tc::smem_u32(c.ybar);
  auto sync = [&]() { group_sync(bar, GT); };

  // the row's label, frame (-1: finished) and the label's score to be, to every CTA of the cluster
  auto publish = [&](int last, int t, float best, int at) {
    if (tid < c.CS)
      send16(map_rank(y_addr, tid),
             make_float4(__int_as_float(last), __int_as_float(t < T ? t : -1), best, __int_as_float(at)), map_rank(y_bar, tid));
  };

  // state of the stream
  const int slot = P.slots[r];
  int last = __ldcg(d.s_last + slot);
  if (!checked(slot >= 0 && slot < d.lm_stride && last >= 0 && last <= V, d.err, 1)) last = V;
  publish(last, 0, 0.f, -1);
  if (tid == 0) {
    s.nl = d.has_lm ? __ldcg(d.s_lm_len + slot) : 0;
    s.nt = d.has_tr ? __ldcg(d.s_tr_len + slot) : 0;
  }
  if (d.has_lm && warp == 0 && lane < kLmChain) {
    s.lm[lane] = __ldcg(d.s_lm_chain + (size_t)slot * kLmChain + lane);
    s.lmr[lane] = __ldcg(d.s_lm_rec + (size_t)slot * kLmChain + lane);
  }
  if (d.has_tr && warp == 1) {
    s.tr[lane] = __ldcg(d.s_tr_chain + (size_t)slot * kTrChain + lane);
    s.trr[lane] = __ldcg(d.s_tr_rec + (size_t)slot * kTrChain + lane);
  }
  sync();
#ifdef TSD_CHECKS
  if (tid == 0) {
    bool ok = checked(s.nl >= 0 && s.nl <= kLmChain && s.nt >= 0 && s.nt <= kTrChain, d.err, 2);
    for (int l = 0; ok && l < s.nl; ++l) {
      const int4 q = s.lmr[l];
      ok = checked(s.lm[l] >= 0 && s.lm[l] < d.lm.n_states, d.err, 4) &&
           checked(q.x >= 0 && q.y >= 0 && (int64_t)q.x + q.y <= d.lm.n_arcs, d.err, 5) &&
           checked(l > 0 || (q.w >= 0 && q.w < d.lm.n_dense), d.err, 6);
    }
    for (int k = 0; ok && k < s.nt; ++k) {
      const int4 q = s.trr[k];
      ok = checked(s.tr[k] > 0 && s.tr[k] < d.tr.n_nodes, d.err, 7) &&
           checked(q.x >= 0 && q.y >= 0 && q.x + q.y <= d.tr.n_children && q.z >= 1 && q.z <= 63, d.err, 8);
    }
    if (!ok) s.nl = s.nt = 0;  // the row goes on from the empty context; the status word says so
  }
  sync();
#endif

  const int4* t4 = reinterpret_cast<const int4*>(d.lm.arc_tok);
  const float4* p4 = reinterpret_cast<const float4*>(d.lm.arc_logp);
  auto copy16 = [](void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
  };
  // level 0 of the deltas: label u's dense row by asynchronous copies (u < 0:
  // no LM state, every delta 0), and levels and depths cleared
  auto begin_deltas = [&](int u) {
    const float* R = d.lm.dense0 + (size_t)max(u, 0) * d.lm.V4;
    for (int q = tid; q < Q; q += GT) {
      if (u >= 0) copy16(term + 4 * q, R + 4 * q);
      else reinterpret_cast<float4*>(term)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
      reinterpret_cast<uint2*>(lev)[q] = reinterpret_cast<uint2*>(dep)[q] = make_uint2(0u, 0u);
    }
  };
  // A thread's group of four arcs of the levels above 0 (level hl, first arc
  // hi) and its groups of children of the trie chain's first nodes: kept from
  // the deltas, which need them, to the search of the next label.  more: the
  // chains have arcs or children that no thread holds.
  int hl = -1, hi = 0;
  int4 ht, ct[kTrHeld];
  bool more = false;
  // the levels above 0 and the trie chain: every arc sets its level's bit,
  // then the deepest level's arc overwrites its label's delta
  // (row_stream.cu); then every label's term c_r + lambda * delta + trie
  auto finish_deltas = [&]() {
    const int nl = s.nl, nt = s.nt;
    float4 hp;
    int G = 0;
    hl = -1;
    for (int l = 1; l < nl; ++l) {
      const int4 q = s.lmr[l];
      const int n = level_groups(q.x, q.y);
      if (tid >= G && tid < G + n) hl = l, hi = (q.x & ~3) + 4 * (tid - G);
      G += n;
    }
    if (hl >= 0) {
      ht = __ldg(t4 + (hi >> 2));
      hp = __ldg(p4 + (hi >> 2));
    }
    more = G > GT || nt > kTrHeld;
#pragma unroll
    for (int k = 0; k < kTrHeld; ++k)
      if (k < nt) {
        const int4 q = s.trr[k];
        const int n = level_groups(q.x, q.y);
        if (tid < n) ct[k] = __ldg(reinterpret_cast<const int4*>(d.tr.ch_tok) + (q.x >> 2) + tid);
        more = more || n > GT;
      }
    if (list && nl > 0) {
      const int4 q = s.lmr[0];
      const int n = level_groups(q.x, q.y);
      for (int g = tid; g < n; g += GT) copy16(list + 4 * g, t4 + (q.x >> 2) + g);
    }
    auto children = [&](int k, int4 tk, int g) {  // node k's children of group g
      const int4 q = s.trr[k];
      const int i0 = (q.x & ~3) + 4 * g;
      const int tv[4] = {tk.x, tk.y, tk.z, tk.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (i0 + j >= q.x && i0 + j < q.x + q.y) dep[tv[j]] = (uint16_t)q.z;
    };
    auto scatter = [&](int k) {
      const int4 q = s.trr[k];
      const int n = level_groups(q.x, q.y);
#pragma unroll
      for (int h = 0; h < kTrHeld; ++h)
        if (h == k && tid < n) children(k, ct[h], tid);
      for (int g = tid + (k < kTrHeld ? GT : 0); g < n; g += GT)
        children(k, __ldg(reinterpret_cast<const int4*>(d.tr.ch_tok) + (q.x >> 2) + g), g);
    };
    // set: the arcs of level l from i0 set its bit (settle false), or the
    // labels whose deepest level it is take its delta
    auto arcs = [&](int l, int i0, int4 tk, float4 lq, bool settle) {
      const int4 q = s.lmr[l];
      const float cum = __int_as_float(q.z);
      const int tv[4] = {tk.x, tk.y, tk.z, tk.w};
      const float pv[4] = {lq.x, lq.y, lq.z, lq.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (i0 + j >= q.x && i0 + j < q.x + q.y && checked(tv[j] >= 0 && tv[j] < V, d.err, 9)) {
          if (!settle) atomicOr(reinterpret_cast<uint32_t*>(lev) + (tv[j] >> 1), 1u << (l + 16 * (tv[j] & 1)));
          else if (nl == 2 || (lev[tv[j]] >> l) == 1) term[tv[j]] = (pv[j] - cum) - uni[tv[j]];
        }
    };
    // past what a thread holds (rare: more than four times GT arcs above level 0)
    auto rest = [&](bool settle) {
#pragma unroll 1
      for (int g0 = tid + GT; g0 < G; g0 += GT) {
        int l = 1, g = g0;
        for (;; ++l) {
          const int n = level_groups(s.lmr[l].x, s.lmr[l].y);
          if (g < n) break;
          g -= n;
        }
        const int i0 = (s.lmr[l].x & ~3) + 4 * g;
        arcs(l, i0, __ldg(t4 + (i0 >> 2)), __ldg(p4 + (i0 >> 2)), settle);
      }
    };
    if (nl > 2) {  // (with one level above 0 every arc of it is its label's deepest)
      if (hl >= 0) arcs(hl, hi, ht, hp, false);
      rest(false);
    }
    if (nt > 0) scatter(nt - 1);  // the trie chain nodes, shallowest first (the deepest overwrites)
    asm volatile("cp.async.wait_all;" ::: "memory");
    sync();
    if (tid < kLmChain) s.lm_hit[tid] = make_int4(-2, 0, 0, 0);  // (the last search's records were read before the barrier)
    if (tid < kTrChain) s.tr_hit[tid] = make_int4(-1, 0, 0, 0);
    if (hl >= 0) arcs(hl, hi, ht, hp, true);
    rest(true);
    for (int k = nt - 2; k >= 0; --k) {
      scatter(k);
      if (k) sync();
    }
    sync();
    const float cr = row::row_constant(lam, nl ? __int_as_float(s.lmr[nl - 1].z) : 0.f, bscale, nt ? s.trr[0].z - 1 : 0);
    for (int q = tid; q < Q; q += GT) {
      const float4 kq = reinterpret_cast<const float4*>(term)[q];
      uint32_t mv[4] = {0u, 0u, 0u, 0u}, rb = 0u;
      if (nt) {
        const uint2 mq = reinterpret_cast<const uint2*>(dep)[q];
        mv[0] = mq.x & 0xffffu, mv[1] = mq.x >> 16, mv[2] = mq.y & 0xffffu, mv[3] = mq.y >> 16;
        if (mv[0] | mv[1] | mv[2] | mv[3]) rb = root[q >> 3] >> ((4 * q) & 31);
      }
      const float x[4] = {kq.x, kq.y, kq.z, kq.w};
      float o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {  // (labels past V never win)
        o[j] = __fmul_rn(lam, x[j]);
        if (mv[j]) o[j] = row::trie_delta(o[j], mv[j], (rb >> j) & 1u, bscale);
        o[j] = 4 * q + j < V ? __fadd_rn(cr, o[j]) : kNegInf;
      }
      reinterpret_cast<float4*>(term)[q] = make_float4(o[0], o[1], o[2], o[3]);
    }
    // (a thread reads back only what it wrote here: no barrier)
  };
  auto find_list = [&](int y) {  // y's place among level 0's labels, or -1 (one warp)
    const int n = s.lmr[0].y;
    const int* a = list + (s.lmr[0].x & 3);
    int lo = 0, hi = n;
    __syncwarp();
    while (hi - lo > 32) {
      const int w = (hi - lo + 31) >> 5, at = lo + lane * w;
      const unsigned m = __ballot_sync(0xffffffffu, at < hi && a[at] <= y);
      if (m == 0) return -1;
      lo += (31 - __clz((int)m)) * w;
      hi = min(hi, lo + w);
    }
    const unsigned m = __ballot_sync(0xffffffffu, lo + lane < hi && a[lo + lane] == y);
    return m ? lo + __ffs((int)m) - 1 : -1;
  };

  int t = 0, sym = 0, cnt = 0, step = 0;
  const uint32_t row_bytes = 32u * (uint32_t)slice_labels(d.N);
  bool ok = true, moved = true;
  begin_deltas(s.nl > 0 ? s.lmr[0].w : -1);
  sync();  // levels and depths are cleared before anyone sets one
  while (t < T) {
    if (tid == 0) tc::mbar_expect_tx(c.lbar + grp, row_bytes);
    if (moved) finish_deltas();
    if (d.cap_rows && step < d.cap_steps && tid == 0) {
      int* q = d.cap_rows + ((size_t)step * P.n + r) * 4;
      q[0] = t;
      q[1] = last;
      q[2] = s.nl ? s.lm[s.nl - 1] : 0;
      q[3] = s.nt ? s.tr[0] : 0;
    }
    // the argmax of (logit + D) + (c_r + delta) over the labels (blank: its logit alone)
    ok = __all_sync(0xffffffffu, wait_cluster(c.lbar + grp, step & 1, d.wait_ns, c.fail));
    float bv = kNegInf;
    int bi = INT_MAX;
    if (ok) {
      for (int q = tid; q < Q; q += GT) {
        const float4 lq = reinterpret_cast<const float4*>(lg)[q];
        const float4 uq = reinterpret_cast<const float4*>(dflt)[q];
        const float4 kq = reinterpret_cast<const float4*>(term)[q];
        const float fv[4] = {(lq.x + uq.x) + kq.x, (lq.y + uq.y) + kq.y, (lq.z + uq.z) + kq.z, (lq.w + uq.w) + kq.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (fv[j] > bv) { bv = fv[j]; bi = 4 * q + j; }
      }
      if (tid == 0) {
        const float fb = lg[V];
        if (fb > bv) { bv = fb; bi = V; }
      }
    }
    __syncwarp();
    {
      const int key = order_key(bv + 0.f), top = __reduce_max_sync(0xffffffffu, key);
      bi = __reduce_min_sync(0xffffffffu, key == top ? bi : INT_MAX);
      bv = key_value(top);
    }
    if (d.cap_logits && step < d.cap_steps) {  // (before the label is out: the next step's logits land here)
      float* cl = d.cap_logits + ((size_t)step * P.n + r) * d.N;
      for (int v = tid; v < d.N; v += GT) cl[v] = lg[v];
    }
    if (lane == 0) s.best[step & 1][warp] = make_int4(__float_as_int(bv), bi, ok ? 1 : 0, 0);
    sync();
    float best = kNegInf;
    int bix = INT_MAX;
#pragma unroll
    for (int w = 0; w < WG; ++w) {
      const int4 q = s.best[step & 1][w];
      best_merge(best, bix, __int_as_float(q.x), q.y);
      ok = ok && q.z;
    }
    if (!ok) {  // the group's threads leave together
      if (tid == 0) atomicOr(d.err, 4);
      *c.fail = 1;
      break;
    }
    const int y = (bix >= 0 && bix <= V) ? bix : V;
    // the row's next position, to every CTA before anything else
    const int t_now = t;
    moved = y != V;
    if (moved) {
      last = y;
      sym += 1;
      if (sym >= d.max_sym) { t += 1; sym = 0; }
    } else {
      t += 1;
      sym = 0;
    }
    publish(last, t, best, moved ? cnt : -1);
    ++step;
    if (!moved) continue;
    // the label's records in every chain element, all in one round: above
    // level 0 a thread that holds the label's arc (or trie child) fetches its
    // record, level 0's labels are searched in shared memory; level 0 of the
    // next deltas is copied meanwhile
    {
      const int nl = s.nl, nt = s.nt;
      auto held = [&](int4 tk, int i0, int4 q) {  // the label's place among four entries from i0 of the range q, or -1
        int at = -1;
        const int tv[4] = {tk.x, tk.y, tk.z, tk.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (tv[j] == y && i0 + j >= q.x && i0 + j < q.x + q.y) at = i0 + j;
        return at;
      };
      int a_lm = hl >= 0 ? held(ht, hi, s.lmr[hl]) : -1;
      int4 r_lm, r_tr[kTrHeld], top;
      if (a_lm >= 0) r_lm = __ldg(d.lm.arc_rec + a_lm);
      int a_tr[kTrHeld];
#pragma unroll
      for (int k = 0; k < kTrHeld; ++k) {
        a_tr[k] = -1;
        if (k < nt) {
          const int4 q = s.trr[k];
          if (tid < level_groups(q.x, q.y)) a_tr[k] = held(ct[k], (q.x & ~3) + 4 * tid, q);
          if (a_tr[k] >= 0) r_tr[k] = __ldg(d.tr.ch_rec + a_tr[k]);
        }
      }
      if (tid == GT - 1) top = d.has_tr ? __ldg(d.tr.root_rec + y) : make_int4(0, 0, 0, 0);
      if (tid == GT - 2) top = lm2 ? __ldg(d.lm.uni_rec + y) : make_int4(-1, 0, 0, 0);
      int a0 = -1;
      int4 r0;
      if (warp == 0 && nl > 0) {
        const int4 q = s.lmr[0];
        a0 = list ? find_list(y) : warp_find_wide<true>(d.lm.arc_tok + q.x, q.y, y, lane, first_load(d.lm.arc_tok + q.x, q.y, lane));
        if (lane == 0 && a0 >= 0) r0 = __ldg(d.lm.arc_rec + q.x + a0);
      }
      if (t < T) begin_deltas(lm2 ? y : -1);
      if (a_lm >= 0) s.lm_hit[hl] = r_lm;
#pragma unroll
      for (int k = 0; k < kTrHeld; ++k)
        if (a_tr[k] >= 0) s.tr_hit[k] = r_tr[k], s.dd[k] = s.trr[k].z + 1;
      if (tid == GT - 1) s.root_hit = top;
      if (tid == GT - 2) s.uni_hit = top;
      if (warp == 0 && lane == 0 && a0 >= 0) s.lm_hit[0] = r0;
      if (tid == 32) {
        const size_t o = (size_t)r * (T * d.max_sym) + cnt;
        P.out_tok[o] = y;
        P.out_frame[o] = t_now;
      }
      if (more) {  // elements whose entries the threads do not all hold: searched by warps
#pragma unroll 1
        for (int task = 1 + warp; task < nl + nt; task += WG) {
          const bool is_lm = task < nl;
          const int4 q = is_lm ? s.lmr[task] : s.trr[task - nl];
          const int32_t* arr = (is_lm ? d.lm.arc_tok : d.tr.ch_tok) + q.x;
          const int at = warp_find_wide<true>(arr, q.y, y, lane, first_load(arr, q.y, lane));
          if (lane == 0 && at >= 0) {
            if (is_lm) s.lm_hit[task] = __ldg(d.lm.arc_rec + q.x + at);
            else s.tr_hit[task - nl] = __ldg(d.tr.ch_rec + q.x + at), s.dd[task - nl] = q.z + 1;
          }
        }
        if (nl == 0 && warp == 0 && nt > 0) {  // (no LM chain: the first task is the deepest trie node)
          const int4 q = s.trr[0];
          const int at = warp_find_wide<true>(d.tr.ch_tok + q.x, q.y, y, lane, first_load(d.tr.ch_tok + q.x, q.y, lane));
          if (lane == 0 && at >= 0) s.tr_hit[0] = __ldg(d.tr.ch_rec + q.x + at), s.dd[0] = q.z + 1;
        }
      }
      sync();
      // the new chains, in place, by every warp alike (the same values, so no
      // barrier follows): the LM chain is y's unigram state, then the targets
      // of y's arcs up to the first level without one; the trie chain y's
      // children of the old nodes, deepest first, then the root's (completing
      // a phrase resets it)
      int ln = 0, tn = 0;
      {
        const int4 h = lane < nl ? s.lm_hit[lane] : make_int4(-2, 0, 0, 0);
        const int4 th = lane < nt ? s.tr_hit[lane] : make_int4(-1, 0, 0, 0);
        const int4 u = s.uni_hit, rh = s.root_hit;
        if (lm2) {
          const bool cont = h.x >= 0 && checked(h.x < d.lm.n_states && h.y >= 0 && h.z >= 0 &&
                                                    (int64_t)h.y + h.z <= d.lm.n_arcs, d.err, 10);
          const unsigned miss = __ballot_sync(0xffffffffu, !cont);
          ln = 1 + min(miss ? __ffs((int)miss) - 1 : 32, kLmChain - 1);
          if (lane == 0) s.lm[0] = 1 + y, s.lmr[0] = make_int4(u.y, u.z, u.w, u.x);
          if (lane + 1 < ln) s.lm[lane + 1] = h.x, s.lmr[lane + 1] = make_int4(h.y, h.z, h.w, 0);
        }
        if (d.has_tr) {
          const bool found = th.x >= 0 && checked(th.x > 0 && th.x < d.tr.n_nodes && th.w >= 0 &&
                                                      th.z + th.w <= d.tr.n_children, d.err, 11);
          const unsigned vm = __ballot_sync(0xffffffffu, found);
          const int nv = __popc(vm), f = __ffs((int)vm) - 1;
          const bool rt = rh.x != 0;
          const int fy = __shfl_sync(0xffffffffu, th.y, f < 0 ? 0 : f);
          const bool reset = nv > 0 ? fy == 0 : (rt && rh.y == 0);
          tn = reset ? 0 : min(nv + (rt ? 1 : 0), kTrChain);
          const int pos = __popc(vm & ((1u << lane) - 1u));
          if (found && pos < tn) s.tr[pos] = th.x, s.trr[pos] = make_int4(th.z, th.w, s.dd[lane], 0);
          if (lane == 0 && rt && nv < tn) s.tr[nv] = rh.x, s.trr[nv] = make_int4(rh.z, rh.w, 2, 0);
        }
        if (lane == 0) s.nl = ln, s.nt = tn;
        __syncwarp();
      }
      cnt += 1;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (!ok) return;
  // the stream's state, once per chunk (and the row's copy of it, which the
  // two-kernel step and its timing replays read)
  if (tid == 0) {
    P.out_count[r] = cnt;
    d.s_last[slot] = last;
    d.m_last[r] = last;
    d.r_t[r] = T;
    d.r_sym[r] = 0;
    d.r_cnt[r] = cnt;
    if (d.has_lm) d.s_lm_len[slot] = s.nl;
    if (d.has_tr) d.s_tr_len[slot] = s.nt;
    d.m_lm_len[r] = s.nl;
    d.m_tr_len[r] = s.nt;
  }
  if (warp == 0 && lane < s.nl) {
    d.s_lm_chain[(size_t)slot * kLmChain + lane] = s.lm[lane];
    d.s_lm_rec[(size_t)slot * kLmChain + lane] = s.lmr[lane];
    d.m_lm[(size_t)r * kLmChain + lane] = s.lm[lane];
    d.m_lmr[(size_t)r * kLmChain + lane] = s.lmr[lane];
  }
  if (warp == 1 && lane < s.nt) {
    d.s_tr_chain[(size_t)slot * kTrChain + lane] = s.tr[lane];
    d.s_tr_rec[(size_t)slot * kTrChain + lane] = s.trr[lane];
    d.m_tr[(size_t)r * kTrChain + lane] = s.tr[lane];
    d.m_trr[(size_t)r * kTrChain + lane] = s.trr[lane];
  }
  if (d.cap_rows)  // steps after the row's last evaluation
    for (int q = step + tid; q < min(d.cap_steps, T * d.max_sym); q += GT)
      reinterpret_cast<int4*>(d.cap_rows)[(size_t)q * P.n + r] = make_int4(-1, -1, -1, -1);
}

// Threads of a row group: with three groups, half as many leave the product's
// warps their registers.
constexpr int group_threads(int RG) { return RG < 3 ? 128 : 64; }

template <int NB, int RG, int FU>
__global__ void __launch_bounds__(kGemm + RG * group_threads(RG), 1)
    k_chunk(const __grid_constant__ DecView d, const __grid_constant__ ChunkArgs P) {
  extern __shared__ __align__(128) unsigned char raw[];
  Ctx c;
  c.sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(raw) + 127) & ~uintptr_t(127));
  c.CS = P.CS;
  c.L = layout(d.N, d.H, d.V4, P.nl, c.CS, NB, RG);
  c.rank = (int)(blockIdx.x % (unsigned)c.CS);
  c.row0 = (int)(blockIdx.x / (unsigned)c.CS) * P.R;
  c.R = min(P.R, P.n - c.row0);
  c.ybar = reinterpret_cast<uint64_t*>(c.sm + c.L.bars);
  c.wbar = c.ybar + 1;
  c.lbar = c.ybar + 2;
  c.sbar = c.lbar + RG;
  int* fail = reinterpret_cast<int*>(c.sbar + kPartBars * RG);
  c.fail = fail;
  c.y = reinterpret_cast<int4*>(c.sm + c.L.y);
  static_assert((2 + (1 + kPartBars) * RG) * 8 + 4 + sizeof(Slice) <= 128, "barrier area");
  Slice* sl = reinterpret_cast<Slice*>(fail + 1);
  c.sl = sl;
  const int tid = threadIdx.x;
  if (tid == 0) {
    const Slice own = slice_of(d.N, c.CS, c.rank);
    *sl = own;
    tc::mbar_init(c.ybar, 1);
    tc::mbar_init(c.wbar, 1);
    for (int g = 0; g < (1 + kPartBars) * RG; ++g) tc::mbar_init(c.lbar + g, 1);  // lbar, then sbar
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tc::mbar_expect_tx(c.ybar, 16u * (uint32_t)c.R);  // the rows' first labels
    // this CTA's labels of W_out, row by row
    tc::mbar_expect_tx(c.wbar, (uint32_t)(own.len * 2 * d.H));
    for (int j = 0; j < own.len; ++j)
      tc::bulk_g2s(c.sm + c.L.w + j * (2 * d.H + kWPad), d.Wt + (size_t)(own.start + j) * d.H, 2u * (uint32_t)d.H, c.wbar);
  }
  // the call's shared rows: the defaults D, log p(v), and the labels that start a phrase
  float* dflt = reinterpret_cast<float*>(c.sm + c.L.dflt);
  float* uni = reinterpret_cast<float*>(c.sm + c.L.uni);
  uint32_t* root = reinterpret_cast<uint32_t*>(c.sm + c.L.root);
  for (int v = tid; v < (d.V4 + 31) / 32 * 32; v += blockDim.x) {
    const bool rc = d.has_tr && v < d.V && __ldg(d.tr.root_child + v) != 0;
    const float u = d.has_lm && v < d.V ? __ldg(d.lm.uni_logp + v) : 0.f;
    if (v < d.V4) dflt[v] = row::default_term(P.lambda, u, rc, P.beta, d.tr.bonus), uni[v] = u;
    const unsigned m = __ballot_sync(0xffffffffu, rc);  // whole warps: the bound is a multiple of 32
    if ((tid & 31) == 0) root[v / 32] = m;
  }
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (tid < kGemm) {
    gemm_loop<NB, RG, FU>(d, P, c);
  } else {
    constexpr int GT = group_threads(RG);
    const int grp = (tid - kGemm) / GT;
    if (grp * c.CS + c.rank < c.R) row_loop<GT>(d, P, c, grp);
  }
  __syncwarp();
  if (*c.fail) {
    // messages and copies in flight land before the CTA's shared memory goes
    tc::mbar_wait(c.wbar, 0);
    const unsigned long long t0 = tc::global_ns();
    while (tc::global_ns() - t0 < 200000ull) __nanosleep(1000);
  }
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The joint kernel of the stateful form with few rows (its label step cannot
// stay in one launch: the prediction network runs between two joint products):
// the same product, sums and softmax partials as the loop above, so that both
// forms give the same bits.  CTA (c, b): slice c of the labels, of rows
// 8 NB b .., its slice of W_out requested before the wait for the joint
// input (further rows follow in steps of the grid); the row pass
// (row_stream.cu) finishes Eq. 1 from the stored logits.
template <int NB>
__global__ void __launch_bounds__(kGemm, 1) k_joint_rows(const __grid_constant__ DecView d, int step, int nl) {
  extern __shared__ __align__(128) unsigned char raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(raw) + 127) & ~uintptr_t(127));
  uint64_t* wbar = reinterpret_cast<uint64_t*>(sm);
  const int H = d.H, U = H / 32, wstride = 2 * H + kWPad;
  const unsigned char* W = sm + 128;
  const int ps = ((nl < kMB ? nl : kMB) + 11) / 16 * 16 + 4;  // as in layout()
  float* part = reinterpret_cast<float*>(sm + 128 + (nl * wstride + 127) / 128 * 128);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, k4 = lane & 3;
  const Slice sl = slice_of(d.N, gridDim.x, blockIdx.x);
  const int n = d.params->n;
  if (tid == 0) {
    tc::mbar_init(wbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tc::mbar_expect_tx(wbar, (uint32_t)(sl.len * 2 * H));
    for (int j = 0; j < sl.len; ++j)
      tc::bulk_g2s(sm + 128 + j * wstride, d.Wt + (size_t)(sl.start + j) * H, 2u * (uint32_t)H, wbar);
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  bool first = true;
#pragma unroll 1
  for (int i0 = blockIdx.y * 8 * NB; i0 < n; i0 += gridDim.y * 8 * NB) {
    uint4 b[kUnits][NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int i = i0 + 8 * j + g;
      const uint4* a = reinterpret_cast<const uint4*>(d.A + (size_t)min(i, n - 1) * H) + k4;
#pragma unroll
      for (int u = 0; u < kUnits; ++u) {
        const int un = warp + 8 * u;
        b[u][j] = un < U && i < n ? __ldcg(a + 4 * un) : make_uint4(0u, 0u, 0u, 0u);
      }
    }
    if (first) {
      first = false;
      const bool ok = __syncthreads_and(tc::mbar_wait(wbar, 0, d.wait_ns) ? 1 : 0);
      if (!ok) {
        if (tid == 0) atomicOr(d.err, 1);
        tc::mbar_wait(wbar, 0);  // the copies land before the CTA's shared memory goes (the long limit)
        return;
      }
    }
    int p0 = sl.part0;
    for (int m0 = 0; m0 < sl.len;) {
      const Block bl = block_at(sl, m0);
      const int left = bl.end - m0;
      if (left > 64) tile_block<10, NB, -1>(W, wstride, sl.len, m0, U, warp, g, k4, b, part, ps);
      else if (left > 32) tile_block<8, NB, -1>(W, wstride, sl.len, m0, U, warp, g, k4, b, part, ps);
      else tile_block<4, NB, -1>(W, wstride, sl.len, m0, U, warp, g, k4, b, part, ps);
      __syncthreads();
      const int lo = lane_labels(sl, bl, m0, lane), v0 = sl.start + m0 + lo;
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const int i = i0 + 8 * j + warp;
        __syncwarp();
        if (i >= n) continue;  // the same for the warp's lanes
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lo >= 0) {
          s = sum_parts<NB>(part, 8 * j + warp, ps, lo);
          const float4 dv = __ldcg(reinterpret_cast<const float4*>(d.dvec + v0));
          *reinterpret_cast<float4*>(d.logits + (size_t)i * d.N_pad + v0) =
              make_float4(s.x + dv.x, s.y + dv.y, s.z + dv.z, s.w + dv.w);
          if (d.cap_logits && step < d.cap_steps) {
            float* cl = d.cap_logits + ((size_t)step * n + i) * d.N + v0;
            const float l[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
            for (int x = 0; x < 4; ++x)
              if (v0 + x < d.N) cl[x] = l[x];
          }
        }
        const float2 p = unit_softmax(s, lo >= 0 ? d.N - v0 : 0, bl.halves, lane);
        if (lane == 0 || (bl.halves && lane == 16))
          d.part[(size_t)i * d.n_ptiles + p0 + (lane >> 4)] = make_float4(p.x, p.y, kNegInf, __int_as_float(INT_MAX));
      }
      __syncthreads();
      m0 = bl.end;
      p0 += 1;
    }
  }
}

int joint_rows_smem(int H, int nl, int NB) {
  const int ps = ((nl < kMB ? nl : kMB) + 11) / 16 * 16 + 4;
  return 128 + 128 + (nl * (2 * H + kWPad) + 127) / 128 * 128 + 8 * 8 * NB * ps * 4;
}

typedef void (*ChunkFn)(DecView, ChunkArgs);
// The kernel of a shape (nullptr: there is none), for hidden size H.  Fixed trip
// counts let the product's loads of W_out be scheduled ahead of its MMAs, where
// there are registers for it.  A chunk of 13 frames without and with them, us:
//   one group, 16 rows a pass: 64 streams, V 1024: H 320 244 / 229, 640 248 / 235,
//     832 267 / 260, 1024 348 / 328;
//   one group, 8 rows: one stream, H 320 181.7 / 180.5, 640 172.7 / 171.9, 832
//     186.4 / 186.5, 1024 164.5 / 166.6; 100 streams, V 2048, H 512, 564 / 548;
//   two groups: 128 streams, V 700, H 320 435 / 368; V 512, H 640 314 / 298, 1024
//     467 / 472; 224 streams, H 832 429 / 420;
//   three groups: V 512, 300 streams, H 320 501 / 451, 336, 640 562 / 512; 128, V 1024,
//     H 640 588 / 520; 224, H 1024 499 / 499.
template <int NB, int RG, int MAX>
ChunkFn fixed_trips(int H) {
  switch (H / 256) {
    case 1: return k_chunk<NB, RG, 1>;
    case 2: return k_chunk<NB, RG, 2>;
    case 3: if constexpr (MAX >= 3) return k_chunk<NB, RG, 3>; break;
    case 4: if constexpr (MAX >= 4) return k_chunk<NB, RG, 4>; break;
  }
  return k_chunk<NB, RG, -1>;
}
ChunkFn kernel_of(int NB, int RG, int H) {
  if (RG == 1) return NB == 1 ? fixed_trips<1, 1, 2>(H) : fixed_trips<2, 1, 4>(H);
  if (RG == 2) return NB == 1 ? k_chunk<1, 2, -1> : fixed_trips<2, 2, 3>(H);
  return NB == 1 ? nullptr : fixed_trips<2, 3, 4>(H);
}

cudaLaunchConfig_t config(const ChunkShape& s, int clusters, cudaLaunchAttribute* a, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * s.CS));
  cfg.blockDim = dim3((unsigned)(kGemm + s.RG * group_threads(s.RG)));
  cfg.dynamicSmemBytes = (size_t)s.smem;
  cfg.stream = st;
  a[0].id = cudaLaunchAttributeClusterDimension;
  a[0].val.clusterDim.x = (unsigned)s.CS;
  a[0].val.clusterDim.y = 1;
  a[0].val.clusterDim.z = 1;
  cfg.attrs = a;
  cfg.numAttrs = 1;
  return cfg;
}

}  // namespace

cudaError_t chunk_cluster_shapes(const DecView& d, std::vector<ChunkShape>& out) {
  out.clear();
  if (d.H > 32 * 8 * kUnits) return cudaSuccess;
  int dev = 0, lim = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  for (int NB = 1; NB <= 2; ++NB)
    for (int RG = 1; RG <= 3; ++RG) {
      const void* f = (const void*)kernel_of(NB, RG, d.H);
      if (!f) continue;
      if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
      if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, lim)) != cudaSuccess) return e;
      for (int CS = 8; CS <= 16; CS *= 2) {
        if (slice_of(d.N, CS, CS - 1).len == 0) continue;  // every CTA sends logits (chunk_partials.h)
        ChunkShape s;
        s.CS = CS, s.RG = RG, s.NB = NB;
        s.nl = slice_of(d.N, CS, 0).len;  // (the largest)
        const Layout L = layout(d.N, d.H, d.V4, s.nl, CS, NB, RG);
        if (L.total > lim) continue;
        s.smem = L.total;
        cudaLaunchAttribute a[1];
        cudaLaunchConfig_t cfg = config(s, 1, a, nullptr);
        if ((e = cudaOccupancyMaxActiveClusters(&s.clusters, f, &cfg)) != cudaSuccess) return e;
        if (s.clusters > 0) out.push_back(s);
      }
    }
  return cudaSuccess;
}

// Where the one launch is no slower than the two-kernel step (7 to 8 us a label
// step at these sizes).  A chunk of 13 frames, one launch / two kernels, us:
//   one group, one pass, always: 112 rows, V 1024, H 1024: 388 / 517; 120, H 640: 346 /
//     478; 112, V 1500, H 512: 305 / 462; V 2048, H 320: 370 / 504;
//   in two passes of 8 rows up to 10 rows a cluster: V 1300, H 896: 70 rows 460 / 481,
//     112: 482 / 481; V 2048, H 512: 57 rows 527 / 491, 112: 578 / 504;
//   two groups, where a slice is one block of the product or H < 512: 200 rows, V 512,
//     H 640: 314 / 482; H 1024: 491 / 528; V 600, H 832: 494 / 491; V 1024, H 320: 342 /
//     467; H 448: 456 / 480; V 1200, H 320: 522 / 515; not V 700, H 512: 506 / 486; H 640:
//     534 / 478;
//   three groups of 64 threads, in clusters of 8, a slice one block, H < 768 and up to
//     170 KB of W_out a step: 300 rows, V 512, H 320 (85 KB): 409 / 480; V 620, H 448
//     (140): 440 / 494; V 639, H 512 (160): 490 / 500; 336, V 512, H 640 (170): 508 / 496;
//     not 260 rows, V 600, H 640 (190): 542 / 494; V 512, H 768: 638 / 514; V 1024, H 320:
//     560 / 486; nor clusters of 16: 200, V 1024, H 640: 665 / 492; 160, V 1500, H 512:
//     741 / 460.
const ChunkShape* chunk_cluster_pick(const std::vector<ChunkShape>& shapes, int n, int H) {
  const ChunkShape* best = nullptr;
  double cost = 0;
  if (n > kChunkMaxRows) return nullptr;
  for (const ChunkShape& s : shapes) {
    const int R = (n + s.clusters - 1) / s.clusters;
    const int passes = (R + 8 * s.NB - 1) / (8 * s.NB);
    if (R > s.CS * s.RG || (passes > 1 && !several_passes(s.NB, s.RG))) continue;
    if (s.RG == 1 && passes > 1 && R > 10) continue;
    if (s.RG == 2 && s.nl > kMB && H >= 512) continue;
    if (s.RG == 3 && (s.CS != 8 || s.nl > kMB || H >= 768 || passes * s.nl * H * 2 > 170 * 1024)) continue;
    // bytes of W_out a CTA reads per step, a pass's overhead, another row group
    const double c = passes * ((double)s.nl * H * 2 + 32768.0 + 16384.0 * s.NB) + 20000.0 * ((R + s.CS - 1) / s.CS);
    if (!best || c < cost) best = &s, cost = c;
  }
  return best;
}

int joint_rows_tiles(int N) { return slice_of(N, 8, 0).parts; }

cudaError_t joint_rows_prepare() {
  int dev = 0, lim = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_joint_rows<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_joint_rows<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  return e;
}

void launch_joint_rows(const ChunkShape& s, const DecView& d, int n, int step, cudaStream_t st, bool pdl) {
  // 16 rows per CTA where their partials fit, and no more CTAs than SMs: most
  // of W_out is then read before the wait.  A chunk of 5 frames (V 1024, H 1024,
  // LSTM 640) in us, against the tensor-core joint kernel: 1 row 387 / 416, 16
  // rows 426 / 441, 64 rows 449 / 454 (8 per CTA: 490), 112 rows 504 / 461.
  const int NB = n > 8 && joint_rows_smem(d.H, s.nl, 2) <= 227 * 1024 ? 2 : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)s.CS, (unsigned)std::min((n + 8 * NB - 1) / (8 * NB), std::max(1, d.sms / s.CS)));
  cfg.blockDim = dim3(kGemm);
  cfg.dynamicSmemBytes = (size_t)joint_rows_smem(d.H, s.nl, NB);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  if (NB == 1) cudaLaunchKernelEx(&cfg, k_joint_rows<1>, d, step, s.nl);
  else cudaLaunchKernelEx(&cfg, k_joint_rows<2>, d, step, s.nl);
}

cudaError_t launch_chunk_cluster(const ChunkShape& s, const DecView& d, ChunkArgs& a, cudaStream_t st) {
  a.CS = s.CS;
  a.nl = s.nl;
  a.R = (a.n + s.clusters - 1) / s.clusters;
  const int clusters = (a.n + a.R - 1) / a.R;
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t cfg = config(s, clusters, at, st);
  return cudaLaunchKernelEx(&cfg, kernel_of(s.NB, s.RG, d.H), d, a);
}

}  // namespace tsd
