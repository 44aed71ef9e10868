// Joint GEMM on the 5th-generation tensor cores (tcgen05) with the selection
// epilogue of pruned fusion.
//
// logits[r][v] = sum_k A[r][k] * Wt[v][k]: A (joint input, bf16 [M][H]) and
// Wt (W_out label-major, bf16 [N_pad][H]) are both K-major, loaded by TMA
// into 128-byte-swizzled shared-memory stages; one elected thread issues
// tcgen05.mma (kind::f16, bf16 x bf16 -> fp32) into a 128 x BN accumulator in
// tensor memory.  Eight epilogue warps read the accumulator back with
// tcgen05.ld (thread = row; two warps per 32-lane quadrant take alternate
// 32-column chunks) and reduce it on chip to the row's selection partial for
// this tile: softmax max and sum over the real labels, and the tile's top K
// logits, ties to the lower label.  Logits never leave the SM.  (Every other
// form stores its logits: joint_greedy.cu.)
//
// Warp roles (320 threads): warp 0 TMA producer, warp 1 TMEM allocator and
// MMA issuer, warps 2-9 epilogue.  Every wait on an mbarrier is bounded in
// time; on expiry the kernel records an error in the decoder's status word,
// drains its own copies and returns.
#include <cuda.h>

#include "decoder.h"
#include "joint_tc.h"
#include "tc_common.cuh"

namespace tsd {

namespace {

using namespace tc;  // kBM, kBK and the tcgen05 / TMA helpers
constexpr int kThreads = 320;
constexpr int kEpiThreads = 256;  // warps 2-9
constexpr float kNegInf = -__builtin_huge_valf();
// Shared memory: [operand stages][barriers].
template <int BN>
struct Smem {
  static constexpr int kStages = (BN == 256) ? 4 : (BN == 128 ? 6 : 8);
  static constexpr int kABytes = kBM * kBK * 2;
  static constexpr int kBBytes = BN * kBK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kBytes = kStages * kStageBytes + 1024 /*align*/ + 256 /*barriers*/;
  static_assert(kBM * 18 * 4 + 16 <= kStages * kStageBytes, "the epilogue halves' exchange (per row 18 floats, 4 flags) fits");
};

// Sum over a chunk of 2^(l[i] * log2 e - s2) in four independent
// accumulators (a single running sum would chain 32 dependent adds).
__device__ __forceinline__ float sum_exp2_32(const float* l, float s2) {
  float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < 32; ++i) a[i & 3] += ex2_approx(fmaf(l[i], kLog2e, -s2));
  return (a[0] + a[1]) + (a[2] + a[3]);
}

// K = d.topk <= 8, the candidate count.
template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
    k_joint_tc(DecView d, int step, const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB) {
  using S = Smem<BN>;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::kStages * S::kStageBytes);
  uint64_t* empty = full + S::kStages;
  uint64_t* accum = empty + S::kStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * BN, m0 = blockIdx.y * kBM;
  const int M = d.params->n * d.K;
  const int KB = d.H / kBK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S::kStages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    mbar_init(accum, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;
  // W_out is constant, so the first stages' W_out tiles are requested before
  // the dependency wait (each stage's barrier expects its A tile as well).
  const int pre = min(KB, S::kStages);
  if (warp == 0 && lane == 0) {
    for (int kb = 0; kb < pre; ++kb) {
      mbar_expect_tx(full + kb, S::kStageBytes);
      tma_load_2d(smem + kb * S::kStageBytes + S::kABytes, &tmB, full + kb, kb * kBK, n0);
    }
  }
  // Programmatic dependent launch: the set-up above overlaps the row pass;
  // its output (the joint input) is read only after the wait.  The next
  // row pass may launch once every CTA is past this point.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;
      for (int kb = 0; kb < KB; ++kb) {
        const int s = kb % S::kStages;
        const uint32_t ph = (uint32_t)(kb / S::kStages) & 1u;
        unsigned char* sa = smem + s * S::kStageBytes;
        if (kb < pre) {  // first use of the stage: W_out already requested
          tma_load_2d(sa, &tmA, full + s, kb * kBK, m0);
          ++issued;
          continue;
        }
        if (!mbar_wait(empty + s, ph ^ 1u, d.wait_ns)) { ok = false; break; }
        mbar_expect_tx(full + s, S::kStageBytes);
        tma_load_2d(sa, &tmA, full + s, kb * kBK, m0);
        tma_load_2d(sa + S::kABytes, &tmB, full + s, kb * kBK, n0);
        ++issued;
      }
      // Never exit with copies in flight: wait for the last use of every
      // stage (its final phase; complete already when the MMAs consumed it,
      // as they do unless a wait expired), with the long limit.
      for (int kb = max(0, issued - S::kStages); kb < issued; ++kb)
        mbar_wait(full + kb % S::kStages, (uint32_t)(kb / S::kStages) & 1u);
      if (!ok) atomicOr(d.err, 1);
    }
    __syncwarp();  // reconverge before the CTA barrier below (bar.sync is warp-aligned)
  } else if (warp == 1) {
    if (elect()) {
      ok = mma_tile<S::kStages, S::kStageBytes, S::kABytes>(tmem, smem_u32(smem), full, empty, KB,
                                                                       idesc_bf16(kBM, BN), d.wait_ns);
      // signals the epilogue once every issued MMA has completed (also after a
      // timeout, so nothing is in flight when TMEM is released)
      mma_commit(accum);
      if (!ok) atomicOr(d.err, 2);
    }
    __syncwarp();
  } else {
    // epilogue: warps 2..9, thread = row of the tile; the two warps of a
    // TMEM lane quadrant take alternate 32-column chunks
    const int q = warp & 3;  // TMEM lane quadrant this warp may access
    const int half = (warp - 2) >> 2;
    const int row = q * 32 + lane;
    const int gr = m0 + row;
    const bool live = gr < M;
    const int N = d.N;
    float mx = kNegInf, se = 0.f;
    const int K = d.topk;
    float tv[8];
    int ti[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) { tv[j] = kNegInf; ti[j] = INT_MAX; }
    float tmin = kNegInf;  // tv[K-1]
    ok = __all_sync(0xffffffffu, mbar_wait(accum, 0, d.wait_ns));  // warp-uniform: tcgen05.ld is .sync.aligned
    if (!ok && lane == 0) atomicOr(d.err, 4);
    fence_after();
    if (ok) {
      const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
      for (int c = half; c < BN / 32; c += 2) {
        __syncwarp();  // the per-chunk selection branches; tcgen05.ld wants the warp whole
        float l[32];
        tmem_ld32(tbase + (uint32_t)(c * 32), l);
        const int c0 = n0 + c * 32;
        // Labels at or past V+1 (padding of the last tile) take no part:
        // their logit becomes -inf.
        if (c0 + 32 > N) {
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (c0 + i >= N) l[i] = kNegInf;
        }
        // the values still to take (b), the chunk's maximum by a tree
        float b[32], u[16];
#pragma unroll
        for (int i = 0; i < 32; ++i) b[i] = l[i];
#pragma unroll
        for (int i = 0; i < 16; ++i) u[i] = fmaxf(b[i], b[i + 16]);
#pragma unroll
        for (int w = 8; w > 0; w >>= 1)
#pragma unroll
          for (int i = 0; i < w; ++i) u[i] = fmaxf(u[i], u[i + w]);
        const float cm = u[0];
        if (cm > tmin) {
          // Take the chunk's values in decreasing order while they beat the
          // K-th kept value: at most K rounds, usually none after the first
          // chunks.  Each round finds the first (lowest-label) position of the
          // chunk maximum, bubbles it into the sorted list (an equal value
          // already kept stays ahead: it has the lower label), masks it out
          // and takes the next maximum.
          float cmx = cm;
#pragma unroll 1
          for (int it = 0; it < K && cmx > tmin; ++it) {
            int jx = 31;
#pragma unroll
            for (int i = 31; i >= 0; --i)
              if (b[i] == cmx) jx = i;
            float cv = cmx;
            int ci = c0 + jx;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if (j < K && cv > tv[j]) {
                const float tf = tv[j]; tv[j] = cv; cv = tf;
                const int tk = ti[j]; ti[j] = ci; ci = tk;
              }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (j == K - 1) tmin = tv[j];
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (i == jx) b[i] = kNegInf;
#pragma unroll
            for (int i = 0; i < 16; ++i) u[i] = fmaxf(b[i], b[i + 16]);
#pragma unroll
            for (int w = 8; w > 0; w >>= 1)
#pragma unroll
              for (int i = 0; i < w; ++i) u[i] = fmaxf(u[i], u[i + w]);
            cmx = u[0];
          }
        }
        if (cm != kNegInf) {
          // online softmax partial: sum of 2^((logit - max) * log2 e)
          const float m2 = fmaxf(mx, cm);
          const float s2 = m2 * kLog2e;
          float acc = (mx == kNegInf) ? 0.f : se * ex2_approx(mx * kLog2e - s2);
          acc += sum_exp2_32(l, s2);
          se = acc;
          mx = m2;
        }
        if (d.cap_logits && step < d.cap_steps && live) {
          float* cl = d.cap_logits + ((size_t)step * M + gr) * N;
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (c0 + i < N) cl[c0 + i] = l[i];
        }
      }
    }
    // never leave with MMAs still writing the accumulator (the long limit
    // whatever wait_ns is)
    if (warp == 2 && lane == 0) mbar_wait(accum, 0);
    __syncwarp();
    // Merge the two halves' partials of each row: the second half leaves its
    // partial in shared memory (the stages are drained: every MMA has
    // completed), the first half combines and stores.
    float* xbase = reinterpret_cast<float*>(smem);
    float* xch = xbase + row * 18;  // (max, sum, then the top 8 (value, label))
    int* xok = reinterpret_cast<int*>(xbase + kBM * 18);  // per quadrant: the second half finished
    if (half == 1) {
      if (ok) {
        xch[0] = mx;
        xch[1] = se;
#pragma unroll
        for (int j = 0; j < 8; ++j) { xch[2 + 2 * j] = tv[j]; xch[3 + 2 * j] = __int_as_float(ti[j]); }
      }
      if (lane == 0) xok[q] = ok ? 1 : 0;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
    if (half == 0 && ok && xok[q] && live) {
      const float m1 = xch[0], s1 = xch[1];
      if (m1 != kNegInf) {
        if (mx == kNegInf) { mx = m1; se = s1; }
        else {
          const float m2 = fmaxf(mx, m1);
          se = se * ex2_approx((mx - m2) * kLog2e) + s1 * ex2_approx((m1 - m2) * kLog2e);
          mx = m2;
        }
      }
      // merge two lists sorted by (value desc, label asc): an entry's
      // place is its index plus the other list's entries ordered before it
      // (unfilled entries (-inf, INT_MAX) of both lists land on the same
      // trailing places with the same contents)
      float2* bp = d.bpart + ((size_t)gr * d.n_ptiles + blockIdx.x) * (1 + K);
      bp[0] = make_float2(mx, se);
      float ov[8];
      int oi[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) { ov[j] = xch[2 + 2 * j]; oi[j] = __float_as_int(xch[3 + 2 * j]); }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (i < K) {
          int pa = i, pb = i;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (j < K) {
              pa += (ov[j] > tv[i] || (ov[j] == tv[i] && oi[j] < ti[i])) ? 1 : 0;
              pb += (tv[j] > ov[i] || (tv[j] == ov[i] && ti[j] < oi[i])) ? 1 : 0;
            }
          }
          if (pa < K) bp[1 + pa] = make_float2(tv[i], __int_as_float(ti[i]));
          if (pb < K) bp[1 + pb] = make_float2(ov[i], __int_as_float(oi[i]));
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN) : "memory");
  }
}

}  // namespace

unsigned long long tc_wait_ns_default() { return kWaitNs; }

int joint_tc_pick_bn(int M_max, int N_pad, int sms) {
  // wider tiles re-read fewer operands; take the widest whose tiles still
  // cover ~80% of the SMs (measured: 256 at 1024 x 4352, 64 at 256 x 1280)
  const int mt = (M_max + kBM - 1) / kBM;
  if (mt * (N_pad / 256) * 5 >= sms * 4) return 256;
  if (mt * (N_pad / 128) * 5 >= sms * 4) return 128;
  return 64;
}

cudaError_t joint_tc_prepare(JointTc* jt, const uint16_t* A, int M_pad, const uint16_t* Wt, int N_pad, int H, int bn,
                             const float* logits) {
  jt->bn = bn;
  if (!make_map(&jt->mapA, A, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, H, M_pad, kBK, kBM)) return cudaErrorInvalidValue;
  if (!make_map(&jt->mapB, Wt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, H, N_pad, kBK, bn)) return cudaErrorInvalidValue;
  // pruned fusion stores no logits
  if (logits && (!make_map(&jt->mapLogits, logits, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, N_pad, M_pad, 32, 32) ||
                 !make_map(&jt->mapLogits16, logits, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, N_pad, M_pad, 32, 16)))
    return cudaErrorInvalidValue;
  if (!make_map(&jt->mapA64, A, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, H, M_pad, kBK, 64)) return cudaErrorInvalidValue;
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = bn == 256   ? cudaFuncSetAttribute(k_joint_tc<256>, attr, Smem<256>::kBytes)
                  : bn == 128 ? cudaFuncSetAttribute(k_joint_tc<128>, attr, Smem<128>::kBytes)
                              : cudaFuncSetAttribute(k_joint_tc<64>, attr, Smem<64>::kBytes);
  if (e == cudaSuccess) e = joint_greedy_prepare(bn);
  return e;
}

namespace {
template <int BN>
void launch_bn(cudaLaunchConfig_t& cfg, const JointTc& jt, const DecView& d, int step) {
  cfg.dynamicSmemBytes = Smem<BN>::kBytes;
  cudaLaunchKernelEx(&cfg, k_joint_tc<BN>, d, step, jt.mapA, jt.mapB);
}
}  // namespace

void launch_joint_tc(const JointTc& jt, const DecView& d, int M, int step, cudaStream_t s, bool pdl) {
  if (d.prune == 0) {
    launch_joint_greedy(jt, d, M, step, s, pdl);
    return;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(d.n_ptiles, (M + kBM - 1) / kBM);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  if (jt.bn == 256) launch_bn<256>(cfg, jt, d, step);
  else if (jt.bn == 128) launch_bn<128>(cfg, jt, d, step);
  else launch_bn<64>(cfg, jt, d, step);
}

}  // namespace tsd
