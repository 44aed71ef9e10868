// Tensor-core GEMMs of the stateful Transducer form (prediction network and
// joint projections), out[r][j] = sum_k A[r][k] * B[j][k] with A and B bf16
// and K-major, on tcgen05 (accumulator in TMEM, TMA loads into
// 128-byte-swizzled stages), each with its own epilogue:
//   kEncProj:   P_enc = enc W_enc + b_enc, stored fp32 (once per chunk);
//   kLstm:      the LSTM cell on the gate pre-activations (columns 4u+q are
//               gate q of unit u): for rows that emitted a label (or start a
//               sequence) c' = s(f) c + s(i) tanh(g), h' = s(o) tanh(c') into
//               the stream's state; every row's h goes on to the projection;
//   kJointIn:   the joint input A = bf16(ReLU(P_enc[t] + h W_pred + b_pred))
//               for the row's current frame t.
// Warp roles: warp 0 TMA producer, warp 1 TMEM allocator and MMA issuer, the
// others epilogue (thread = row and, for the LSTM, four units).  Every mbarrier wait is
// bounded in time; on expiry the kernel records an error and returns.
#include <cuda.h>

#include "decoder.h"
#include "gemm_tc.h"
#include "tc_common.cuh"

namespace tsd {

namespace {

using namespace tc;

// Output tiles.  The per-step GEMMs are bound by what an SM takes in from L2
// after the dependency wait (about 60 bytes a clock; the first stages of the
// weights are there by then), so a 64-row tile is taken while every tile has
// an SM of its own, and narrow 128-row tiles otherwise.  256 rows: the LSTM
// (N 2560, K 1280) reads 426 KB per CTA in 128 x 64 tiles, 246 in 64 x 80; the
// joint input (N 1024, K 640) 164 and 82.
// The cell is 20 divisions and exponentials per unit and row: every epilogue
// warp has four units of its rows.  A chunk of 256 streams x 5 frames (D 640):
// 554 us with 128-row tiles and four epilogue warps, 510 with these.
template <int EPI, int BM>
struct Shape {
  static constexpr int BN = EPI == kEncProj ? 128 : (EPI == kLstm ? (BM == 64 ? 80 : 64) : 32);
  static constexpr int CW = EPI == kLstm ? 16 : 32;             // columns per epilogue block
  static constexpr int EW = EPI == kLstm ? BN / CW : 1;         // epilogue warps per TMEM lane quadrant
  static constexpr int Threads = 64 + 128 * EW;
  static constexpr int Tmem = BN <= 32 ? 32 : (BN <= 64 ? 64 : 128);  // TMEM columns (a power of two)
  static constexpr int ABytes = BM * kBK * 2;
  static constexpr int BBytes = BN * kBK * 2;
  static constexpr int StageBytes = ABytes + BBytes;
  static constexpr int Stages = (200 * 1024) / StageBytes;
  static constexpr int Smem = Stages * StageBytes + 1024 /*align*/ + 512 /*barriers*/ + BN * 4 /*bias*/;
  static_assert((2 * Stages + 1) * 8 + 4 <= 512, "barrier area");
};
constexpr int kGBar = 512;  // mbarriers and the TMEM address

__device__ __forceinline__ float sigm(float x) { return 1.f / (1.f + expf(-x)); }

__device__ __forceinline__ uint16_t bf16_bits(float v) {
  const __nv_bfloat16 b = __float2bfloat16_rn(v);
  return *reinterpret_cast<const uint16_t*>(&b);
}

template <int EPI, int BM>
__global__ void __launch_bounds__((Shape<EPI, BM>::Threads), 1)
    k_gemm_tc(DecView d, GemmArgs g, const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB) {
  using S = Shape<EPI, BM>;
  constexpr int kGN = S::BN;
  constexpr int kGStages = S::Stages;
  constexpr int kGABytes = S::ABytes;
  constexpr int kGStageBytes = S::StageBytes;
  constexpr int kQRows = BM / 4;  // rows of a TMEM lane quadrant (its first lanes)
  static_assert(kGN % S::CW == 0 && kGStageBytes % 1024 == 0, "tile shape");
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kGStages * kGStageBytes);
  uint64_t* empty = full + kGStages;
  uint64_t* accum = empty + kGStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum + 1);
  float* s_bias = reinterpret_cast<float*>(smem + kGStages * kGStageBytes + kGBar);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * kGN, m0 = blockIdx.y * BM;
  const int KB = g.K / kBK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kGStages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    mbar_init(accum, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(S::Tmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (warp >= 2) {
    // the tile's bias (a constant weight) to shared memory
    const int j = threadIdx.x - 64;
    if (j < kGN) s_bias[j] = n0 + j < g.N ? g.bias[n0 + j] : 0.f;
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;
  // the weights are constant: the first stages' B tiles go out before the
  // dependency wait
  const int pre = min(KB, kGStages);
  if (warp == 0 && lane == 0) {
    for (int kb = 0; kb < pre; ++kb) {
      mbar_expect_tx(full + kb, kGStageBytes);
      tma_load_2d(smem + kb * kGStageBytes + kGABytes, &tmB, full + kb, kb * kBK, n0);
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;
      for (int kb = 0; kb < KB; ++kb) {
        const int s = kb % kGStages;
        const uint32_t ph = (uint32_t)(kb / kGStages) & 1u;
        unsigned char* sa = smem + s * kGStageBytes;
        if (kb < pre) {
          tma_load_2d(sa, &tmA, full + s, kb * kBK, m0);
          ++issued;
          continue;
        }
        if (!mbar_wait(empty + s, ph ^ 1u)) { ok = false; break; }
        mbar_expect_tx(full + s, kGStageBytes);
        tma_load_2d(sa, &tmA, full + s, kb * kBK, m0);
        tma_load_2d(sa + kGABytes, &tmB, full + s, kb * kBK, n0);
        ++issued;
      }
      if (!ok) {
        for (int kb = max(0, issued - kGStages); kb < issued; ++kb)
          mbar_wait(full + kb % kGStages, (uint32_t)(kb / kGStages) & 1u);
        atomicOr(d.err, 64);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (elect()) {
      ok = mma_tile<kGStages, kGStageBytes, kGABytes>(tmem, smem_u32(smem), full, empty, KB,
                                                                 idesc_bf16(BM, kGN), kWaitNs);
      mma_commit(accum);
      if (!ok) atomicOr(d.err, 128);
    }
    __syncwarp();
  } else {
    const int q = warp & 3;
    const int gr = m0 + q * kQRows + lane;
    // Per-row operands the epilogue combines with the accumulator are loaded
    // into registers before the accumulator is ready: with the stores that
    // follow (possibly aliasing, to the compiler) they would otherwise each
    // cost a dependent round trip to memory.
    const Params* P = d.params;
    const bool live = lane < kQRows && gr < g.M;
    int slot = 0, flag = 0, t = 0, T = 1;
    float4 pre4[EPI == kJointIn ? kGN / 4 : 1];
    uint2 h4 = make_uint2(0u, 0u);
    const int D = d.pred_D;
    const int c0 = EPI == kLstm ? ((warp - 2) >> 2) * 16 : 0;  // kLstm: this warp's columns of the tile
    const int u0 = (n0 + c0) / 4;                              // and their first LSTM unit
    const bool mine = live && n0 + c0 < g.N;
    if (EPI == kLstm && mine) {
      slot = P->slots[gr];
      flag = d.pflag[gr];
      if (flag) pre4[0] = *reinterpret_cast<const float4*>(d.pred_c + (size_t)slot * D + u0);
      else h4 = *reinterpret_cast<const uint2*>(d.pred_h + (size_t)slot * D + u0);
    }
    if (EPI == kJointIn && live) {
      t = d.r_t[gr];
      T = P->T;
      if (t < T) {
        const float4* pe = reinterpret_cast<const float4*>(d.pred_penc + ((size_t)gr * T + t) * g.ld + n0);
#pragma unroll
        for (int i = 0; i < kGN / 4; ++i)
          if (n0 + 4 * i < g.N) pre4[i] = pe[i];  // N is a multiple of 32: whole chunks
      }
    }
    ok = __all_sync(0xffffffffu, mbar_wait(accum, 0));
    if (!ok && lane == 0) atomicOr(d.err, 256);
    fence_after();
    if (ok) {
      const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16);
      __syncwarp();
      if constexpr (EPI == kLstm) {
        // columns 4u+q of the block: gates (i, f, g, o) of units u0 .. u0+3
        float v[16];
        tmem_ld16(tbase + (uint32_t)c0, v);
        if (mine) {
          const float* bb = s_bias + c0;
          const size_t base = (size_t)slot * D + u0;
          uint2 hv = h4;
          if (flag) {
            float cn[4];
            const float cprev[4] = {pre4[0].x, pre4[0].y, pre4[0].z, pre4[0].w};
            uint16_t* hb = reinterpret_cast<uint16_t*>(&hv);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float gi = sigm(v[4 * j] + bb[4 * j]);
              const float gf = sigm(v[4 * j + 1] + bb[4 * j + 1]);
              const float gg = tanhf(v[4 * j + 2] + bb[4 * j + 2]);
              const float go = sigm(v[4 * j + 3] + bb[4 * j + 3]);
              cn[j] = gf * cprev[j] + gi * gg;
              hb[j] = bf16_bits(go * tanhf(cn[j]));
            }
            *reinterpret_cast<float4*>(d.pred_c + base) = make_float4(cn[0], cn[1], cn[2], cn[3]);
            *reinterpret_cast<uint2*>(d.pred_h + base) = hv;
          }
          *reinterpret_cast<uint2*>(d.pred_hin + (size_t)gr * D + u0) = hv;
        }
      } else {
#pragma unroll
        for (int c = 0; c < kGN / 32; ++c) {
          __syncwarp();
          float v[32];
          tmem_ld32(tbase + (uint32_t)(c * 32), v);
          const int c1 = n0 + c * 32;
          if (!live || c1 >= g.N) continue;
          const float* bb = s_bias + c * 32;
          if (EPI == kEncProj) {
            float* out = g.out + (size_t)gr * g.ld + c1;
#pragma unroll
            for (int i = 0; i < 32; i += 4)
              *reinterpret_cast<float4*>(out + i) =
                  make_float4(v[i] + bb[i], v[i + 1] + bb[i + 1], v[i + 2] + bb[i + 2], v[i + 3] + bb[i + 3]);
          } else if (t < T) {  // kJointIn
            const float* pe = reinterpret_cast<const float*>(&pre4[8 * c]);
            uint16_t* a = d.A + (size_t)gr * d.H + c1;
#pragma unroll
            for (int i = 0; i < 32; i += 8) {
              uint4 o;
              uint16_t* ob = reinterpret_cast<uint16_t*>(&o);
#pragma unroll
              for (int k = 0; k < 8; ++k) ob[k] = bf16_bits(fmaxf(pe[i + k] + (v[i + k] + bb[i + k]), 0.f));
              *reinterpret_cast<uint4*>(a + i) = o;
            }
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::Tmem) : "memory");
  }
}

}  // namespace

bool gemm_tc_maps(GemmMaps* m, int epi, const uint16_t* A, int a_rows, const uint16_t* B, int b_rows, int K) {
  const auto bf16 = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  const int bn = epi == kEncProj ? Shape<kEncProj, 128>::BN : (epi == kLstm ? Shape<kLstm, 128>::BN : Shape<kJointIn, 128>::BN);
  const int bn64 = epi == kLstm ? Shape<kLstm, 64>::BN : Shape<kJointIn, 64>::BN;
  return make_map(&m->a, A, bf16, 2, K, a_rows, kBK, 128) && make_map(&m->b, B, bf16, 2, K, b_rows, kBK, bn) &&
         make_map(&m->a64, A, bf16, 2, K, a_rows, kBK, 64) && make_map(&m->b64, B, bf16, 2, K, b_rows, kBK, bn64);
}

namespace {
template <int EPI, int BM>
cudaError_t prepare_one() {
  return cudaFuncSetAttribute(k_gemm_tc<EPI, BM>, cudaFuncAttributeMaxDynamicSharedMemorySize, Shape<EPI, BM>::Smem);
}

template <int EPI, int BM>
void launch_one(const DecView& d, const GemmArgs& g, const CUtensorMap& a, const CUtensorMap& b, cudaStream_t s,
                bool pdl) {
  using S = Shape<EPI, BM>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((g.N + S::BN - 1) / S::BN, (g.M + BM - 1) / BM);
  cfg.blockDim = dim3(S::Threads);
  cfg.dynamicSmemBytes = S::Smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k_gemm_tc<EPI, BM>, d, g, a, b);
}

template <int EPI>
void launch_step(const DecView& d, const GemmArgs& g, const GemmMaps& m, cudaStream_t s, bool pdl) {
  constexpr int BN = Shape<EPI, 64>::BN;
  if ((g.M + 63) / 64 * ((g.N + BN - 1) / BN) <= d.sms) launch_one<EPI, 64>(d, g, m.a64, m.b64, s, pdl);
  else launch_one<EPI, 128>(d, g, m.a, m.b, s, pdl);
}
}  // namespace

cudaError_t gemm_tc_prepare() {
  cudaError_t e = prepare_one<kEncProj, 128>();
  if (e == cudaSuccess) e = prepare_one<kLstm, 128>();
  if (e == cudaSuccess) e = prepare_one<kLstm, 64>();
  if (e == cudaSuccess) e = prepare_one<kJointIn, 128>();
  if (e == cudaSuccess) e = prepare_one<kJointIn, 64>();
  return e;
}

void launch_gemm_tc(int epi, const DecView& d, const GemmArgs& g, const GemmMaps& m, cudaStream_t s, bool pdl) {
  if (epi == kEncProj) launch_one<kEncProj, 128>(d, g, m.a, m.b, s, pdl);
  else if (epi == kLstm) launch_step<kLstm>(d, g, m, s, pdl);
  else launch_step<kJointIn>(d, g, m, s, pdl);
}

}  // namespace tsd
