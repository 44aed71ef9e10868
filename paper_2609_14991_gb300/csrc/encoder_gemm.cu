// Tensor-core GEMM of the cache-aware encoder: out = A . B^T with A [M][K]
// and B [N][K] bf16 K-major (B = a weight stored [out][in]), fp32 accumulate
// in TMEM.  Persistent: one CTA (or CTA pair) per SM (pair) walks the tile
// list (tiles of one weight column block are adjacent, so concurrent CTAs
// share B in L2).  Warp 0 streams A and B k-blocks by TMA into a ring of
// 128-byte-swizzled stages that continues across tiles; warp 1 issues the
// MMAs of tile i into accumulator i mod 2; warps 2-17 run the epilogue of tile
// i (thread = output row; warp w reads TMEM lanes 32 (w mod 4) .., the four
// warps of a lane quadrant take different columns) while the MMAs of tile
// i+1 run, then hand the accumulator back.  The epilogue applies the bias and
// one of: the fp32 stream's start (x = acc + b), its residual update (x +=
// alpha (acc + b)), Swish to bf16, plain bf16 (q/k/v), GLU to bf16.
//
// Tile shapes, all with the same order of the sum over K (a row's result does
// not depend on the batch):
//   256 x 256 over two CTAs (cta_group::2): each CTA stages its 128 rows of A
//          and half of B, 32 KB per 64-deep k-block for twice the product of
//          a 128 x 128 tile.  A 128 x 128 tile needs 126 bytes per clock and SM
//          from L2 at the tensor rate, twice what arrives (measured: 50-62,
//          15-19 TB/s over the chip); the pair needs 64;
//   128 x 128, 128 x 64, 128 x 32 on one CTA, for fewer rows or narrow
//          outputs: narrower tiles put more SMs on the weights; calls of at
//          most 64 rows stage 64 rows of A.
// What bounds them (0.6B shape, 3328 x 4096 x 1024 with Swish, 20.5 us in the
// kernel): 1.5 us to the first operands, 5.2 us per tile and pair of which the
// MMAs are 4.2 (the operands' way from L2 is the rest), 2.4 us of epilogue
// after the last tile.  With 128 x 128 tiles for everything, a division's range
// check per value and row-per-thread stores the same rows took two launches of
// 26.7 us, 18.5 us of each without the epilogue.  Swish and GLU give the bits of
// 1 / (1 + expf(-x)), checked for range once per block of 32 values and reckoned
// in pairs (tc::sigmoid2); the hardware's 2^x and reciprocal alone were 3 to 5%
// of a chunk faster (about 2 us a launch, in the last epilogue; the figures above
// are with them), with twice the error.  Blocks of 32 rows leave through
// shared memory by TMA: bf16 stores, and for the residual update an fp32
// add in L2 (one writer per element), so x is not read at all.
//
// Every mbarrier wait is bounded in time; on expiry the kernel records an
// error bit and the other roles run out their own bounded waits.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "encoder.h"
#include "tc_common.cuh"

namespace tsd {

namespace {

using namespace tc;

constexpr int kEpiWarps = 16;
constexpr int kThreads = 64 + 32 * kEpiWarps;  // warp 0 TMA, warp 1 MMA, warps 2-17 epilogue
int g_sms = 148;

// One tile shape: BN output columns, PAIR: two CTAs (each with BN / 2 rows of
// B), AR rows of A staged per CTA (64: a call of at most 64 rows; the rest of
// the MMA's 128 rows are whatever shared memory holds, and never stored).
template <int BN, bool PAIR, int AR>
struct Shape {
  static constexpr int kABytes = AR * kBK * 2;
  static constexpr int kBRows = PAIR ? BN / 2 : BN;
  static constexpr int kStageBytes = kABytes + kBRows * kBK * 2;
  static constexpr int kBlk = BN == 256 ? 64 : 32;                 // columns an epilogue warp takes at a time
  static constexpr int kParts = BN / kBlk < 4 ? BN / kBlk : 4;     // warps of a lane quadrant with work
  static constexpr int kStgBytes = 4 * kParts * 4096;              // staging: a 4 KB block for each of them
  // as many stages as fit (at most 16; the MMA reads 128 rows of A from the last one)
  static constexpr int kFit = (227 * 1024 - 1024 - 512 - kStgBytes - (kBM - AR) * kBK * 2) / kStageBytes;
  static constexpr int kStages = kFit < 16 ? kFit : 16;
  static constexpr int kStgOff = kStages * kStageBytes + (kBM - AR) * kBK * 2;
  static constexpr int kBarOff = kStgOff + kStgBytes;
  static constexpr int kSmem = kBarOff + 512 + 1024 /*align*/;
  static_assert((2 * kStages + 4) * 8 + 4 <= 512, "barrier area");
  static_assert(kSmem <= 227 * 1024 && kStages >= 4, "shared memory per CTA");
};

__device__ __forceinline__ uint32_t pack_bf16(uint64_t x) {
  float a, b;
  unpair(x, a, b);
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// TMA load whose bytes complete on a barrier of this CTA or its pair's leader.
template <bool PAIR>
__device__ __forceinline__ void load_2d(void* dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  if constexpr (PAIR)
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

template <bool PAIR>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if constexpr (PAIR)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
  else
    mma_bf16(d, a, b, idesc, acc);
}

// The MMAs issued so far, on completion, arrive on the barrier (of both CTAs of a pair).
template <bool PAIR>
__device__ __forceinline__ void commit(uint64_t* bar) {
  if constexpr (PAIR)
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"((uint16_t)3)
        : "memory");
  else
    mma_commit(bar);
}

// fp32 add of a staged box to global memory.
__device__ __forceinline__ void tma_add_2d(const CUtensorMap* map, const void* src, int x, int y) {
  asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(src)), "r"(x), "r"(y)
               : "memory");
}

// fp32 adds of four values to global memory (no value comes back to wait for).
__device__ __forceinline__ void add4(float4* p, float4 v) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}

// 32 accumulator columns from `taddr` with their bias (the same addresses for every lane), as pairs
__device__ __forceinline__ void load_cols(uint32_t taddr, const float* bias, uint64_t (&v)[16]) {
  float f[32];
  tmem_ld32(taddr, f);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(bias) + i);
    v[2 * i] = add2(pair_of(f[4 * i], f[4 * i + 1]), pair_of(q.x, q.y));
    v[2 * i + 1] = add2(pair_of(f[4 * i + 2], f[4 * i + 3]), pair_of(q.z, q.w));
  }
}

template <int EPI, int BN, bool PAIR, int AR>
__global__ void __launch_bounds__(kThreads, 1)
    k_egemm(EGemm g, const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
            const __grid_constant__ CUtensorMap tmO) {
  using S = Shape<BN, PAIR, AR>;
  constexpr int kStages = S::kStages, kABytes = S::kABytes;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::kBarOff);
  uint64_t* empty = full + kStages;
  uint64_t* accf = empty + kStages;  // [2] accumulator holds a finished tile
  uint64_t* acce = accf + 2;         // [2] accumulator read out by the epilogue (of both CTAs)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acce + 2);

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int rank = PAIR ? (int)(blockIdx.x & 1) : 0;
  const int first = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x, stride = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  const int KB = g.K / kBK;
  constexpr int kTM = PAIR ? 2 * kBM : kBM;  // rows per tile
  const int Mt = (g.M + kTM - 1) / kTM, Nt = (g.N + BN - 1) / BN;
  const int tiles = Mt * Nt;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf + b, 1);
      mbar_init(acce + b, kEpiWarps * (PAIR ? 2 : 1));  // one arrival per epilogue warp
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(2 * BN)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(2 * BN)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  fence_before();
  if constexpr (PAIR)  // the pair's barriers and accumulators exist before either CTA uses them
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (elect()) {
      int it = 0;
      bool ok = true;
      auto bar = [&](int st) { return PAIR ? map_rank(smem_u32(full + st), 0) : smem_u32(full + st); };
      auto load_b = [&](int st, int t, int kb) {
        if (rank == 0) mbar_expect_tx(full + st, (PAIR ? 2 : 1) * S::kStageBytes);
        load_2d<PAIR>(smem + st * S::kStageBytes + kABytes, &tmB, bar(st), kb * kBK, (t / Mt) * BN + rank * S::kBRows);
      };
      // B is a weight, A the previous kernel's output: the first stages'
      // tiles of B are requested before the wait
      const int pre = first < tiles ? min(KB, kStages) : 0;
      for (int kb = 0; kb < pre; ++kb) load_b(kb, first, kb);
      asm volatile("griddepcontrol.wait;" ::: "memory");
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      for (int t = first; t < tiles && ok; t += stride) {
        const int m0 = g.m0 + (t % Mt) * kTM + rank * kBM;
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = it % kStages;
          const uint32_t ph = (uint32_t)(it / kStages) & 1u;
          if (it >= kStages && !mbar_wait(empty + s, ph ^ 1u)) { ok = false; break; }
          if (it >= pre) load_b(s, t, kb);
          load_2d<PAIR>(smem + s * S::kStageBytes, &tmA, bar(s), kb * kBK, m0);
        }
      }
      if (!ok) {
        // drain the copies still in flight (the leader's barriers count the pair's)
        if (rank == 0)
          for (int j = max(0, it - kStages); j < it; ++j) mbar_wait(full + j % kStages, (uint32_t)(j / kStages) & 1u);
        atomicOr(g.err, 1u);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (rank == 0 && elect()) {
      const uint32_t idesc = idesc_bf16(kTM, BN);
      int tl = 0, s = 0;
      uint32_t ph = 0;
      bool ok = true, ready = mbar_test(full, 0);
      for (int t = first; t < tiles && ok; t += stride, ++tl) {
        const int buf = tl & 1, use = tl >> 1;
        if (tl >= 2 && !mbar_wait(acce + buf, (uint32_t)(use - 1) & 1u)) { ok = false; break; }
        fence_after();
        const uint32_t acc = tmem + (uint32_t)(buf * BN);
        for (int kb = 0; kb < KB; ++kb) {
          if (!ready && !mbar_wait(full + s, ph)) { ok = false; break; }
          // the next stage's barrier is read while this stage's MMAs are issued
          const int s1 = s + 1 == kStages ? 0 : s + 1;
          const uint32_t ph1 = s1 == 0 ? ph ^ 1u : ph;
          ready = mbar_test(full + s1, ph1);
          fence_after();
          const uint32_t sa = smem_u32(smem + s * S::kStageBytes);
          const uint64_t ad = sw128_desc(sa), bd = sw128_desc(sa + kABytes);
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)
            mma<PAIR>(acc, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), idesc, (kb | k) ? 1u : 0u);
          commit<PAIR>(empty + s);
          s = s1;
          ph = ph1;
        }
        commit<PAIR>(accf + buf);  // also after a timeout: nothing is left in flight
      }
      if (!ok) atomicOr(g.err, 2u);
    }
    __syncwarp();
  } else {
    // x (the residual update) and the buffers written here belong to kernels before this one
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int q = warp & 3;             // TMEM lane quadrant this warp may access
    const int part = (warp - 2) >> 2;   // this warp among the quadrant's
    unsigned char* stg = smem + S::kStgOff + (warp - 2) * 4096;
    int tl = 0;
    bool ok = true;
    // the staged block may be written again once its store has read it
    auto stage = [&]() {
      if (lane == 0) tma_store_wait_read<0>();
      __syncwarp();
      return stg;
    };
    auto ship = [&](const unsigned char* src, int x, int y, bool add) {
      fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        if (add) tma_add_2d(&tmO, src, x, y);
        else tma_store_2d(&tmO, src, x, y);
        tma_store_commit();
      }
    };
    for (int t = first; t < tiles && ok; t += stride, ++tl) {
      const int buf = tl & 1, use = tl >> 1;
      const int m0 = g.m0 + (t % Mt) * kTM + rank * kBM, n0 = (t / Mt) * BN;
      const int r0 = m0 + q * 32, gr = r0 + lane;
      const int end = g.m0 + g.M;
      const bool live = gr < end;
      const bool whole = r0 + 32 <= end;  // all 32 rows of the warp are this call's (branch's): boxes by TMA
      ok = __all_sync(0xffffffffu, mbar_wait(accf + buf, (uint32_t)use & 1u));
      if (!ok) {
        if (lane == 0) atomicOr(g.err, 4u);
        break;
      }
      fence_after();
      const uint32_t tbase = tmem + (uint32_t)(buf * BN) + ((uint32_t)(q * 32) << 16);
      constexpr int kBlk = EPI == kEGlu ? 64 : S::kBlk;
      if (r0 < end) {
        // blocks of kBlk columns in turn
#pragma unroll 1
        for (int p = part; p < BN / kBlk; p += kEpiWarps / 4) {
          const int c0 = n0 + kBlk * p;
          if (c0 >= g.N) break;
          const uint32_t tc0 = tbase + (uint32_t)(kBlk * p);
          unsigned char* st = nullptr;
          if constexpr (EPI == kEGlu) {
            // columns [64 p, 64 p + 32) are values, [64 p + 32, 64 p + 64) their gates
            __syncwarp();
            uint64_t a[16], b[16];
            load_cols(tc0 + 32, g.bias + c0 + 32, b);
            sigmoid2(b, b);
            load_cols(tc0, g.bias + c0, a);
            uint32_t w[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = pack_bf16(mul2(a[i], b[i]));
            if (whole) st = stage();
            uint16_t* o = static_cast<uint16_t*>(g.out) + (size_t)gr * g.ld + c0 / 2;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const uint4 x = make_uint4(w[4 * e], w[4 * e + 1], w[4 * e + 2], w[4 * e + 3]);
              if (whole) *reinterpret_cast<uint4*>(st + lane * 64 + ((e ^ ((lane >> 1) & 3)) << 4)) = x;
              else if (live) reinterpret_cast<uint4*>(o)[e] = x;
            }
            if (whole) ship(st, c0 / 2, r0, false);
          } else {
#pragma unroll
            for (int h = 0; h < kBlk / 32; ++h) {
              __syncwarp();
              uint64_t v[16];
              load_cols(tc0 + (uint32_t)(32 * h), g.bias + c0 + 32 * h, v);
              if constexpr (EPI == kEInit || EPI == kEResid) {
                if (EPI == kEResid) {
#pragma unroll
                  for (int i = 0; i < 16; ++i) v[i] = mul2(v[i], pair_of(g.alpha, g.alpha));
                }
                if (whole) st = stage();
                float4* xp = reinterpret_cast<float4*>(static_cast<float*>(g.out) + (size_t)gr * g.ld + c0 + 32 * h);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                  float4 x;
                  unpair(v[2 * e], x.x, x.y);
                  unpair(v[2 * e + 1], x.z, x.w);
                  if (whole) {
                    *reinterpret_cast<float4*>(st + lane * 128 + ((e ^ (lane & 7)) << 4)) = x;
                  } else if (live) {
                    if (EPI == kEResid) add4(xp + e, x);
                    else xp[e] = x;
                  }
                }
                if (whole) ship(st, c0 + 32 * h, r0, EPI == kEResid);
              } else {
                if (EPI == kESwish) {
                  uint64_t g16[16];
                  sigmoid2(v, g16);
#pragma unroll
                  for (int i = 0; i < 16; ++i) v[i] = mul2(v[i], g16[i]);
                }
                uint32_t w[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) w[i] = pack_bf16(v[i]);
                if (whole && h == 0) st = stage();
                uint16_t* o = static_cast<uint16_t*>(g.out) + (size_t)gr * g.ld + c0 + 32 * h;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const uint4 x = make_uint4(w[4 * e], w[4 * e + 1], w[4 * e + 2], w[4 * e + 3]);
                  if (whole)
                    *reinterpret_cast<uint4*>(st + (kBlk == 64 ? lane * 128 + (((4 * h + e) ^ (lane & 7)) << 4)
                                                               : lane * 64 + ((e ^ ((lane >> 1) & 3)) << 4))) = x;
                  else if (live)
                    reinterpret_cast<uint4*>(o)[e] = x;
                }
                if (whole && h == kBlk / 32 - 1) ship(st, c0, r0, false);
              }
            }
          }
        }
      }
      // this warp's reads of the accumulator are done: hand it back
      fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0) mbar_arrive(acce + buf);
        else
          asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(map_rank(smem_u32(acce + buf), 0))
                       : "memory");
      }
    }
    // the staged blocks must have been read before the CTA's shared memory
    // goes; the stores' writes complete with the grid
    if (lane == 0) tma_store_wait_read<0>();
    __syncwarp();
  }
  fence_before();
  __syncthreads();
  if constexpr (PAIR)  // neither CTA leaves while the other may still signal it or read its operands
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp == 1) {
    fence_after();
    if constexpr (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
  }
}

// Clocks of a GEMM on a tile shape: rounds of tiles over the SMs, each
// k-block the larger of its MMAs (measured per 16-deep MMA: 129 clocks at 256
// columns over a pair, 65 at 128, 49 at 64, 41 at 32) and its operands at 64
// bytes per clock and SM, and a launch's fill and last epilogue.
double cost(int M, int N, int K, int BN, bool pair, int a_rows) {
  const int tm = pair ? 2 * kBM : kBM;
  const int tiles = ((M + tm - 1) / tm) * ((N + BN - 1) / BN);
  const int slots = pair ? g_sms / 2 : g_sms;
  const double mma = 4.0 * (pair ? 129 : BN == 128 ? 65 : BN == 64 ? 49 : 41);
  const double load = ((pair ? kBM : a_rows) + (pair ? BN / 2 : BN)) * 128.0 / 64.0;
  const int rounds = (tiles + slots - 1) / slots;
  return rounds * (K / kBK) * std::max(mma, load) + 1000.0 + 12.0 * BN;
}

template <int EPI, int BN, bool PAIR, int AR>
cudaError_t launch_shape(const EGemm& g, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& o, cudaStream_t s,
                         bool pdl) {
  constexpr int tm = PAIR ? 2 * kBM : kBM;
  const int tiles = ((g.M + tm - 1) / tm) * ((g.N + BN - 1) / BN);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(PAIR ? 2 * std::min(tiles, g_sms / 2) : std::min(tiles, g_sms)));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = Shape<BN, PAIR, AR>::kSmem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  int n = 0;
  if (PAIR) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = 2;
    at[n].val.clusterDim.y = 1;
    at[n++].val.clusterDim.z = 1;
  }
  if (pdl) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = (unsigned)n;
  return cudaLaunchKernelEx(&cfg, k_egemm<EPI, BN, PAIR, AR>, g, a, b, o);
}

template <int EPI>
void launch_one(const EGemm& g, const EncMapA& A, const EncMapB& B, const EncMapO& O, cudaStream_t s, bool pdl) {
  // a call of at most 64 rows stages 64 rows of A
  const bool few = g.m0 == 0 && g.M <= 64;
  const int ar = few ? 64 : kBM;
  double best = few ? 1e30 : cost(g.M, g.N, g.K, 256, true, kBM);
  int pick = 0;
  const int bns[3] = {128, 64, 32};
  for (int i = few ? 1 : 0; i < (EPI == kEGlu ? 2 : 3); ++i) {  // GLU pairs need 64 columns
    const double c = cost(g.M, g.N, g.K, bns[i], false, ar);
    if (c < best) best = c, pick = 1 + i;
  }
  const CUtensorMap& o = (EPI == kESwish || EPI == kEPlain) ? O.m[pick == 0 ? 0 : 1] : O.m[EPI == kEGlu ? 1 : 0];
  if (pick == 0) launch_shape<EPI, 256, true, 128>(g, A.m[0], B.m[0], o, s, pdl);
  else if (pick == 1) launch_shape<EPI, 128, false, 128>(g, A.m[0], B.m[0], o, s, pdl);
  else if (pick == 2 && few) launch_shape<EPI, 64, false, 64>(g, A.m[1], B.m[1], o, s, pdl);
  else if (pick == 2) launch_shape<EPI, 64, false, 128>(g, A.m[0], B.m[1], o, s, pdl);
  else if constexpr (EPI != kEGlu) {
    if (few) launch_shape<EPI, 32, false, 64>(g, A.m[1], B.m[2], o, s, pdl);
    else launch_shape<EPI, 32, false, 128>(g, A.m[0], B.m[2], o, s, pdl);
  }
}

template <int EPI, int BN, bool PAIR, int AR>
void prepare_shape(cudaError_t& e) {
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_egemm<EPI, BN, PAIR, AR>, cudaFuncAttributeMaxDynamicSharedMemorySize, Shape<BN, PAIR, AR>::kSmem);
}

template <int EPI>
void prepare_one(cudaError_t& e) {
  prepare_shape<EPI, 256, true, 128>(e);
  prepare_shape<EPI, 128, false, 128>(e);
  prepare_shape<EPI, 64, false, 128>(e);
  prepare_shape<EPI, 64, false, 64>(e);
  if constexpr (EPI != kEGlu) {
    prepare_shape<EPI, 32, false, 128>(e);
    prepare_shape<EPI, 32, false, 64>(e);
  }
}

}  // namespace

bool egemm_map_a(EncMapA* m, const uint16_t* A, int rows, int K) {
  for (int i = 0; i < 2; ++i)
    if (!tc::make_map(&m->m[i], A, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, K, rows, tc::kBK, tc::kBM >> i)) return false;
  return true;
}

bool egemm_map_b(EncMapB* m, const uint16_t* B, int rows, int K) {
  for (int i = 0; i < 3; ++i)
    if (!tc::make_map(&m->m[i], B, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, K, rows, tc::kBK, 128 >> i)) return false;
  return true;
}

bool egemm_map_out(EncMapO* m, bool fp32, void* out, int rows, int ld) {
  // boxes of 32 rows: 32 fp32 columns; 64 bf16 columns, or 32 (the narrow tiles, GLU)
  if (fp32) return tc::make_map(&m->m[0], out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, ld, rows, 32, 32);
  return tc::make_map(&m->m[0], out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ld, rows, 64, 32) &&
         tc::make_map(&m->m[1], out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ld, rows, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B);
}

cudaError_t egemm_prepare() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
  prepare_one<kEInit>(e);
  prepare_one<kEResid>(e);
  prepare_one<kESwish>(e);
  prepare_one<kEPlain>(e);
  prepare_one<kEGlu>(e);
  return e;
}

void launch_egemm(int epi, const EGemm& g, const EncMapA& a, const EncMapB& b, const EncMapO& o, cudaStream_t s, bool pdl) {
  switch (epi) {
    case kEInit: launch_one<kEInit>(g, a, b, o, s, pdl); break;
    case kEResid: launch_one<kEResid>(g, a, b, o, s, pdl); break;
    case kESwish: launch_one<kESwish>(g, a, b, o, s, pdl); break;
    case kEPlain: launch_one<kEPlain>(g, a, b, o, s, pdl); break;
    default: launch_one<kEGlu>(g, a, b, o, s, pdl); break;
  }
}

}  // namespace tsd
