// Building blocks of the tcgen05 GEMM kernels (device) and their TMA
// tensor maps (host), shared by the joint kernel and the generic GEMM.
#pragma once

#include <cuda.h>

#include <cstdint>

namespace tsd {
namespace tc {

constexpr int kBM = 128, kBK = 64;
constexpr unsigned long long kWaitNs = 1000000000ull;  // 1 s bound on any barrier wait
constexpr float kLog2e = 1.4426950408889634f;

// 2^x by the hardware approximation (relative error ~2^-22; 2^-inf = 0).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Pairs of fp32 values in one instruction (each rounded as the scalar ones).
__device__ __forceinline__ uint64_t pair_of(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpair(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// 1 / x for x in [1, 2^125], correctly rounded: the hardware's approximation
// and one Newton step with fused multiply-adds (P. Markstein, IBM J. Res. Dev.
// 34, 1990).
constexpr float kRecipMax = 0x1p125f;
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ uint64_t recip2(uint64_t x) {
  float a, b;
  unpair(x, a, b);
  a = rcp_approx(a), b = rcp_approx(b);
  const uint64_t r = pair_of(a, b);
  return fma2(r, fma2(x, pair_of(-a, -b), pair_of(1.f, 1.f)), r);
}

// y = 1 / (1 + e^-x), the bits of 1.f / (1.f + expf(-x)) at every x (0 where e^-x
// overflows).  One range check for the whole block: a division's own, per
// value, keeps the values apart.
template <int N>
__device__ __forceinline__ void sigmoid2(const uint64_t (&x)[N], uint64_t (&y)[N]) {
  float top = 0.f;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    float a, b;
    unpair(x[i], a, b);
    a = expf(-a), b = expf(-b);
    top = fmaxf(top, fmaxf(a, b));
    y[i] = add2(pair_of(a, b), pair_of(1.f, 1.f));
  }
  if (top < kRecipMax) {
#pragma unroll
    for (int i = 0; i < N; ++i) y[i] = recip2(y[i]);
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      float a, b;
      unpair(y[i], a, b);
      y[i] = pair_of(1.f / a, 1.f / b);
    }
  }
}

// y = x / (1 + e^-x), the bits of x / (1.f + expf(-x)) at every x: a quotient from
// the correctly rounded reciprocal and one remainder (as above) is correctly
// rounded while it and its remainder are normal numbers.
template <int N>
__device__ __forceinline__ void swish2(const uint64_t (&x)[N], uint64_t (&y)[N]) {
  uint64_t d[N];
  bool plain = true;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    float a, b;
    unpair(x[i], a, b);
    const float e = expf(-a), f = expf(-b);
    plain = plain && fmaxf(e, f) < 0x1p40f && fminf(fabsf(a), fabsf(b)) > 0x1p-80f && fmaxf(fabsf(a), fabsf(b)) < 0x1p100f;
    d[i] = add2(pair_of(e, f), pair_of(1.f, 1.f));
  }
  if (plain) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const uint64_t r = recip2(d[i]), q = mul2(x[i], r);
      float a, b;
      unpair(d[i], a, b);
      y[i] = fma2(fma2(pair_of(-a, -b), q, x[i]), r, q);
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      float a, b, u, v;
      unpair(x[i], a, b);
      unpair(d[i], u, v);
      y[i] = pair_of(a / u, b / v);
    }
  }
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// A shared-memory address in the CTA of that rank of the cluster.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}

// Untiled bulk copy global -> shared (both addresses 16-byte aligned, bytes a
// multiple of 16), completing its bytes on the barrier.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// True in one lane of a converged warp: MMAs issued by it go out closer than by a
// lane picked by its number (49 clocks apart against 57 at 128 x 64 x 16).
__device__ __forceinline__ bool elect() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Whether the phase has completed, without waiting.
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Waits for the phase of the given parity; false if it did not complete
// within limit_ns nanoseconds.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, unsigned long long limit_ns = kWaitNs) {
  if (mbar_try(b, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (!mbar_try(b, parity)) {
    if (global_ns() - t0 > limit_ns) return false;
  }
  return true;
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// TMA store of a 2-D box from shared memory (bulk-group completion), and its
// ordering helpers: the generic-proxy writes of the box must be fenced
// before the async proxy reads them; a buffer may be rewritten once its
// store has read it; the CTA waits for its stores before it exits.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(src)), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// at most N of this thread's store groups may still be reading shared memory
template <int N>
__device__ __forceinline__ void tma_store_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major tile stored with the 128-byte
// swizzle: rows of 64 bf16 (128 B), 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address
  d |= (uint64_t)1 << 16;                      // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;            // stride byte offset: next 8-row group
  d |= (uint64_t)1 << 46;                      // descriptor version
  d |= (uint64_t)2 << 61;                      // 128-byte swizzle
  return d;
}

// Instruction descriptor: kind::f16, A = B = bf16, D = f32, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// The MMAs of one tile over KB operand stages (A, then B at A_BYTES, 64-deep,
// 128-byte swizzle) by the calling thread; each stage is handed back to the
// producer when its MMAs have completed.  False if a wait expired.  The next
// stage's barrier is read while this stage's MMAs are issued: a narrow tile's
// stage otherwise takes 315 clocks (64 x 64) with its operands long there.
template <int STAGES, int STAGE_BYTES, int A_BYTES>
__device__ __forceinline__ bool mma_tile(uint32_t tmem, uint32_t smem, uint64_t* full, uint64_t* empty, int KB,
                                         uint32_t idesc, unsigned long long limit_ns) {
  int s = 0;
  uint32_t ph = 0;
  bool ready = mbar_test(full, 0);
  for (int kb = 0; kb < KB; ++kb) {
    if (!ready && !mbar_wait(full + s, ph, limit_ns)) return false;
    const int s1 = s + 1 == STAGES ? 0 : s + 1;
    const uint32_t ph1 = s1 == 0 ? ph ^ 1u : ph;
    ready = kb + 1 < KB && mbar_test(full + s1, ph1);
    fence_after();
    const uint64_t ad = sw128_desc(smem + s * STAGE_BYTES), bd = sw128_desc(smem + s * STAGE_BYTES + A_BYTES);
#pragma unroll
    for (int k = 0; k < kBK / 16; ++k)  // K = 16 per instruction: +32 bytes in the swizzle atom
      mma_bf16(tmem, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), idesc, (kb | k) ? 1u : 0u);
    mma_commit(empty + s);
    s = s1;
    ph = ph1;
  }
  return true;
}

// 32 consecutive fp32 columns of this warp's 32 TMEM lanes (one per thread).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}


// 16 consecutive fp32 columns of this warp's 32 TMEM lanes (one per thread).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Host: the driver's tensor-map encoder.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// 2-D row-major map (by default with the 128-byte swizzle): `inner` elements
// per row, boxes of box_inner x box_rows.
inline bool make_map(CUtensorMap* m, const void* base, CUtensorMapDataType dtype, int elem_bytes, int inner, int rows,
              int box_inner, int box_rows, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)inner * elem_bytes};
  cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return fn(m, dtype, 2, const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}


}  // namespace tc
}  // namespace tsd
