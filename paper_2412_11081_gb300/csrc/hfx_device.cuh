// Device helpers shared by the split-precision translation units
// (hfx_mixed.cu, hfx_t1umma.cu): index lookups, operand splitting, warp sums and
// the tcgen05 / mbarrier / bulk-copy wrappers (inline PTX).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "hfx_internal.h"

namespace hfx {
namespace dev {

__device__ __forceinline__ int rup16(int x) { return (x + 15) & ~15; }

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Split modes (the plan's precision): every operand is two 16-bit pieces
// x = p0 + p1 + r, p0 the round-to-nearest of x and p1 of what p0 leaves.
//   kSplitBf16 (HFX_BF16X3): bf16 pieces, 16 significant bits, any FP32 range
//   kSplitHalf (HFX_BF16X6): fp16 pieces, 22 significant bits.  fp16 has
//     five exponent bits, so the stores hold x times a power of two
//     (SplitScale, per atom) that keeps every element's magnitude within 2^15:
//     the low piece is exact to 2^-25 of the stored scale, so elements down to
//     2^-18 of that bound keep all 22 bits and the rest an absolute error of
//     2^-40 of it.  Three products of two such pieces carry what six products of
//     three bf16 pieces did, at half the tensor-core work and two thirds of
//     the operand bytes.
constexpr int NP = kPieces;

// 2^e, e held within what the type has (terms that far from the largest of
// their sum round to nothing).
__device__ __forceinline__ float p2f(int e) { return __int_as_float((max(-126, min(127, e)) + 127) << 23); }
__device__ __forceinline__ double p2d(int e) { return __hiloint2double((max(-1022, min(1023, e)) + 1023) << 20, 0); }

// The factor between a value and its store, 2^e: 1 (and no multiplication) with bf16 pieces.
template <int SP>
__device__ __forceinline__ float pscale(int e) {
  return SP == kSplitHalf ? p2f(e) : 1.f;
}
template <int SP>
__device__ __forceinline__ double pscale_d(int e) {
  return SP == kSplitHalf ? p2d(e) : 1.0;
}

// Exponents of the fp16 pieces of Y^{XZ} (HFX_BF16X3), V_AB, and the product <Y^{AB}, Y^{BA}>.
__device__ __forceinline__ int y_exp(const DevPlan& P, int X, int Z) { return max(-120, min(120, P.sc.y[X] + P.sc.d[Z])); }
__device__ __forceinline__ int v_exp(const DevPlan& P, int A, int B) { return P.sc.q[A] - P.sc.d[B] - P.sc.y[B]; }
__device__ __forceinline__ int r2_exp(const DevPlan& P, int A, int B) { return P.sc.y[A] + P.sc.d[B] + P.sc.y[B] + P.sc.d[A]; }

template <int SP>
__device__ __forceinline__ void split_f(float x, uint16_t (&p)[NP]) {
  if (SP == kSplitHalf) {
    const __half h = __float2half_rn(x);
    p[0] = __half_as_ushort(h);
    p[1] = __half_as_ushort(__float2half_rn(x - __half2float(h)));
  } else {
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    p[0] = __bfloat16_as_ushort(h);
    p[1] = __bfloat16_as_ushort(__float2bfloat16_rn(x - __bfloat162float(h)));
  }
}

// The pieces of two values, x0 in the low half of each word.
template <int SP>
__device__ __forceinline__ void split2(float x0, float x1, uint32_t (&p)[NP]) {
  if (SP == kSplitHalf) {
    const __half2 h = __floats2half2_rn(x0, x1);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(x0 - f.x, x1 - f.y);
    p[0] = *reinterpret_cast<const uint32_t*>(&h);
    p[1] = *reinterpret_cast<const uint32_t*>(&l);
  } else {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - __low2float(h), x1 - __high2float(h));
    p[0] = *reinterpret_cast<const uint32_t*>(&h);
    p[1] = *reinterpret_cast<const uint32_t*>(&l);
  }
}

// The same for four consecutive values (element 0 in the low half of .x).
template <int SP>
__device__ __forceinline__ void split4(const float (&x)[4], uint2 (&p)[NP]) {
  uint32_t a[NP], b[NP];
  split2<SP>(x[0], x[1], a);
  split2<SP>(x[2], x[3], b);
#pragma unroll
  for (int i = 0; i < NP; ++i) p[i] = make_uint2(a[i], b[i]);
}

__device__ __forceinline__ int ylut_get(const DevPlan& P, int i, int j, int r0, int r1, int r2) {
  if (r0 < -P.HY0 || r0 > P.HY0 || r1 < -P.HY1 || r1 > P.HY1 || r2 < -P.HY2 || r2 > P.HY2) return -1;
  const long long n0 = 2 * P.HY0 + 1, n1 = 2 * P.HY1 + 1, n2 = 2 * P.HY2 + 1;
  const long long idx = (((((long long)i * P.N + j) * n0 + (r0 + P.HY0)) * n1 + (r1 + P.HY1)) * n2) + (r2 + P.HY2);
  return P.ylut[idx];
}

__device__ __forceinline__ int dlut_get(const DevPlan& P, int i, int j, int r0, int r1, int r2) {
  if (r0 < -P.HD0 || r0 > P.HD0 || r1 < -P.HD1 || r1 > P.HD1 || r2 < -P.HD2 || r2 > P.HD2) return -1;
  const long long n0 = 2 * P.HD0 + 1, n1 = 2 * P.HD1 + 1, n2 = 2 * P.HD2 + 1;
  const long long idx = (((((long long)i * P.N + j) * n0 + (r0 + P.HD0)) * n1 + (r1 + P.HD1)) * n2) + (r2 + P.HD2);
  return P.dlut[idx];
}

// ------------------------------------------------------------- warp-level MMA
// m16n8k16 MMAs on the pieces with FP32 accumulation, the split products and
// the ldmatrix loads of their fragments.
__device__ __forceinline__ uint32_t pack2(uint16_t lo, uint16_t hi) { return (uint32_t)lo | ((uint32_t)hi << 16); }

template <int SP>
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  if (SP == kSplitHalf)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// The piece products (0,1), (1,0), (0,0), smallest first.
template <int SP>
__device__ __forceinline__ void mma_split(float (&c)[4], const uint32_t (&a)[NP][4], const uint32_t (&b)[NP][2]) {
  mma16816<SP>(c, a[0], b[1]);
  mma16816<SP>(c, a[1], b[0]);
  mma16816<SP>(c, a[0], b[0]);
}

// Two independent accumulators with their product chains interleaved, so the
// dependent MMAs of one tile overlap the other's.
template <int SP>
__device__ __forceinline__ void mma_split2(float (&c0)[4], const uint32_t (&a0)[NP][4], const uint32_t (&b0)[NP][2],
                                           float (&c1)[4], const uint32_t (&a1)[NP][4], const uint32_t (&b1)[NP][2]) {
  mma16816<SP>(c0, a0[0], b0[1]);
  mma16816<SP>(c1, a1[0], b1[1]);
  mma16816<SP>(c0, a0[1], b0[0]);
  mma16816<SP>(c1, a1[1], b1[0]);
  mma16816<SP>(c0, a0[0], b0[0]);
  mma16816<SP>(c1, a1[0], b1[0]);
}

__device__ __forceinline__ void ldm_x4(uint32_t (&r)[4], const void* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}

__device__ __forceinline__ void ldm_x2(uint32_t (&r)[2], const void* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}

__device__ __forceinline__ void ldm_x2_trans(uint32_t (&r)[2], const void* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}

// ------------------------------------------------------------- tcgen05 / TMA
constexpr long long kWaitCycles = 1ll << 31;   // limit of one mbarrier wait (1 s at 2.07 GHz)

// Shared-memory matrix descriptor, no swizzle: start address, the byte
// distance between core matrices adjacent in K (lbo) and between core
// matrices adjacent in M/N (sbo), descriptor version 1 of the sm_100 family.
// The same two fields serve K-major and MN-major operands: lbo always steps
// along K, sbo along M/N.
__device__ __forceinline__ uint64_t sdesc2(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor of kind::f16 with A and B of the split's piece type
// (fp16 or bf16, both operands alike), FP32 accumulator; b_mn = 1 reads B as
// MN-major.
template <int SP>
__host__ __device__ constexpr uint32_t idesc_split(int M, int N, int b_mn) {
  return (1u << 4) | (SP == kSplitHalf ? 0u : (1u << 7) | (1u << 10)) | ((uint32_t)b_mn << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// One potentially blocking test: the thread may sleep in hardware up to
// kTryNs for the phase instead of polling the barrier through the shared-
// memory pipe (which the tensor cores' operand reads also use).
constexpr uint32_t kTryNs = 20000;

template <uint32_t HintNs = kTryNs>
__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
  uint32_t done;
  if (HintNs) {
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done)
                 : "r"(mbar), "r"(parity), "r"(HintNs)
                 : "memory");
  } else {
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done)
                 : "r"(mbar), "r"(parity)
                 : "memory");
  }
  return done != 0;
}

// Wait for the phase of the given parity to complete; false once kWaitCycles
// have passed without it (the caller then records an error and stops).  HintNs is
// the suspend-time hint of each test (0: the hardware's own default).
template <uint32_t HintNs = kTryNs>
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
  // One test in a small loop (unrolled at every wait, the tests grew the
  // tcgen05 kernels to 250 KB of code, past the instruction cache), and the
  // limit by the SM's cycle counter: a read of the wall clock in the loop
  // holds the thread for longer than the waits it bounds.  First product of
  // the 64-atom Si cell: 17.1 ms unrolled, 17.6 with the wall clock in the
  // loop, 13.5 as here; of the 8-atom minimal cell 0.62, 0.53, 0.37 ms.
  const long long t0 = clock64();
#pragma unroll 1
  while (!mbar_try<HintNs>(mbar, parity))
    if (clock64() - t0 > kWaitCycles) return false;
  return true;
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mbar), "r"(count));
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mbar), "r"(bytes) : "memory");
}

// Bulk asynchronous copy global -> shared (both 16-byte aligned, size a
// multiple of 16), completion counted in bytes on mbar.
__device__ __forceinline__ void bulk_g2s(uint32_t sdst, const void* gsrc, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(sdst),
               "l"(gsrc), "r"(bytes), "r"(mbar)
               : "memory");
}

__device__ __forceinline__ void umma_f16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
               " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
               "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void umma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// 32 lanes x 16 (or 8) consecutive 32-bit columns of tensor memory; the values are
// there after tmem_wait_ld.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }

// 32 lanes x 32 consecutive 32-bit columns of tensor memory (lane = thread of
// the warp's quarter), waited on.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

}  // namespace dev
}  // namespace hfx
