// Device helpers of the warp-specialised decode-attention kernels: barriers and staged copies, shared-memory accesses by
// 32-bit address, tensor-core tiles and small conversions.
#pragma once

#include "common.cuh"

namespace mixkvq {
namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
// Polls a phase of a barrier up to max_polls times; false if it never completed.
__device__ __forceinline__ bool mbar_wait_polls(uint32_t bar, uint32_t parity, uint32_t max_polls) {
  uint32_t ok;
  asm volatile(
      "{\n\t"
      ".reg .pred p, q;\n\t"
      ".reg .u32 n;\n\t"
      "mov.u32 n, 0;\n"
      "MIXKVQ_WAIT:\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n\t"
      "@p bra MIXKVQ_DONE;\n\t"
      "add.u32 n, n, 1;\n\t"
      "setp.lt.u32 q, n, %3;\n\t"
      "@q bra MIXKVQ_WAIT;\n"
      "MIXKVQ_DONE:\n\t"
      "selp.u32 %0, 1, 0, p;\n\t"
      "}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(max_polls)
      : "memory");
  return ok != 0;
}
// one lane of the (converged) warp arrives on the barrier
__device__ __forceinline__ void mbar_arrive_one(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\t@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(bar)
      : "memory");
}
// one lane of the (converged) warp stages `bytes` from global memory at shared address dst and arms the barrier for
// bytes + extra (extra > 0 only in the test of the give-up path); nothing happens when `enabled` is 0
__device__ __forceinline__ void stage_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar, uint32_t extra,
                                           uint32_t enabled) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t.reg .u32 tx;\n\t"
      "setp.ne.u32 e, %5, 0;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "and.pred p, p, e;\n\t"
      "add.u32 tx, %2, %4;\n\t"
      "@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%3], tx;\n\t"
      "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n\t"
      "}" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar), "r"(extra), "r"(enabled)
      : "memory");
}
// the same for a unit whose key-group scales do not lie directly before it: two copies on one barrier
__device__ __forceinline__ void stage_copy2(uint32_t dst_a, const void* src_a, uint32_t bytes_a, uint32_t dst_b,
                                            const void* src_b, uint32_t bytes_b, uint32_t bar, uint32_t extra, uint32_t enabled) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t.reg .u32 tx;\n\t"
      "setp.ne.u32 e, %8, 0;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "and.pred p, p, e;\n\t"
      "add.u32 tx, %2, %5;\n\t"
      "add.u32 tx, tx, %7;\n\t"
      "@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%6], tx;\n\t"
      "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%6];\n\t"
      "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%3], [%4], %5, [%6];\n\t"
      "}" ::"r"(dst_a),
      "l"(src_a), "r"(bytes_a), "r"(dst_b), "l"(src_b), "r"(bytes_b), "r"(bar), "r"(extra), "r"(enabled)
      : "memory");
}
// 16 bytes from global to shared memory, asynchronously (cp.async groups)
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// shared-memory accesses by 32-bit shared address (the offsets added at the call sites fold into the instruction)
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t a) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts128(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t x) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}
__device__ __forceinline__ void sts16(uint32_t a, uint32_t x) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((uint16_t)x) : "memory");
}

__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                        uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// d = a * b + c with the accumulator input in other registers than the result
__device__ __forceinline__ void mma_f16_to(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                           uint32_t b1, float c0, float c1, float c2, float c3) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
               : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// k = 8: A holds two words per lane, B one
__device__ __forceinline__ void mma_bf16_k8(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
  uint32_t y;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}
__device__ __forceinline__ uint32_t hfma2_u(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ uint32_t hmul2_u(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
// 2^x by the special-function unit alone (no range fix-up): inputs here are at most about 0, or -inf
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t pack_bf162(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
// two bf16 in one word -> two fp16 in one word (exact inside the fp16 range)
__device__ __forceinline__ uint32_t bf16x2_to_f16x2(uint32_t w) { return pack_half2(bf_lo(w), bf_hi(w)); }

// ---- The rotation of a fused decode step, on the query rows in shared memory.  A thread has one channel pair (i, i + 64) of every
// kThreads / 64-th row, one row behind another, so that it needs hardly any registers: rotated 16 bytes at a time on the way from global
// memory to the table, the main loops of a third of the kernels spilled, and the step without rotation needed kernels of its own.
// us per decode step, so / here: three tiers, 7b shape, 8 x 20011 tokens, 14 layers, rotating 497 / 487; 8 x 32768, not rotating 730 / 710;
// two tiers, 28 layers, not rotating 1056 / 1045; one sequence of 1024 tokens, 28 layers, rotating 177 / 174, not 159 / 155.
struct RopeInput {
  float c, s;               // of the thread's channel pair
  uint32_t k0, k1;          // the pair of the new key (the last 64 threads)
};
template <int kThreads>
__device__ __forceinline__ RopeInput rope_request(const LayerView& lv, int s) {
  static_assert(kThreads % 64 == 0, "a thread keeps its channel pair");
  const int i = threadIdx.x & 63;
  RopeInput in{lv.rope_cos[i], lv.rope_sin[i], 0u, 0u};
  if ((int)threadIdx.x >= kThreads - 64) {
    in.k0 = lv.new_k[(size_t)s * kD + i];
    in.k1 = lv.new_k[(size_t)s * kD + i + 64];
  }
  return in;
}
// Rotates the g rows of the table at qb16 (kStride halves apart; their fp16 copies at qf16 if kHalf) and the new key, which goes to
// key_row, its place in the residual window, unless that is null.  out_q: the rows in the caller's tensor, to be left rotated as the
// key there is (null: the merge does that).
template <int kThreads, int kStride, bool kHalf>
__device__ __forceinline__ void rope_rotate(const LayerView& lv, int s, int g, const RopeInput& in, uint32_t qb16, uint32_t qf16, uint16_t* key_row,
                                            uint16_t* out_q) {
  const int i = threadIdx.x & 63;
  auto pair = [&](uint32_t& lo, uint32_t& hi) {
    const float x0 = bf16_bits_to_float(lo), x1 = bf16_bits_to_float(hi);
    lo = pack_bf162(rotate_one(x0, x1, in.c, in.s, true), 0.f) & 0xFFFFu;
    hi = pack_bf162(rotate_one(x1, x0, in.c, in.s, false), 0.f) & 0xFFFFu;
  };
#pragma unroll 1
  for (int h = threadIdx.x >> 6; h < g; h += kThreads / 64) {
    const uint32_t at = qb16 + (h * kStride + i) * 2;
    uint32_t lo = lds16(at), hi = lds16(at + 128);
    pair(lo, hi);
    sts16(at, lo);
    sts16(at + 128, hi);
    if (kHalf) {
      sts16(qf16 + (h * kStride + i) * 2, bf16x2_to_f16x2(lo));
      sts16(qf16 + (h * kStride + i) * 2 + 128, bf16x2_to_f16x2(hi));
    }
    if (out_q != nullptr) {
      out_q[h * kD + i] = (uint16_t)lo;
      out_q[h * kD + i + 64] = (uint16_t)hi;
    }
  }
  if ((int)threadIdx.x >= kThreads - 64) {
    uint32_t lo = in.k0, hi = in.k1;
    pair(lo, hi);
    if (key_row != nullptr) {
      key_row[i] = (uint16_t)lo;
      key_row[i + 64] = (uint16_t)hi;
    }
    if (out_q != nullptr) {
      uint16_t* out_k = const_cast<uint16_t*>(lv.new_k) + (size_t)s * kD;
      out_k[i] = (uint16_t)lo;
      out_k[i + 64] = (uint16_t)hi;
    }
  }
}

}  // namespace
}  // namespace mixkvq
