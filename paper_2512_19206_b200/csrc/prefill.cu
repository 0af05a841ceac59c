// Causal full-precision attention over a prompt (the prefill phase of Section 4.2: the prompt is attended in full
// precision, then quantized into the cache) on the tcgen05 tensor cores with tensor-memory accumulators.
//
// Two kernels.  prefill_pack_kernel rewrites K (bf16) and V (converted to fp16) of the prompt into images of 128-token
// tiles in the tensor core's canonical shared-memory layout, so that a tile reaches shared memory as ONE 32 KB bulk
// copy.  prefill_attention_kernel runs one CTA of 384 threads per 256 (short prompts: 128) query rows of a stream (batch element and KV head; a token's
// query heads side by side):
//   warps 0-3, 4-7   two softmax groups, one per 128 query rows (thread = row = lane of tensor memory);
//   warp 8           one thread issues every tcgen05.mma;
//   warp 9           one thread issues the bulk copies of the K and V tiles into two-stage rings.
// Per key tile j and row group g:
//   S_g = Q_g K_j^T   bf16 operands from shared memory, fp32 accumulator in tensor memory;
//   softmax           the thread reads its row of S (tcgen05.ld), applies scale and causal mask, and writes its row of P as
//                     fp16 over columns that S occupied (tcgen05.st);
//   O_g = P_g V_j     A operand from tensor memory, V from shared memory (MN-major).  The thread adds its row of the product to
//                     an fp32 sum in registers at the start of the next tile; when the maximum of a row of the warp has risen,
//                     the warp rescales its sums first (after the first tiles that is rare: a third of the 256 tiles at L = 32768).
// The issue order S_A(j+1) behind P_A V(j), S_B(j+1) behind P_B V(j) keeps the tensor core busy on one row group while
// the other one is in its softmax; the softmax threads never wait for a P V product (products complete in issue order, so S(j)
// being there means that P V(j-1) is done).  P and V are fp16 (11 significant bits): bf16 probabilities alone would cost up to
// 2^-9 of the value range.  Every wait on a barrier is bounded; a wait that runs out sets the status word and the
// role that saw it stops, after which the others run out too and the CTA finishes.
// Why the sum over the tiles is not left to the tensor core: its fp32 accumulator truncates, a bias of half a unit in the last
// place per product, and 8 products per tile add up.  Against fp64, values with a mean (|N(0,1)| + 0.5), relative error at 777 /
// 8192 / 32768 / 65536 tokens: 3.8e-5 / 3.8e-5 / 10.4e-5 / 17.8e-5 accumulated in tensor memory (bias -1.4e-4 at 32768);
// 3.8e-5 / 2.8e-5 / 2.8e-5 / 2.8e-5 with the sum in registers, the rounding of P.  Sums over 2, 4, 8 or 16 tiles in tensor memory: 2.83,
// 2.85, 2.91, 3.09e-5 at 32768, and no faster than 2 % (the registers cost the time, not the additions).
// B200, whole call per layer (us), sum in tensor memory / in registers, both with 256 rows of one head per CTA: prompt of 32768 tokens (7b
// shape) 6492 / 6811, 8192: 530 / 558, 333: 29.4 / 29.5; 4 x 777 tokens (8b shape) 100.7 / 103.5.  (Waiting for each product right behind its
// issue, and with the tensor core idle meanwhile: 7447, 699, 104, 169.)
// Tensor memory is read 16 columns at a time, the next 16 in flight, on the diagonal too: blocks of 32 registers beside the 128 of the sum
// spilled 96 to 356 bytes, whatever the split.  By 32 columns / by 16, on the diagonal one after another / in flight everywhere, 32768 tokens 6782 /
// 6919 / 6757, 8192 542 / 547 / 539.
// Rows: with 256 rows of one head per CTA the last row tile of 4 x 777 tokens (8b shape) held 9 rows of 256 and the diagonal tiles were
// half empty; side by side the heads take 13 row tiles with 49 key tiles per stream instead of 16 with 76: attention 75 -> 54 us,
// whole call 108 -> 93 us per layer.
#include "common.cuh"

namespace mixkvq {

namespace {

constexpr int kTile = 128;                       // query rows and key rows per tile
constexpr int kTileBytes = kTile * kD * 2;       // one 128 x 128 tile of 16-bit elements
constexpr int kQRows = 2 * kTile;                // query rows per CTA, or kTile (the rule is at the launch)
constexpr int kThreads = 384;
constexpr int kBars = 17;
constexpr int kSmem = 6 * kTileBytes + 256;      // two Q tiles, two K and two V stages; barriers and tensor-memory slot
enum Bar { kKFull = 0, kVFull = 2, kKEmpty = 4, kVEmpty = 6, kSFull = 8, kPHalf = 10, kPReady = 12, kDoneA = 14, kDoneB = 15, kDone = 16 };
constexpr uint32_t kPolls = 1u << 21;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Canonical layout without swizzle: 8-row x 16-byte core matrices; row r, 16-bit element k of a 128 x 128 K-major tile
// sits at byte (r / 8) * 2048 + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
// instruction descriptor of kind::f16: fp32 accumulator; operand formats 0 = fp16, 1 = bf16; B K-major (0) or MN-major (1)
__device__ __forceinline__ constexpr uint32_t make_idesc(int M, int N, int fmt, int b_mn_major) {
  return (1u << 4) | ((uint32_t)fmt << 7) | ((uint32_t)fmt << 10) | ((uint32_t)b_mn_major << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ bool mbar_wait_polls(uint32_t bar, uint32_t parity, uint32_t max_polls) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .u32 n;\n\tmov.u32 n, 0;\n"
      "PREFILL_WAIT:\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n\t"
      "@p bra PREFILL_DONE;\n\t"
      "add.u32 n, n, 1;\n\t"
      "setp.lt.u32 q, n, %3;\n\t"
      "@q bra PREFILL_WAIT;\n"
      "PREFILL_DONE:\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(max_polls)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D (tensor memory) = A (shared memory) * B (shared memory) [+ D]
__device__ __forceinline__ void tc_mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// A load of 16 columns of the thread's tensor-memory lane.  The registers are valid only after tmem_wait_ld16 on them (the wait names
//  the registers as operands, so that no use of them is scheduled before it).  tcgen05.wait::ld covers every load
// the thread has issued, so a load issued before a block of arithmetic and waited for after it runs under that arithmetic.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&u)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
        "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait_ld16(uint32_t (&u)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]), "+r"(u[4]), "+r"(u[5]), "+r"(u[6]), "+r"(u[7]), "+r"(u[8]),
                 "+r"(u[9]), "+r"(u[10]), "+r"(u[11]), "+r"(u[12]), "+r"(u[13]), "+r"(u[14]), "+r"(u[15])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&w)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(w[0]), "r"(w[1]),
               "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t bf16x2_to_f16x2(uint32_t w) {
  return pack_half2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}


__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// D (tensor memory) = A (tensor memory, 16-bit pairs per column) * B (shared memory) [+ D]
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// K, V [B * Hkv][L][128] bf16 -> tile images [B * Hkv][n_tiles][32 KB]: K as the K-major B operand of Q K^T (bf16),
// V as the MN-major B operand of P V (fp16); rows past L are zero.  Consecutive threads write consecutive 16 bytes.
__global__ void __launch_bounds__(256)
prefill_pack_kernel(const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v, unsigned char* __restrict__ kt,
                    unsigned char* __restrict__ vt, int L, int n_tiles) {
  dependency_wait();
  const int t = blockIdx.x, s = blockIdx.y;
  const __nv_bfloat16* kg = k + ((size_t)s * L + (size_t)t * kTile) * kD;
  const __nv_bfloat16* vg = v + ((size_t)s * L + (size_t)t * kTile) * kD;
  uint4* kd = reinterpret_cast<uint4*>(kt + ((size_t)s * n_tiles + t) * kTileBytes);
  uint4* vd = reinterpret_cast<uint4*>(vt + ((size_t)s * n_tiles + t) * kTileBytes);
  const int rows = min(kTile, L - t * kTile);
  // all of a thread's loads are in flight at once
  constexpr int kEach = kTile * 16 / 256;
  uint4 x[kEach], y[kEach];
#pragma unroll
  for (int n = 0; n < kEach; ++n) {
    const int i = threadIdx.x + 256 * n;
    // K: byte offset (r / 8) * 2048 + c * 128 + (r % 8) * 16 of row r, 16-byte chunk c; V: c * 2048 + (r / 8) * 128 + (r % 8) * 16
    const int kr = 8 * (i >> 7) + (i & 7), kc = (i >> 3) & 15, vr = i & 127, vc = i >> 7;
    x[n] = y[n] = make_uint4(0u, 0u, 0u, 0u);
    if (kr < rows) x[n] = *reinterpret_cast<const uint4*>(kg + (size_t)kr * kD + 8 * kc);
    if (vr < rows) y[n] = *reinterpret_cast<const uint4*>(vg + (size_t)vr * kD + 8 * vc);
  }
#pragma unroll
  for (int n = 0; n < kEach; ++n) {
    const int i = threadIdx.x + 256 * n;
    kd[i] = x[n];
    vd[i] = make_uint4(bf16x2_to_f16x2(y[n].x), bf16x2_to_f16x2(y[n].y), bf16x2_to_f16x2(y[n].z), bf16x2_to_f16x2(y[n].w));
  }
}

// Two fp32 values in one 64-bit register: the FMA pipe does both halves of these with one instruction.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ uint64_t pack2u(uint32_t a, uint32_t b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t x, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Calls f(piece, columns) for the pieces of 16 columns below n_pieces of the thread's tensor-memory row, the next piece in flight.
template <bool kAll, typename F>
__device__ __forceinline__ void for_pieces(uint32_t taddr, int n_pieces, F f) {
  if constexpr (kAll) {
    uint32_t a[16], b[16];
    tmem_ld16_issue(taddr, a);
#pragma unroll
    for (int h = 0; h < 8; h += 2) {
      tmem_wait_ld16(a);
      tmem_ld16_issue(taddr + 16 * h + 16, b);
      f(h, a);
      tmem_wait_ld16(b);
      if (h < 6) tmem_ld16_issue(taddr + 16 * h + 32, a);
      f(h + 1, b);
    }
  } else {
    uint32_t a[16], b[16];
    tmem_ld16_issue(taddr, a);
#pragma unroll 1
    for (int h = 0; h < n_pieces; h += 2) {
      tmem_wait_ld16(a);
      if (h + 1 < n_pieces) tmem_ld16_issue(taddr + 16 * h + 16, b);
      f(h, a);
      if (h + 1 < n_pieces) {
        tmem_wait_ld16(b);
        if (h + 2 < n_pieces) tmem_ld16_issue(taddr + 16 * h + 32, a);
        f(h + 1, b);
      }
    }
  }
}

// Adds the row's P V product in tensor memory to the sum kept in registers.
__device__ __forceinline__ void add_output(uint32_t o_addr, float (&sum_o)[128]) {
  for_pieces<true>(o_addr, 8, [&](int h, const uint32_t (&x)[16]) {
#pragma unroll
    for (int k = 0; k < 16; k += 2)
      unpack2(add2(pack2u(x[k], x[k + 1]), pack2(sum_o[16 * h + k], sum_o[16 * h + k + 1])), sum_o[16 * h + k], sum_o[16 * h + k + 1]);
  });
}

// One 128-key tile of one row group's softmax.  The thread owns one row of S (128 fp32 columns of its tensor-memory lane at
// s_addr) and of the last product P V (at o_addr), which goes to its sum.  Writes P (fp16 pairs) over columns [0, 64) of S.  kDiag: the
// tile on the diagonal: the thread's row sees the columns <= last, none of the warp's rows sees those > warp_last; the product takes the
// pieces of 16 keys below n_write (rows that see none of a piece have zeros there).
template <bool kDiag>
__device__ __forceinline__ void softmax_tile(uint32_t s_addr, uint32_t o_addr, int warp_last, int last, int n_write, bool first, float scale_log2e,
                                             float& m_ref, float& l_run, uint32_t half_bar, float (&sum_o)[128]) {
  if (!first) add_output(o_addr, sum_o);             // the product of the tile before
  // ---- the row's maximum
  float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};      // four independent chains
  const int n_seen = kDiag ? (warp_last >> 4) + 1 : 8;              // pieces of 16 columns that some row of the warp sees
  for_pieces<!kDiag>(s_addr, n_seen, [&](int h, const uint32_t (&u)[16]) {
    const int lim = last - 16 * h;
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      const float x0 = kDiag && i > lim ? -INFINITY : __uint_as_float(u[i]);
      const float x1 = kDiag && i + 1 > lim ? -INFINITY : __uint_as_float(u[i + 1]);
      mx4[(i >> 1) & 3] = fmaxf(fmaxf(mx4[(i >> 1) & 3], x0), x1);
    }
  });
  const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * scale_log2e;
  if (first) {
    m_ref = mx;
  } else if (__any_sync(0xffffffffu, mx > m_ref)) {
    // raise the reference and rescale the sum of the products before this tile
    const float m_new = fmaxf(m_ref, mx), alpha = ex2(m_ref - m_new);
    const uint64_t alpha2 = pack2(alpha, alpha);
#pragma unroll
    for (int d = 0; d < 128; d += 2) unpack2(mul2(pack2(sum_o[d], sum_o[d + 1]), alpha2), sum_o[d], sum_o[d + 1]);
    l_run *= alpha;
    m_ref = m_new;
  }
  // P of the first 64 keys is handed over on its own: its products run while the other half is computed
  auto half_ready = [&]() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    tc_fence_before();
    mbar_arrive(half_bar);
  };
  // ---- probabilities, 16 columns at a time, the next ones in flight; P piece h (8 columns of fp16 pairs) lies inside the S columns of
  // pieces <= h, which are already in registers
  const uint64_t scale2 = pack2(scale_log2e, scale_log2e), ref2 = pack2(-m_ref, -m_ref);
  uint64_t sum[2] = {0ull, 0ull};
  auto probs = [&](const uint32_t (&u)[16], int h) {
    uint32_t wd[8];
    const int lim = last - 16 * h;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float x0, x1;
      unpack2(fma2(pack2u(u[2 * i], u[2 * i + 1]), scale2, ref2), x0, x1);
      float p0 = ex2(x0), p1 = ex2(x1);
      if constexpr (kDiag) {
        p0 = 2 * i <= lim ? p0 : 0.f;
        p1 = 2 * i + 1 <= lim ? p1 : 0.f;
      }
      sum[i & 1] = add2(sum[i & 1], pack2(p0, p1));
      wd[i] = pack_half2(p0, p1);
    }
    tmem_st8(s_addr + 8 * h, wd);
  };
  for_pieces<!kDiag>(s_addr, n_seen, [&](int h, const uint32_t (&u)[16]) {
    probs(u, h);
    if (h == 3) half_ready();
  });
  if constexpr (kDiag) {
    for (int h = n_seen; h < n_write; ++h) {
      const uint32_t zero[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
      tmem_st8(s_addr + 8 * h, zero);
      if (h == 3) half_ready();
    }
    if (max(n_seen, n_write) < 4) half_ready();
  }
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  float s0, s1;
  unpack2(add2(sum[0], sum[1]), s0, s1);
  l_run += s0 + s1;
}

// q [B, Hq, L, 128] bf16; kt, vt the tile images of prefill_pack_kernel; out [B, Hq, L, 128] fp32.  A stream's query rows are numbered
// token by token, its g heads side by side: row x is head x % g of token x / g.  A CTA takes 256 such rows, two groups of 128.  128
// tokens are g whole groups, so that a group's tokens lie in one key tile, its last, and a group of 128 / g tokens does less than a
// group of 128 tokens of one head where it lies at the diagonal, and a prompt that is no multiple of 256 leaves fewer rows idle.
// blockIdx.x / n_streams counts the row tiles from the last one down (it has the most key tiles: the long CTAs start first),
// blockIdx.x % n_streams = b * Hkv + hk.
__global__ void __launch_bounds__(kThreads, 1)
prefill_attention_kernel(const __nv_bfloat16* __restrict__ q, const unsigned char* __restrict__ kt,
                         const unsigned char* __restrict__ vt, float* __restrict__ out, int n_streams, int g_heads, int L,
                         int n_tiles, int n_qtiles, int q_rows, float scale_log2e, uint32_t* status, uint32_t max_polls, uint32_t debug_extra_tx,
                         uint32_t debug_extra_v) {
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* Qs = smem;                              // two tiles
  unsigned char* Ks = smem + 2 * kTileBytes;             // two stages
  unsigned char* Vs = smem + 4 * kTileBytes;             // two stages
  const uint32_t bars = smem_u32(smem + 6 * kTileBytes);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + 6 * kTileBytes + 8 * kBars);
  auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int qt = n_qtiles - 1 - (int)blockIdx.x / n_streams, s = (int)blockIdx.x % n_streams;
  const uint32_t g_inv = 65536u / (uint32_t)g_heads + 1u;              // x / g = x * g_inv >> 16 for x < 512
  struct Rows {          // of a row tile: the first row's token and head
    int tok0, rem0, L;
    uint32_t inv;
    __device__ int token(int row) const { return min(tok0 + (int)((uint32_t)(rem0 + row) * inv >> 16), L - 1); }
  };
  auto rows_of = [&](int tile) {
    const int tok0 = tile * q_rows / g_heads;
    return Rows{tok0, tile * q_rows - tok0 * g_heads, L, g_inv};
  };
  const unsigned char* ktg = kt + (size_t)s * n_tiles * kTileBytes;
  const unsigned char* vtg = vt + (size_t)s * n_tiles * kTileBytes;
  // The two groups: the last token (rows past the prompt see what its last token sees and are not stored), its key tiles (n_b = 0: no
  // row of the prompt in group B; n_a <= n_b otherwise) and the columns of the last of them that some row sees
  const Rows rows = rows_of(qt);
  const int tok0 = rows.tok0, rem0 = rows.rem0;
  const int last_a = rows.token(kTile - 1), last_b = rows.token(kQRows - 1);
  const int n_a = last_a / kTile + 1, n_b = q_rows == kQRows && qt * kQRows + kTile < L * g_heads ? last_b / kTile + 1 : 0, n = max(n_a, n_b);
  const int seen_a = last_a % kTile + 1, seen_b = last_b % kTile + 1;

  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  int issued = 0;                  // K and V tiles requested (the copying thread)
  // (test hooks: the barrier of the first key tile, or of the last value tile where that is odd or the prompt's last, can be armed for
  // more bytes than arrive, so that it never completes.  Not of every last value tile: some CTAs end as usual beside those that give up.)
  const int armed_v = (n & 1) == 0 || n == n_tiles ? n - 1 : -1;
  auto copy_tile = [&](int j, bool keys) {
    const int st = j & 1, full = (keys ? kKFull : kVFull) + st;
    mbar_expect_tx(bar(full), kTileBytes + (keys ? (j == 0 ? debug_extra_tx : 0u) : (j == armed_v ? debug_extra_v : 0u)));
    bulk_copy(smem_u32((keys ? Ks : Vs) + st * kTileBytes), (keys ? ktg : vtg) + (size_t)j * kTileBytes, kTileBytes, bar(full));
  };
  if (tid == 9 * 32) {
    for (int i = 0; i < kBars; ++i) mbar_init(bar(i), i >= kPHalf && i < kDoneA ? kTile : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    // the first tiles are under way while Q is loaded (Q was written before the kernel that packs the tiles: only the tiles
    // wait for that kernel)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (; issued < min(2, n); ++issued) {
      copy_tile(issued, true);
      copy_tile(issued, false);
    }
  }
  // both Q tiles: piece i of a tile is 16 bytes at byte 16 i of its image (rows past L are zero).  All of a thread's loads are
  // in flight at once (one after the other they took 8000 to 12000 cycles of a CTA that needs 3900 per key tile).
  {
    constexpr int kPieces = 2 * kTile * 16, kEach = (kPieces + kThreads - 1) / kThreads;
    uint4 x[kEach];
#pragma unroll
    for (int k = 0; k < kEach; ++k) {
      const int i = tid + k * kThreads, ii = i & 2047, c = (ii >> 3) & 15;
      const uint32_t r = (uint32_t)(rem0 + (i >> 11) * kTile + 8 * (ii >> 7) + (ii & 7)), tk = r * g_inv >> 16;
      x[k] = make_uint4(0u, 0u, 0u, 0u);
      if (i < q_rows * 16 && tok0 + (int)tk < L)
        x[k] = *reinterpret_cast<const uint4*>(q + (((size_t)s * g_heads + (r - tk * g_heads)) * L + tok0 + tk) * kD + 8 * c);
    }
#pragma unroll
    for (int k = 0; k < kEach; ++k)
      if (tid + k * kThreads < kPieces) reinterpret_cast<uint4*>(Qs)[tid + k * kThreads] = x[k];
  }
  // Every thread waits for the kernel before: nothing below runs, and no successor starts, before that is complete.
  dependency_wait();
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");        // Q is read by the tensor core
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = *tmem_slot;
  // tensor-memory columns: S_A / P_A at 0, S_B / P_B at 128, O_A at 256, O_B at 384
  bool dead = false;
  auto wait = [&](int i, uint32_t parity) {
    if (!dead && !mbar_wait_polls(bar(i), parity, max_polls)) {
      dead = true;
      atomicOr(status, (uint32_t)MIXKVQ_DEV_COPY_TIMEOUT);
    }
    return !dead;
  };

  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;" ::: "memory");
    if (warp == 8 && lane == 0) {
      // ---------------------------------------------------------------- tensor-core issue
      const uint32_t idesc_qk = make_idesc(128, 128, 1, 0), idesc_pv = make_idesc(128, 128, 0, 1);
      // S_g = Q_g K_j^T; of a group's last key tile only the columns that some row sees
      auto issue_s = [&](int g, int j, int seen) {
        const uint64_t qd = make_desc(smem_u32(Qs + g * kTileBytes), 128, 2048);
        const uint64_t kd = make_desc(smem_u32(Ks + (j & 1) * kTileBytes), 128, 2048);
        const uint32_t idesc = seen == kTile ? idesc_qk : make_idesc(128, (seen + 15) & ~15, 1, 0);
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) tc_mma_ss(tbase + 128 * g, qd + (uint64_t)(ks * 16), kd + (uint64_t)(ks * 16), idesc, ks > 0);
        tc_commit(bar(kSFull + g));
      };
      // O_g = P_g V_j, 64 of the tile's keys at a time, as soon as each half of P_g is there (a product of its own per tile).  Whole tiles
      // without a decision between the instructions: the issuing thread's own time counts.
      auto issue_o = [&](int g, int j, int seen) {
        const uint64_t vd = make_desc(smem_u32(Vs + (j & 1) * kTileBytes), 128, 2048);
        const uint32_t o = tbase + 256 + 128 * g, p = tbase + 128 * g;
        if (!wait(kPHalf + g, (uint32_t)j & 1u)) return false;
        tc_fence_after();
        if (seen == kTile) {
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) tc_mma_ts(o, p + 8 * ks, vd + (uint64_t)(ks * 16), idesc_pv, ks > 0);
        } else {
          for (int ks = 0; ks < 4 && 16 * ks < seen; ++ks) tc_mma_ts(o, p + 8 * ks, vd + (uint64_t)(ks * 16), idesc_pv, ks > 0);
        }
        if (!wait(kPReady + g, (uint32_t)j & 1u)) return false;
        tc_fence_after();
        if (seen == kTile) {
#pragma unroll
          for (int ks = 4; ks < 8; ++ks) tc_mma_ts(o, p + 8 * ks, vd + (uint64_t)(ks * 16), idesc_pv, 1);
        } else {
          for (int ks = 4; 16 * ks < seen; ++ks) tc_mma_ts(o, p + 8 * ks, vd + (uint64_t)(ks * 16), idesc_pv, 1);
        }
        return true;
      };
      if (wait(kKFull, 0)) {
        tc_fence_after();
        issue_s(0, 0, n_a == 1 ? seen_a : kTile);
        if (n_b > 0) issue_s(1, 0, n_b == 1 ? seen_b : kTile);
        tc_commit(bar(kKEmpty));
      }
      for (int j = 0; j < n && !dead; ++j) {
        const int st = j & 1, nx = (j + 1) & 1;
        const uint32_t ph = (uint32_t)(j >> 1) & 1u, ph_nx = (uint32_t)((j + 1) >> 1) & 1u;
        if (!wait(kVFull + st, ph)) break;
        if (j < n_a) {
          if (!issue_o(0, j, j + 1 == n_a ? seen_a : kTile)) break;
          if (n_b == 0) tc_commit(bar(kVEmpty + st));
          if (j + 1 == n_a) tc_commit(bar(kDoneA));
          if (j + 1 < n_a) {
            if (!wait(kKFull + nx, ph_nx)) break;
            tc_fence_after();
            issue_s(0, j + 1, j + 2 == n_a ? seen_a : kTile);
            if (n_b == 0) tc_commit(bar(kKEmpty + nx));
          }
        }
        if (n_b == 0) continue;
        if (!issue_o(1, j, j + 1 == n_b ? seen_b : kTile)) break;
        tc_commit(bar(kVEmpty + st));
        if (j + 1 == n_b) tc_commit(bar(kDoneB));        // (not when a wait ran out: group B must not take an unfinished product)
        if (j + 1 < n_b) {
          if (!wait(kKFull + nx, ph_nx)) break;
          tc_fence_after();
          issue_s(1, j + 1, j + 2 == n_b ? seen_b : kTile);
          tc_commit(bar(kKEmpty + nx));
        }
      }
      tc_commit(bar(kDone));                             // every product issued above has finished when this one fires
      dead = false;
      wait(kDone, 0);
    } else if (warp == 9 && lane == 0) {
      // ---------------------------------------------------------------- bulk copies of the K and V tiles
      for (int j = 2; j < n; ++j) {
        const int st = j & 1;
        const uint32_t ph_prev = (uint32_t)((j >> 1) - 1) & 1u;
        if (!wait(kKEmpty + st, ph_prev)) break;
        copy_tile(j, true);
        issued = j + 1;
        if (!wait(kVEmpty + st, ph_prev)) {               // the K copy above is awaited below like the others
          mbar_expect_tx(bar(kVFull + st), 0);
          break;
        }
        copy_tile(j, false);
      }
      // no copy may be in flight when the CTA ends: the last copy into each stage has landed once its barrier's phase is over
      for (int j = max(0, issued - 2); j < issued; ++j) {
        dead = false;                                    // every one of these waits is made, whatever the others did
        wait(kKFull + (j & 1), (uint32_t)(j >> 1) & 1u);
        dead = false;
        wait(kVFull + (j & 1), (uint32_t)(j >> 1) & 1u);
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 216;" ::: "memory");
    // ------------------------------------------------------------------ softmax and output rows
    const int g = warp >> 2;
    const uint32_t lane_base = tbase + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t s_addr = lane_base + 128 * g, o_addr = lane_base + 256 + 128 * g;
    const int n_g = g == 0 ? n_a : n_b;
    // worked out again where it is needed: the loop has no registers to keep it in
    auto rows_again = [&]() {
      int again = qt;
      asm volatile("" : "+r"(again));
      return rows_of(again);
    };
    float m_ref = -INFINITY, l_run = 0.f;
    float sum_o[128];
#pragma unroll
    for (int d = 0; d < 128; ++d) sum_o[d] = 0.f;
    int j = 0;
    auto s_ready = [&]() {
      if (!wait(kSFull + g, (uint32_t)j & 1u)) return false;
      tc_fence_after();
      return true;
    };
    auto p_ready = [&]() {
      tc_fence_before();
      mbar_arrive(bar(kPReady + g));
    };
#pragma unroll 1
    for (; j + 1 < n_g; ++j) {
      if (!s_ready()) break;
      softmax_tile<false>(s_addr, o_addr, 0, 0, 8, j == 0, scale_log2e, m_ref, l_run, bar(kPHalf + g), sum_o);
      p_ready();
    }
    if (n_g > 0 && !dead && s_ready()) {       // the tile on the diagonal
      const Rows at = rows_again();
      const int r = g * kTile + (tid & 127), c0 = j * kTile;
      softmax_tile<true>(s_addr, o_addr, at.token(r | 31) - c0, at.token(r) - c0, (at.token(g * kTile + 127) - c0 + 16) >> 4, j == 0,
                         scale_log2e, m_ref, l_run, bar(kPHalf + g), sum_o);
      p_ready();
    }
    // Output rows.  The rows of a warp are 512 bytes or more apart, so direct stores cost a wavefront per lane (10 thousand cycles for
    // 256 rows at once, about half for 128).  Where group A is done a tile earlier than group B it stores directly, in 32-byte
    // pieces where the caller's buffer allows, under B's last tile; otherwise the rows go through the shared memory, which nobody needs
    // any more once B's last product is there, and leave as one bulk copy each.
    const bool direct = g == 0 && n_a < n_b;
    if (n_g > 0 && wait(g == 0 ? kDoneA : kDoneB, 0) && (direct || n_b == 0 || wait(kDoneB, 0))) {
      tc_fence_after();
      add_output(o_addr, sum_o);
      const float inv = 1.f / l_run;
      const Rows at = rows_again();
      const int row = tid & 127;
      const uint32_t x = (uint32_t)(at.rem0 + g * kTile + row), tk = x * g_inv >> 16;
      const bool valid = at.tok0 + (int)tk < L;
      float* dst = out + (((size_t)s * g_heads + (x - tk * g_heads)) * L + at.tok0 + tk) * kD;
      const bool wide = (reinterpret_cast<uintptr_t>(out) & 31u) == 0;
      const uint32_t staged = smem_u32(smem) + (uint32_t)(g * kTile + row) * 528u;      // (a row's 16-byte pieces on the banks of no other lane)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float y[32];
#pragma unroll
        for (int d = 0; d < 32; ++d) y[d] = sum_o[32 * c + d] * inv;
        if (!direct) {
#pragma unroll
          for (int d = 0; d < 32; d += 4)
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(staged + 4 * (32 * c + d)), "f"(y[d]), "f"(y[d + 1]),
                         "f"(y[d + 2]), "f"(y[d + 3])
                         : "memory");
        } else if (valid) {
#pragma unroll
          for (int d = 0; d < 32; d += 8) {
            if (wide) {
              asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + 32 * c + d), "f"(y[d]), "f"(y[d + 1]),
                           "f"(y[d + 2]), "f"(y[d + 3]), "f"(y[d + 4]), "f"(y[d + 5]), "f"(y[d + 6]), "f"(y[d + 7])
                           : "memory");
            } else {
              reinterpret_cast<float4*>(dst + 32 * c + d)[0] = make_float4(y[d], y[d + 1], y[d + 2], y[d + 3]);
              reinterpret_cast<float4*>(dst + 32 * c + d)[1] = make_float4(y[d + 4], y[d + 5], y[d + 6], y[d + 7]);
            }
          }
        }
      }
      if (!direct && valid) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(staged), "r"(kD * 4) : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(512) : "memory");
}

}  // namespace

cudaError_t prefill_attention_setup() {
  return cudaFuncSetAttribute(prefill_attention_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
}

size_t prefill_scratch_bytes(int B, int Hkv, int L) {
  return (size_t)2 * B * Hkv * ((L + kTile - 1) / kTile) * kTileBytes;
}

cudaError_t launch_prefill_attention(const void* q, const void* k, const void* v, float* out, void* scratch, int B, int Hq,
                                     int Hkv, int L, float scale, uint32_t* status, uint32_t max_polls, uint32_t debug_extra_tx,
                                     uint32_t debug_extra_v, int n_sms, cudaStream_t stream) {
  const int g = Hq / Hkv, n_tiles = (L + kTile - 1) / kTile;
  // A short prompt's row tiles leave most SMs idle: 128 rows per CTA as long as every CTA has an SM to itself and a sixth of the SMs is left
  // for the append, which runs beside the attention (no SM has the registers for both).  us per layer of the whole call, 256 / 128 rows: one prompt
  // of the 7b shape, 60 tokens (16 CTAs with 128 rows) 19.2 / 17.3, 333 (76) 27.2 / 25.5, 550 (124) 31.3 / 28.6, 621 (136) 37.3 / 38.9, 655 (144)
  // 33.7 / 46.7; 8b shape 450 (120) 29.6 / 26.9, 540 (136) 30.9 / 32.8; 4 prompts of the 7b shape, 100 (96) 29.4 / 27.0, 130 (128) 26.3 / 27.8.
  const int q_rows = ((long long)L * g + kTile - 1) / kTile * B * Hkv <= n_sms * 5 / 6 ? kTile : kQRows;
  const int n_qtiles = (int)(((long long)L * g + q_rows - 1) / q_rows);
  unsigned char* kt = static_cast<unsigned char*>(scratch);
  unsigned char* vt = kt + (size_t)B * Hkv * n_tiles * kTileBytes;
  const cudaError_t e = launch_dependent(prefill_pack_kernel, dim3((unsigned)n_tiles, (unsigned)(B * Hkv)), 256, 0, stream,
                                         static_cast<const __nv_bfloat16*>(k), static_cast<const __nv_bfloat16*>(v), kt, vt, L, n_tiles);
  if (e != cudaSuccess) return e;
  return launch_dependent(prefill_attention_kernel, dim3((unsigned)(n_qtiles * B * Hkv)), kThreads, kSmem, stream,
                          static_cast<const __nv_bfloat16*>(q), kt, vt, out, B * Hkv, g, L, n_tiles, n_qtiles, q_rows,
                          scale * 1.4426950408889634f, status, max_polls ? max_polls : kPolls, debug_extra_tx, debug_extra_v);
}

}  // namespace mixkvq
