// The lazy update of Appendix D.1 for full windows of R tokens: channel statistics, salience and tiers (Section 4.2),
// per-channel mixed-precision key quantization and per-token value quantization (Eq. 2), and bit-packing into the block
// layout.
//
// Work is cut into roles, one CTA of 256 threads each:
//   tiers    (bulk only) one window: importance from its queries, key extrema, the 128 tiers, the tier counts; the last
//            CTA of a stream to finish turns the stream's counts into places in the promoted-channel arena
//   keys     one window: key codes, scales, promoted channels and high planes, packed
//   values   one window: value codes and scales, packed
//   tail     (bulk only) one stream: the last 1..R tokens of the append go to the residual window
// Decode flushes the residual window in one launch of a keys CTA (which finds the tiers itself) and a values CTA per
// stream.  A bulk append quantizes complete windows straight from the tensors in two launches, tiers and values first,
// then keys and tails, because a block's place in the arena depends on the tier counts of the blocks before it.
//
// What bounds it: a bulk append reads g + 3 rows of 256 bytes per token and KV head (queries, keys twice, values) and
// writes about 100 bytes, so HBM by design; the quantization itself is about 8 instructions per code.  Figures at
// launch_flush_bulk.
#include "window.cuh"

namespace mixkvq {

namespace {

struct BulkSrc {
  const uint16_t* k;      // [S][n_tokens][128] bf16 bits
  const uint16_t* v;      // [S][n_tokens][128]
  const uint16_t* q;      // [B][Hq][n_tokens][128]
  int n_tokens, t0;       // tokens per stream in the tensors, first token of block 0 of this call
  int nb;                 // blocks of this call
  int tail;               // tokens behind them that go to the residual window
  int behind_prefill;     // the kernel before the first launch is the prefill attention of the same tensors
};

constexpr int kKeyRow = 68;      // 32-bit words per staged key row: rows r = 0..7 start 4 banks apart
constexpr int kValRow = 66;      // ... value row: rows 2t, t = 0..3, start 4 banks apart
// bytes 128.. of a still unwritten block hold its window's cumulative importance between two launches
constexpr int kSnapshotOff = 128, kSnapshotCntOff = 128 + 1024;
// per-stream state, a word of its zero padding: windows of the current launch that are done (0 between launches)
constexpr int kDoneOff = 1032;

__host__ __device__ inline uint32_t flush_extras_bytes(const LayerView& lv, int n16, int n4) {
  return lv.tile ? tile_extras_header_bytes(n16, n4) + tile_extras_body_bytes(n16, n4)
                 : extras_header_bytes(n16, n4) + (uint32_t)lv.U * extras_unit_bytes(n16, n4, lv.dense_hi != 0);
}

constexpr uint32_t kNegInf2 = 0xFF80FF80u, kPosInf2 = 0x7F807F80u;
__device__ __forceinline__ float lo_f(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_f(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// Reciprocal of a stored scale for the code computation; 0 for s = 0 (a constant group, or a channel without codes): every
// code is then 0.  A scale of 2^-128 or less has none in fp32: NaN, which sends every code of the group to the division.
__device__ __forceinline__ float code_reciprocal(float s) {
  const float r = __frcp_rn(s);
  return s == 0.0f ? 0.0f : (fabsf(r) == INFINITY ? __int_as_float(0x7FFFFFFF) : r);
}

// The code of Eq. 2 (quant_code in common.cuh) without its division: p = t * r with t = x - z rounded as there and
// r = RN(1 / s) differs from the IEEE quotient by less than 2e-6 (codes are at most 15), so it rounds to the same
// integer unless it lies within 4e-6 of a half-integer.  Adding 1.5 * 2^23 rounds p to an integer, to nearest even, in
// the low bits of the sum; `off` collects the largest distance from p to its integer (NaN if any is: an element that is NaN or
// infinite, or a scale without a reciprocal), and the caller settles a batch of codes one by one when it comes that close
// to one half.  With bf16 data that is mostly an exact tie, x - z = (c + 1/2) s
// (about one code in a thousand, so every third batch of a warp): settled by one FMA, which is zero exactly then; only
// what is left takes the division (all of them dividing: 44 us for the keys of 992 windows, 34 us so).
constexpr float kMagic = 12582912.0f, kHalfMargin = 0.5f - 4e-6f;
__device__ __forceinline__ float max_or_nan(float a, float b) {
  float y;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
  return y;
}
__device__ __forceinline__ bool settled(float off) { return off <= kHalfMargin; }      // (not for a NaN)
__device__ __forceinline__ uint32_t code_bits(float x, float z, float r, float& off) {
  const float t = __fsub_rn(x, z);
  const float m = __fmaf_rn(t, r, kMagic);
  off = max_or_nan(off, fabsf(__fmaf_rn(t, r, -__fsub_rn(m, kMagic))));
  return __float_as_uint(m);            // the code in the low four bits
}
// a code that came close to one half, or whose product is NaN
__device__ __noinline__ uint32_t close_code(float x, float z, float r, float s, int max_code) {
  const float t = __fsub_rn(x, z);
  const float c = __fsub_rn(__fmaf_rn(t, r, kMagic), kMagic), d = __fmaf_rn(t, r, -c);
  const int ci = (int)c;
  if (__fmaf_rn(c + copysignf(0.5f, d), s, -t) == 0.0f) return (uint32_t)((ci & 1) ? (d > 0.f ? ci + 1 : ci - 1) : ci);   // a tie: the even code
  return (uint32_t)quant_code(x, z, s, max_code);
}
// one code by itself, settled
__device__ __forceinline__ uint32_t settle_code(float x, float z, float r, float s, int max_code) {
  float off = 0.f;
  const uint32_t c = code_bits(x, z, r, off) & 15u;
  return settled(off) ? c : close_code(x, z, r, s, max_code);
}
// stored metadata word {s, z} -> {r, z}
__device__ __forceinline__ float2 code_params(uint32_t meta) { return make_float2(code_reciprocal(lo_f(meta)), hi_f(meta)); }

__host__ __device__ inline int key_rows_bytes(int R) { return R * kKeyRow * 4; }
__host__ __device__ inline int key_smem_bytes(int R, int NG) {
  return key_rows_bytes(R) + (R / 32) * 64 * 8 + NG * 128 * 8 + NG * 128 * 4 + 3 * 128 + 64 + 1024;
}
__host__ __device__ inline int value_smem_bytes(int R, int VG, int v_bits) {
  return R * kValRow * 4 + R * VG * 8 + R * VG * 4 + (R / 32) * 1024 * (v_bits == 4 ? 2 : 1);
}
__host__ __device__ inline int tiers_smem_bytes() { return kAbsSumSmem > 2 * 8 * 64 * 4 ? kAbsSumSmem + 1024 : 2 * 8 * 64 * 4 + 1024; }

// tier of channel d from its salience inputs; threads 0..127 call it with their channel, all 256 reach the barriers
__device__ inline uint8_t window_tier(const LayerView& lv, int d, bool active, double acc, uint32_t cnt, float mx, float mn,
                                      double* aS) {
  uint8_t tier = kU2;
  if (active) {
    double A;
    tier = salience_tier(acc, cnt, mx, mn, lv.score_bits, lv.tau_bf16, lv.tau_u4, &A, lv.importance_mode == 2);
    aS[d] = A;
  }
  if (lv.budget_bf16 + lv.budget_u4 > 0) {     // fixed budget: the rank among the window's saliences decides
    __syncthreads();
    if (active) tier = budget_tier(aS, d, lv.budget_bf16, lv.budget_u4);
  }
  return tier;
}

// ================================================================================================ tiers role
// One window of a bulk append.  Its 128 tiers go to the first bytes of the block (rewritten by the keys role), the counts
// to the table entry.  The CTA that finishes a stream's last window gives the stream's new blocks their places in the
// arena, in order.  A block that does not fit gets nothing there and a table entry without promoted channels, and the
// status word says so: the same rule as for a single flush.
__device__ inline void tiers_role(const LayerView& lv, const BulkSrc& src, unsigned char* smem, int s, int w) {
  const int tid = threadIdx.x, R = lv.R, g = lv.g;
  char* blk = lv.base + (size_t)s * lv.base_stride + (size_t)(lv.n_blocks + w) * lv.base_bytes;
  char* state = lv.state + (size_t)s * lv.state_stride;
  double* aS = reinterpret_cast<double*>(smem + tiers_smem_bytes() - 1024);
  __shared__ int cntS[8];
  __shared__ int lastS;
  // ---- importance of the window
  double acc = 0.0;
  uint32_t cnt = (uint32_t)(R * g);
  if (lv.importance_mode == 1) {
    // cumulative: left here by the launch before
    if (tid < kD) acc = reinterpret_cast<const double*>(blk + kSnapshotOff)[tid];
    cnt = *reinterpret_cast<const uint32_t*>(blk + kSnapshotCntOff);
  } else if (lv.importance_mode == 0) {
    const int b = s / lv.Hkv, hk = s % lv.Hkv;
    const uint16_t* qw = src.q + (((size_t)b * lv.Hq + hk * g) * src.n_tokens + src.t0 + (size_t)w * R) * kD;
    int unit;
    acc = abs_sum_256(qw, (size_t)src.n_tokens * kD, R, g, 0.0, smem, &unit);
    __syncthreads();
  }
  // ---- key extrema
  uint32_t* mxS = reinterpret_cast<uint32_t*>(smem);        // [8 warps][64] channel pairs
  uint32_t* mnS = mxS + 8 * 64;
  {
    const int c = tid & 15, rg = tid >> 4;
    const uint4* kw = reinterpret_cast<const uint4*>(src.k + ((size_t)s * src.n_tokens + src.t0 + (size_t)w * R) * kD);
    uint32_t mx[4], mn[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      mx[i] = kNegInf2;
      mn[i] = kPosInf2;
    }
    for (int j = rg; j < R; j += 16 * 8) {
      uint4 x[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = kw[(j + 16 * k < R ? j + 16 * k : j) * 16 + c];     // (a repeated row changes nothing)
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const uint32_t v[4] = {x[k].x, x[k].y, x[k].z, x[k].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          mx[i] = max_bf162(mx[i], v[i]);
          mn[i] = min_bf162(mn[i], v[i]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      mx[i] = max_bf162(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], 16));
      mn[i] = min_bf162(mn[i], __shfl_xor_sync(0xffffffffu, mn[i], 16));
    }
    if ((tid & 31) < 16) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        mxS[(tid >> 5) * 64 + 4 * c + i] = mx[i];
        mnS[(tid >> 5) * 64 + 4 * c + i] = mn[i];
      }
    }
  }
  __syncthreads();
  float wmx = 0.f, wmn = 0.f;
  if (tid < kD) {
    uint32_t mx = mxS[tid >> 1], mn = mnS[tid >> 1];
#pragma unroll
    for (int i = 1; i < 8; ++i) {
      mx = max_bf162(mx, mxS[i * 64 + (tid >> 1)]);
      mn = min_bf162(mn, mnS[i * 64 + (tid >> 1)]);
    }
    wmx = (tid & 1) ? hi_f(mx) : lo_f(mx);
    wmn = (tid & 1) ? hi_f(mn) : lo_f(mn);
  }
  const uint8_t tier = window_tier(lv, tid, tid < kD, acc, cnt, wmx, wmn, aS);
  if (tid < kD) {
    const unsigned m16 = __ballot_sync(0xffffffffu, tier == kBF16), m4 = __ballot_sync(0xffffffffu, tier == kU4);
    if ((tid & 31) == 0) {
      cntS[tid >> 5] = __popc(m16);
      cntS[4 + (tid >> 5)] = __popc(m4);
    }
    reinterpret_cast<uint8_t*>(blk)[tid] = tier;
  }
  __syncthreads();
  uint2* table = reinterpret_cast<uint2*>(lv.table + (size_t)s * lv.table_stride) + lv.n_blocks;
  uint32_t* done = reinterpret_cast<uint32_t*>(state + kDoneOff);
  if (tid == 0) {
    table[w] = make_uint2(0u, (uint32_t)(cntS[0] + cntS[1] + cntS[2] + cntS[3]) |
                                  ((uint32_t)(cntS[4] + cntS[5] + cntS[6] + cntS[7]) << 8));
    __threadfence();
    lastS = atomicAdd(done, 1u) == (uint32_t)(src.nb - 1) ? 1 : 0;
  }
  __syncthreads();
  if (!lastS) return;
  // ---- the stream's last window: places in the arena
  __threadfence();
  uint32_t* used = reinterpret_cast<uint32_t*>(state + 1028);
  uint32_t* sumS = reinterpret_cast<uint32_t*>(smem);               // [8] warp totals
  const uint32_t used0 = *used;
  auto need16 = [&](uint2 e) { return flush_extras_bytes(lv, e.y & 0xFF, (e.y >> 8) & 0xFF) / 16; };
  unsigned long long total = used0;
  for (int pass = 0; pass < 2; ++pass) {
    // pass 0: does everything fit?  pass 1 (only then): offsets by a running prefix sum
    uint32_t run = used0;
    for (int i0 = 0; i0 < src.nb; i0 += 256) {
      const int i = i0 + tid;
      uint2 e = make_uint2(0u, 0u);
      uint32_t x = 0;
      if (i < src.nb) {
        e = __ldcg(&table[i]);
        x = need16(e);
      }
      uint32_t inc = x;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, off);
        if ((tid & 31) >= off) inc += y;
      }
      __syncthreads();
      if ((tid & 31) == 31) sumS[tid >> 5] = inc;
      __syncthreads();
      uint32_t before = run, all = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (k < (tid >> 5)) before += sumS[k];
        all += sumS[k];
      }
      if (pass == 1 && i < src.nb) {
        e.x = before + inc - x;
        table[i] = e;
      }
      run += all;
      if (pass == 0) total += all;
    }
    if (pass == 0 && total * 16 > lv.extras_budget) break;
    if (pass == 1 && tid == 0) *used = run;
  }
  if (tid == 0) {
    if (total * 16 > lv.extras_budget) {
      // not everything fits: block by block, those that fit are placed
      uint32_t off16 = used0;
      for (int i = 0; i < src.nb; ++i) {
        uint2 e = __ldcg(&table[i]);
        const uint32_t x = need16(e);
        e.x = off16;
        if ((uint64_t)(off16 + (uint64_t)x) * 16 > lv.extras_budget) {
          atomicOr(lv.status, (uint32_t)MIXKVQ_DEV_EXTRAS_FULL);
          e.y = 0u;
        } else {
          off16 += x;
        }
        table[i] = e;
      }
      *used = off16;
    }
    *done = 0u;
  }
}

// ================================================================================================ keys role
// One window: `rows` its R rows of 256 bytes.  bulk: the tiers role has been here; otherwise the tiers and the place in
// the arena are found here.
template <int G, bool kTile>
__device__ inline void keys_role(const LayerView& lv, unsigned char* smem, const uint4* __restrict__ rows, int s, int block_index,
                                 bool bulk) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int R = lv.R, U = lv.U, NG = lv.NG;
  constexpr int UPG = G / 32;
  uint32_t* kS = reinterpret_cast<uint32_t*>(smem);                                   // [R][kKeyRow] channel pairs
  uint2* mmS = reinterpret_cast<uint2*>(smem + key_rows_bytes(R));                    // [U][64] {max, min} per channel pair
  float2* prmS = reinterpret_cast<float2*>(reinterpret_cast<unsigned char*>(mmS) + U * 64 * 8);    // [NG][128] {1 / s, z}
  uint32_t* metaS = reinterpret_cast<uint32_t*>(prmS + NG * kD);                      // [NG][128] stored {s, z}
  double* aS = reinterpret_cast<double*>(metaS + NG * kD);                            // [128]
  uint8_t* tierS = reinterpret_cast<uint8_t*>(aS + kD);                               // [128]
  uint8_t* chan16S = tierS + kD;                                                      // [128]
  uint8_t* chan4S = chan16S + kD;                                                     // [128]
  int* cntS = reinterpret_cast<int*>(chan4S + kD);                                    // [8], then n16, n4, place, whether it has one
  auto key_at = [&](int j, int d) { return reinterpret_cast<const uint16_t*>(kS + j * kKeyRow)[d]; };

  char* state = lv.state + (size_t)s * lv.state_stride;
  char* blk = lv.base + (size_t)s * lv.base_stride + (size_t)block_index * lv.base_bytes;
  uint2* table_entry = reinterpret_cast<uint2*>(lv.table + (size_t)s * lv.table_stride) + block_index;

  for (int i0 = 0; i0 < R * 16; i0 += 8 * 256) {
    uint4 x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (i0 + tid + 256 * k < R * 16) x[k] = rows[i0 + tid + 256 * k];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = i0 + tid + 256 * k;
      if (i < R * 16) *reinterpret_cast<uint4*>(kS + (i >> 4) * kKeyRow + 4 * (i & 15)) = x[k];
    }
  }
  uint8_t tier = kU2;
  if (bulk && tid < kD) tier = reinterpret_cast<const uint8_t*>(blk)[tid];            // before anything is written there
  double acc = 0.0;
  uint32_t cnt = 1;
  if (!bulk) {
    if (tid < kD) acc = reinterpret_cast<const double*>(state)[tid];
    cnt = *reinterpret_cast<const uint32_t*>(state + 1024);
  }
  __syncthreads();

  // ---- extrema of every 32-token unit
  {
    const int w = tid & 63;
    for (int u = tid >> 6; u < U; u += 4) {
      uint32_t mx = kNegInf2, mn = kPosInf2;
#pragma unroll 8
      for (int j = 0; j < 32; ++j) {
        const uint32_t x = kS[(32 * u + j) * kKeyRow + w];
        mx = max_bf162(mx, x);
        mn = min_bf162(mn, x);
      }
      mmS[u * 64 + w] = make_uint2(mx, mn);
    }
  }
  __syncthreads();
  // ---- tiers
  if (!bulk) {
    float wmx = 0.f, wmn = 0.f;
    if (tid < kD) {
      uint32_t mx = kNegInf2, mn = kPosInf2;
      for (int u = 0; u < U; ++u) {
        const uint2 m = mmS[u * 64 + (tid >> 1)];
        mx = max_bf162(mx, m.x);
        mn = min_bf162(mn, m.y);
      }
      wmx = (tid & 1) ? hi_f(mx) : lo_f(mx);
      wmn = (tid & 1) ? hi_f(mn) : lo_f(mn);
    }
    tier = window_tier(lv, tid, tid < kD, acc, cnt, wmx, wmn, aS);
  }
  unsigned m16 = 0, m4 = 0;
  if (tid < kD) {
    tierS[tid] = tier;
    m16 = __ballot_sync(0xffffffffu, tier == kBF16);
    m4 = __ballot_sync(0xffffffffu, tier == kU4);
    if (lane == 0) {
      cntS[warp] = __popc(m16);
      cntS[4 + warp] = __popc(m4);
    }
  }
  __syncthreads();
  // ---- channel lists (ascending channel order inside each tier), place in the arena, scales
  if (tid < kD) {
    int b16 = 0, b4 = 0;
    for (int w2 = 0; w2 < warp; ++w2) {
      b16 += cntS[w2];
      b4 += cntS[4 + w2];
    }
    const unsigned below = (1u << lane) - 1u;
    if (m16 & (1u << lane)) chan16S[b16 + __popc(m16 & below)] = (uint8_t)tid;
    if (m4 & (1u << lane)) chan4S[b4 + __popc(m4 & below)] = (uint8_t)tid;
  } else if (tid == kD) {
    int n16 = cntS[0] + cntS[1] + cntS[2] + cntS[3], n4 = cntS[4] + cntS[5] + cntS[6] + cntS[7];
    const uint32_t need = flush_extras_bytes(lv, n16, n4);
    uint32_t off16 = 0;
    bool placed = true;
    if (bulk) {
      // the tiers role placed the block (and cleared the counts if the arena was full)
      off16 = table_entry->x;
      placed = (uint64_t)off16 * 16 + need <= lv.extras_budget;
      if (!placed) n16 = n4 = 0;
    } else {
      uint32_t* used = reinterpret_cast<uint32_t*>(state + 1028);
      off16 = *used;
      if ((uint64_t)off16 * 16 + need > lv.extras_budget) {
        atomicOr(lv.status, (uint32_t)MIXKVQ_DEV_EXTRAS_FULL);
        placed = false;
        n16 = n4 = 0;      // nothing goes to the arena and the entry records no promoted channel; the status word says so
      } else {
        *used = off16 + need / 16;
      }
      *table_entry = make_uint2(off16, (uint32_t)n16 | ((uint32_t)n4 << 8));
    }
    cntS[8] = n16;
    cntS[9] = n4;
    cntS[10] = (int)off16;
    cntS[11] = placed ? 1 : 0;
  }
  for (int i = tid; i < NG * kD; i += 256) {
    const int kg = i >> 7, d = i & 127;
    uint32_t meta = 0;
    if (tierS[d] != kBF16) {
      uint32_t mx = kNegInf2, mn = kPosInf2;
#pragma unroll
      for (int k = 0; k < UPG; ++k) {
        const uint2 m = mmS[(kg * UPG + k) * 64 + (d >> 1)];
        mx = max_bf162(mx, m.x);
        mn = min_bf162(mn, m.y);
      }
      const float gmx = (d & 1) ? hi_f(mx) : lo_f(mx), gmn = (d & 1) ? hi_f(mn) : lo_f(mn);
      const float sc = stored_scale(gmx, gmn, tierS[d] == kU4 ? 15.0f : 3.0f);
      meta = float_to_bf16_bits_exact(sc) | (float_to_bf16_bits_exact(gmn) << 16);
    }
    prmS[i] = code_params(meta);             // promoted channels: every code 0
    metaS[i] = meta;
    reinterpret_cast<uint32_t*>(blk + (kTile ? (uint32_t)kg * 512u : frag_meta_off(kg, G, lv.unit_bytes)))[d] = meta;
  }
  __syncthreads();

  const int n16 = cntS[8], n4 = cntS[9], n16p = (n16 + 1) >> 1, n4p = ((n4 + 1) >> 1) << 1;
  char* ex = lv.extras + (size_t)s * lv.extras_stride + (size_t)cntS[10] * 16;
  const uint32_t hdr = extras_header_bytes(n16, n4), exunit = extras_unit_bytes(n16, n4, lv.dense_hi != 0);
  // one code by itself (for the gathered high plane)
  auto code_of = [&](int j, int d) {
    const int i = (j / G) * kD + d;
    const float2 p = prmS[i];
    return settle_code(__uint_as_float((uint32_t)key_at(j, d) << 16), p.y, p.x, lo_f(metaS[i]), tierS[d] == kU4 ? 15 : 3);
  };
  const bool dense = !kTile && lv.dense_hi && n4 > 0;

  if constexpr (kTile) {
    // ---- low plane: a token's key codes are 32 contiguous bytes (two 16-byte halves)
    for (int i = tid; i < 2 * 128; i += 256) {
      const int j = i & 127, hh = i >> 7;
      uint32_t w[4] = {0u, 0u, 0u, 0u};
      const float4* prm4 = reinterpret_cast<const float4*>(prmS + (j / G) * kD + 64 * hh);
#pragma unroll
      for (int wi = 0; wi < 4; ++wi) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const uint4 x = *reinterpret_cast<const uint4*>(kS + j * kKeyRow + 32 * hh + 8 * wi + 4 * half);
          const uint32_t xx[4] = {x.x, x.y, x.z, x.w};
          uint32_t part = 0;
          float off = 0.f;
#pragma unroll
          for (int f = 0; f < 4; ++f) {
            const float4 p = prm4[8 * wi + 4 * half + f];
            part |= (code_bits(lo_f(xx[f]), p.y, p.x, off) & 3u) << (2 * (4 * half + f));
            part |= (code_bits(hi_f(xx[f]), p.w, p.z, off) & 3u) << (16 + 2 * (4 * half + f));
          }
          if (!settled(off)) {
            part = 0;
            for (int f = 0; f < 4; ++f)
              for (int e = 0; e < 2; ++e)
                part |= (code_of(j, 64 * hh + 16 * wi + 8 * half + 2 * f + e) & 3u) << (16 * e + 2 * (4 * half + f));
          }
          w[wi] |= part;
        }
      }
      *reinterpret_cast<uint4*>(blk + NG * 512 + hh * 2048 + j * 16) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    const int n4w = (n4 + 15) >> 4;
    const uint32_t thdr = tile_extras_header_bytes(n16, n4);
    for (int i = tid; i < (int)thdr; i += 256) {
      uint8_t b = 0;
      if (i < 2 * n16p) b = (i < n16) ? chan16S[i] : 0xFF;
      else if (i < 2 * n16p + 16 * n4w) b = (i - 2 * n16p < n4) ? chan4S[i - 2 * n16p] : 0xFF;
      ex[i] = (char)b;
    }
    uint32_t* xw = reinterpret_cast<uint32_t*>(ex + thdr);
    for (int i = tid; i < n16p * 128; i += 256) {
      const int p = i >> 7, j = i & 127;
      uint32_t w = key_at(j, chan16S[2 * p]);
      if (2 * p + 1 < n16) w |= (uint32_t)key_at(j, chan16S[2 * p + 1]) << 16;
      xw[i] = w;
    }
    for (int i = tid; i < n4w * 128; i += 256) {
      const int wq = i >> 7, j = i & 127;
      uint32_t w = 0;
      for (int k = 0; k < 16 && 16 * wq + k < n4; ++k) w |= (code_of(j, chan4S[16 * wq + k]) >> 2) << (16 * (k & 1) + 2 * (k >> 1));
      xw[n16p * 128 + i] = w;
    }
  } else {
    // ---- low plane (and, with a 4-bit base, the dense high plane), fragment order: a thread makes the four words of a
    // 16-byte piece: tokens r and r + 8 of an m-tile, channels 16 kt + {0, 8} + 2t + {0, 1} of all eight k-tiles
    for (int i = tid; i < U * 64; i += 256) {
      const int u = i >> 6, mt = (i >> 5) & 1, r = lane >> 2, t = lane & 3;
      const int ja = 32 * u + 16 * mt + r;
      const float4* prm4 = reinterpret_cast<const float4*>(prmS + ((32 * u) / G) * kD) + t;
      const uint32_t* rowa = kS + ja * kKeyRow + t;
      uint32_t lo[4] = {0u, 0u, 0u, 0u}, hi[4] = {0u, 0u, 0u, 0u};        // [2 ch + rh]
#pragma unroll 2
      for (int kt = 0; kt < 8; ++kt) {
        uint32_t c[2][2][2];                  // [ch][rh][e]
        float off = 0.f;
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          const float4 p = prm4[8 * kt + 4 * ch];
#pragma unroll
          for (int rh = 0; rh < 2; ++rh) {
            const uint32_t x = rowa[8 * rh * kKeyRow + 8 * kt + 4 * ch];
            c[ch][rh][0] = code_bits(lo_f(x), p.y, p.x, off);
            c[ch][rh][1] = code_bits(hi_f(x), p.w, p.z, off);
          }
        }
        if (!settled(off)) {
#pragma unroll
          for (int ch = 0; ch < 2; ++ch) {
            const float4 p = prm4[8 * kt + 4 * ch];
            const int d = 16 * kt + 8 * ch + 2 * t;
            const float s0 = lo_f(metaS[((32 * u) / G) * kD + d]), s1 = lo_f(metaS[((32 * u) / G) * kD + d + 1]);
#pragma unroll
            for (int rh = 0; rh < 2; ++rh) {
              const uint32_t x = rowa[8 * rh * kKeyRow + 8 * kt + 4 * ch];
              c[ch][rh][0] = settle_code(lo_f(x), p.y, p.x, s0, tierS[d] == kU4 ? 15 : 3);
              c[ch][rh][1] = settle_code(hi_f(x), p.w, p.z, s1, tierS[d + 1] == kU4 ? 15 : 3);
            }
          }
        }
#pragma unroll
        for (int ch = 0; ch < 2; ++ch)
#pragma unroll
          for (int rh = 0; rh < 2; ++rh) {
            lo[2 * ch + rh] |= ((c[ch][rh][0] & 3u) << (2 * kt)) | ((c[ch][rh][1] & 3u) << (16 + 2 * kt));
            if (dense) hi[2 * ch + rh] |= (((c[ch][rh][0] >> 2) & 3u) << (2 * kt)) | (((c[ch][rh][1] >> 2) & 3u) << (16 + 2 * kt));
          }
      }
      reinterpret_cast<uint4*>(blk + frag_unit_off(u, G, lv.unit_bytes))[32 * mt + lane] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      if (dense)
        reinterpret_cast<uint4*>(ex + hdr + (size_t)u * exunit + 128 * n16p)[32 * mt + lane] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    }
    // ---- extras: header, BF16 pairs, UINT4 high plane
    for (int i = tid; i < (int)hdr; i += 256) {
      uint8_t b = 0;
      if (i < 2 * n16p) b = (i < n16) ? chan16S[i] : 0xFF;
      else if (i < 2 * n16p + n4p) b = (i - 2 * n16p < n4) ? chan4S[i - 2 * n16p] : 0xFF;
      ex[i] = (char)b;
    }
    for (int i = tid; i < R * n16p; i += 256) {
      const int p = i / R, j = i - p * R;
      uint32_t w = key_at(j, chan16S[2 * p]);
      if (2 * p + 1 < n16) w |= (uint32_t)key_at(j, chan16S[2 * p + 1]) << 16;
      reinterpret_cast<uint32_t*>(ex + hdr + (size_t)(j >> 5) * exunit)[32 * p + (j & 31)] = w;
    }
    if (!lv.dense_hi) {
      for (int i = tid; i < U * n4p * 2; i += 256) {
        const int u = i / (n4p * 2), rem = i - u * (n4p * 2), p = rem >> 2, wj = rem & 3;
        uint32_t w = 0;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (2 * p + e >= n4) continue;
          const int d = chan4S[2 * p + e];
#pragma unroll
          for (int rhi = 0; rhi < 2; ++rhi)
#pragma unroll
            for (int m = 0; m < 4; ++m)        // m = 2 mt + rh
              w |= (code_of(32 * u + 8 * m + wj + 4 * rhi, d) >> 2) << (16 * e + 8 * rhi + 2 * m);
        }
        reinterpret_cast<uint32_t*>(ex + hdr + (size_t)u * exunit + 128 * n16p)[rem] = w;
      }
    } else if (n4 == 0 && cntS[11]) {
      // 4-bit base, no channel in UINT4 (all promoted, or saliences that are NaN): the dense plane exists and is zero
      for (int i = tid; i < U * 64; i += 256)
        reinterpret_cast<uint4*>(ex + hdr + (size_t)(i >> 6) * exunit + 128 * n16p)[i & 63] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  // ---- window importance: the accumulator restarts with the next window (Section 4.2)
  if (!bulk && lv.importance_mode != 1) {
    if (tid < kD) reinterpret_cast<double*>(state)[tid] = 0.0;
    if (tid == 0) *reinterpret_cast<uint32_t*>(state + 1024) = 0u;
  }
}

// ================================================================================================ values role
template <int G, bool kTile>
__device__ inline void values_role(const LayerView& lv, unsigned char* smem, const uint4* __restrict__ rows, int s,
                                   int block_index) {
  constexpr int VG = kD / G;
  const int tid = threadIdx.x, R = lv.R, U = lv.U, NG = lv.NG;
  const bool v4 = lv.v_bits == 4;
  uint32_t* vS = reinterpret_cast<uint32_t*>(smem);                            // [R][kValRow] channel pairs
  float2* prmS = reinterpret_cast<float2*>(smem + R * kValRow * 4);            // [R][VG] {1 / s, z}
  uint32_t* metaS = reinterpret_cast<uint32_t*>(prmS + R * VG);                // [R][VG] stored {s, z}
  uint32_t* packS = metaS + R * VG;                                            // [U][256] packed words, then the high plane's
  char* blk = lv.base + (size_t)s * lv.base_stride + (size_t)block_index * lv.base_bytes;

  // ---- load; extrema of a token's group of G channels: G / 8 neighbouring threads of the 16 that hold a row
  for (int i0 = 0; i0 < R * 16; i0 += 8 * 256) {
    uint4 x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      x[k] = make_uint4(0u, 0u, 0u, 0u);
      if (i0 + tid + 256 * k < R * 16) x[k] = rows[i0 + tid + 256 * k];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = i0 + tid + 256 * k, j = i >> 4, c = i & 15;
      uint32_t mx = max_bf162(max_bf162(x[k].x, x[k].y), max_bf162(x[k].z, x[k].w));
      uint32_t mn = min_bf162(min_bf162(x[k].x, x[k].y), min_bf162(x[k].z, x[k].w));
#pragma unroll
      for (int off = 1; off < G / 8; off <<= 1) {
        mx = max_bf162(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        mn = min_bf162(mn, __shfl_xor_sync(0xffffffffu, mn, off));
      }
      if (i < R * 16) {
        uint2* dst = reinterpret_cast<uint2*>(vS + j * kValRow + 4 * c);
        dst[0] = make_uint2(x[k].x, x[k].y);
        dst[1] = make_uint2(x[k].z, x[k].w);
        if ((c & (G / 8 - 1)) == 0)          // {max, min}, for now
          metaS[j * VG + c / (G / 8)] = float_to_bf16_bits_exact(fmaxf(lo_f(mx), hi_f(mx))) |
                                        (float_to_bf16_bits_exact(fminf(lo_f(mn), hi_f(mn))) << 16);
      }
    }
  }
  __syncthreads();
  // ---- scales
  for (int i = tid; i < R * VG; i += 256) {
    const uint32_t ext = metaS[i];                       // {max, min}
    const float gmx = lo_f(ext), gmn = hi_f(ext);
    const float sc = stored_scale(gmx, gmn, v4 ? 15.0f : 3.0f);
    const uint32_t meta = float_to_bf16_bits_exact(sc) | (float_to_bf16_bits_exact(gmn) << 16);
    prmS[i] = code_params(meta);
    metaS[i] = meta;
    const int j = i / VG, vg = i - j * VG;
    uint32_t* dst = kTile ? reinterpret_cast<uint32_t*>(blk + NG * 512 + 8192) + i
                          : reinterpret_cast<uint32_t*>(blk + frag_unit_off(j >> 5, G, lv.unit_bytes) + 2048) + (j & 31) * VG + vg;
    *dst = meta;
  }
  __syncthreads();
  const int max_code = v4 ? 15 : 3;
  auto code_of = [&](int j, int c) {
    const int i = j * VG + c / G;
    const float2 p = prmS[i];
    return settle_code(__uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(vS + j * kValRow)[c] << 16), p.y, p.x,
                       lo_f(metaS[i]), max_code);
  };
  if constexpr (kTile) {
    // ---- a channel's value codes over the 128 tokens are 32 contiguous bytes: a thread makes the words of two channels
    // over 16 tokens
    for (int i = tid; i < 8 * 64; i += 256) {
      const int W = i >> 6, cp = i & 63;
      uint32_t w[2] = {0u, 0u};
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        float off = 0.f;
        uint32_t part[2] = {0u, 0u};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int j = 16 * W + 8 * half + k, bit = 16 * (k & 1) + 2 * (4 * half + (k >> 1));
          const float2 p = prmS[j * VG + (2 * cp) / G];
          const uint32_t x = vS[j * kValRow + cp];
          part[0] |= (code_bits(lo_f(x), p.y, p.x, off) & 3u) << bit;
          part[1] |= (code_bits(hi_f(x), p.y, p.x, off) & 3u) << bit;
        }
        if (!settled(off)) {
          part[0] = part[1] = 0;
          for (int k = 0; k < 8; ++k)
            for (int e = 0; e < 2; ++e)
              part[e] |= (code_of(16 * W + 8 * half + k, 2 * cp + e) & 3u) << (16 * (k & 1) + 2 * (4 * half + (k >> 1)));
        }
        w[0] |= part[0];
        w[1] |= part[1];
      }
#pragma unroll
      for (int e = 0; e < 2; ++e)
        *reinterpret_cast<uint32_t*>(blk + NG * 512 + 4096 + (W >> 2) * 2048 + (2 * cp + e) * 16 + (W & 3) * 4) = w[e];
    }
  } else {
    // ---- fragment order: a thread makes the words of channel tile ct, rows r = 2rp and 2rp + 1 (two channels each, 8
    // apart), lane column t (eight tokens).  The lanes of a warp take t, rp and two tiles 2 apart: all 32 banks.
    for (int i = tid; i < U * 128; i += 256) {
      const int t = i & 3, rp = (i >> 2) & 3, ct = 2 * ((i >> 4) & 1) + ((i >> 5) & 1) + 4 * ((i >> 6) & 1), u = i >> 7;
      const int vg = (16 * ct) / G;
      uint32_t lo[2] = {0u, 0u}, hi[2] = {0u, 0u};
#pragma unroll
      for (int ks = 0; ks < 2; ++ks)
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          uint32_t c[2][2][2];               // [e][rh][row]
          float off = 0.f;
          const int j = 32 * u + 16 * ks + 8 * ch + 2 * t;
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float2 p = prmS[(j + e) * VG + vg];
#pragma unroll
            for (int rh = 0; rh < 2; ++rh) {
              const uint32_t x = vS[(j + e) * kValRow + 8 * ct + 4 * rh + rp];
              c[e][rh][0] = code_bits(lo_f(x), p.y, p.x, off);
              c[e][rh][1] = code_bits(hi_f(x), p.y, p.x, off);
            }
          }
          if (!settled(off)) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float2 p = prmS[(j + e) * VG + vg];
              const float sc = lo_f(metaS[(j + e) * VG + vg]);
#pragma unroll
              for (int rh = 0; rh < 2; ++rh) {
                const uint32_t x = vS[(j + e) * kValRow + 8 * ct + 4 * rh + rp];
                c[e][rh][0] = settle_code(lo_f(x), p.y, p.x, sc, max_code);
                c[e][rh][1] = settle_code(hi_f(x), p.y, p.x, sc, max_code);
              }
            }
          }
#pragma unroll
          for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int rh = 0; rh < 2; ++rh)
#pragma unroll
              for (int b = 0; b < 2; ++b) {
                const int bit = 16 * e + 2 * (4 * rh + 2 * ks + ch);
                lo[b] |= (c[e][rh][b] & 3u) << bit;
                if (v4) hi[b] |= ((c[e][rh][b] >> 2) & 3u) << bit;
              }
        }
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int wi = (ct >> 2) * 128 + (4 * (2 * rp + b) + t) * 4 + (ct & 3);
        packS[u * 256 + wi] = lo[b];
        if (v4) packS[(U + u) * 256 + wi] = hi[b];
      }
    }
    __syncthreads();
    for (int i = tid; i < U * 64; i += 256) {
      const int u = i >> 6;
      char* dst = blk + frag_unit_off(u, G, lv.unit_bytes);
      reinterpret_cast<uint4*>(dst + 1024)[i & 63] = reinterpret_cast<const uint4*>(packS)[i];
      // 4-bit values: the high plane in the same bit order, after the unit's value scales
      if (v4) reinterpret_cast<uint4*>(dst + 2048 + 128 * VG)[i & 63] = reinterpret_cast<const uint4*>(packS)[U * 64 + i];
    }
  }
}

// ================================================================================================ kernels
// Flush of the residual window: blockIdx.y 0 = keys, 1 = values.
template <int G, bool kTile>
__global__ void __launch_bounds__(256, 2) flush_kernel(LayerView lv) {
  extern __shared__ __align__(16) unsigned char smem[];
  dependency_wait();
  const int s = blockIdx.x;
  int block_index = lv.n_blocks;
  if (lv.seq != nullptr) {
    // ragged batch: the sequences whose window is full take part, each with its own block count
    const int4 f = lv.seq[s / lv.Hkv];
    if (f.y != lv.R) return;
    block_index = f.x;
  }
  if (blockIdx.y == 0)
    keys_role<G, kTile>(lv, smem, reinterpret_cast<const uint4*>(lv.resk + (size_t)s * lv.resk_stride), s, block_index, false);
  else
    values_role<G, kTile>(lv, smem, reinterpret_cast<const uint4*>(lv.resv + (size_t)s * lv.resv_stride), s, block_index);
}

// Bulk append, first launch: blockIdx.y = window, blockIdx.z 0 = tiers, 1 = values.
template <int G, bool kTile>
__global__ void __launch_bounds__(256, 4) bulk_tiers_values_kernel(LayerView lv, BulkSrc src) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int s = blockIdx.x, w = blockIdx.y;
  // Behind the prefill attention, which neither writes what is read here nor touches the cache, the work starts as soon as an
  // SM is free of it, and only the end waits.  (With importance mode 1 the kernel before this one is another.)
  const bool early = src.behind_prefill != 0 && lv.importance_mode != 1;
  if (!early) dependency_wait();
  if (blockIdx.z == 0) {
    tiers_role(lv, src, smem, s, w);
  } else {
    const uint16_t* rows = src.v + ((size_t)s * src.n_tokens + src.t0 + (size_t)w * lv.R) * kD;
    values_role<G, kTile>(lv, smem, reinterpret_cast<const uint4*>(rows), s, lv.n_blocks + w);
  }
  if (early) dependency_wait();
}

// Bulk append, second launch: blockIdx.y < nb: keys of that window, blockIdx.y == nb: the stream's tail (if there is one).
template <int G, bool kTile>
__global__ void __launch_bounds__(256, 4) bulk_keys_tail_kernel(LayerView lv, BulkSrc src) {
  extern __shared__ __align__(16) unsigned char smem[];
  dependency_wait();
  const int s = blockIdx.x, w = blockIdx.y;
  if (w < src.nb) {
    const uint16_t* rows = src.k + ((size_t)s * src.n_tokens + src.t0 + (size_t)w * lv.R) * kD;
    keys_role<G, kTile>(lv, smem, reinterpret_cast<const uint4*>(rows), s, lv.n_blocks + w, true);
  } else {
    append_rows(lv, src.k, src.v, src.q, src.n_tokens, src.t0 + src.nb * lv.R, src.tail, 0, s, smem);
  }
}

// Cumulative importance (Appendix D.2) in a bulk append: the running |q| sums continue across the windows.  Each CTA sums
// one window on top of nothing; the last CTA of a stream then runs the sums through the stream's windows in order and
// leaves every window's running sum and count where the tiers role reads them, and the final values in the state.  The
// defined sum is one serial chain; a window's sum may be added as a whole only if no addition of that chain rounds.
// Every window reports the exponent of its smallest magnitude for that check; when it fails, the CTA walks the queries
// in order instead.
__global__ void __launch_bounds__(256, 4) bulk_importance_kernel(LayerView lv, BulkSrc src) {
  __shared__ __align__(16) unsigned char smem[kAbsSumSmem];
  __shared__ int lastS;
  dependency_wait();
  const int s = blockIdx.x, w = blockIdx.y, tid = threadIdx.x, g = lv.g, R = lv.R;
  const int b = s / lv.Hkv, hk = s % lv.Hkv;
  char* state = lv.state + (size_t)s * lv.state_stride;
  const uint16_t* q0 = src.q + (((size_t)b * lv.Hq + hk * g) * src.n_tokens + src.t0) * kD;
  const size_t head_stride = (size_t)src.n_tokens * kD;
  char* blk0 = lv.base + (size_t)s * lv.base_stride + (size_t)lv.n_blocks * lv.base_bytes;
  auto blk = [&](int i) { return blk0 + (size_t)i * lv.base_bytes; };
  int unit;
  const double sum = abs_sum_256(q0 + (size_t)w * R * kD, head_stride, R, g, 0.0, smem, &unit);
  if (tid < kD) reinterpret_cast<double*>(blk(w) + kSnapshotOff)[tid] = sum;
  if (tid == 0) *reinterpret_cast<int*>(blk(w) + kSnapshotCntOff) = unit;
  uint32_t* done = reinterpret_cast<uint32_t*>(state + kDoneOff);
  __threadfence();
  __syncthreads();
  if (tid == 0) lastS = atomicAdd(done, 1u) == (uint32_t)(src.nb - 1) ? 1 : 0;
  __syncthreads();
  if (!lastS) return;
  __threadfence();
  double a = tid < kD ? reinterpret_cast<const double*>(state)[tid] : 0.0;
  const uint32_t cnt0 = *reinterpret_cast<const uint32_t*>(state + 1024);
  int all_unit = 0x7FFFFFFF;
  for (int i = tid; i < src.nb; i += 256) all_unit = min(all_unit, __ldcg(reinterpret_cast<const int*>(blk(i) + kSnapshotCntOff)));
  all_unit = __reduce_min_sync(0xffffffffu, all_unit);
  int* minS = reinterpret_cast<int*>(smem);
  if ((tid & 31) == 0) minS[tid >> 5] = all_unit;
  __syncthreads();
  for (int i = 0; i < 8; ++i) all_unit = min(all_unit, minS[i]);
  double total = a;
  if (tid < kD) {
#pragma unroll 16
    for (int i = 0; i < src.nb; ++i) total = __dadd_rn(total, __ldcg(reinterpret_cast<const double*>(blk(i) + kSnapshotOff) + tid));
  }
  const bool exact = tid >= kD || (all_unit != kAbsSumRounded && sum_is_exact(a, total, all_unit));
  const bool all_exact = __syncthreads_and(exact ? 1 : 0) != 0;
  auto snap = [&](int i) { return reinterpret_cast<double*>(blk(i) + kSnapshotOff) + tid; };
  if (tid < kD) {
    for (int i0 = 0; i0 < src.nb; i0 += 16) {
      double x[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) x[k] = i0 + k < src.nb ? __ldcg(snap(i0 + k)) : 0.0;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int i = i0 + k;
        if (i >= src.nb) break;
        if (all_exact) {
          a = __dadd_rn(a, x[k]);
        } else {
          for (int j = i * R; j < (i + 1) * R; ++j)
            for (int h = 0; h < g; ++h)
              a = __dadd_rn(a, (double)fabsf(bf16_bits_to_float(q0[(size_t)h * head_stride + (size_t)j * kD + tid])));
        }
        *snap(i) = a;
      }
    }
  }
  for (int i = tid; i < src.nb; i += 256) *reinterpret_cast<uint32_t*>(blk(i) + kSnapshotCntOff) = cnt0 + (uint32_t)(i + 1) * (uint32_t)(R * g);
  const uint32_t cnt = cnt0 + (uint32_t)src.nb * (uint32_t)(R * g);
  if (tid < kD) reinterpret_cast<double*>(state)[tid] = a;
  if (tid == 0) {
    *reinterpret_cast<uint32_t*>(state + 1024) = cnt;
    *done = 0u;
  }
}

inline int key_smem(const LayerView& lv) {
  const int a = key_smem_bytes(lv.R, lv.NG);
  return a > kAbsSumSmem ? a : kAbsSumSmem;
}
inline int value_smem(const LayerView& lv) { return value_smem_bytes(lv.R, lv.VG, lv.v_bits); }

template <typename K>
cudaError_t allow_smem(K kernel) {
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024);
  if (e != cudaSuccess) return e;
  // four CTAs of 42 KB (R = 128) only fit an SM with the largest shared-memory carve-out
  return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
}
template <int G, bool kTile>
cudaError_t setup_one() {
  cudaError_t e = allow_smem(flush_kernel<G, kTile>);
  if (e == cudaSuccess) e = allow_smem(bulk_tiers_values_kernel<G, kTile>);
  if (e == cudaSuccess) e = allow_smem(bulk_keys_tail_kernel<G, kTile>);
  return e;
}
template <int G, bool kTile>
cudaError_t single(const LayerView& lv, cudaStream_t stream) {
  const int a = key_smem(lv), b = value_smem(lv);
  return launch_dependent(flush_kernel<G, kTile>, dim3(lv.B * lv.Hkv, 2), 256, a > b ? a : b, stream, lv);
}
template <int G, bool kTile>
cudaError_t bulk(const LayerView& lv, const BulkSrc& src, cudaStream_t stream) {
  const int S = lv.B * lv.Hkv, b = value_smem(lv), t = tiers_smem_bytes();
  cudaError_t e = cudaSuccess;
  if (lv.importance_mode == 1) e = launch_dependent(bulk_importance_kernel, dim3(S, src.nb), 256, 0, stream, lv, src);
  if (e == cudaSuccess)
    e = launch_dependent(bulk_tiers_values_kernel<G, kTile>, dim3(S, src.nb, 2), 256, t > b ? t : b, stream, lv, src);
  if (e == cudaSuccess) e = launch_dependent(bulk_keys_tail_kernel<G, kTile>, dim3(S, src.nb + (src.tail > 0 ? 1 : 0)), 256, key_smem(lv), stream, lv, src);
  return e;
}

}  // namespace

cudaError_t flush_setup() {
  cudaError_t e = setup_one<32, false>();
  if (e == cudaSuccess) e = setup_one<64, false>();
  if (e == cudaSuccess) e = setup_one<128, false>();
  if (e == cudaSuccess) e = setup_one<32, true>();
  if (e == cudaSuccess) e = setup_one<64, true>();
  if (e == cudaSuccess) e = setup_one<128, true>();
  return e;
}

cudaError_t launch_flush(const LayerView& lv, cudaStream_t stream) {
  if (lv.tile) return lv.G == 32 ? single<32, true>(lv, stream) : lv.G == 64 ? single<64, true>(lv, stream) : single<128, true>(lv, stream);
  return lv.G == 32 ? single<32, false>(lv, stream) : lv.G == 64 ? single<64, false>(lv, stream) : single<128, false>(lv, stream);
}

// nb complete R-token windows starting at token t0 of the append's tensors go straight to packed blocks, and the `tail`
// (1..R) tokens behind them to the residual window: two launches, three with cumulative importance.  Precondition (checked
// by the caller): empty residual window.
// B200, 31 windows of R = 128 of 32 streams, g = 7 (292 MB read: 45 us at the measured copy rate): 67 + 34 us, against
// 79 + 9 + 79 + 26 us for two passes of one CTA doing everything per window around a serial prefix sum and a separate
// append of the tail.  The first launch is bound by instruction issue (67 % of the slots, the magnitude sums first among
// them) and its loads, the second by its second wave of CTAs (1024 on 592 places).
cudaError_t launch_flush_bulk(const LayerView& lv, const void* k, const void* v, const void* q, int n_tokens, int t0,
                              int nb, int tail, bool behind_prefill, cudaStream_t stream) {
  const BulkSrc src{static_cast<const uint16_t*>(k), static_cast<const uint16_t*>(v), static_cast<const uint16_t*>(q), n_tokens,
                    t0, nb, tail, behind_prefill ? 1 : 0};
  if (lv.tile) return lv.G == 32 ? bulk<32, true>(lv, src, stream) : lv.G == 64 ? bulk<64, true>(lv, src, stream) : bulk<128, true>(lv, src, stream);
  return lv.G == 32 ? bulk<32, false>(lv, src, stream) : lv.G == 64 ? bulk<64, false>(lv, src, stream) : bulk<128, false>(lv, src, stream);
}

}  // namespace mixkvq
