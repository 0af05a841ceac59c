// Log-sum-exp merge of the split partials of decode attention.
#include "common.cuh"

namespace mixkvq {

// Partials live at ws[slot * kPartialFloats + h * 130 + {0: m (log2 domain), 1: l, 2..129: o}].
// mode 0: stream s owns slots [s*n, s*n + n).  mode 1: the attention grid of `n` CTAs split the
// S*units_per_stream work units evenly; CTA c wrote its part of stream s to slot c + s.
//
// One CTA per (stream, head).  What bounds it is latency: a stream has between 1 partial (many streams) and 74 (four
// streams, 296 CTAs), 0.5 KB each.  The warps of the CTA take the partials in turn (warp w: w, w + W, ...), kChunk of
// them in flight per warp, so that up to W * kChunk partials cost one round trip to memory; the warps' results meet in
// shared memory.  B200, attention + merge per layer from a graph: one sequence of 4000 tokens (74 partials) 17.2 us with
// one thread per channel walking chunks of 12, 9.6 us so; 8 sequences of 32768 tokens (9 partials) 41.7 and
// 40.4 us.
// The kernel behind a merge is let go before the merge waits for its split kernel: the next layer's split kernel then takes the places of
// this one's CTAs as they finish, and its set-up and first copies run under their tail (28 layers of the 7b shape, 32768 tokens
// x 8: 1138 -> 1104 us per decode step).  What is still running when that kernel starts are this merge and the split kernel before it, which
// write partials, outputs, residual windows and accumulators, no packed block; its wait covers both, the merge's own included.  Not with
// little work per CTA or one CTA per SM (`early` = false; the rule is at the launch): the next CTAs are then placed around those still
// there, two on some SMs and none on others.
constexpr int kCombineChunk = 8;
constexpr int kCombineMaxWarps = 8;

// A decode step that rotates: the split kernel has rotated as it read; here, behind it, the rows in the caller's tensors are.  One warp's
// part: lanes 0 .. 15 the query row `row`, lanes 16 .. 31 (with the stream's head 0) its new key row.  Requested before the merge
// (rope_load) and stored behind it.
struct RopeRows {
  uint16_t *q, *k;                       // [B Hq][128], [S][128]
  const float *cos_row, *sin_row;
};
struct RopeWork {
  uint4 *at, y;
};
__device__ __forceinline__ RopeWork rope_load(const RopeRows& r, size_t row, int s, int h, int lane) {
  RopeWork w;
  w.at = nullptr;
  if (lane < 16 || h == 0) {
    uint4* base = reinterpret_cast<uint4*>(lane < 16 ? r.q + row * kD : r.k + (size_t)s * kD);
    const int c = lane & 15;
    w.at = base + c;
    w.y = rotate_chunk(base[c], base[c ^ 8], r.cos_row, r.sin_row, c);
  }
  return w;
}
// (the whole warp has loaded before one of its lanes stores)
__device__ __forceinline__ void rope_store(const RopeWork& w) {
  __syncwarp();
  if (w.at != nullptr) *w.at = w.y;
}

// (Rope: nothing, or the RopeRows of a step that rotates: the other merges do not carry its parameters)
template <typename... Rope>
__global__ void __launch_bounds__(kCombineMaxWarps * 32)
combine_kernel(const float* __restrict__ ws, float* __restrict__ out, int g, int Hkv, int Hq, int mode, int n,
               long long units_per_stream, int S, const int4* __restrict__ seq, const int* __restrict__ seq_prefix,
               float* __restrict__ lse_out, bool early, Rope... rope) {
  constexpr bool kRope = sizeof...(Rope) > 0;
  __shared__ float mlS[kCombineMaxWarps][2];
  __shared__ __align__(16) float oS[kCombineMaxWarps][kD];
  if (early) let_successor_start();
  const int s = blockIdx.x / g, h = blockIdx.x % g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5;
  int first, count;
  // started early (programmatic dependent launch): waits for the kernel that wrote the partials once it knows where they are
  // (a ragged batch's table is read for that)
  if (seq != nullptr) dependency_wait();
  if (mode == 0) {
    first = s * n;
    count = n;
  } else if (seq != nullptr) {
    // ragged batch: each of sequence b's streams has (prefix[b + 1] - prefix[b]) / Hkv CTAs of its own (none if it is empty)
    const int bq = s / Hkv, p0 = seq_prefix[bq];
    count = (seq_prefix[bq + 1] - p0) / Hkv;
    first = p0 + (s % Hkv) * count + s;
  } else {
    const long long total = units_per_stream * S;
    const long long x0 = units_per_stream * s, x1 = units_per_stream * (s + 1) - 1;
    const int c0 = (int)(((x0 + 1) * n - 1) / total), c1 = (int)(((x1 + 1) * n - 1) / total);
    first = c0 + s;
    count = c1 - c0 + 1;
  }
  dependency_wait();
  RopeWork rotated{};
  if constexpr (kRope) {
    if (warp == W - 1) rotated = rope_load(rope..., ((size_t)(s / Hkv) * Hq + (s % Hkv) * g + h), s, h, lane);
  }
  // ---- this warp's partials: one pass with a running maximum; a lane has channels 2 lane, 2 lane + 1 and 64 more
  const float* base = ws + (size_t)first * kPartialFloats + h * 130;
  float M = -INFINITY, l = 0.f;
  float2 oa = make_float2(0.f, 0.f), ob = make_float2(0.f, 0.f);
  for (int i0 = warp; i0 < count; i0 += W * kCombineChunk) {
    float2 ml[kCombineChunk], xa[kCombineChunk], xb[kCombineChunk];
#pragma unroll
    for (int j = 0; j < kCombineChunk; ++j) {
      const int i = i0 + j * W;
      ml[j] = make_float2(-INFINITY, 0.f);
      xa[j] = xb[j] = make_float2(0.f, 0.f);
      if (i < count) {
        const float2* p = reinterpret_cast<const float2*>(base + (size_t)i * kPartialFloats);
        ml[j] = p[0];
        xa[j] = p[1 + lane];
        xb[j] = p[33 + lane];
      }
    }
    float Mn = M;
#pragma unroll
    for (int j = 0; j < kCombineChunk; ++j) Mn = fmaxf(Mn, ml[j].x);
    const float f0 = (M == -INFINITY) ? 0.f : exp2f(M - Mn);
    l *= f0;
    oa.x *= f0; oa.y *= f0; ob.x *= f0; ob.y *= f0;
#pragma unroll
    for (int j = 0; j < kCombineChunk; ++j) {
      const float f = (ml[j].x == -INFINITY) ? 0.f : exp2f(ml[j].x - Mn);
      l += f * ml[j].y;
      oa.x += f * xa[j].x; oa.y += f * xa[j].y;
      ob.x += f * xb[j].x; ob.y += f * xb[j].y;
    }
    M = Mn;
  }
  if (kRope && warp == W - 1) rope_store(rotated);
  // ---- the warps' results
  if (lane == 0) {
    mlS[warp][0] = M;
    mlS[warp][1] = l;
  }
  *reinterpret_cast<float2*>(&oS[warp][2 * lane]) = oa;
  *reinterpret_cast<float2*>(&oS[warp][64 + 2 * lane]) = ob;
  __syncthreads();
  const int c = threadIdx.x;
  if (c >= kD) return;
  float Mt = -INFINITY, lt = 0.f, ot = 0.f;
  for (int w = 0; w < W; ++w) Mt = fmaxf(Mt, mlS[w][0]);
  for (int w = 0; w < W; ++w) {
    const float mw = mlS[w][0], f = (mw == -INFINITY) ? 0.f : exp2f(mw - Mt);
    lt += f * mlS[w][1];
    ot += f * oS[w][c];
  }
  // lt == 0 only when every split gave up (its partial is then m = -inf, l = 0, o = 0 and the status word says so) or
  // when the sequence of a ragged batch holds no token
  const int b = s / Hkv, hk = s % Hkv;
  out[((size_t)b * Hq + hk * g + h) * kD + c] = lt > 0.f ? ot / lt : 0.f;
  // natural logarithm of the softmax denominator (the maximum is kept in the base-2 domain)
  if (lse_out != nullptr && c == 0)
    lse_out[(size_t)b * Hq + hk * g + h] = lt > 0.f ? (Mt + log2f(lt)) * 0.6931471805599453f : -INFINITY;
}

// The same for streams with few partials (mode 1): one CTA per stream, warp h merges head h by itself, all of a row's partials
// in flight (attention and merge per layer, a CTA per head / per stream: 32b shape, 512 streams with one to three partials, 236.2 /
// 231.6 us; 32 streams with nine partials 15.7 / 15.9; 16 streams with 18, 37.4 / 37.9).
constexpr int kRowsChunk = 8, kRowsMaxPartials = 8;

template <typename... Rope>
__global__ void __launch_bounds__(256)
combine_rows_kernel(const float* __restrict__ ws, float* __restrict__ out, int g, int Hkv, int Hq, int n, long long units_per_stream,
                    int S, float* __restrict__ lse_out, bool early, Rope... rope) {
  constexpr bool kRope = sizeof...(Rope) > 0;
  if (early) let_successor_start();
  const int s = blockIdx.x, h = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long total = units_per_stream * S;
  const long long x0 = units_per_stream * s, x1 = units_per_stream * (s + 1) - 1;
  const int c0 = (int)(((x0 + 1) * n - 1) / total), c1 = (int)(((x1 + 1) * n - 1) / total), count = c1 - c0 + 1;
  const float* base = ws + (size_t)(c0 + s) * kPartialFloats + h * 130;
  dependency_wait();
  RopeWork rotated{};
  if constexpr (kRope) rotated = rope_load(rope..., (size_t)s * g + h, s, h, lane);
  float M = -INFINITY, l = 0.f;
  float2 oa = make_float2(0.f, 0.f), ob = make_float2(0.f, 0.f);
  for (int i0 = 0; i0 < count; i0 += kRowsChunk) {
    float2 ml[kRowsChunk], xa[kRowsChunk], xb[kRowsChunk];
#pragma unroll
    for (int j = 0; j < kRowsChunk; ++j) {
      ml[j] = make_float2(-INFINITY, 0.f);
      xa[j] = xb[j] = make_float2(0.f, 0.f);
      if (i0 + j < count) {
        const float2* p = reinterpret_cast<const float2*>(base + (size_t)(i0 + j) * kPartialFloats);
        ml[j] = p[0];
        xa[j] = p[1 + lane];
        xb[j] = p[33 + lane];
      }
    }
    float Mn = M;
#pragma unroll
    for (int j = 0; j < kRowsChunk; ++j) Mn = fmaxf(Mn, ml[j].x);
    const float f0 = (M == -INFINITY) ? 0.f : exp2f(M - Mn);
    l *= f0;
    oa.x *= f0; oa.y *= f0; ob.x *= f0; ob.y *= f0;
#pragma unroll
    for (int j = 0; j < kRowsChunk; ++j) {
      const float f = (ml[j].x == -INFINITY) ? 0.f : exp2f(ml[j].x - Mn);
      l += f * ml[j].y;
      oa.x += f * xa[j].x; oa.y += f * xa[j].y;
      ob.x += f * xb[j].x; ob.y += f * xb[j].y;
    }
    M = Mn;
  }
  if (kRope) rope_store(rotated);
  const size_t row = (size_t)s * g + h;             // (b Hkv + hk) g + h = b Hq + hk g + h
  float2* dst = reinterpret_cast<float2*>(out + row * kD);
  dst[lane] = l > 0.f ? make_float2(oa.x / l, oa.y / l) : make_float2(0.f, 0.f);
  dst[32 + lane] = l > 0.f ? make_float2(ob.x / l, ob.y / l) : make_float2(0.f, 0.f);
  if (lse_out != nullptr && lane == 0) lse_out[row] = l > 0.f ? (M + log2f(l)) * 0.6931471805599453f : -INFINITY;
}

cudaError_t launch_combine(const float* ws, float* out, int g, int Hkv, int Hq, int mode, int n,
                           long long units_per_stream, int S, cudaStream_t stream, const int4* seq, const int* seq_prefix,
                           float* lse_out, bool early, void* rope_q, void* rope_k, const float* rope_cos, const float* rope_sin) {
  const bool rows = mode == 1 && seq == nullptr && n / S + 2 <= kRowsMaxPartials;
  // eight warps when four with a chunk each do not cover a stream's partials in one round trip (a ragged batch may give
  // nearly all CTAs to one sequence), four otherwise: more warps only lengthen the last step
  const int partials = mode == 0 ? n : (seq != nullptr ? n : n / S + 1);
  auto launch = [&](auto... rope) {
    if (rows)
      return launch_dependent(combine_rows_kernel<decltype(rope)...>, dim3((unsigned)S), 32 * g, 0, stream, ws, out, g, Hkv, Hq, n, units_per_stream, S, lse_out,
                              early, rope...);
    return launch_dependent(combine_kernel<decltype(rope)...>, dim3((unsigned)(S * g)), partials > 4 * kCombineChunk ? kCombineMaxWarps * 32 : 128, 0, stream, ws,
                            out, g, Hkv, Hq, mode, n, units_per_stream, S, seq, seq_prefix, lse_out, early, rope...);
  };
  if (rope_q != nullptr) return launch(RopeRows{static_cast<uint16_t*>(rope_q), static_cast<uint16_t*>(rope_k), rope_cos, rope_sin});
  return launch();
}

// The table of a ragged batch, from the host's per-sequence fill (kernel arguments: no copy, ordered in the stream).
__global__ void seq_table_kernel(SeqTableArgs a, int4* __restrict__ seq, int* __restrict__ seq_prefix) {
  // a link of the chain of dependent launches: started early, waits for everything before it (a kernel that still
  // reads the table's previous contents included), and only then lets the attention kernel behind it start
  dependency_wait();
  const int b = threadIdx.x;
  if (b < a.n) seq[b] = make_int4(a.fill[3 * b], a.fill[3 * b + 1], a.fill[3 * b + 2], a.w[b]);
  if (b == 0) {
    int acc = 0;
    for (int i = 0; i < a.n; ++i) {
      seq_prefix[i] = acc;
      acc += a.Hkv * a.ctas[i];
    }
    seq_prefix[a.n] = acc;
  }
}

cudaError_t launch_seq_table(const SeqTableArgs& a, int4* seq, int* seq_prefix, cudaStream_t stream) {
  return launch_dependent(seq_table_kernel, dim3(1), kMaxRaggedBatch, 0, stream, a, seq, seq_prefix);
}

// Softmax attention over the union of disjoint token sets from the per-set results: o = sum_r w_r o_r / sum_r w_r with
// w_r = exp(lse_r - max_r lse_r).  o_parts [n_parts][rows][128], lse_parts [n_parts][rows]; a part with lse = -inf
// (no tokens) has weight 0; all parts empty: zeros.
__global__ void __launch_bounds__(128)
merge_partials_kernel(const float* __restrict__ o_parts, const float* __restrict__ lse_parts, int n_parts, int rows,
                      float* __restrict__ out) {
  const int row = blockIdx.x, c = threadIdx.x;
  float top = -INFINITY;
  for (int r = 0; r < n_parts; ++r) top = fmaxf(top, lse_parts[(size_t)r * rows + row]);
  float den = 0.f, num = 0.f;
  if (top != -INFINITY) {
    for (int r = 0; r < n_parts; ++r) {
      const float w = expf(lse_parts[(size_t)r * rows + row] - top);
      den += w;
      num += w * o_parts[((size_t)r * rows + row) * kD + c];
    }
  }
  out[(size_t)row * kD + c] = den > 0.f ? num / den : 0.f;
}

// The partial of a cache that holds no token: zeros and lse = -inf.
__global__ void __launch_bounds__(128) empty_partial_kernel(float* __restrict__ out, float* __restrict__ lse) {
  out[(size_t)blockIdx.x * kD + threadIdx.x] = 0.f;
  if (threadIdx.x == 0) lse[blockIdx.x] = -INFINITY;
}

cudaError_t launch_empty_partial(float* out, float* lse, int rows, cudaStream_t stream) {
  empty_partial_kernel<<<rows, 128, 0, stream>>>(out, lse);
  return cudaGetLastError();
}

cudaError_t launch_merge_partials(const float* o_parts, const float* lse_parts, int n_parts, int rows, float* out,
                                  cudaStream_t stream) {
  merge_partials_kernel<<<rows, 128, 0, stream>>>(o_parts, lse_parts, n_parts, rows, out);
  return cudaGetLastError();
}

// Two sets of partials per stream (packed blocks, residual window), each written by a grid that split its
// S * units work items evenly over n CTAs or groups: member c of set k wrote its part of stream s to slot
// base_k + c + s.
__device__ inline void slot_range(int s, int S, int n, long long units, int* first, int* count) {
  const long long total = units * S;
  const long long x0 = units * s, x1 = units * (s + 1) - 1;
  const int c0 = (int)(((x0 + 1) * n - 1) / total), c1 = (int)(((x1 + 1) * n - 1) / total);
  *first = c0 + s;
  *count = c1 - c0 + 1;
}

__global__ void __launch_bounds__(128)
combine2_kernel(const float* __restrict__ ws, float* __restrict__ out, int g, int Hkv, int Hq, int S, int n1,
                long long units1, int slot2, int n2, long long units2) {
  const int s = blockIdx.x / g, h = blockIdx.x % g, c = threadIdx.x;
  int f1, c1, f2, c2;
  slot_range(s, S, n1, units1, &f1, &c1);
  slot_range(s, S, n2, units2, &f2, &c2);
  f2 += slot2;
  const int b = s / Hkv, hk = s % Hkv;
  float M = -INFINITY;
  for (int i = 0; i < c1 + c2; ++i) {
    const int slot = i < c1 ? f1 + i : f2 + (i - c1);
    M = fmaxf(M, ws[(size_t)slot * kPartialFloats + h * 130]);
  }
  float l = 0.f, o = 0.f;
#pragma unroll 4
  for (int i = 0; i < c1 + c2; ++i) {
    const int slot = i < c1 ? f1 + i : f2 + (i - c1);
    const float* p = ws + (size_t)slot * kPartialFloats + h * 130;
    const float m = p[0];
    const float f = (m == -INFINITY) ? 0.f : exp2f(m - M);
    l += f * p[1];
    o += f * p[2 + c];
  }
  out[((size_t)b * Hq + hk * g + h) * kD + c] = l > 0.f ? o / l : 0.f;
}

cudaError_t launch_combine2(const float* ws, float* out, int g, int Hkv, int Hq, int S, int n1, long long units1,
                            int slot2, int n2, long long units2, cudaStream_t stream) {
  combine2_kernel<<<S * g, 128, 0, stream>>>(ws, out, g, Hkv, Hq, S, n1, units1, slot2, n2, units2);
  return cudaGetLastError();
}

}  // namespace mixkvq
