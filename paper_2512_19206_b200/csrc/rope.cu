// Rotary position embedding of the keys and queries of an append, in place (Appendix D: importance scores and keys
// are taken after the rotation, so every caller rotates right before it appends).
//
// (The arithmetic is rotate_chunk in common.cuh; a fused decode step rotates in the split kernel instead.)
#include "common.cuh"

namespace mixkvq {

namespace {

// rows: the B * Hkv * n key rows, then the B * Hq * n query rows; token index of a row = row % n.
// One thread rotates eight pairs of one row: channels 8c .. 8c+7 and 64 + 8c .. 64 + 8c+7.
__global__ void __launch_bounds__(256)
rope_kernel(__nv_bfloat16* __restrict__ k, __nv_bfloat16* __restrict__ q, const float* __restrict__ cos_t,
            const float* __restrict__ sin_t, long long k_rows, long long rows, int n_tokens, int pos0) {
  dependency_wait();
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long row = idx >> 3;
  const int c = (int)(idx & 7);
  if (row >= rows) return;
  __nv_bfloat16* x = (row < k_rows ? k + row * kD : q + (row - k_rows) * kD) + 8 * c;
  const int pos = pos0 + (int)(row % n_tokens);
  const float *cos_row = cos_t + (size_t)pos * 64, *sin_row = sin_t + (size_t)pos * 64;
  const uint4 lo = *reinterpret_cast<const uint4*>(x), hi = *reinterpret_cast<const uint4*>(x + 64);
  *reinterpret_cast<uint4*>(x) = rotate_chunk(lo, hi, cos_row, sin_row, c);
  *reinterpret_cast<uint4*>(x + 64) = rotate_chunk(hi, lo, cos_row, sin_row, c + 8);
}

}  // namespace

cudaError_t launch_rope(void* k, void* q, const float* cos_t, const float* sin_t, int B, int Hkv, int Hq, int n_tokens,
                        int pos0, cudaStream_t stream) {
  const long long k_rows = (long long)B * Hkv * n_tokens, rows = k_rows + (long long)B * Hq * n_tokens;
  const long long threads = rows * 8;
  return launch_dependent(rope_kernel, dim3((unsigned)((threads + 255) / 256)), 256, 0, stream, static_cast<__nv_bfloat16*>(k),
                          static_cast<__nv_bfloat16*>(q), cos_t, sin_t, k_rows, rows, n_tokens, pos0);
}

}  // namespace mixkvq
