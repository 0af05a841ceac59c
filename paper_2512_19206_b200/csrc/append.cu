// Residual append and query-magnitude accumulation (Appendix D.1 first step, Appendix D.2).
#include "window.cuh"

namespace mixkvq {

// One CTA per stream: m tokens (input tokens t0..t0+m-1) into residual slots r0..r0+m-1 (append_rows).  Latency-bound: at
// m = 128, g = 7 the serial chain of 896 fp64 additions per channel was most of its 38 us.
__global__ void __launch_bounds__(256)
append_tokens_kernel(LayerView lv, const uint16_t* __restrict__ k, const uint16_t* __restrict__ v,
                     const uint16_t* __restrict__ q, int n_tokens, int t0, int m, int r0) {
  __shared__ __align__(16) unsigned char smem[kAbsSumSmem];
  dependency_wait();
  append_rows(lv, k, v, q, n_tokens, t0, m, r0, blockIdx.x, smem);
}

// Sink tokens: m rows of keys and of values go to sink slots n_sink .. n_sink + m - 1 of every stream, nothing else happens.
__global__ void __launch_bounds__(256)
sink_append_kernel(LayerView lv, const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v, int n_tokens,
                   int t0, int m) {
  dependency_wait();
  const int s = blockIdx.x, tid = threadIdx.x;
  const uint4* ksrc = reinterpret_cast<const uint4*>(k + ((size_t)s * n_tokens + t0) * kD);
  const uint4* vsrc = reinterpret_cast<const uint4*>(v + ((size_t)s * n_tokens + t0) * kD);
  uint4* kdst = reinterpret_cast<uint4*>(lv.sink + (size_t)s * lv.sink_stride) + (size_t)lv.n_sink * 16;
  uint4* vdst = kdst + (size_t)lv.sink_len * 16;
  for (int i = tid; i < m * 16; i += 256) {
    kdst[i] = ksrc[i];
    vdst[i] = vsrc[i];
  }
}

cudaError_t launch_sink_append(const LayerView& lv, const void* k, const void* v, int n_tokens, int t0, int m,
                               cudaStream_t stream) {
  return launch_dependent(sink_append_kernel, dim3(lv.B * lv.Hkv), 256, 0, stream, lv, static_cast<const __nv_bfloat16*>(k),
                          static_cast<const __nv_bfloat16*>(v), n_tokens, t0, m);
}

cudaError_t launch_append(const LayerView& lv, const void* k, const void* v, const void* q, int n_tokens, int t0,
                          int m, cudaStream_t stream) {
  return launch_dependent(append_tokens_kernel, dim3(lv.B * lv.Hkv), 256, 0, stream, lv, static_cast<const uint16_t*>(k),
                          static_cast<const uint16_t*>(v), static_cast<const uint16_t*>(q), n_tokens, t0, m, lv.r);
}

}  // namespace mixkvq
