// What the append and the bulk append share: the sum of the query magnitudes of a window, and the rows that go to the
// residual window.
#pragma once

#include "common.cuh"

namespace mixkvq {

__device__ __forceinline__ uint32_t max_bf162(uint32_t a, uint32_t b) {
  const __nv_bfloat162 m = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&m);
}
__device__ __forceinline__ uint32_t min_bf162(uint32_t a, uint32_t b) {
  const __nv_bfloat162 m = __hmin2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&m);
}

// ---- Sum of query magnitudes with the defined result of the serial fp64 sum (token-major, heads ascending), by all 256
// threads of a CTA.
//
// The serial sum is one chain of n * g dependent additions per channel (896 at n = 128, g = 7).  bf16 magnitudes have
// 8 significant bits, so as long as their exponents do not spread too far every partial sum, in ANY order, is a multiple
// of the smallest element's last bit that needs at most 53 bits: then no addition rounds and every order gives the
// serial sum's bits.  The threads therefore add in parallel and check afterwards that this held (smallest non-zero
// magnitude against the total, per channel); if it did not, the sum is taken again in the defined order.
constexpr int kAbsSumSmem = 8 * kD * 8 + 16;      // bytes of scratch: partial sums of the 8 warps, smallest magnitude
constexpr int kAbsSumRounded = -0x7FFFFFFF, kAbsSumZero = 0x7FFFFFFF;

// 2^-640 times a normal bf16 magnitude as fp64, from the bits x << 13 (exponent and mantissa in place, anything elsewhere):
// two logic operations per element with the shift.  0 becomes 2^-127 (times 2^-640) and subnormals a wrong value below
// 2^-126: see the check.
__device__ __forceinline__ double scaled_magnitude(uint32_t shifted) {
  return __hiloint2double((int)((shifted & 0x0FFFE000u) | 0x10000000u), 0);
}
constexpr double kMagnitudeScale = 4.562440617622195e+192;           // 2^640

// Whether a0 >= 0 plus addends that are all multiples of 2^unit, with the (rounded) sum `total`, can be added in any order
// without rounding: every partial sum is at most the total and a multiple of the smallest last bit.
__device__ inline bool sum_is_exact(double a0, double total, int unit) {
  if (a0 != 0.0) {
    const long long bits = __double_as_longlong(a0);
    const int ea = (int)((bits >> 52) & 0x7FF);
    if (ea == 0 || ea == 0x7FF) return false;
    unit = min(unit, ea - 1075 + __ffsll((bits & 0xFFFFFFFFFFFFFll) | (1ll << 52)) - 1);      // a0's last set bit
  }
  if (unit == kAbsSumZero) return true;
  return unit > -900 && unit < 900 && total < __hiloint2double((unit + 53 + 1023) << 20, 0);
}

// The queries of n tokens and g heads: qw[h * head_stride + j * 128 + d], bf16 bits.  Returns a0 plus the sum of channel
// threadIdx.x in threads 0..127 (others: undefined), and in *unit the exponent of a common last bit of all magnitudes
// (kAbsSumZero: all are zero; kAbsSumRounded: the sum was taken in order).  `smem`: kAbsSumSmem bytes, 16-byte aligned,
// free on entry.  All 256 threads call it; it contains barriers.
__device__ inline double abs_sum_256(const uint16_t* __restrict__ qw, size_t head_stride, int n, int g, double a0,
                                     unsigned char* smem, int* unit) {
  double* redS = reinterpret_cast<double*>(smem);                      // [8 warps][128]
  uint32_t* minS = reinterpret_cast<uint32_t*>(smem + 8 * kD * 8);     // smallest |q| bits - 1 (0xFFFF: all zero)
  const int tid = threadIdx.x, c = tid & 15, rg = tid >> 4;            // 8 channels of every 16th row
  if (tid == 0) *minS = 0xFFFFu;
  double a[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = 0.0;
  // smallest non-zero magnitude, as bf16 pairs -(bits - 1): the largest of them; zeros become NaNs, which the maximum ignores
  uint32_t mn = 0x7FFF7FFFu;
  constexpr int kDepth = 8;                                            // 16-byte loads in flight per thread
  const int rows = n * g, dh = 16 / n, dj = 16 - dh * n;               // rows head by head; 16 rows further
  int h = rg / n, j = rg - h * n;
  for (int row = rg; row < rows; row += 16 * kDepth) {
    uint4 x[kDepth];
#pragma unroll
    for (int k = 0; k < kDepth; ++k) {
      x[k] = make_uint4(0u, 0u, 0u, 0u);
      if (row + 16 * k < rows) x[k] = *reinterpret_cast<const uint4*>(qw + (size_t)h * head_stride + (size_t)(j * kD + 8 * c));
      j += dj;
      h += dh;
      if (j >= n) {
        j -= n;
        ++h;
      }
    }
#pragma unroll
    for (int k = 0; k < kDepth; ++k) {                                 // rows past the end are zeros: they add 2^-127
      const uint32_t w[4] = {x[k].x, x[k].y, x[k].z, x[k].w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[2 * i] = __dadd_rn(a[2 * i], scaled_magnitude(w[i] << 13));
        a[2 * i + 1] = __dadd_rn(a[2 * i + 1], scaled_magnitude(w[i] >> 3));
        mn = max_bf162(mn, (w[i] | 0x80008000u) - 0x00010001u);
      }
    }
  }
  __syncthreads();                                                     // minS is set
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = __dadd_rn(a[i], __shfl_xor_sync(0xffffffffu, a[i], 16));
  if ((tid & 31) < 16) {
#pragma unroll
    for (int i = 0; i < 8; ++i) redS[(tid >> 5) * kD + 8 * c + i] = a[i];
  }
  const uint32_t lo = mn & 0xFFFFu, hi = mn >> 16;                     // bits - 1 with the sign set, or the NaN 0x7FFF
  const uint32_t m1 = __reduce_min_sync(0xffffffffu, min(lo >= 0x8000u ? lo - 0x8000u : 0xFFFFu, hi >= 0x8000u ? hi - 0x8000u : 0xFFFFu));
  if ((tid & 31) == 0) atomicMin(minS, m1);
  __syncthreads();
  double total = a0;
  bool exact = true;
  const uint32_t smallest = *minS;
  const bool none = smallest == 0xFFFFu;                                // nothing but zeros (and NaNs)
  const int e = none ? 0 : (int)((smallest + 1u) >> 7);                 // biased exponent of the smallest magnitude
  *unit = none ? kAbsSumZero : e - 134;                                 // all magnitudes are multiples of 2^unit
  if (tid < kD) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s = __dadd_rn(s, redS[w * kD + tid]);
    s = __dmul_rn(s, kMagnitudeScale);
    // Zeros went in as 2^-127.  With every other magnitude at least 2^-47 they disappear in the first one they meet (at
    // most 2^12 of them with the rows past the end, 2^-115 against a half unit of 2^-100), and a channel of zeros alone stays below 2^-100.
    if (s < 7.888609052210118e-31) s = 0.0;
    total = __dadd_rn(a0, s);
    // (a sum of 2^128 or more: possibly infinities, or NaNs, which went in as 2^128 and more and which the search for the
    // smallest magnitude passes over)
    exact = s < 3.402823669209385e38 && (none || (e >= 80 && sum_is_exact(a0, total, *unit)));
  }
  if (!__syncthreads_and(exact ? 1 : 0)) {
    *unit = kAbsSumRounded;
    if (tid < kD) {
      total = a0;
      for (int jj = 0; jj < n; ++jj)
        for (int hh = 0; hh < g; ++hh)
          total = __dadd_rn(total, (double)fabsf(bf16_bits_to_float(qw[(size_t)hh * head_stride + (size_t)jj * kD + tid])));
    }
  }
  return total;
}

// ---- One stream's part of a residual append (one CTA of 256 threads): input tokens t0 .. t0 + m - 1 go to residual slots
// r0 .. r0 + m - 1 by 16-byte copies, and |q| of the g heads of the group is added to the importance accumulator.
// `smem`: kAbsSumSmem bytes.
__device__ inline void append_rows(const LayerView& lv, const uint16_t* __restrict__ k, const uint16_t* __restrict__ v,
                                   const uint16_t* __restrict__ q, int n_tokens, int t0, int m, int r0, int s,
                                   unsigned char* smem) {
  const int tid = threadIdx.x, b = s / lv.Hkv, hk = s % lv.Hkv, g = lv.g;
  const uint4* ksrc = reinterpret_cast<const uint4*>(k + ((size_t)s * n_tokens + t0) * kD);
  const uint4* vsrc = reinterpret_cast<const uint4*>(v + ((size_t)s * n_tokens + t0) * kD);
  uint4* kdst = reinterpret_cast<uint4*>(lv.resk + (size_t)s * lv.resk_stride) + (size_t)r0 * 16;
  uint4* vdst = reinterpret_cast<uint4*>(lv.resv + (size_t)s * lv.resv_stride) + (size_t)r0 * 16;
#pragma unroll 4
  for (int i = tid; i < m * 16; i += 256) {
    const uint4 a = ksrc[i], c = vsrc[i];
    kdst[i] = a;
    vdst[i] = c;
  }
  double* acc = reinterpret_cast<double*>(lv.state + (size_t)s * lv.state_stride);
  const uint16_t* qw = q + (((size_t)b * lv.Hq + hk * g) * n_tokens + t0) * kD;
  int unit;
  const double a = abs_sum_256(qw, (size_t)n_tokens * kD, m, g, tid < kD ? acc[tid] : 0.0, smem, &unit);
  if (tid < kD) acc[tid] = a;
  if (tid == 0) *reinterpret_cast<uint32_t*>(lv.state + (size_t)s * lv.state_stride + 1024) += (uint32_t)(m * g);
}

}  // namespace mixkvq
