// FFT pieces shared by the point-cloud transforms and the synthesis: complex
// product, bit reversal, a per-CTA twiddle table and the in-place shared-memory
// transform.
//
// The transform is radix-2 decimation in time, three stages at a time: a thread
// holds eight points in registers, so a 4096-point transform passes four times
// through shared memory, with four barriers, instead of twelve; the butterflies
// and their operands are those of single stages.  These transforms are chains of
// dependent shared-memory round trips in a few CTAs, so passes are what they cost
// (k_fft_rows, 4 rows of 4096: 22.0 -> 7.7 us; 1,536 rows of 256: 8.3 -> 6.1 us).
// Points and twiddles sit at padded slots: strides of 8, 32, 128, ... points (the
// bit-reversed stores, the first passes) would otherwise share banks.
#pragma once

#include <cuda_runtime.h>

namespace sbr {
namespace fft {

__device__ inline float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ inline int bitrev(int x, int bits) { return (int)(__brev((unsigned)x) >> (32 - bits)); }

// Slot of point i, and the slots n points take.
__host__ __device__ constexpr int slot(int i) { return i + (i >> 3) + (i >> 7); }
__host__ __device__ constexpr int slots(int n) { return slot(n) + 1; }

// Twiddles e^{sign 2 pi i j / n}, j < n / 2, at tw[slot(j)]; the stage of length
// len = 2^m takes entry j << (logn - m) (the same float argument 2 j / len as a
// direct evaluation: both quotients are exact).  slots(n / 2) entries.
__device__ inline void fill_twiddles(float2* tw, int n, float sign, int lanes, int lane) {
  for (int j = lane; j < (n >> 1); j += lanes) {
    float sn, cs;
    sincospif(sign * 2.f * (float)j / (float)n, &sn, &cs);
    tw[slot(j)] = make_float2(cs, sn);
  }
}

// Stages m .. m + R - 1 for the 2^R points of unit u.
template <int R>
__device__ inline void stages(float2* s, const float2* tw, int logn, int m, int u) {
  const int half = 1 << (m - 1), j = u & (half - 1), base = ((u >> (m - 1)) << (m - 1 + R)) + j;
  float2 x[1 << R];
#pragma unroll
  for (int k = 0; k < (1 << R); ++k) x[k] = s[slot(base + k * half)];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int k = 0; k < (1 << R); ++k) {
      if (k & (1 << r)) continue;
      const float2 w = tw[slot((j + (k & ((1 << r) - 1)) * half) << (logn - m - r))];
      const float2 t = cmul(x[k | (1 << r)], w), a = x[k];
      x[k] = make_float2(a.x + t.x, a.y + t.y);
      x[k | (1 << r)] = make_float2(a.x - t.x, a.y - t.y);
    }
#pragma unroll
  for (int k = 0; k < (1 << R); ++k) s[slot(base + k * half)] = x[k];
}

// In-place transforms of 2^logb rows of n = 2^logn points, row b at s + b ld, points
// at their slots in bit-reversed order, all threads of the block cooperating.
// kRowFast: consecutive threads take consecutive rows (ld odd), else points.
template <bool kRowFast>
__device__ inline void smem_fft_rows(float2* s, int ld, int logb, const float2* tw, int logn, int lanes, int lane) {
  int m = 1;
  while (m <= logn) {
    const int left = (logn - m + 1) % 3, r = left ? left : 3, logu = logn - r;  // the short pass first
    for (int i = lane; i < 1 << (logu + logb); i += lanes) {
      const int b = kRowFast ? i & ((1 << logb) - 1) : i >> logu, u = kRowFast ? i >> logb : i & ((1 << logu) - 1);
      float2* row = s + b * ld;
      if (r == 3) stages<3>(row, tw, logn, m, u);
      else if (r == 2) stages<2>(row, tw, logn, m, u);
      else stages<1>(row, tw, logn, m, u);
    }
    m += r;
    __syncthreads();
  }
}

// One row.
__device__ inline void smem_fft(float2* s, const float2* tw, int logn, int lanes, int lane) {
  smem_fft_rows<false>(s, 0, 0, tw, logn, lanes, lane);
}

}  // namespace fft
}  // namespace sbr
