// Small DFTs in registers, shared by the FFT kernels (NUFFT tier, range-Doppler maps).
#pragma once

#include <cuda_runtime.h>

namespace rsim {

__device__ __forceinline__ float2 cmul(float2 a, float2 w) {
  return make_float2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
}

// exp(+j 2 pi m / 16) for 0 <= m < 8: cosines and sines of multiples of pi / 8
__device__ __forceinline__ float2 unit16(int m) {
  constexpr float c1 = 0.92387953251128676f, s1 = 0.38268343236508977f, h = 0.70710678118654752f;
  switch (m) {
    case 0: return make_float2(1.f, 0.f);
    case 1: return make_float2(c1, s1);
    case 2: return make_float2(h, h);
    case 3: return make_float2(s1, c1);
    case 4: return make_float2(0.f, 1.f);
    case 5: return make_float2(-s1, c1);
    case 6: return make_float2(-h, h);
    default: return make_float2(-c1, s1);
  }
}

__host__ __device__ constexpr int rev_bits(int i, int bits) {
  int r = 0;
  for (int b = 0; b < bits; ++b) r |= ((i >> b) & 1) << (bits - 1 - b);
  return r;
}

__host__ __device__ constexpr int log2_c(int r) { return r <= 1 ? 0 : 1 + log2_c(r >> 1); }

// In-register inverse-sign DFT of R <= 16 points, natural order in and out:
// A_m = sum_j a_j exp(+j 2 pi j m / R), by radix-2 decimation in time.
template <int R>
__device__ __forceinline__ void dft_inv(float2 (&a)[R]) {
  constexpr int bits = log2_c(R);
  float2 b[R];
#pragma unroll
  for (int i = 0; i < R; ++i) b[rev_bits(i, bits)] = a[i];
#pragma unroll
  for (int h = 1; h < R; h <<= 1) {
#pragma unroll
    for (int i0 = 0; i0 < R; i0 += 2 * h) {
#pragma unroll
      for (int k = 0; k < h; ++k) {
        const int m = k * (8 / h);  // exp(+j 2 pi k / (2 h)) = unit16(k 16 / (2 h))
        const float2 u = b[i0 + k];
        float2 t = b[i0 + k + h];
        if (m == 4)
          t = make_float2(-t.y, t.x);
        else if (m != 0)
          t = cmul(t, unit16(m));
        b[i0 + k] = make_float2(u.x + t.x, u.y + t.y);
        b[i0 + k + h] = make_float2(u.x - t.x, u.y - t.y);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i) a[i] = b[i];
}

}  // namespace rsim
