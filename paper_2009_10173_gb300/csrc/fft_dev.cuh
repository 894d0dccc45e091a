// The 16-point twiddle constants and bit reversal of the power-of-two register
// passes, used by the lateral-FFT operator form (sizes above 512) and by the
// band-pass filter along time.
#pragma once

#include <cuda_runtime.h>

namespace oam {
namespace fftdev {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ __forceinline__ int bitrev(int x, int lg) { return (int)(__brev((unsigned)x) >> (32 - lg)); }

constexpr float kRsqrt2 = 0.70710678118654752f;  // cos(pi/4) = sin(pi/4)
constexpr float kCosPi8 = 0.92387953251128676f;  // cos(pi/8)
constexpr float kSinPi8 = 0.38268343236508977f;  // sin(pi/8)

// W_N^u = exp(-2 pi i u / N) for N <= 16 (u < N/2), from the constants above.
__device__ __forceinline__ float2 w16(int N, int u) {
  switch (u * (16 / N)) {  // in sixteenths of a turn
    case 0: return make_float2(1.0f, 0.0f);
    case 1: return make_float2(kCosPi8, -kSinPi8);
    case 2: return make_float2(kRsqrt2, -kRsqrt2);
    case 3: return make_float2(kSinPi8, -kCosPi8);
    case 4: return make_float2(0.0f, -1.0f);
    case 5: return make_float2(-kSinPi8, -kCosPi8);
    case 6: return make_float2(-kRsqrt2, -kRsqrt2);
    default: return make_float2(-kCosPi8, -kSinPi8);  // 7
  }
}

}  // namespace fftdev
}  // namespace oam
