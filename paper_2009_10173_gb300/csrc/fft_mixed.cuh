// Mixed-radix transforms of interleaved complex lines: P = R1 x R2 points, each
// factor a transform in one thread's registers, one trip through shared memory.
//
// Forward (sign -1), with i = i1 R2 + i2 and f = k1 + R1 k2:
//   pass 1, per (line, i2): Y[k1] = sum_i1 x[i1 R2 + i2] W_R1^(i1 k1),
//           times W_P^(i2 k1);
//   pass 2, per (line, k1): X[k1 + R1 k2] = sum_i2 Y[k1][i2] W_R2^(i2 k2).
// Both ends are in natural order, so global reads and writes stay coalesced
// along the lines and nothing is permuted.  The inverse (sign +1) is the
// forward transform of values with real and imaginary parts exchanged.
//
// Why these sizes: a lateral-FFT application is bound by reading the slab's
// spectrum, whose bytes grow with P^2, so the next power of two costs up to
// 3.2x.  One application, GB300, from power-of-two sizes, with the products' kernel of
// that form: 256x256x384 adjoint (P 512 -> 288) 2.19 -> 0.65 ms, 200x200x300 forward
// (256 -> 240) 0.509 -> 0.428 ms, 64x64x128 forward (128 -> 96) 86 -> 57 us (with
// k_fft_apply 0.54 and 0.32 ms, 47 us).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace oam {
namespace mixfft {

// cos and sin of 2 pi k / n at compile time: the angle is reduced to the first
// eighth of a turn with integers, then summed as a Taylor series.
constexpr double kPi = 3.14159265358979323846;
constexpr double taylor(double x, bool cosine) {
  double term = cosine ? 1.0 : x, sum = term;
  for (int i = cosine ? 1 : 2; i < 24; i += 2) {
    term *= -x * x / (double)(i * (i + 1));
    sum += term;
  }
  return sum;
}
constexpr double turn_cos(int k, int n) {  // 0 <= k < n
  if (2 * k > n) return turn_cos(n - k, n);
  if (4 * k > n) return -turn_cos(n - 2 * k, 2 * n);
  return 8 * k > n ? taylor(kPi / 2 * (double)(n - 4 * k) / n, false) : taylor(2 * kPi * k / n, true);
}
constexpr double turn_sin(int k, int n) { return turn_cos((4 * k + 3 * n) % (4 * n), 4 * n); }

template <int I>
using Int = std::integral_constant<int, I>;
template <int I, int N, class F>
__device__ __forceinline__ void static_for(F f) {
  if constexpr (I < N) {
    f(Int<I>{});
    static_for<I + 1, N>(f);
  }
}

// The transforms below are written for any complex type with these operations; a type
// of another file brings its own.
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 cadd_i(float2 a, float2 b) { return make_float2(a.x - b.y, a.y + b.x); }  // a + i b
__device__ __forceinline__ float2 csub_i(float2 a, float2 b) { return make_float2(a.x + b.y, a.y - b.x); }  // a - i b
__device__ __forceinline__ float2 cturn(float2 a) { return make_float2(a.y, -a.x); }                        // -i a
__device__ __forceinline__ float2 cscale(float s, float2 a) { return make_float2(s * a.x, s * a.y); }
__device__ __forceinline__ float2 caxpy(float s, float2 a, float2 b) {  // s a + b
  return make_float2(fmaf(s, a.x, b.x), fmaf(s, a.y, b.y));
}
__device__ __forceinline__ float2 caxpy_i(float s, float2 a, float2 b) {  // b - i s a
  return make_float2(fmaf(s, a.y, b.x), fmaf(-s, a.x, b.y));
}
__device__ __forceinline__ float2 croot(float2 a, float c, float s) {  // a (c - i s)
  return make_float2(a.x * c + a.y * s, a.y * c - a.x * s);
}
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// a W_N^K, W_N = exp(-2 pi i / N)
template <int N, int K, class T>
__device__ __forceinline__ T mul_root(T a) {
  constexpr int k = K % N;
  if constexpr (k == 0) return a;
  else if constexpr (4 * k == N) return cturn(a);
  else if constexpr (2 * k == N) return cneg(a);
  else if constexpr (4 * k == 3 * N) return cneg(cturn(a));
  else return croot(a, (float)turn_cos(k, N), (float)turn_sin(k, N));
}

// In-register forward transform of N points (N a product of 2, 3 and 5).
template <int N, class T>
__device__ __forceinline__ void dft(T (&v)[N]) {
  if constexpr (N == 1) {
  } else if constexpr (N == 2) {
    const T a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  } else if constexpr (N == 3) {
    constexpr float s = (float)turn_sin(1, 3);
    const T t = cadd(v[1], v[2]), d = csub(v[1], v[2]), m = caxpy(-0.5f, t, v[0]);
    v[0] = cadd(v[0], t);
    v[1] = caxpy_i(s, d, m);
    v[2] = caxpy_i(-s, d, m);
  } else if constexpr (N == 4) {
    const T a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
    v[0] = cadd(a, c);
    v[2] = csub(a, c);
    v[1] = csub_i(b, d);
    v[3] = cadd_i(b, d);
  } else if constexpr (N == 5) {
    constexpr float c1 = (float)turn_cos(1, 5), c2 = (float)turn_cos(2, 5);
    constexpr float s1 = (float)turn_sin(1, 5), s2 = (float)turn_sin(2, 5);
    const T t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]), d1 = csub(v[1], v[4]), d2 = csub(v[2], v[3]);
    const T m1 = caxpy(c2, t2, caxpy(c1, t1, v[0])), m2 = caxpy(c1, t2, caxpy(c2, t1, v[0]));
    const T n1 = caxpy(s2, d2, cscale(s1, d1)), n2 = caxpy(-s1, d2, cscale(s2, d1));
    v[0] = cadd(v[0], cadd(t1, t2));
    v[1] = csub_i(m1, n1);
    v[4] = cadd_i(m1, n1);
    v[2] = csub_i(m2, n2);
    v[3] = cadd_i(m2, n2);
  } else {
    constexpr int A = N % 4 == 0 ? 4 : N % 2 == 0 ? 2 : N % 3 == 0 ? 3 : 5, B = N / A;
    static_assert(A * B == N && (N % 2 == 0 || N % 3 == 0 || N % 5 == 0), "factors 2, 3 and 5 only");
    T w[N];
    static_for<0, B>([&](auto j) {
      T t[A];
      static_for<0, A>([&](auto i) { t[i()] = v[i() * B + j()]; });
      dft<A>(t);
      static_for<0, A>([&](auto i) { w[i() * B + j()] = mul_root<N, i() * j()>(t[i()]); });
    });
    static_for<0, A>([&](auto i) {
      T t[B];
      static_for<0, B>([&](auto j) { t[j()] = w[i() * B + j()]; });
      dft<B>(t);
      static_for<0, B>([&](auto j) { v[i() + A * j()] = t[j()]; });
    });
  }
}

// Shared slot of intermediate (k1, i2) of line l among KL lines: lines fastest.
// With 16 lines a half-warp's 8-byte accesses are one 128-byte row; with fewer,
// a pad of KL slots after each k1 row keeps the rows that a half-warp reads
// together in pass 2 in distinct banks.
template <int R2, int KL>
__host__ __device__ constexpr int mix_stride() {
  return R2 * KL + (KL < 16 ? KL : 0);
}
template <int R1, int R2, int KL>
__host__ __device__ constexpr size_t mix_smem() {
  return sizeof(float2) * (size_t)R1 * mix_stride<R2, KL>();
}
// Threads of a block: one per pass-1 or pass-2 item, whichever is more, up to 256.
template <int R1, int R2, int KL>
__host__ __device__ constexpr int mix_threads() {
  constexpr int n = (R1 > R2 ? R1 : R2) * KL;
  return n > 256 ? 256 : (n + 31) / 32 * 32;
}

// One transform of KL lines, in two passes with a barrier between.  src(i2, l, v)
// fills v[m] with points m R2 + i2 (all of a thread's loads together, so that
// they are in flight at once), dst(f, l, v) takes frequency f (inverse: src fills
// frequencies, dst takes a point).  tw holds W_P^j, j < P (global memory, read
// through L1).
template <int R1, int R2, int KL, bool kInverse, class Src>
__device__ __forceinline__ void mix_pass1(float2 *a, const float2 *__restrict__ tw, Src src) {
  constexpr int RS = mix_stride<R2, KL>();
  for (int id = threadIdx.x; id < R2 * KL; id += blockDim.x) {
    const int l = id % KL, i2 = id / KL;
    float2 v[R1];
    src(i2, l, v);
    if (kInverse) {
#pragma unroll
      for (int m = 0; m < R1; ++m) v[m] = make_float2(v[m].y, v[m].x);
    }
    dft<R1>(v);
    a[i2 * KL + l] = v[0];
#pragma unroll
    for (int m = 1; m < R1; ++m) a[m * RS + i2 * KL + l] = cmulc(v[m], __ldg(tw + m * i2));
  }
}
template <int R1, int R2, int KL, bool kInverse, class Dst>
__device__ __forceinline__ void mix_pass2(float2 *a, Dst dst) {
  constexpr int RS = mix_stride<R2, KL>();
  for (int id = threadIdx.x; id < R1 * KL; id += blockDim.x) {
    const int l = id % KL, k1 = id / KL;
    float2 v[R2];
#pragma unroll
    for (int m = 0; m < R2; ++m) v[m] = a[k1 * RS + m * KL + l];
    dft<R2>(v);
#pragma unroll
    for (int m = 0; m < R2; ++m) dst(k1 + R1 * m, l, kInverse ? make_float2(v[m].y, v[m].x) : v[m]);
  }
}
template <int R1, int R2, int KL, bool kInverse, class Src, class Dst>
__device__ __forceinline__ void mix_transform(float2 *a, const float2 *__restrict__ tw, Src src, Dst dst) {
  mix_pass1<R1, R2, KL, kInverse>(a, tw, src);
  __syncthreads();
  mix_pass2<R1, R2, KL, kInverse>(a, dst);
}

// The transform sizes, smallest first: even, at most 512, steps of at most a third
// from 12 on and a quarter or less over most of 64 .. 320 (the batched scans with a
// 61-wide window need 94, 126, 158, 190, 230 and 286 points).
#define OAM_MIX_SIZES(X)                                                                                     \
  X(4, 2, 2) X(8, 2, 4) X(12, 3, 4) X(16, 4, 4) X(20, 4, 5) X(24, 4, 6) X(32, 4, 8) X(40, 5, 8) X(48, 6, 8) \
  X(64, 8, 8) X(80, 8, 10) X(96, 8, 12) X(128, 8, 16) X(160, 10, 16) X(192, 12, 16) X(240, 15, 16)         \
  X(256, 16, 16) X(288, 16, 18) X(320, 16, 20) X(384, 16, 24) X(512, 16, 32)
constexpr int kMixMax = 512;

// Smallest size >= need (need <= kMixMax).
inline int mix_size(int need) {
#define OAM_X(P, R1, R2) \
  if (need <= P) return P;
  OAM_MIX_SIZES(OAM_X)
#undef OAM_X
  return 0;
}

}  // namespace mixfft
}  // namespace oam
