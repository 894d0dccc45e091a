// Line transforms of the split-BF16 operators: the scan's y axis is taken to the
// lateral frequency domain around the tensor-core correlation along x (op_tc.cu).
//
// Forward transform, per (x, channel block): the real y line of the operator
// input, zero-padded to P, as re and im rows of the packed correlation input.
// Inverse, per (x, channel block): the correlation's re and im rows back to a
// real y line of the output.  Both move the volume or the signals once and the
// half spectrum (about 1.2x the lines, the inverse once per partial sum) once; 32
// channels per block, two neighbours per thread, make every global access a whole
// 128-byte line per point, and all of a thread's loads are issued before its first
// use.  At 200x200x300 (cold caches) 40 us forward, issue-bound, and 30, 62, 67 us
// inverse with 1, 2 and, at three blocks per SM instead of two, 3 partial sums, bound
// by the loads' latency (18 us of bytes forward, 26 + 9 per sum inverse, at 6.8 TB/s).
// The output's channels beyond the accumulator are zeroed by a spare warp of the
// correlation kernel where its products hide that (35 us here), else by blocks of the
// inverse (op_tc.cu, zeros_in_inverse).
//
// The correlation has compact support: a position whose window holds only zeros
// gets exact zeros, and a non-finite input reaches only the positions whose window
// holds it, and of those the samples (depths) that the slab couples with its channel.
// A transform along y would spread both over the line.  So the forward transform marks
// the positions that hold a non-zero and, per 32 channels, those that hold a non-finite
// value (taken as zero by the transform), one bit each; a spare warp of the correlation
// kernel grows the marks by the window while the products run (op_tc.cu); the inverse
// writes zeros where the window of an output position holds no input, NaN in the 32
// channels that a non-finite one reaches, and clears the marks.
#include <algorithm>
#include <cfloat>

#include "fft_mixed.cuh"
#include "internal.cuh"

using namespace oam;
using namespace oam::mixfft;

namespace {

constexpr int kLineCh = 32;  // channels per block: sixteen complex lines of two neighbouring real channels
constexpr int kKH = kLineCh / 2;

// The bits of `bits` belong to rows y0 .. y0 + 31 of one column's mark words.
__device__ __forceinline__ void mark_rows(unsigned *col, int y0, unsigned bits) {
  const int w = y0 >> 5, s = y0 & 31;  // marked rows lie in the grid, so non-empty words are valid
  const unsigned lo = bits << s, hi = s ? bits >> (32 - s) : 0u;
  if (lo && (__ldcg(col + w) & lo) != lo) atomicOr(col + w, lo);
  if (hi && (__ldcg(col + w + 1) & hi) != hi) atomicOr(col + w + 1, hi);
}

// kVec: input rows are a whole number of float2 from an 8-byte boundary.
template <int R1, int R2, bool kVec>
__global__ void __launch_bounds__(mix_threads<R1, R2, kKH>())
    k_line_r2c(const LineShape s, const float *__restrict__ X, const float2 *__restrict__ tw, float *__restrict__ out) {
  constexpr int P = R1 * R2, Q = P / 2 + 1, RS = mix_stride<R2, kKH>();
  extern __shared__ float2 sm[];
  __shared__ uint8_t some[P], bad[P];
  __shared__ unsigned umax[Q];
  const int x = blockIdx.y, cb = blockIdx.x * kLineCh, y0 = s.first_row(blockIdx.z);
  for (int i = threadIdx.x; i < P; i += blockDim.x) some[i] = bad[i] = 0;
  __syncthreads();
  const float *col = X + (size_t)x * s.len + s.in_lo + cb;
  const size_t stride = (size_t)s.px * s.len;
  const int live = min(s.elems, s.len - s.in_lo) - cb;  // channels that exist
  auto load = [&](int i2, int l, float2 (&v)[R1]) {
    const bool ok0 = 2 * l < live, ok1 = 2 * l + 1 < live;
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const int y = y0 + m * R2 + i2;
      const bool in = y >= 0 && y < s.py;
      const float *p = col + (ptrdiff_t)y * (ptrdiff_t)stride + 2 * l;
      if (kVec) {
        v[m] = in && ok0 ? *reinterpret_cast<const float2 *>(p) : make_float2(0.0f, 0.0f);
      } else {
        v[m].x = in && ok0 ? p[0] : 0.0f;
        v[m].y = in && ok1 ? p[1] : 0.0f;
      }
    }
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      if (v[m].x != 0.0f || v[m].y != 0.0f) some[m * R2 + i2] = 1;  // also true for NaN
      if (!(fabsf(v[m].x) <= FLT_MAX && fabsf(v[m].y) <= FLT_MAX)) {
        bad[m * R2 + i2] = 1;
        if (!(fabsf(v[m].x) <= FLT_MAX)) v[m].x = 0.0f;
        if (!(fabsf(v[m].y) <= FLT_MAX)) v[m].y = 0.0f;
      }
    }
  };
  auto keep = [&](int f, int l, float2 v) { sm[(f % R1) * RS + (f / R1) * kKH + l] = v; };  // its own pass-2 slots
  mix_transform<R1, R2, kKH, false>(sm, tw, load, keep);
  __syncthreads();
  // untangle the two channels of each line; a half-warp holds one frequency of all lines
  float *o0 = out + ((size_t)s.R + (size_t)(2 * blockIdx.z) * s.wp + x) * s.elems + cb;
  const size_t im_off = (size_t)s.wp * s.elems, f_off = (size_t)s.rows * s.elems;
  for (int i = threadIdx.x; i < (Q * kKH + 31) / 32 * 32; i += blockDim.x) {
    const int l = i % kKH, u = i / kKH, un = u == 0 ? 0 : P - u;
    float top = 0.0f;
    if (u < Q) {
      const float2 z = sm[(u % R1) * RS + (u / R1) * kKH + l], w = sm[(un % R1) * RS + (un / R1) * kKH + l];
      const float2 re = make_float2(0.5f * (z.x + w.x), 0.5f * (z.y + w.y));
      const float2 im = make_float2(0.5f * (z.y - w.y), 0.5f * (w.x - z.x));
      if (2 * l < live) {  // channels beyond the input stay zero (a pair's second is zero then)
        float *o = o0 + (size_t)u * f_off + 2 * l;
        *reinterpret_cast<float2 *>(o) = re;
        *reinterpret_cast<float2 *>(o + im_off) = im;
      }
      top = fmaxf(fmaxf(fabsf(re.x), fabsf(re.y)), fmaxf(fabsf(im.x), fabsf(im.y)));
    }
    // the frequency's largest magnitude on this line (non-negative floats compare as integers)
    unsigned t = __float_as_uint(top);
#pragma unroll
    for (int off = kKH / 2; off; off >>= 1) t = max(t, __shfl_xor_sync(0xffffffffu, t, off));
    if (l == 0 && u < Q) umax[u] = t;
  }
  for (int w = threadIdx.x >> 5; 32 * w < P; w += blockDim.x >> 5) {
    const int i = 32 * w + (threadIdx.x & 31);
    const unsigned b = __ballot_sync(0xffffffffu, i < P && some[i]), n = __ballot_sync(0xffffffffu, i < P && bad[i]);
    if ((threadIdx.x & 31) == 0) {
      mark_rows(s.marks + (size_t)x * s.words, y0 + 32 * w, b);
      if (n) {
        mark_rows(s.marks + ((size_t)(1 + blockIdx.x) * s.px + x) * s.words, y0 + 32 * w, n);
        *s.any_bad = 1;
      }
    }
  }
  __syncthreads();
  for (int u = threadIdx.x; u < Q; u += blockDim.x)
    if (umax[u]) atomicMax(s.vmax + (size_t)u * s.px + x, umax[u]);
}

// kVec: output rows are a whole number of float2 from an 8-byte boundary.
template <int R1, int R2, bool kVec>
__global__ void __launch_bounds__(mix_threads<R1, R2, kKH>(), R1 >= 15 && R2 <= 20 ? 3 : 2)
    k_line_c2r(const LineShape s, const float *__restrict__ part, const float2 *__restrict__ tw, float scale,
               float *__restrict__ out) {
  constexpr int P = R1 * R2, Q = P / 2 + 1;
  extern __shared__ float2 sm[];
  __shared__ unsigned words[2][P / 32 + 2];  // grown marks of the rows written: some input, a non-finite one
  const int x = blockIdx.y, ob = (s.zeros ? 0 : s.out_lo / kLineCh * kLineCh) + blockIdx.x * kLineCh;
  const int y0 = s.first_row(blockIdx.z), ya = s.out_row(blockIdx.z), yb = min(s.py, ya + s.valid);  // rows written
  float *col = out + (size_t)x * s.out_len + ob;
  const size_t stride = (size_t)s.px * s.out_len;
  const int cols = min(kLineCh, s.out_len - ob);
  const bool spoiled = __ldg(s.spoiled) != 0;
  // this application's marks are grown: clear them for the next
  if (blockIdx.x == 0 && blockIdx.z == 0) {
    const int planes = spoiled ? s.planes : 1;
    for (int i = threadIdx.x; i < planes * s.words; i += blockDim.x)
      s.marks[((size_t)(i / s.words) * s.px + x) * s.words + i % s.words] = 0;
    for (int i = threadIdx.x; i < Q; i += blockDim.x) s.vmax[(size_t)i * s.px + x] = 0;
    if (x == 0 && threadIdx.x == 0) *s.any_bad = 0;
  }
  if (ob + kLineCh <= s.out_lo || ob >= s.out_lo + s.acc) {  // outside the accumulator (whole float4 there)
    for (int i = threadIdx.x; i < (yb - ya) * (kLineCh / 4); i += blockDim.x) {
      const int y = ya + i / (kLineCh / 4), c = 4 * (i % (kLineCh / 4));
      if (c < cols) *reinterpret_cast<float4 *>(col + (size_t)y * stride + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    return;
  }
  const int w0 = ya >> 5, nw = ((yb - 1) >> 5) - w0 + 1;
  const int z0 = ob - s.out_lo;  // accumulator column of the block's first channel (even: out_lo is 16-aligned)
  for (int i = threadIdx.x; i < nw; i += blockDim.x) {
    const size_t at = (size_t)x * s.words + w0 + i, plane = (size_t)s.px * s.words;
    words[0][i] = __ldg(s.grown + at);
    unsigned bad = 0;
    if (spoiled)
      for (int b = 0; b < s.planes - 1; ++b)
        if (s.reach[b].x < z0 + kLineCh && s.reach[b].y > z0) bad |= __ldg(s.grown + (1 + b) * plane + at);
    words[1][i] = bad;
  }
  const size_t f_off = (size_t)s.nr * s.px * s.acc, im_off = (size_t)s.px * s.acc, p_off = Q * f_off;
  const float *zc = part + ((size_t)(2 * blockIdx.z) * s.px + x) * s.acc + z0;
  auto load = [&](int i2, int l, float2 (&v)[R1]) {
    const bool ok = z0 + 2 * l >= 0 && z0 + 2 * l < s.acc;
#pragma unroll
    for (int m = 0; m < R1; ++m) v[m] = make_float2(0.0f, 0.0f);
    if (!ok) return;
    for (int q = 0; q < s.parts; ++q) {
      const float *zp = zc + q * p_off + 2 * l;
      float2 re[R1], im[R1];
#pragma unroll
      for (int m = 0; m < R1; ++m) {
        const int f = m * R2 + i2, fh = f < Q ? f : P - f;  // Hermitian source row
        re[m] = *reinterpret_cast<const float2 *>(zp + fh * f_off);
        im[m] = *reinterpret_cast<const float2 *>(zp + fh * f_off + im_off);
      }
#pragma unroll
      for (int m = 0; m < R1; ++m) {
        const int f = m * R2 + i2;
        const float sg = f == 0 || f == (P >> 1) ? 0.0f : f < Q ? 1.0f : -1.0f;
        v[m] = cadd(v[m], make_float2(fmaf(-sg, im[m].y, re[m].x), fmaf(sg, im[m].x, re[m].y)));
      }
    }
  };
  auto store = [&](int i, int l, float2 v) {
    const int y = y0 + i;
    if (y < ya || y >= yb || 2 * l >= cols) return;
    const int j = (y >> 5) - w0;
    const unsigned bit = 1u << (y & 31);
    const int st = words[1][j] & bit ? 2 : words[0][j] & bit ? 1 : 0;
    const bool in = z0 + 2 * l >= 0 && z0 + 2 * l < s.acc;  // acc is even: both channels or none
    const float fill = in && st == 2 ? __int_as_float(0x7fffffff) : 0.0f;
    const float2 w = in && st == 1 ? make_float2(v.x * scale, v.y * scale) : make_float2(fill, fill);
    float *p = col + (size_t)y * stride + 2 * l;
    if (kVec) {
      *reinterpret_cast<float2 *>(p) = w;
    } else {
      p[0] = w.x;
      if (2 * l + 1 < cols) p[1] = w.y;
    }
  };
  mix_transform<R1, R2, kKH, true>(sm, tw, load, store);
}

template <int R1, int R2, bool kVec>
oam_status run(bool inverse, cudaStream_t st, const LineShape &s, const float *in, const float2 *tw, float *out) {
  constexpr size_t sm = mix_smem<R1, R2, kKH>();
  constexpr int threads = mix_threads<R1, R2, kKH>();
  if (inverse) {
    if (sm > 40 * 1024)  // static shared memory comes on top
      OAM_CUDA_TRY(
          cudaFuncSetAttribute(k_line_c2r<R1, R2, kVec>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    int z0, z1;
    line_channels(s, &z0, &z1);
    if (s.zeros) z0 = 0, z1 = s.out_len;
    k_line_c2r<R1, R2, kVec><<<dim3((z1 - z0 + kLineCh - 1) / kLineCh, s.px, s.segs), threads, sm, st>>>(
        s, in, tw, 1.0f / (float)(R1 * R2), out);
  } else {
    if (sm > 40 * 1024)
      OAM_CUDA_TRY(
          cudaFuncSetAttribute(k_line_r2c<R1, R2, kVec>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    k_line_r2c<R1, R2, kVec><<<dim3((std::min(s.elems, s.len - s.in_lo) + kLineCh - 1) / kLineCh, s.px, s.segs),
                               threads, sm, st>>>(s, in, tw, out);
  }
  OAM_LAUNCHED();
  return OAM_OK;
}

oam_status dispatch(int P, bool inverse, cudaStream_t st, LineShape s, const float *in, const float2 *tw, float *out) {
  // volumes of an odd depth count have rows off the 8-byte grid (nt is a multiple of 4)
  const bool vec = inverse ? s.out_len % 2 == 0 : s.len % 2 == 0 && s.in_lo % 2 == 0;
  switch (P) {
#define OAM_X(N, R1, R2)                                               \
  case N:                                                              \
    return vec ? run<R1, R2, true>(inverse, st, s, in, tw, out)        \
               : run<R1, R2, false>(inverse, st, s, in, tw, out);
    OAM_MIX_SIZES(OAM_X)
#undef OAM_X
  }
  return OAM_ERR_UNSUPPORTED;
}

}  // namespace

// The 32-channel blocks of the output that meet the accumulator, up to the row's end.
void oam::line_channels(const LineShape &s, int *z0, int *z1) {
  *z0 = s.out_lo / kLineCh * kLineCh;
  *z1 = std::min(s.out_len, (s.out_lo + s.acc + kLineCh - 1) / kLineCh * kLineCh);
}

oam_status oam::line_r2c(int P, cudaStream_t st, const LineShape &s, const float *in, const float2 *tw, float *packed) {
  return dispatch(P, false, st, s, in, tw, packed);
}
oam_status oam::line_c2r(int P, cudaStream_t st, const LineShape &s, const float *part, const float2 *tw, float *out) {
  return dispatch(P, true, st, s, part, tw, out);
}
