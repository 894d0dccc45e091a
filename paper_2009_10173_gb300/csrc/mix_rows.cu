// Row transforms of the lateral-FFT form at the mixed-radix sizes (fft_mixed.cuh):
// real rows along x to the half spectrum, and back.
#include "fft_mixed.cuh"
#include "internal.cuh"

using namespace oam;
using namespace oam::mixfft;

namespace {

constexpr int kRowCh = 32;  // channels per block: sixteen complex lines of two neighbouring real channels

// Real rows -> half spectrum along x.  X[py][px][Ctot] (channels c0 .. c0+C-1
// used), Y[Q][py][CO] complex, CO a multiple of 4.  Block (channel block, y).
// Channels 2l and 2l + 1 ride as the real and imaginary parts of complex line l; with
// Z = FFT(x + i y), X(u) = (Z(u) + conj Z(-u)) / 2 and Y(u) = (Z(u) - conj Z(-u)) / 2i.
// kVec: the rows' channel pairs lie on 8-byte boundaries.
template <int R1, int R2, int KC, bool kVec>
__global__ void __launch_bounds__(mix_threads<R1, R2, KC / 2>())
    k_mix_rows_r2c(const float *__restrict__ X, int py, int px, int Ctot, int c0, int C, int CO,
                   const float2 *__restrict__ tw, float2 *__restrict__ Y) {
  constexpr int KH = KC / 2, P = R1 * R2, Q = P / 2 + 1, RS = mix_stride<R2, KH>();
  extern __shared__ float2 sm[];
  const int y = blockIdx.y, cb = blockIdx.x * KC;
  const float *row = X + (size_t)y * px * Ctot + c0 + cb;
  auto load = [&](int i2, int l, float2 (&v)[R1]) {
    const bool ok0 = cb + 2 * l < C, ok1 = cb + 2 * l + 1 < C;
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const int x = m * R2 + i2;
      const float *p = row + (size_t)x * Ctot + 2 * l;
      if (kVec && ok1) {
        v[m] = x < px ? *reinterpret_cast<const float2 *>(p) : make_float2(0.0f, 0.0f);
      } else {
        v[m].x = x < px && ok0 ? p[0] : 0.0f;
        v[m].y = x < px && ok1 ? p[1] : 0.0f;
      }
    }
  };
  auto keep = [&](int f, int l, float2 v) { sm[(f % R1) * RS + (f / R1) * KH + l] = v; };  // its own pass-2 slots
  mix_transform<R1, R2, KH, false>(sm, tw, load, keep);
  __syncthreads();
  for (int i = threadIdx.x; i < Q * KH; i += blockDim.x) {
    const int u = i / KH, l = i % KH, un = u == 0 ? 0 : P - u;
    if (cb + 2 * l >= C) continue;
    const float2 z = sm[(u % R1) * RS + (u / R1) * KH + l], w = sm[(un % R1) * RS + (un / R1) * KH + l];
    *reinterpret_cast<float4 *>(Y + ((size_t)u * py + y) * CO + cb + 2 * l) =
        make_float4(0.5f * (z.x + w.x), 0.5f * (z.y - w.y), 0.5f * (z.y + w.y), 0.5f * (w.x - z.x));
  }
}

// Half spectrum along x -> real rows, scaled.  Z[Q][py][CO] (CO a multiple of 4)
// holds channels c0 .. c0+C-1 of the output X[py][px][Ctot] (c0 a multiple of 4);
// every other output channel is written as zero.  Block (output channel block, y).
// Channels 2l and 2l + 1 share one complex line W = X + i Y (each extended
// Hermitian, the imaginary parts of its u = 0 and u = P/2 terms dropped): the
// inverse transform's real and imaginary parts are the two real rows.
template <int R1, int R2, int KC, bool kVec>
__global__ void __launch_bounds__(mix_threads<R1, R2, KC / 2>())
    k_mix_rows_c2r(const float2 *__restrict__ Z, int py, int px, int Ctot, int c0, int C, int CO,
                   const float2 *__restrict__ tw, float scale, float *__restrict__ X) {
  constexpr int KH = KC / 2, P = R1 * R2, Q = P / 2 + 1;
  extern __shared__ float2 sm[];
  const int y = blockIdx.y, ob = blockIdx.x * KC;
  float *row = X + (size_t)y * px * Ctot + ob;
  const int cols = min(KC, Ctot - ob);
  auto put = [&](int x, int l, float2 v) {
    float *p = row + (size_t)x * Ctot + 2 * l;
    if (kVec) {
      if (2 * l < cols) *reinterpret_cast<float2 *>(p) = v;
    } else {
      if (2 * l < cols) p[0] = v.x;
      if (2 * l + 1 < cols) p[1] = v.y;
    }
  };
  if (ob >= c0 + C || ob + KC <= c0) {  // block entirely outside the band: zeros
    for (int i = threadIdx.x; i < px * KH; i += blockDim.x) put(i / KH, i % KH, make_float2(0.0f, 0.0f));
    return;
  }
  auto load = [&](int i2, int l, float2 (&v)[R1]) {
    const int z = ob + 2 * l - c0;  // even
    const bool okx = z >= 0 && z < C, oky = z >= 0 && z + 1 < C;
    float4 xy[R1];
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const int f = m * R2 + i2, fh = f < Q ? f : P - f;  // Hermitian source column
      xy[m] = okx ? *reinterpret_cast<const float4 *>(Z + ((size_t)fh * py + y) * CO + z)
                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const int f = m * R2 + i2;
      const float sg = f == 0 || f == (P >> 1) ? 0.0f : f < Q ? 1.0f : -1.0f;
      if (!oky) xy[m].z = xy[m].w = 0.0f;
      v[m] = make_float2(fmaf(-sg, xy[m].w, xy[m].x), fmaf(sg, xy[m].y, xy[m].z));
    }
  };
  auto store = [&](int x, int l, float2 v) {
    if (x < px) put(x, l, make_float2(v.x * scale, v.y * scale));  // channels outside the band transform zeros
  };
  mix_transform<R1, R2, KH, true>(sm, tw, load, store);
}

template <int R1, int R2, bool kVec>
oam_status rows_r2c(cudaStream_t st, const float *X, int py, int px, int Ctot, int c0, int C, int CO,
                    const float2 *tw, float2 *Y) {
  constexpr size_t sm = mix_smem<R1, R2, kRowCh / 2>();
  if (sm > 48 * 1024)
    OAM_CUDA_TRY(cudaFuncSetAttribute(k_mix_rows_r2c<R1, R2, kRowCh, kVec>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k_mix_rows_r2c<R1, R2, kRowCh, kVec>
      <<<dim3((C + kRowCh - 1) / kRowCh, py), mix_threads<R1, R2, kRowCh / 2>(), sm, st>>>(X, py, px, Ctot, c0, C, CO,
                                                                                          tw, Y);
  OAM_LAUNCHED();
  return OAM_OK;
}

template <int R1, int R2, bool kVec>
oam_status rows_c2r(cudaStream_t st, const float2 *Z, int py, int px, int Ctot, int c0, int C, int CO,
                    const float2 *tw, float scale, float *X) {
  constexpr size_t sm = mix_smem<R1, R2, kRowCh / 2>();
  if (sm > 48 * 1024)
    OAM_CUDA_TRY(cudaFuncSetAttribute(k_mix_rows_c2r<R1, R2, kRowCh, kVec>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k_mix_rows_c2r<R1, R2, kRowCh, kVec>
      <<<dim3((Ctot + kRowCh - 1) / kRowCh, py), mix_threads<R1, R2, kRowCh / 2>(), sm, st>>>(Z, py, px, Ctot, c0, C,
                                                                                             CO, tw, scale, X);
  OAM_LAUNCHED();
  return OAM_OK;
}

}  // namespace

oam_status oam::mix_rows_r2c(int P, cudaStream_t st, const float *X, int py, int px, int Ctot, int c0, int C, int CO,
                             const float2 *tw, float2 *Y) {
  const bool vec = Ctot % 2 == 0 && c0 % 2 == 0;
  switch (P) {
#define OAM_X(N, R1, R2)                                                          \
  case N:                                                                         \
    return vec ? rows_r2c<R1, R2, true>(st, X, py, px, Ctot, c0, C, CO, tw, Y)    \
               : rows_r2c<R1, R2, false>(st, X, py, px, Ctot, c0, C, CO, tw, Y);
    OAM_MIX_SIZES(OAM_X)
#undef OAM_X
  }
  return OAM_ERR_UNSUPPORTED;
}

oam_status oam::mix_rows_c2r(int P, cudaStream_t st, const float2 *Z, int py, int px, int Ctot, int c0, int C, int CO,
                             const float2 *tw, float scale, float *X) {
  const bool vec = Ctot % 2 == 0;
  switch (P) {
#define OAM_X(N, R1, R2)                                                                 \
  case N:                                                                                \
    return vec ? rows_c2r<R1, R2, true>(st, Z, py, px, Ctot, c0, C, CO, tw, scale, X)    \
               : rows_c2r<R1, R2, false>(st, Z, py, px, Ctot, c0, C, CO, tw, scale, X);
    OAM_MIX_SIZES(OAM_X)
#undef OAM_X
  }
  return OAM_ERR_UNSUPPORTED;
}
