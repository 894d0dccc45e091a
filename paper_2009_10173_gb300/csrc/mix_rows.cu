// Row transforms of the lateral-FFT form at the mixed-radix sizes (fft_mixed.cuh):
// real rows along x to the half spectrum, and back.
#include "fft_mixed.cuh"
#include "internal.cuh"

using namespace oam;
using namespace oam::mixfft;

namespace {

constexpr int kRowCh = 16;  // channels per block: eight complex lines of two real channels

// Real rows -> half spectrum along x.  X[py][px][Ctot] (channels c0 .. c0+C-1
// used), Y[Q][py][C] complex.  Block (channel block of KC, y).  Channels l and
// l + KC/2 ride as the real and imaginary parts of one complex line; with
// Z = FFT(x + i y), X(u) = (Z(u) + conj Z(-u)) / 2 and Y(u) = (Z(u) - conj Z(-u)) / 2i.
template <int R1, int R2, int KC>
__global__ void __launch_bounds__(mix_threads<R1, R2, KC / 2>())
    k_mix_rows_r2c(const float *__restrict__ X, int py, int px, int Ctot, int c0, int C, const float2 *__restrict__ tw,
                   float2 *__restrict__ Y) {
  constexpr int KH = KC / 2, P = R1 * R2, Q = P / 2 + 1, RS = mix_stride<R2, KH>();
  extern __shared__ float2 sm[];
  const int y = blockIdx.y, cb = blockIdx.x * KC;
  const float *row = X + (size_t)y * px * Ctot + c0 + cb;
  auto load = [&](int i2, int l, float2 (&v)[R1]) {
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const int x = m * R2 + i2;
      const float *p = row + (size_t)x * Ctot;
      v[m].x = x < px && cb + l < C ? p[l] : 0.0f;
      v[m].y = x < px && cb + l + KH < C ? p[l + KH] : 0.0f;
    }
  };
  auto keep = [&](int f, int l, float2 v) { sm[(f % R1) * RS + (f / R1) * KH + l] = v; };  // its own pass-2 slots
  mix_transform<R1, R2, KH, false>(sm, tw, load, keep);
  __syncthreads();
  for (int i = threadIdx.x; i < Q * KC; i += blockDim.x) {
    const int u = i / KC, c = i % KC, l = c % KH, un = u == 0 ? 0 : P - u;
    if (cb + c >= C) continue;
    const float2 z = sm[(u % R1) * RS + (u / R1) * KH + l], w = sm[(un % R1) * RS + (un / R1) * KH + l];
    Y[((size_t)u * py + y) * C + cb + c] = c < KH ? make_float2(0.5f * (z.x + w.x), 0.5f * (z.y - w.y))
                                                  : make_float2(0.5f * (z.y + w.y), 0.5f * (w.x - z.x));
  }
}

// Half spectrum along x -> real rows, scaled.  Z[Q][py][C] holds channels
// c0 .. c0+C-1 of the output X[py][px][Ctot]; every other output channel is
// written as zero.  Block (output channel block of KC, y).  Channels l and
// l + KC/2 share one complex line W = X + i Y (each extended Hermitian, the
// imaginary parts of its u = 0 and u = P/2 terms dropped): the inverse
// transform's real and imaginary parts are the two real rows.
template <int R1, int R2, int KC>
__global__ void __launch_bounds__(mix_threads<R1, R2, KC / 2>())
    k_mix_rows_c2r(const float2 *__restrict__ Z, int py, int px, int Ctot, int c0, int C,
                   const float2 *__restrict__ tw, float scale, float *__restrict__ X) {
  constexpr int KH = KC / 2, P = R1 * R2, Q = P / 2 + 1;
  extern __shared__ float2 sm[];
  const int y = blockIdx.y, ob = blockIdx.x * KC;
  float *row = X + (size_t)y * px * Ctot;
  if (ob >= c0 + C || ob + KC <= c0) {  // block entirely outside the band: zeros
    for (int i = threadIdx.x; i < px * KC; i += blockDim.x) {
      const int x = i / KC, c = i % KC;
      if (ob + c < Ctot) row[(size_t)x * Ctot + ob + c] = 0.0f;
    }
    return;
  }
  auto load = [&](int i2, int l, float2 (&v)[R1]) {
    const int zx = ob + l - c0, zy = ob + l + KH - c0;
    const bool okx = zx >= 0 && zx < C, oky = zy >= 0 && zy < C;
    float2 xs[R1], ys[R1];
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const int f = m * R2 + i2, fh = f < Q ? f : P - f;  // Hermitian source column
      const float2 *z = Z + ((size_t)fh * py + y) * C;
      xs[m] = okx ? z[zx] : make_float2(0.0f, 0.0f);
      ys[m] = oky ? z[zy] : make_float2(0.0f, 0.0f);
    }
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const int f = m * R2 + i2;
      const float sg = f == 0 || f == (P >> 1) ? 0.0f : f < Q ? 1.0f : -1.0f;
      v[m] = make_float2(fmaf(-sg, ys[m].y, xs[m].x), fmaf(sg, xs[m].y, ys[m].x));
    }
  };
  auto store = [&](int x, int l, float2 v) {
    if (x >= px) return;
    float *p = row + (size_t)x * Ctot;
    const int o0 = ob + l, o1 = ob + l + KH;
    if (o0 < Ctot) p[o0] = (o0 - c0 >= 0 && o0 - c0 < C) ? v.x * scale : 0.0f;
    if (o1 < Ctot) p[o1] = (o1 - c0 >= 0 && o1 - c0 < C) ? v.y * scale : 0.0f;
  };
  mix_transform<R1, R2, KH, true>(sm, tw, load, store);
}

template <int R1, int R2>
oam_status rows_r2c(cudaStream_t st, const float *X, int py, int px, int Ctot, int c0, int C, const float2 *tw,
                    float2 *Y) {
  constexpr size_t sm = mix_smem<R1, R2, kRowCh / 2>();
  static_assert(sm <= 48 * 1024, "default shared memory");
  k_mix_rows_r2c<R1, R2, kRowCh><<<dim3((C + kRowCh - 1) / kRowCh, py), mix_threads<R1, R2, kRowCh / 2>(), sm, st>>>(
      X, py, px, Ctot, c0, C, tw, Y);
  OAM_LAUNCHED();
  return OAM_OK;
}

template <int R1, int R2>
oam_status rows_c2r(cudaStream_t st, const float2 *Z, int py, int px, int Ctot, int c0, int C, const float2 *tw,
                    float scale, float *X) {
  constexpr size_t sm = mix_smem<R1, R2, kRowCh / 2>();
  k_mix_rows_c2r<R1, R2, kRowCh><<<dim3((Ctot + kRowCh - 1) / kRowCh, py), mix_threads<R1, R2, kRowCh / 2>(), sm,
                                   st>>>(Z, py, px, Ctot, c0, C, tw, scale, X);
  OAM_LAUNCHED();
  return OAM_OK;
}

}  // namespace

oam_status oam::mix_rows_r2c(int P, cudaStream_t st, const float *X, int py, int px, int Ctot, int c0, int C,
                             const float2 *tw, float2 *Y) {
  switch (P) {
#define OAM_X(N, R1, R2) \
  case N: return rows_r2c<R1, R2>(st, X, py, px, Ctot, c0, C, tw, Y);
    OAM_MIX_SIZES(OAM_X)
#undef OAM_X
  }
  return OAM_ERR_UNSUPPORTED;
}

oam_status oam::mix_rows_c2r(int P, cudaStream_t st, const float2 *Z, int py, int px, int Ctot, int c0, int C,
                             const float2 *tw, float scale, float *X) {
  switch (P) {
#define OAM_X(N, R1, R2) \
  case N: return rows_c2r<R1, R2>(st, Z, py, px, Ctot, c0, C, tw, scale, X);
    OAM_MIX_SIZES(OAM_X)
#undef OAM_X
  }
  return OAM_ERR_UNSUPPORTED;
}
