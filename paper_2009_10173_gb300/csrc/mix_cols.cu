// Column transforms of the lateral-FFT form at the mixed-radix sizes
// (fft_mixed.cuh), and the table of roots that every mixed-radix kernel reads.
#include <cmath>
#include <vector>

#include "fft_mixed.cuh"
#include "internal.cuh"

using namespace oam;
using namespace oam::mixfft;

namespace {

constexpr int kColCh = 16;  // complex channels per block

// Complex transform along the row index of Z[Q][nin][C] -> W[Q][nout][C]
// (rows >= nin read as zero, rows >= nout dropped).  Block (channel block, u).
template <int R1, int R2, int KC, bool kInverse>
__global__ void __launch_bounds__(mix_threads<R1, R2, KC>())
    k_mix_cols(const float2 *__restrict__ Z, int nin, int nout, int C, const float2 *__restrict__ tw,
               float2 *__restrict__ W) {
  extern __shared__ float2 sm[];
  const int u = blockIdx.y, cb = blockIdx.x * KC;
  const float2 *zin = Z + (size_t)u * nin * C + cb;
  float2 *wout = W + (size_t)u * nout * C + cb;
  auto load = [&](int i2, int l, float2 (&v)[R1]) {
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const int i = m * R2 + i2;
      v[m] = (i < nin && cb + l < C) ? zin[(size_t)i * C + l] : make_float2(0.0f, 0.0f);
    }
  };
  auto store = [&](int i, int l, float2 v) {
    if (i < nout && cb + l < C) wout[(size_t)i * C + l] = v;
  };
  mix_transform<R1, R2, KC, kInverse>(sm, tw, load, store);
}

template <int R1, int R2, bool kInverse>
oam_status cols(cudaStream_t st, const float2 *Z, int Q, int nin, int nout, int C, const float2 *tw, float2 *W) {
  constexpr size_t sm = mix_smem<R1, R2, kColCh>();
  if (sm > 48 * 1024)
    OAM_CUDA_TRY(cudaFuncSetAttribute(k_mix_cols<R1, R2, kColCh, kInverse>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k_mix_cols<R1, R2, kColCh, kInverse><<<dim3((C + kColCh - 1) / kColCh, Q), mix_threads<R1, R2, kColCh>(), sm, st>>>(
      Z, nin, nout, C, tw, W);
  OAM_LAUNCHED();
  return OAM_OK;
}

}  // namespace

oam_status oam::mix_cols(int P, bool inverse, cudaStream_t st, const float2 *Z, int nin, int nout, int C,
                         const float2 *tw, float2 *W) {
  const int Q = P / 2 + 1;
  switch (P) {
#define OAM_X(N, R1, R2)                                                      \
  case N:                                                                     \
    return inverse ? cols<R1, R2, true>(st, Z, Q, nin, nout, C, tw, W)        \
                   : cols<R1, R2, false>(st, Z, Q, nin, nout, C, tw, W);
    OAM_MIX_SIZES(OAM_X)
#undef OAM_X
  }
  return OAM_ERR_UNSUPPORTED;
}

// W_P^j = exp(-2 pi i j / P), j < P, rounded from FP64 (exact at the quarter turns).
std::vector<float2> oam::mix_roots(int P) {
  std::vector<float2> w(P);
  for (int j = 0; j < P; ++j) w[j] = make_float2((float)turn_cos(j, P), (float)-turn_sin(j, P));
  return w;
}
int oam::mix_size_for(int need) { return need <= kMixMax ? mix_size(need) : 0; }
