// Lateral-FFT form of the forward and adjoint operators (FP32).
//
// A and A^T are 2-D correlations of the single-position slab with the volume
// over the scan grid (Methods, Efficient reconstruction based on scanning
// symmetries: the model is the same for every scanning position).  With the
// volume and the signals zero-padded to P x P, P >= max(py, px) + R one of the
// mixed-radix transform sizes up to 512 or a power of two, no circular wrap
// reaches the output window, and the correlation theorem restates both operators
// exactly per lateral frequency (v, u):
//   A:    s^(v,u,n) = sum_k S^(v,u,k,n) H^(v,u,k)
//   A^T:  H^(v,u,k) = sum_n S^(v,u,k,n) s^(v,u,n)
// The slab is mirror-symmetric in both lateral offsets (the patch set is;
// Results, axial symmetry), so its lateral DFT
//   S^(v,u,k,n) = sum_{b,a} S[b][a][k][n] cos(2 pi v b / P) cos(2 pi u a / P)
// is real and even in v and in u (and symmetric in (v, u) when dx = dy), and
// conj(S^) = S^.  Ŝ is therefore stored once per frequency orbit
// {(+-v, +-u)} (and (u, v)), each orbit row holding, for every depth k, the
// union band of samples [klo_k, klo_k + klen_k) over all lateral offsets.
//
// One application is five launches: FFT along x of real rows (half spectrum
// u in [0, P/2]), FFT along y, the per-orbit banded real matrix times up to
// four complex frequency vectors, inverse FFT along y, inverse FFT along x
// back to real rows (Hermitian extension) with zero fill outside the band.
// The transforms keep their points in registers between trips through shared
// memory; every sum runs in a fixed order, so results are deterministic.
#include <algorithm>
#include <cmath>
#include <set>
#include <vector>

#include "f32x2.cuh"
#include "fft_dev.cuh"
#include "internal.cuh"

using namespace oam;

namespace oam {

// S^ for one direction: per frequency orbit a row of `stride` floats that holds, for
// each input element e (forward: depth, adjoint: sample), the outputs of the
// four-output groups [glo, ghi) that its band meets (zeros outside the band).
struct ApplyRows {
  int n_in = 0, n_out = 0;    // elements
  int windows = 0;            // 32-output windows
  long long stride = 0;       // floats per orbit row (a multiple of 4)
  int2 *d_elem = nullptr;     // [n_in] (float4 index of group 0 in the row, glo | ghi << 16)
  int2 *d_window = nullptr;   // [windows] input elements [x, y) whose groups meet the window
  float *d_s = nullptr;       // [n_rep][stride]
};

struct FftLayout {
  int P = 0, lgP = 0, Q = 0;  // transform size, its log2 (powers of two above 512), half-spectrum columns P/2 + 1
  int KC = 0;                 // channels per FFT block (power-of-two kernels)
  float2 *d_tw = nullptr;     // [P] roots W_P^j of the mixed-radix kernels; none for P > 512
  bool mixed = false;         // a mixed-radix size
  bool d4 = false;            // S^(v,u) = S^(u,v)
  int n_rep = 0;              // frequency orbits
  int n0 = 0, NS = 0;         // support: samples n0 .. n0 + NS - 1 (n0: n_lo rounded down to 4)
  int CZ = 0, CS = 0;         // channel strides of the work buffers: nz and NS rounded up to 4
  int4 *d_members = nullptr;  // [n_rep] half-spectrum indices u*P + v (-1 unused)
  ApplyRows rows[2];          // S^ by depth (forward), by sample (adjoint)
  float2 *d_w1 = nullptr, *d_w2 = nullptr;  // [Q][P][max(CZ, CS)] work buffers
  double flops = 0;                         // flops of one application (matrix part + FFTs)
  double bytes = 0;                         // device bytes read + written per application
};

}  // namespace oam

namespace {

using namespace oam::fftdev;

constexpr int kFftThreads = 256;
constexpr int kApplyWarps = 5;  // spectral products: warps per block
constexpr unsigned kAhead = 48 * 1024;  // bytes of a row prefetched to L2
constexpr int kUnroll = 4;      // 16-byte row loads per lane and step, two steps in flight
constexpr int kStep = 4 * kUnroll;  // input elements per step
constexpr int kBuildThreads = 128;


// ---- power-of-two transforms in register passes (P = 1024, 2048) -----------
// Sizes up to 512 run in the mixed-radix kernels (mix_rows.cu, mix_cols.cu).
// The kernels below run up to four stages per pass in registers: a forward transform is
// decimation in frequency (natural order in, bit-reversed out: the point at
// position i ends as frequency bitrev(i), which goes to global row bitrev(i)),
// an inverse transform decimation in time (position i loads frequency
// bitrev(i), natural order out), so no permutation pass is needed, the first
// pass reads global memory and the last writes it.  Passes cover stages
// k .. k + r - 1 (spans 2^k .. 2^(k+r-1)) with k a multiple of 4: the first
// forward pass has r0 = log2 P - 4 (ceil(log2 P / 4) - 1) stages, every other
// pass four.

// Shared-memory slot of point i of line l among KL lines: lines fastest, and
// for KL < 16 a pad of KL slots after every 16 points, so that the 16 lines x
// points a half-warp touches in a pass fall in distinct banks.
template <int KL>
__device__ __forceinline__ int xslot(int i, int l) {
  return i * KL + l + (KL < 16 ? (i >> 4) * KL : 0);
}
template <int KL>
__host__ __device__ constexpr size_t xslots(int P) {
  return (size_t)P * KL + (KL < 16 ? (size_t)(P >> 4) * KL : 0);
}

// One pass of r stages over the points i0 + m 2^k (m < 2^r) of each group
// (line l, q < 2^k, block blk; i0 = blk 2^(k+r) + q).  Forward (decimation in
// frequency, spans from large to small): span S = 2^(k+j) maps (u, w) at
// (n, n + S) to (u + w, (u - w) W_2S^(n mod S)), n mod S = q + (m mod 2^j) 2^k,
// twiddle W_2S^q W_2^(j+1)^(m mod 2^j), the first factor a power of
// b = W_2^(k+r)^q (one sincospif, then squarings).  Inverse (decimation in
// time, spans from small to large, sign +1): (u, w) go to (u + w conj(W),
// u - w conj(W)).  src(i, l) yields point i before the pass, dst(i, l, v)
// takes it after.
template <int KL, int r, bool kForward, class Src, class Dst>
__device__ __forceinline__ void xpass(int P, int k, Src src, Dst dst) {
  constexpr int R = 1 << r;
  const int groups = P >> r;
  for (int id = threadIdx.x; id < groups * KL; id += blockDim.x) {
    const int l = id % KL, t = id / KL;
    const int q = t & ((1 << k) - 1), blk = t >> k;
    const int i0 = (blk << (k + r)) | q;
    float2 v[R];
#pragma unroll
    for (int m = 0; m < R; ++m) v[m] = src(i0 + (m << k), l);
    float2 pw[r];
    sincospif(-2.0f * (float)q / (float)(1 << (k + r)), &pw[r - 1].y, &pw[r - 1].x);
#pragma unroll
    for (int j = r - 2; j >= 0; --j) pw[j] = cmul(pw[j + 1], pw[j + 1]);
    if (kForward) {
#pragma unroll
      for (int j = r - 1; j >= 0; --j) {
        const int S = 1 << j;
#pragma unroll
        for (int m = 0; m < R; ++m) {
          if (m & S) continue;
          const float2 u = v[m], w = v[m + S];
          v[m] = make_float2(u.x + w.x, u.y + w.y);
          const int um = m & (S - 1);
          const float2 tw = um == 0 ? pw[j] : cmul(pw[j], w16(2 * S, um));
          v[m + S] = cmul(make_float2(u.x - w.x, u.y - w.y), tw);
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < r; ++j) {
        const int S = 1 << j;
#pragma unroll
        for (int m = 0; m < R; ++m) {
          if (m & S) continue;
          const int um = m & (S - 1);
          const float2 tw = um == 0 ? pw[j] : cmul(pw[j], w16(2 * S, um));
          const float2 u = v[m], w = cmul(v[m + S], make_float2(tw.x, -tw.y));
          v[m] = make_float2(u.x + w.x, u.y + w.y);
          v[m + S] = make_float2(u.x - w.x, u.y - w.y);
        }
      }
    }
#pragma unroll
    for (int m = 0; m < R; ++m) dst(i0 + (m << k), l, v[m]);
  }
}

// A whole transform of KL lines of P = 2^lgP points (lgP 10 or 11: one pass of two or
// three stages and two of four) through the shared slots `a`: `first` reads the input
// (forward: natural point i; inverse: the point at position i, i.e. frequency bitrev(i)),
// `last` takes position i's result (forward: frequency bitrev(i); inverse: point i).  With
// kLastToSmem the last pass writes the slots too (followed by a barrier) and `last` is not
// called.
template <int KL, bool kForward, bool kLastToSmem, class First, class Last>
__device__ __forceinline__ void xtransform(float2 *a, int P, int lgP, First first, Last last) {
  auto from_smem = [&](int i, int l) { return a[xslot<KL>(i, l)]; };
  auto to_smem = [&](int i, int l, float2 v) { a[xslot<KL>(i, l)] = v; };
  auto short_pass = [&](auto src, auto dst) {  // stages 8 and up
    if (lgP == 10) xpass<KL, 2, kForward>(P, 8, src, dst);
    else xpass<KL, 3, kForward>(P, 8, src, dst);
  };
  if (kForward) short_pass(first, to_smem);
  else xpass<KL, 4, kForward>(P, 0, first, to_smem);
  __syncthreads();
  xpass<KL, 4, kForward>(P, 4, from_smem, to_smem);
  __syncthreads();
  if constexpr (kForward) {
    if constexpr (kLastToSmem) xpass<KL, 4, kForward>(P, 0, from_smem, to_smem);
    else xpass<KL, 4, kForward>(P, 0, from_smem, last);
  } else {
    short_pass(from_smem, last);
  }
  if (kLastToSmem) __syncthreads();
}

// Real rows -> half spectrum along x (arguments and results as k_mix_rows_r2c).
template <int KC>
__global__ void __launch_bounds__(kFftThreads) k_xfft_rows_r2c(const float *__restrict__ X, int py, int px, int Ctot,
                                                               int c0, int C, int CO, int P, int lgP, int Q,
                                                               float2 *__restrict__ Y) {
  constexpr int KH = KC / 2;
  extern __shared__ float2 sm[];
  float2 *a = sm;
  const int y = blockIdx.x, cb = blockIdx.y * KC;
  const float *row = X + (size_t)y * px * Ctot + c0 + cb;
  auto load = [&](int x, int l) {
    float re = 0.0f, im = 0.0f;
    if (x < px) {
      const float *p = row + (size_t)x * Ctot;
      if (cb + l < C) re = p[l];
      if (cb + l + KH < C) im = p[l + KH];
    }
    return make_float2(re, im);
  };
  auto none = [](int, int, float2) {};
  xtransform<KH, true, true>(a, P, lgP, load, none);
  for (int i = threadIdx.x; i < Q * KC; i += blockDim.x) {
    const int u = i / KC, c = i % KC, l = c % KH;
    if (cb + c >= C) continue;
    const float2 z = a[xslot<KH>(bitrev(u, lgP), l)], w = a[xslot<KH>(bitrev((P - u) & (P - 1), lgP), l)];
    Y[((size_t)u * py + y) * CO + cb + c] = c < KH ? make_float2(0.5f * (z.x + w.x), 0.5f * (z.y - w.y))
                                                  : make_float2(0.5f * (z.y + w.y), 0.5f * (w.x - z.x));
  }
}

// Complex transform along the row index (as k_mix_cols).
template <int KC, bool kInverse>
__global__ void __launch_bounds__(kFftThreads) k_xfft_cols(const float2 *__restrict__ Z, int nin, int nout, int C,
                                                           int P, int lgP, float2 *__restrict__ W) {
  extern __shared__ float2 sm[];
  const int u = blockIdx.x, cb = blockIdx.y * KC;
  const float2 *zin = Z + (size_t)u * nin * C + cb;
  float2 *wout = W + (size_t)u * nout * C + cb;
  auto load = [&](int i, int l) {
    const int row = kInverse ? bitrev(i, lgP) : i;
    return (row < nin && cb + l < C) ? zin[(size_t)row * C + l] : make_float2(0.0f, 0.0f);
  };
  auto store = [&](int i, int l, float2 v) {
    const int row = kInverse ? i : bitrev(i, lgP);
    if (row < nout && cb + l < C) wout[(size_t)row * C + l] = v;
  };
  xtransform<KC, !kInverse, false>(sm, P, lgP, load, store);
}

// Half spectrum along x -> real rows (as k_mix_rows_c2r).
template <int KC>
__global__ void __launch_bounds__(kFftThreads) k_xfft_rows_c2r(const float2 *__restrict__ Z, int py, int px, int Ctot,
                                                               int c0, int C, int CO, int P, int lgP, int Q,
                                                               float scale, float *__restrict__ X) {
  constexpr int KH = KC / 2;
  extern __shared__ float2 sm[];
  const int y = blockIdx.x, ob = blockIdx.y * KC;
  if (ob >= c0 + C || ob + KC <= c0) {  // block entirely outside the band: zeros
    for (int i = threadIdx.x; i < px * KC; i += blockDim.x) {
      const int x = i / KC, c = i % KC;
      if (ob + c < Ctot) X[((size_t)y * px + x) * Ctot + ob + c] = 0.0f;
    }
    return;
  }
  // position i takes frequency f = bitrev(i) of W = X + i Y, the two real
  // channels' Hermitian-extended spectra (imaginary parts of f = 0, P/2 dropped)
  auto load = [&](int i, int l) {
    const int f = bitrev(i, lgP);
    const int fh = f < Q ? f : P - f;
    float2 xs = make_float2(0.0f, 0.0f), ys = make_float2(0.0f, 0.0f);
    const int zx = ob + l - c0, zy = ob + l + KH - c0;
    if (zx >= 0 && zx < C) xs = Z[((size_t)fh * py + y) * CO + zx];
    if (zy >= 0 && zy < C) ys = Z[((size_t)fh * py + y) * CO + zy];
    if (f == 0 || f == (P >> 1)) {
      xs.y = 0.0f;
      ys.y = 0.0f;
    } else if (f >= Q) {
      xs.y = -xs.y;
      ys.y = -ys.y;
    }
    return make_float2(xs.x - ys.y, xs.y + ys.x);
  };
  auto store = [&](int x, int l, float2 v) {
    if (x >= px) return;
    float *p = X + ((size_t)y * px + x) * Ctot;
    const int o0 = ob + l, o1 = ob + l + KH;
    if (o0 < Ctot) p[o0] = (o0 - c0 >= 0 && o0 - c0 < C) ? v.x * scale : 0.0f;
    if (o1 < Ctot) p[o1] = (o1 - c0 >= 0 && o1 - c0 < C) ? v.y * scale : 0.0f;
  };
  xtransform<KH, false, false>(sm, P, lgP, load, store);
}

// Spectral products of one frequency orbit r and direction: out_f[o] = sum_e S^_r[e][o]
// in_f[e] for the orbit's up to four member frequencies f.  A warp serves a window of
// 32 outputs: lanes hold eight groups of four outputs, their four quarters walk
// interleaved input elements of the window's range; a lane reads its four outputs'
// S^ with one 16-byte load and multiplies them with the element's four complex values
// from shared memory as packed (re, im) pairs.
//
// What bounds it: reading S^ once from HBM.  Four outputs per load and packed products
// take 7 issue slots per S^ value instead of 20 (a lane per output, scalar loads), and
// the next step's loads are issued before this step's products.  200x200x300 (0.77 GB),
// cold caches: 200 us forward, 191 adjoint (3.9 TB/s), against 270 and 217 for the scalar
// form with its own kernel per direction.  What remains is the loads' latency at 20 warps
// per SM (registers); a block therefore starts by asking L2 for the first 48 KB of its row:
// a whole application 338 -> 321 us (adjoint 316 -> 309), 256x256x384 573 -> 547 (522 ->
// 512), 128x128x192 123 -> 119, 64x64x128 41 both.  24 KB give 327 and 559, 64 KB 331 and
// 566.  Asking for whole rows or for the rows of later blocks evicts the vectors (adjoint
// 256x256x384 547, 652), loading S^ as evict-first loses what L2 keeps of it (forward 349).

// Sums over the quarters of a warp's [output][member] sums; quarter ph keeps member ph.
__device__ __forceinline__ void sum_quarters(const uint64_t (&acc)[4][4], int ph, uint64_t (&c)[4]) {
  const bool hi = ph & 2, odd = ph & 1;
  uint64_t b[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
      b[i][j] = f2_add(hi ? acc[i][2 + j] : acc[i][j],
                     __shfl_xor_sync(0xffffffffu, hi ? acc[i][j] : acc[i][2 + j], 16));
#pragma unroll
  for (int i = 0; i < 4; ++i)
    c[i] = f2_add(odd ? b[i][1] : b[i][0], __shfl_xor_sync(0xffffffffu, odd ? b[i][0] : b[i][1], 8));
}
// Eight FP32 values' exponents below the largest.
__device__ __forceinline__ bool all_finite(const uint64_t (&c)[4]) {
  bool ok = true;
#pragma unroll
  for (int i = 0; i < 4; ++i) ok = ok && (~c[i] & 0x7f800000u) && (~c[i] >> 32 & 0x7f800000u);
  return ok;
}

__global__ void __launch_bounds__(32 * kApplyWarps, 4)
    k_fft_apply(const float *__restrict__ S, long long stride, const int4 *__restrict__ members,
                const int2 *__restrict__ elem, const int2 *__restrict__ window, int windows, int n_in, int in_stride,
                int n_out, int out_stride, const float2 *__restrict__ in, float2 *__restrict__ out) {
  extern __shared__ ulonglong2 sma[];
  // members (0, 1) and (2, 3) as (re, im) pairs; kStep elements beyond the last meet no output
  ulonglong2 *X = sma;                                            // [n_in + kStep][2]
  int2 *E = reinterpret_cast<int2 *>(X + 2 * (n_in + kStep));     // [n_in + kStep]
  const int r = blockIdx.x;
  const float4 *row = reinterpret_cast<const float4 *>(S + (size_t)r * stride);
  if (threadIdx.x == 0)  // the row's start to L2, under the loads of the vectors
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(row),
                 "r"((unsigned)min(stride * (long long)sizeof(float), (long long)kAhead))
                 : "memory");
  const int4 mem = members[r];
  {
    float2 *X2 = reinterpret_cast<float2 *>(X);
    const float2 z = make_float2(0.0f, 0.0f);
    for (int e = threadIdx.x; e < n_in + kStep; e += blockDim.x) {
      const bool ok = e < n_in;
      const float2 x0 = ok && mem.x >= 0 ? in[(size_t)mem.x * in_stride + e] : z;
      const float2 x1 = ok && mem.y >= 0 ? in[(size_t)mem.y * in_stride + e] : z;
      const float2 x2 = ok && mem.z >= 0 ? in[(size_t)mem.z * in_stride + e] : z;
      const float2 x3 = ok && mem.w >= 0 ? in[(size_t)mem.w * in_stride + e] : z;
      X2[4 * e] = x0;
      X2[4 * e + 1] = x1;
      X2[4 * e + 2] = x2;
      X2[4 * e + 3] = x3;
      E[e] = ok ? elem[e] : make_int2(0, 0);
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, ph = lane >> 3;
  for (int w = threadIdx.x >> 5; w < windows; w += blockDim.x >> 5) {
    const int g = 8 * w + (lane & 7);
    const int2 win = window[w];
    uint64_t acc[4][4];  // [output][member]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0;
    auto load = [&](int e) {
      const int2 d = E[e];
      const bool in_band = g >= (d.y & 0xffff) && g < (int)((unsigned)d.y >> 16);
      return in_band ? __ldg(row + d.x + g) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto add = [&](int e, float4 v) {
      const ulonglong2 h0 = X[2 * e], h1 = X[2 * e + 1];
      const uint64_t h[4] = {h0.x, h0.y, h1.x, h1.y}, s[4] = {f2_splat(v.x), f2_splat(v.y), f2_splat(v.z), f2_splat(v.w)};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = f2_fma(s[i], h[j], acc[i][j]);
    };
    // the next step's loads are issued before this step's products
    float4 v[kUnroll], next[kUnroll];
#pragma unroll
    for (int q = 0; q < kUnroll; ++q) v[q] = load(win.x + 4 * q + ph);
    for (int e0 = win.x; e0 < win.y; e0 += kStep) {
      const bool more = e0 + kStep < win.y;
#pragma unroll
      for (int q = 0; q < kUnroll; ++q)
        next[q] = more ? load(e0 + kStep + 4 * q + ph) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int q = 0; q < kUnroll; ++q) add(e0 + 4 * q + ph, v[q]);
#pragma unroll
      for (int q = 0; q < kUnroll; ++q) v[q] = next[q];
    }
    // sum the quarters, each keeping the member of its number
    uint64_t c[4];
    sum_quarters(acc, ph, c);
    // A lane added zeros for the elements that do not meet its group; where the sums are
    // not finite they are taken again without those elements, so that a non-finite one
    // reaches no sample beyond its band's groups.  (1 to 3 us of an application; predicated
    // products cost 10 %, a look at the vectors while they are loaded 2 to 4 %.)
    if (__any_sync(0xffffffffu, !all_finite(c))) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0;
      for (int e = win.x + ph; e < win.y; e += 4)
        if (g >= (E[e].y & 0xffff) && g < (int)((unsigned)E[e].y >> 16)) add(e, load(e));
      __syncwarp();
      sum_quarters(acc, ph, c);
    }
    const int f = ph == 0 ? mem.x : ph == 1 ? mem.y : ph == 2 ? mem.z : mem.w;
    if (f >= 0 && 4 * g < n_out) {  // whole groups: out_stride is a multiple of 4
      ulonglong2 *o = reinterpret_cast<ulonglong2 *>(out + (size_t)f * out_stride + 4 * g);
      o[0] = make_ulonglong2(c[0], c[1]);
      o[1] = make_ulonglong2(c[2], c[3]);
    }
  }
}

// ---------------------------------------------------------------- S^ build
// Pass 1: T[b'][u][e] = sum_{a'=0..R} w_a' cos(2 pi u a' / P) S[b'][a'][k_e][n_e]
// for every row entry e = (k_e, n_e); w_0 = 1, w_{>0} = 2 (the +-a' pair).
// Block (entry block, b').  tw: the roots rounded from FP64 (none above 512 points):
// cospif of a rounded 2 m / P, exact for powers of two alone, is off by up to 2e-7.
__device__ __forceinline__ void load_cosines(float *cosT, const float2 *tw, int P) {
  for (int m = threadIdx.x; m < P; m += blockDim.x) cosT[m] = tw ? tw[m].x : cospif(2.0f * (float)m / (float)P);
  __syncthreads();
}
__global__ void __launch_bounds__(kBuildThreads) k_shat_pass1(const float *__restrict__ band,
                                                              const int *__restrict__ band_lo,
                                                              const int *__restrict__ band_hi, int band_w,
                                                              const int *__restrict__ tap_orbit, int R, int W,
                                                              int nz, const int2 *__restrict__ entry_kn,
                                                              long long row_len, int P, int Q,
                                                              const float2 *__restrict__ tw, float *__restrict__ T) {
  extern __shared__ float smb[];
  float *cosT = smb;           // [P]
  float *sv = smb + P;         // [R+1][blockDim]: weighted slab values of this thread's entry
  load_cosines(cosT, tw, P);
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int bp = blockIdx.y;
  if (e >= row_len) return;
  const int2 kn = entry_kn[e];
  const int ts = blockDim.x, tid = threadIdx.x;
  for (int ap = 0; ap <= R; ++ap) {
    const int o = tap_orbit[(bp + R) * W + (ap + R)];
    const int lo = band_lo[o * nz + kn.x], hi = band_hi[o * nz + kn.x];
    float v = 0.0f;
    if (kn.y >= lo && kn.y < hi) v = band[((size_t)o * nz + kn.x) * band_w + (kn.y - lo)];
    sv[ap * ts + tid] = ap == 0 ? v : 2.0f * v;
  }
  for (int u = 0; u < Q; ++u) {
    float acc = 0.0f;
    for (int ap = 0, j = 0; ap <= R; ++ap) {  // j = u ap mod P
      acc = fmaf(cosT[j], sv[ap * ts + tid], acc);
      j += u;
      if (j >= P) j -= P;
    }
    T[((size_t)bp * Q + u) * row_len + e] = acc;
  }
}

// Pass 2: S^[r][e] = sum_{b'=0..R} w_b' cos(2 pi v0 b' / P) T[b'][u0][e] for
// every orbit r = (v0, u0) with this u0.  Block (entry block, u0).
__global__ void __launch_bounds__(kBuildThreads) k_shat_pass2(const float *__restrict__ T, long long row_len, int R,
                                                              int P, int Q, const float2 *__restrict__ tw,
                                                              const int *__restrict__ rep_of,
                                                              const int2 *__restrict__ entry_kn, int n0,
                                                              const int2 *__restrict__ by_depth,
                                                              const int2 *__restrict__ by_sample,
                                                              long long stride, long long stride_t,
                                                              float *__restrict__ shat, float *__restrict__ shat_t) {
  extern __shared__ float smb[];
  float *cosT = smb;    // [P]
  float *tv = smb + P;  // [R+1][blockDim]
  load_cosines(cosT, tw, P);
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int u0 = blockIdx.y;
  if (e >= row_len) return;
  const int ts = blockDim.x, tid = threadIdx.x;
  for (int bp = 0; bp <= R; ++bp) {
    const float t = T[((size_t)bp * Q + u0) * row_len + e];
    tv[bp * ts + tid] = bp == 0 ? t : 2.0f * t;
  }
  const int2 kn = entry_kn[e];
  const int jn = kn.y - n0;
  const long long ef = 4LL * by_depth[kn.x].x + jn, et = 4LL * by_sample[jn].x + kn.x;  // its place in the two rows
  for (int v0 = 0; v0 < Q; ++v0) {
    const int r = rep_of[v0 * Q + u0];
    if (r < 0) continue;
    float acc = 0.0f;
    for (int bp = 0, j = 0; bp <= R; ++bp) {  // j = v0 bp mod P
      acc = fmaf(cosT[j], tv[bp * ts + tid], acc);
      j += v0;
      if (j >= P) j -= P;
    }
    shat[(size_t)r * stride + ef] = acc;
    shat_t[(size_t)r * stride_t + et] = acc;
  }
}

// Host tables of the lateral-FFT layout, planned from the model's bands.
struct FftPlan {
  std::vector<int2> elem[2], window[2], entry_kn;  // entry_kn: (depth, sample) of the S^ entries of an orbit
  std::vector<int> rep_of;
  std::vector<int4> members;
};

// Row layout of one direction: lo[e] .. hi[e] - 1 are the outputs that element e meets.
void plan_apply(const std::vector<int> &lo, const std::vector<int> &hi, int n_out, ApplyRows *A,
                std::vector<int2> *elem, std::vector<int2> *window) {
  A->n_in = (int)lo.size();
  A->n_out = n_out;
  A->windows = (n_out + 31) / 32;
  elem->assign(A->n_in, make_int2(0, 0));
  window->assign(A->windows, make_int2(A->n_in, 0));
  int used = 0;  // groups
  for (int e = 0; e < A->n_in; ++e) {
    if (hi[e] <= lo[e]) continue;
    const int glo = lo[e] / 4, ghi = (hi[e] + 3) / 4;
    (*elem)[e] = make_int2(used - glo, glo | (ghi << 16));
    used += ghi - glo;
    for (int w = glo / 8; w <= (ghi - 1) / 8; ++w) {
      (*window)[w].x = std::min((*window)[w].x, e);
      (*window)[w].y = e + 1;
    }
  }
  for (int2 &w : *window)
    if (w.y <= w.x) w = make_int2(0, 0);
  A->stride = 4LL * std::max(used, 1);
}

// Fill L's sizes and the host tables (no device call).
oam_status fft_plan(const oam_model *m, FftLayout *L, FftPlan &pl) {
  const int R = m->R, W = m->W, nz = m->grid.nz;
  // The transform size is the smallest mixed-radix one that the scan and its
  // halo fit (S^ grows with its square: 96 for 64 positions and R = 30, 160
  // for 128, 288 for 256); beyond 512 the next power of two.
  const int need = std::max(m->grid.py, m->grid.px) + R;
  int P = mix_size_for(need), lgP = 0;
  L->mixed = P > 0;
  if (!P) {
    P = 1024;
    lgP = 10;
    while (P < need) {
      P <<= 1;
      ++lgP;
    }
  }
  if (P > 2048) return OAM_ERR_UNSUPPORTED;
  L->P = P;
  L->lgP = lgP;
  L->Q = P / 2 + 1;
  L->KC = 4096 / P;  // power-of-two kernels: 4 or 2
  const int Q = L->Q;
  // D4 when the tap -> orbit map is symmetric under b <-> a
  L->d4 = true;
  for (int b = -R; b <= R && L->d4; ++b)
    for (int a = -R; a <= R; ++a)
      if (m->h_tap_orbit[(b + R) * W + (a + R)] != m->h_tap_orbit[(a + R) * W + (b + R)]) {
        L->d4 = false;
        break;
      }
  // union band per depth over all orbits, and the depths per sample
  L->n0 = m->n_lo & ~3;
  L->NS = std::max(1, m->n_hi - L->n0);
  L->CZ = (nz + 3) & ~3;
  L->CS = (L->NS + 3) & ~3;
  std::vector<int> klo(nz, 0), khi(nz, 0), slo(L->NS, nz), shi(L->NS, 0);  // samples from n0
  pl.entry_kn.clear();
  for (int k = 0; k < nz; ++k) {
    int lo = 1 << 30, hi = -1;
    for (int o = 0; o < m->n_orb; ++o) {
      const int bl = m->h_band_lo[(size_t)o * nz + k], bh = m->h_band_hi[(size_t)o * nz + k];
      if (bh > bl) {
        lo = std::min(lo, bl);
        hi = std::max(hi, bh);
      }
    }
    if (hi <= lo) continue;
    klo[k] = lo - L->n0;
    khi[k] = hi - L->n0;
    for (int j = klo[k]; j < khi[k]; ++j) {
      slo[j] = std::min(slo[j], k);
      shi[j] = k + 1;
      pl.entry_kn.push_back(make_int2(k, L->n0 + j));
    }
  }
  if (pl.entry_kn.empty()) pl.entry_kn.push_back(make_int2(0, L->n0));  // an empty slab: one zero entry
  if (nz > 4 * 65535 || L->NS > 4 * 65535) return OAM_ERR_UNSUPPORTED;  // 16-bit group indices (beyond the API's sizes)
  plan_apply(klo, khi, L->NS, &L->rows[0], &pl.elem[0], &pl.window[0]);
  plan_apply(slo, shi, nz, &L->rows[1], &pl.elem[1], &pl.window[1]);
  // frequency orbits and their members in the half spectrum (index u*P + v)
  std::vector<int> &rep_of = pl.rep_of;
  std::vector<int4> &members = pl.members;
  rep_of.assign((size_t)Q * Q, -1);
  members.clear();
  long long covered = 0;
  for (int u0 = 0; u0 < Q; ++u0)
    for (int v0 = 0; v0 < (L->d4 ? u0 + 1 : Q); ++v0) {
      std::set<int> fs;
      for (int v : {v0, (P - v0) % P}) fs.insert(u0 * P + v);
      if (L->d4)
        for (int v : {u0, (P - u0) % P}) fs.insert(v0 * P + v);
      int4 mm = make_int4(-1, -1, -1, -1);
      int *slot = &mm.x;
      int i = 0;
      for (int f : fs) slot[i++] = f;
      covered += i;
      rep_of[(size_t)v0 * Q + u0] = (int)members.size();
      members.push_back(mm);
    }
  if (covered != (long long)Q * P) return OAM_ERR_DEVICE;  // orbit plan must cover the half spectrum once
  L->n_rep = (int)members.size();
  return OAM_OK;
}

// Device bytes fft_build allocates and keeps (host only).
oam_status fft_layout_bytes(const FftLayout &L, const FftPlan &pl, size_t *bytes) {
  size_t b = (L.mixed ? alloc_bytes<float2>(L.P) : 0) + alloc_bytes<int4>(pl.members.size()) +
             2 * alloc_bytes<float2>((size_t)L.Q * L.P * std::max(L.CZ, L.CS));
  for (const ApplyRows &A : L.rows)
    b += alloc_bytes<int2>(A.n_in) + alloc_bytes<int2>(A.windows) + alloc_bytes<float>((size_t)L.n_rep * A.stride);
  *bytes = b;
  return OAM_OK;
}

}  // namespace

oam_status oam::fft_plan_bytes(const oam_model *m, size_t *bytes) {
  FftLayout L;
  FftPlan pl;
  oam_status rc = fft_plan(m, &L, pl);
  if (rc) return rc;
  return fft_layout_bytes(L, pl, bytes);
}

oam_status oam::fft_build(oam_model *m, cudaStream_t st) {
  const int R = m->R, W = m->W, nz = m->grid.nz;
  FftLayout *L = new (std::nothrow) FftLayout();
  if (!L) return OAM_ERR_OOM;
  m->fft = L;
  FftPlan pl;
  {
    oam_status rc0 = fft_plan(m, L, pl);
    if (rc0) return rc0;
  }
  const int P = L->P, Q = L->Q;
  const std::vector<int> &rep_of = pl.rep_of;
  const std::vector<int2> &entry_kn = pl.entry_kn;
  const std::vector<int4> &members = pl.members;
  const long long entries = (long long)entry_kn.size();
  oam_status rc;
  const size_t chan = (size_t)Q * P * std::max(L->CZ, L->CS);
  if ((rc = dev_alloc(m, &L->d_members, members.size())) || (rc = dev_alloc(m, &L->d_w1, chan)) ||
      (rc = dev_alloc(m, &L->d_w2, chan)))
    return rc;
  std::vector<float2> roots;
  if (L->mixed) {
    if ((rc = dev_alloc(m, &L->d_tw, (size_t)P))) return rc;
    roots = mix_roots(P);
    OAM_CUDA_TRY(cudaMemcpyAsync(L->d_tw, roots.data(), sizeof(float2) * P, cudaMemcpyHostToDevice, st));
  }
  OAM_CUDA_TRY(cudaMemcpyAsync(L->d_members, members.data(), sizeof(int4) * members.size(), cudaMemcpyHostToDevice,
                               st));
  for (int d = 0; d < 2; ++d) {
    ApplyRows &A = L->rows[d];
    if ((rc = dev_alloc(m, &A.d_elem, (size_t)A.n_in)) || (rc = dev_alloc(m, &A.d_window, (size_t)A.windows)) ||
        (rc = dev_alloc(m, &A.d_s, (size_t)L->n_rep * A.stride)))
      return rc;
    OAM_CUDA_TRY(cudaMemcpyAsync(A.d_elem, pl.elem[d].data(), sizeof(int2) * A.n_in, cudaMemcpyHostToDevice, st));
    OAM_CUDA_TRY(
        cudaMemcpyAsync(A.d_window, pl.window[d].data(), sizeof(int2) * A.windows, cudaMemcpyHostToDevice, st));
    // outputs of a group that the element's band does not meet stay zero
    OAM_CUDA_TRY(cudaMemsetAsync(A.d_s, 0, sizeof(float) * (size_t)L->n_rep * A.stride, st));
  }
  // build S^ (temporaries: entry table, band_hi, rep table, T)
  int2 *d_entry = nullptr;
  int *d_band_hi = nullptr, *d_rep_of = nullptr;
  float *d_T = nullptr;
  const size_t nb = (size_t)m->n_orb * nz;
  if (cudaMallocAsync((void **)&d_entry, sizeof(int2) * entry_kn.size(), st) != cudaSuccess ||
      cudaMallocAsync((void **)&d_band_hi, sizeof(int) * nb, st) != cudaSuccess ||
      cudaMallocAsync((void **)&d_rep_of, sizeof(int) * rep_of.size(), st) != cudaSuccess ||
      cudaMallocAsync((void **)&d_T, sizeof(float) * (size_t)(R + 1) * Q * entries, st) != cudaSuccess) {
    cudaGetLastError();
    if (d_entry) cudaFreeAsync(d_entry, st);
    if (d_band_hi) cudaFreeAsync(d_band_hi, st);
    if (d_rep_of) cudaFreeAsync(d_rep_of, st);
    if (d_T) cudaFreeAsync(d_T, st);
    return OAM_ERR_OOM;
  }
  cudaMemcpyAsync(d_entry, entry_kn.data(), sizeof(int2) * entry_kn.size(), cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(d_band_hi, m->h_band_hi.data(), sizeof(int) * nb, cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(d_rep_of, rep_of.data(), sizeof(int) * rep_of.size(), cudaMemcpyHostToDevice, st);
  const unsigned eblocks = (unsigned)((entries + kBuildThreads - 1) / kBuildThreads);
  const size_t sb = sizeof(float) * ((size_t)P + (size_t)(R + 1) * kBuildThreads);
  if (sb > 48 * 1024) {  // one limit for every model: builds from several threads would lower each other's
    const int limit = std::max<int>((int)sb, 227 * 1024);
    OAM_CUDA_TRY(cudaFuncSetAttribute(k_shat_pass1, cudaFuncAttributeMaxDynamicSharedMemorySize, limit));
    OAM_CUDA_TRY(cudaFuncSetAttribute(k_shat_pass2, cudaFuncAttributeMaxDynamicSharedMemorySize, limit));
  }
  k_shat_pass1<<<dim3(eblocks, R + 1), kBuildThreads, sb, st>>>(
      m->d_band, m->d_band_lo, d_band_hi, m->band_w, m->d_tap_orbit, R, W, nz, d_entry, entries, P, Q, L->d_tw, d_T);
  OAM_LAUNCHED();
  k_shat_pass2<<<dim3(eblocks, Q), kBuildThreads, sb, st>>>(d_T, entries, R, P, Q, L->d_tw, d_rep_of, d_entry, L->n0,
                                                            L->rows[0].d_elem, L->rows[1].d_elem, L->rows[0].stride,
                                                            L->rows[1].stride, L->rows[0].d_s, L->rows[1].d_s);
  OAM_LAUNCHED();
  OAM_CUDA_TRY(cudaStreamSynchronize(st));  // host tables above go out of scope
  cudaFreeAsync(d_entry, st);
  cudaFreeAsync(d_band_hi, st);
  cudaFreeAsync(d_rep_of, st);
  cudaFreeAsync(d_T, st);
  // cost of one application: the banded matrix over all member frequencies
  // (real x complex: 4 flops per entry) and 5 N log2 N per complex transform
  const double half = (double)Q * P;
  const double fft_lines = (double)m->grid.py * m->grid.nz + half / P * m->grid.nz + half / P * L->NS +
                           (double)m->grid.py * L->NS;
  L->flops = 4.0 * half * (double)entries + 5.0 * P * std::log2((double)P) * fft_lines;
  const double c8 = sizeof(float2);
  L->bytes = 4.0 * (double)L->n_rep * entries +                              // S^
             4.0 * vol_elems(m) + 4.0 * (double)m->grid.py * m->grid.px * m->grid.nt +  // input, output
             c8 * Q * m->grid.py * (nz + L->NS) * 2 +                            // row-transform buffers
             c8 * half * (nz + L->NS) * 2;                                       // column-transform buffers
  return OAM_OK;
}

void oam::fft_free(oam_model *m, cudaStream_t st) {
  FftLayout *L = m->fft;
  if (!L) return;
  for (void *p : {(void *)L->d_tw, (void *)L->d_members, (void *)L->d_w1, (void *)L->d_w2})
    if (p) cudaFreeAsync(p, st);
  for (ApplyRows &A : L->rows)
    for (void *p : {(void *)A.d_elem, (void *)A.d_window, (void *)A.d_s})
      if (p) cudaFreeAsync(p, st);
  delete L;
  m->fft = nullptr;
}

double oam::fft_flops(const oam_model *m) { return m->fft ? m->fft->flops : 0.0; }
double oam::fft_bytes(const oam_model *m) { return m->fft ? m->fft->bytes : 0.0; }

namespace {

oam_status set_smem(const void *fn, size_t bytes) {
  if (bytes > 48 * 1024)
    OAM_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  return OAM_OK;
}

}  // namespace

namespace {

// Threads for a register-pass transform block: one per group of the
// four-stage passes (KL lines x P/16 groups), 64 to 256.
int xthreads(int P, int KL) { return std::max(64, std::min(kFftThreads, (((P >> 4) * KL + 31) / 32) * 32)); }

// The transforms of one application, KC channels per block; the spectral
// products are launched by run_fft between them.  Register passes (P = 1024, 2048).
template <int KC>
struct XKernels {
  static oam_status rows_r2c(const FftLayout *L, cudaStream_t st, const float *X, int py, int px, int Ctot, int c0,
                             int C, int CO, float2 *Y) {
    const size_t sm = sizeof(float2) * xslots<KC / 2>(L->P);
    oam_status rc = set_smem((const void *)k_xfft_rows_r2c<KC>, sm);
    if (rc) return rc;
    k_xfft_rows_r2c<KC><<<dim3(py, (C + KC - 1) / KC), xthreads(L->P, KC / 2), sm, st>>>(
        X, py, px, Ctot, c0, C, CO, L->P, L->lgP, L->Q, Y);
    OAM_LAUNCHED();
    return OAM_OK;
  }
  template <bool kInverse>
  static oam_status cols(const FftLayout *L, cudaStream_t st, const float2 *Z, int nin, int nout, int C, float2 *W) {
    const size_t sm = sizeof(float2) * xslots<KC>(L->P);
    oam_status rc = set_smem((const void *)k_xfft_cols<KC, kInverse>, sm);
    if (rc) return rc;
    k_xfft_cols<KC, kInverse><<<dim3(L->Q, (C + KC - 1) / KC), xthreads(L->P, KC), sm, st>>>(Z, nin, nout, C, L->P,
                                                                                            L->lgP, W);
    OAM_LAUNCHED();
    return OAM_OK;
  }
  static oam_status rows_c2r(const FftLayout *L, cudaStream_t st, const float2 *Z, int py, int px, int Ctot, int c0,
                             int C, int CO, float scale, float *X) {
    const size_t sm = sizeof(float2) * xslots<KC / 2>(L->P);
    oam_status rc = set_smem((const void *)k_xfft_rows_c2r<KC>, sm);
    if (rc) return rc;
    k_xfft_rows_c2r<KC><<<dim3(py, (Ctot + KC - 1) / KC), xthreads(L->P, KC / 2), sm, st>>>(
        Z, py, px, Ctot, c0, C, CO, L->P, L->lgP, L->Q, scale, X);
    OAM_LAUNCHED();
    return OAM_OK;
  }
};

// The same in the mixed-radix kernels (P <= 512).
struct MKernels {
  static oam_status rows_r2c(const FftLayout *L, cudaStream_t st, const float *X, int py, int px, int Ctot, int c0,
                             int C, int CO, float2 *Y) {
    return mix_rows_r2c(L->P, st, X, py, px, Ctot, c0, C, CO, L->d_tw, Y);
  }
  template <bool kInverse>
  static oam_status cols(const FftLayout *L, cudaStream_t st, const float2 *Z, int nin, int nout, int C, float2 *W) {
    return mix_cols(L->P, kInverse, st, Z, nin, nout, C, L->d_tw, W);
  }
  static oam_status rows_c2r(const FftLayout *L, cudaStream_t st, const float2 *Z, int py, int px, int Ctot, int c0,
                             int C, int CO, float scale, float *X) {
    return mix_rows_c2r(L->P, st, Z, py, px, Ctot, c0, C, CO, L->d_tw, scale, X);
  }
};

template <class K>
oam_status run_fft(const oam_model *m, const FftLayout *L, bool fwd, const float *in, float *out, cudaStream_t st) {
  const int P = L->P, nz = m->grid.nz, nt = m->grid.nt, py = m->grid.py, px = m->grid.px, NS = L->NS;
  const float scale = 1.0f / ((float)P * (float)P);
  const ApplyRows &A = L->rows[fwd ? 0 : 1];
  // input and output: row lengths, first channels, channels and work-buffer strides
  const int il = fwd ? nz : nt, i0 = fwd ? 0 : L->n0, ic = fwd ? nz : NS, is = fwd ? L->CZ : L->CS;
  const int ol = fwd ? nt : nz, o0 = fwd ? L->n0 : 0, oc = fwd ? NS : nz, os = fwd ? L->CS : L->CZ;
  oam_status rc;
  if ((rc = K::rows_r2c(L, st, in, py, px, il, i0, ic, is, L->d_w2))) return rc;
  if ((rc = K::template cols<false>(L, st, L->d_w2, py, P, is, L->d_w1))) return rc;
  const size_t sa = (2 * sizeof(ulonglong2) + sizeof(int2)) * (A.n_in + kStep);
  // both directions and every model share the kernel: one limit for all, or calls from several threads would
  // lower each other's between setting it and the launch
  if (sa > 48 * 1024 && (rc = set_smem((const void *)k_fft_apply, std::max<size_t>(sa, 227 * 1024)))) return rc;
  const int rounds = (A.windows + kApplyWarps - 1) / kApplyWarps, warps = (A.windows + rounds - 1) / rounds;
  k_fft_apply<<<L->n_rep, 32 * warps, sa, st>>>(A.d_s, A.stride, L->d_members, A.d_elem, A.d_window, A.windows,
                                                A.n_in, is, A.n_out, os, L->d_w1, L->d_w2);
  OAM_LAUNCHED();
  if ((rc = K::template cols<true>(L, st, L->d_w2, P, py, os, L->d_w1))) return rc;
  return K::rows_c2r(L, st, L->d_w1, py, px, ol, o0, oc, os, scale, out);
}

oam_status run_fft_any(const oam_model *m, bool fwd, const float *in, float *out, cudaStream_t st) {
  const FftLayout *L = m->fft;
  if (!L) return OAM_ERR_UNSUPPORTED;
  ProfScope prof(m, st, fwd);
  if (L->d_tw) return run_fft<MKernels>(m, L, fwd, in, out, st);
  return L->KC == 4 ? run_fft<XKernels<4>>(m, L, fwd, in, out, st) : run_fft<XKernels<2>>(m, L, fwd, in, out, st);
}

}  // namespace

oam_status oam::forward_fft(const oam_model *m, const float *H, float *s, cudaStream_t st) {
  return run_fft_any(m, true, H, s, st);
}

oam_status oam::adjoint_fft(const oam_model *m, const float *s, float *H, cudaStream_t st) {
  return run_fft_any(m, false, s, H, st);
}
