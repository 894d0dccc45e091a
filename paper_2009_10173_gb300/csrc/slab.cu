// Model slab builder (Methods, Forward modeling, Eqs. 1-4): per-orbit bands
// of the single-position model, and the FP32 operator layouts packed from them.
//
// Distances use the cancellation-free form d - F = (2F r.n + |r|^2) / (d + F)
// in FP64, so the arrival sample fs*(d/c - t0) = (fs/c)(d - F) + fs(F/c - t0)
// keeps full precision; the EIR derivative, a polynomial in the fraction of a sample
// between an arrival and its nearest sample, is summed over patches as moments
// (k_slab_moments), or evaluated in FP32 per patch (k_slab_values).
#include <algorithm>
#include <climits>
#include <cmath>

#include "internal.cuh"

using namespace oam;

namespace {

struct Geo {
  double F, dx, dy, dz, z0;
  double ks;      // fs / c, samples per metre
  double G;       // fs * (F/c - t0)
  double cut;     // truncation, samples
  float inv2s2;   // 1 / (2 sigma_s^2)
  float env2;     // log2(e) / (2 sigma_s^2): envelope exp(-tau^2 / (2 sigma_s^2)) = 2^(-env2 tau^2)
  float invs2;    // 1 / sigma_s^2
  float omega;    // 2 pi fc / fs
  float cyc;      // 2 fc / fs: the phase omega * tau in units of pi
};

// d - F for the voxel at lateral offset (a dx, b dy), depth k, and patch normal n.
__device__ __forceinline__ double delta_dist(const Geo &g, int b, int a, int k, Patch p) {
  double rx = a * g.dx, ry = b * g.dy, rz = g.z0 + k * g.dz;
  double rn = __dadd_rn(__dadd_rn(__dmul_rn(rx, p.x), __dmul_rn(ry, p.y)), __dmul_rn(rz, p.z));
  double r2 = __dadd_rn(__dadd_rn(__dmul_rn(rx, rx), __dmul_rn(ry, ry)), __dmul_rn(rz, rz));
  double num = __dadd_rn(__dmul_rn(2.0 * g.F, rn), r2);
  double d = sqrt(__dadd_rn(__dmul_rn(g.F, g.F), num));
  return __ddiv_rn(num, __dadd_rn(d, g.F));
}

// ---------------------------------------------------------------- double-word FP32
// A pair (h, l) of floats with |l| <= ulp(h)/2 carries about 48 significand
// bits, enough for patch arrivals to 1e-11 samples, at FP32 instruction rates
// (this GPU's FP64 rate is far lower).  Error-free transforms and the add,
// multiply, divide and square-root steps follow Joldes, Muller and Popescu,
// "Tight and rigorous error bounds for basic building blocks of double-word
// arithmetic" (ACM TOMS 2017); the _rn intrinsics keep the compiler from
// contracting or reordering them.
struct DW {
  float h, l;
};
__device__ __forceinline__ DW fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ DW two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), ap = __fsub_rn(s, b), bp = __fsub_rn(s, ap);
  return {s, __fadd_rn(__fsub_rn(a, ap), __fsub_rn(b, bp))};
}
__device__ __forceinline__ DW two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ DW dw_add(DW x, DW y) {
  const DW s = two_sum(x.h, y.h), t = two_sum(x.l, y.l);
  const DW v = fast_two_sum(s.h, __fadd_rn(s.l, t.h));
  return fast_two_sum(v.h, __fadd_rn(t.l, v.l));
}
__device__ __forceinline__ DW dw_mul(DW x, DW y) {
  const DW c = two_prod(x.h, y.h);
  const float t = __fmaf_rn(x.l, y.h, __fmaf_rn(x.h, y.l, __fmul_rn(x.l, y.l)));
  return fast_two_sum(c.h, __fadd_rn(c.l, t));
}
__device__ __forceinline__ DW dw_mul_f(DW x, float y) {
  const DW c = two_prod(x.h, y);
  const DW t = fast_two_sum(c.h, __fmul_rn(x.l, y));
  return fast_two_sum(t.h, __fadd_rn(t.l, c.l));
}
__device__ __forceinline__ DW dw_div(DW x, DW y) {
  const float th = __fdiv_rn(x.h, y.h);
  const DW r = dw_mul_f(y, th);
  const float d = __fadd_rn(__fsub_rn(x.h, r.h), __fsub_rn(x.l, r.l));
  return fast_two_sum(th, __fdiv_rn(d, y.h));
}
__device__ __forceinline__ DW dw_sqrt(DW x) {  // x > 0: one Newton step from the FP32 root
  const float s = __fsqrt_rn(x.h);
  const float e = __fadd_rn(__fmaf_rn(-s, s, x.h), x.l);
  return fast_two_sum(s, __fdiv_rn(e, __fmul_rn(2.0f, s)));
}
__device__ __forceinline__ DW to_dw(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}

// Patch normal as double words and weight in mm^2 per metre of distance.
struct __align__(32) PatchDW {
  float xh, xl, yh, yl, zh, zl, w, pad;
};

__global__ void k_patch_dw(const Patch *__restrict__ patch, int M, PatchDW *__restrict__ out) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < M; j += gridDim.x * blockDim.x) {
    const Patch p = patch[j];
    const DW x = to_dw(p.x), y = to_dw(p.y), z = to_dw(p.z);
    out[j] = PatchDW{x.h, x.l, y.h, y.l, z.h, z.l, (float)(p.w * 1e-3), 0.0f};
  }
}

// d - F in plain FP32 (same cancellation-free form).  Its error is below
// 4e-7 |r|, r the voxel offset (|d - F| <= |r|).
__device__ __forceinline__ float delta_dist_f(float rx, float ry, float rz, float r2, float F, const PatchDW &p) {
  const float rn = rx * p.xh + ry * p.yh + rz * p.zh;
  const float num = 2.0f * F * rn + r2;
  const float d = sqrtf(F * F + num);
  return num / (d + F);
}

template <bool kMax>
__device__ __forceinline__ float block_ext(float v, float *sh) {
  for (int off = 16; off; off >>= 1) {
    const float o = __shfl_xor_sync(0xffffffffu, v, off);
    v = kMax ? fmaxf(v, o) : fminf(v, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  v = sh[0];
  for (int i = 1; i < (int)(blockDim.x >> 5); ++i) v = kMax ? fmaxf(v, sh[i]) : fminf(v, sh[i]);
  return v;
}

// Per (orbit, depth): min and max of d - F over the patches, exactly as FP64
// evaluates them.  Plain FP32 distances locate the extremes; only patches
// within 1e-5 |r| of the FP32 extremes (a bound 25x the FP32 error) are
// evaluated in FP64, so the true FP64 extremes are always among them.
__global__ void k_delta_range(Geo g, const Patch *__restrict__ patch, const PatchDW *__restrict__ pdw, int M,
                              const int *orb_b, const int *orb_a, int nz, double2 *out) {
  __shared__ float shf[32];
  __shared__ double slo[32], shi[32];
  const int o = blockIdx.x, k = blockIdx.y;
  const int b = orb_b[o], a = orb_a[o];
  const double rxd = a * g.dx, ryd = b * g.dy, rzd = g.z0 + k * g.dz;
  const float rx = (float)rxd, ry = (float)ryd, rz = (float)rzd;
  const float r2 = (float)(rxd * rxd + ryd * ryd + rzd * rzd), F = (float)g.F;
  float lo32 = INFINITY, hi32 = -INFINITY;
  for (int j = threadIdx.x; j < M; j += blockDim.x) {
    const float dd = delta_dist_f(rx, ry, rz, r2, F, pdw[j]);
    lo32 = fminf(lo32, dd);
    hi32 = fmaxf(hi32, dd);
  }
  lo32 = block_ext<false>(lo32, shf);
  hi32 = block_ext<true>(hi32, shf);
  const float tol = 1e-5f * sqrtf(r2);
  double lo = INFINITY, hi = -INFINITY;
  for (int j = threadIdx.x; j < M; j += blockDim.x) {
    const float dd = delta_dist_f(rx, ry, rz, r2, F, pdw[j]);
    if (dd <= lo32 + tol || dd >= hi32 - tol) {
      const double d64 = delta_dist(g, b, a, k, patch[j]);
      if (dd <= lo32 + tol) lo = fmin(lo, d64);
      if (dd >= hi32 - tol) hi = fmax(hi, d64);
    }
  }
  for (int off = 16; off; off >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, off));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, off));
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    slo[w] = lo;
    shi[w] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) {
      lo = fmin(lo, slo[i]);
      hi = fmax(hi, shi[i]);
    }
    out[o * nz + k] = make_double2(lo, hi);
  }
}

// ---------------------------------------------------------------- trilinear voxels
// The paper's discretisation of Eq. 1 (Methods, Forward modeling): the
// surface integral of the trilinear interpolation of the voxel values, and a
// central finite difference in time.  A voxel is the tent
// L(x/dx) L(y/dy) L(z/dz), L(u) = max(0, 1 - |u|); across its support the
// sphere |x - x'| = ct is a plane, so the integral is the tent's planar
// Radon transform along e = (v - q)/|v - q|: the hats of half-width
// a = |e_i| d_i (area d_i) convolve, i.e. a six-box spline
//   sum over sign vectors s of prod(s) (u + sum s_i c_i/2)_+^5 / 5!,
// with an axis whose a < 1e-3 max(a) taken as a spike of mass d_i.  FP64:
// the signed sum cancels heavily.
__device__ double tent_radon(double dx, double dy, double dz, double ex, double ey, double ez, double u) {
  const double d[3] = {dx, dy, dz}, e[3] = {fabs(ex), fabs(ey), fabs(ez)};
  double a[3], amax = 0.0;
  for (int i = 0; i < 3; ++i) {
    a[i] = e[i] * d[i];
    amax = fmax(amax, a[i]);
  }
  double c[6], scale = 1.0;
  int n = 0;
  for (int i = 0; i < 3; ++i) {
    if (a[i] < 1e-3 * amax) {
      scale *= d[i];
    } else {
      c[n++] = a[i];
      c[n++] = a[i];
      scale *= d[i] / (a[i] * a[i]);
    }
  }
  double fact = 1.0;
  for (int i = 2; i < n; ++i) fact *= i;
  double sum = 0.0;
  for (int mask = 0; mask < (1 << n); ++mask) {
    double x = u, sign = 1.0;
    for (int i = 0; i < n; ++i) {
      if (mask & (1 << i)) {
        x -= 0.5 * c[i];
        sign = -sign;
      } else {
        x += 0.5 * c[i];
      }
    }
    if (x > 0.0) {
      double pw = 1.0;
      for (int q = 1; q < n; ++q) pw *= x;
      sum += sign * pw;
    }
  }
  return scale * sum / fact;
}

struct Geo33 {
  double F, dx, dy, dz, z0;  // mm
  double c;                  // mm / s
  double fs, t0;             // Hz, s
  double sigma, omega;       // EIR in samples: std dev, rad per sample
  int T;                     // EIR taps each side (whole samples within the cut)
  int len;                   // samples of a patch's finite-difference support held per patch
};

constexpr int k33Chunk = 128;  // patches per shared-memory chunk

// Block (orbit o, depth k): band values S[o][k][lo .. hi) =
//   sum_j w_j sum_m e(n - m) D_j(m),  D_j(m) = (I_j(m+1) - I_j(m-1)) / 2,
//   I_j(m) = R_j(c t_m - r_j) / (c t_m),  t_m = t0 + m / fs,
// patches in index order, each patch's sum over m first (FP64 throughout).
__global__ void k_slab33_values(Geo33 g, const Patch *__restrict__ patch, int M, const int *orb_b, const int *orb_a,
                                int nz, int nt, const int *band_lo, const int *band_hi, int band_w,
                                float *__restrict__ band) {
  extern __shared__ double sm33[];
  double *e = sm33;                           // [2T + 1]
  double *D = e + 2 * g.T + 1;                // [k33Chunk][len]
  int *m0s = reinterpret_cast<int *>(D + (size_t)k33Chunk * g.len);  // [k33Chunk]
  double *ws = reinterpret_cast<double *>(m0s + k33Chunk + (k33Chunk & 1));  // [k33Chunk] (8-byte aligned)
  const int o = blockIdx.x, k = blockIdx.y;
  const double vx = orb_a[o] * g.dx, vy = orb_b[o] * g.dy, vz = g.z0 + k * g.dz;
  const int lo = band_lo[(size_t)o * nz + k], hi = band_hi[(size_t)o * nz + k];
  for (int i = threadIdx.x; i <= 2 * g.T; i += blockDim.x) {
    const double tau = i - g.T;
    e[i] = exp(-tau * tau / (2.0 * g.sigma * g.sigma)) * cos(g.omega * tau);
  }
  constexpr int kPer = 4;  // band samples per thread (band_w <= 4 * blockDim)
  double acc[kPer];
#pragma unroll
  for (int q = 0; q < kPer; ++q) acc[q] = 0.0;
  const double h = g.dx + g.dy + g.dz;
  for (int j0 = 0; j0 < M; j0 += k33Chunk) {
    __syncthreads();
    for (int i = threadIdx.x; i < k33Chunk; i += blockDim.x) {
      const int j = j0 + i;
      if (j >= M) {
        m0s[i] = INT_MIN / 2;
        continue;
      }
      const Patch pj = patch[j];
      const double ux = vx + g.F * pj.x, uy = vy + g.F * pj.y, uz = vz + g.F * pj.z;  // v - q, q = -F n
      const double r = sqrt(ux * ux + uy * uy + uz * uz);
      const double ex = ux / r, ey = uy / r, ez = uz / r;
      const int m0 = (int)floor(g.fs * ((r - h) / g.c - g.t0)) - 1;
      m0s[i] = m0;
      ws[i] = pj.w;
      for (int q = 0; q < g.len; ++q) {
        const int m = m0 + q;
        double dv = 0.0;
        if (m >= -1 && m <= nt) {
          const double rho1 = g.c * (g.t0 + (m + 1) / g.fs), rho0 = g.c * (g.t0 + (m - 1) / g.fs);
          const double i1 = tent_radon(g.dx, g.dy, g.dz, ex, ey, ez, rho1 - r) / rho1;
          const double i0 = tent_radon(g.dx, g.dy, g.dz, ex, ey, ez, rho0 - r) / rho0;
          dv = 0.5 * (i1 - i0);
        }
        D[(size_t)i * g.len + q] = dv;
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int n = lo + threadIdx.x + q * blockDim.x;
      if (n >= hi) continue;
      for (int i = 0; i < k33Chunk; ++i) {
        const int m0 = m0s[i];
        if (n < m0 - g.T || n > m0 + g.len - 1 + g.T) continue;
        double sj = 0.0;
        for (int qq = 0; qq < g.len; ++qq) {
          const int dm = n - (m0 + qq);
          if (dm >= -g.T && dm <= g.T) sj += e[dm + g.T] * D[(size_t)i * g.len + qq];
        }
        acc[q] += ws[i] * sj;
      }
    }
  }
  float *row = band + ((size_t)o * nz + k) * band_w;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int i = threadIdx.x + q * blockDim.x;
    if (i < band_w) row[i] = lo + i < hi ? (float)acc[q] : 0.0f;
  }
}

constexpr int kPatchChunk = 512;

// Band values: thread i of block (o, k) owns sample lo + i (+ blockDim.x ...).
// Each patch's arrival D = (fs/c)(d - F) + fs(F/c - t0) (samples, double-word
// FP32, ~1e-11 samples) is split into the nearest sample n_ref and a fraction
// f = D - n_ref in [-1/2, 1/2], so tau = (n - n_ref) - f is the FP32 rounding
// of the offset.  The phase omega*tau is a rotation: the patch's own
// (cos, sin)(-omega f) turned by a table entry (cos, sin)(omega t) for the
// integer t = n - n_ref (|t| <= cut + 1/2); both arguments are small, so the
// result stays within a few ulp.  The envelope is exp2 of a pre-scaled
// argument and the patch sum is a compensated (Kahan) FP32 sum.  Patches are
// visited in index order, so every entry is a fixed-order sum.
__global__ void k_slab_values(Geo g, const PatchDW *__restrict__ pdw, int M, const int *orb_b,
                              const int *orb_a, int nz, const int *band_lo, const int *band_hi,
                              int band_w, int T0, float *band) {
  extern __shared__ float2 rot[];  // [2 T0 + 1]: (cos, sin)(omega t), t = -T0 .. T0
  const int o = blockIdx.x, k = blockIdx.y;
  const int b = orb_b[o], a = orb_a[o];
  const int lo = band_lo[o * nz + k], hi = band_hi[o * nz + k];
  __shared__ float4 sP[kPatchChunk];  // (n_ref, f, cos(omega f), -sin(omega f))
  __shared__ float sW[kPatchChunk];
  for (int t = threadIdx.x; t <= 2 * T0; t += blockDim.x) {
    float sn, cs;
    sincospif(g.cyc * (float)(t - T0), &sn, &cs);
    rot[t] = make_float2(cs, sn);
  }
  const int per = (band_w + blockDim.x - 1) / blockDim.x;  // samples per thread (<= 4)
  const float cut = (float)g.cut;
  float sum[4] = {0, 0, 0, 0}, comp[4] = {0, 0, 0, 0};
  // block constants as double words (voxel offset, |r|^2, F, 2F, F^2, fs/c, G)
  const double rxd = a * g.dx, ryd = b * g.dy, rzd = g.z0 + k * g.dz;
  const DW rx = to_dw(rxd), ry = to_dw(ryd), rz = to_dw(rzd), r2 = to_dw(rxd * rxd + ryd * ryd + rzd * rzd);
  const DW Fw = to_dw(g.F), F2w = to_dw(2.0 * g.F), FFw = to_dw(g.F * g.F), ks = to_dw(g.ks), G = to_dw(g.G);
  for (int j0 = 0; j0 < M; j0 += kPatchChunk) {
    const int cnt = min(kPatchChunk, M - j0);
    __syncthreads();
    for (int j = threadIdx.x; j < cnt; j += blockDim.x) {
      const PatchDW p = pdw[j0 + j];
      const DW rn = dw_add(dw_add(dw_mul(rx, DW{p.xh, p.xl}), dw_mul(ry, DW{p.yh, p.yl})), dw_mul(rz, DW{p.zh, p.zl}));
      const DW num = dw_add(dw_mul(F2w, rn), r2);
      const DW d = dw_sqrt(dw_add(FFw, num));
      const DW dd = dw_div(num, dw_add(d, Fw));        // d - F, metres
      const DW D = dw_add(dw_mul(ks, dd), G);           // arrival, samples
      const float nr = rintf(D.h);
      const float f = __fadd_rn(__fsub_rn(D.h, nr), D.l);  // D.h - nr is exact
      float sn, cs;
      sincospif(g.cyc * f, &sn, &cs);
      sP[j] = make_float4(nr, f, cs, -sn);
      sW[j] = __fdiv_rn(p.w, dw_add(Fw, dd).h);         // (mm^2 / 1e3) / metres = mm^2 / mm
    }
    __syncthreads();
    for (int r = 0; r < per; ++r) {
      const int n = lo + threadIdx.x + r * blockDim.x;
      if (n >= hi) break;
      const float nf = (float)n;
      float s = sum[r], c = comp[r];
      for (int j = 0; j < cnt; ++j) {
        const float4 q = sP[j];
        const float t = nf - q.x;  // exact integer
        const float tau = t - q.y;
        if (fabsf(tau) <= cut) {
          const float2 e = rot[__float2int_rn(t) + T0];  // |t| <= cut + 1/2 < T0
          const float cs = e.x * q.z - e.y * q.w;        // cos(omega t - omega f)
          const float sn = e.y * q.z + e.x * q.w;        // sin(omega t - omega f)
          const float env = exp2f(-tau * tau * g.env2);
          const float v = -env * (tau * g.invs2 * cs + g.omega * sn);
          const float y = sW[j] * v - c;
          const float u = s + y;
          c = (u - s) - y;
          s = u;
        }
      }
      sum[r] = s;
      comp[r] = c;
    }
  }
  float *row = band + ((size_t)o * nz + k) * band_w;
  for (int r = 0; r < per; ++r) {
    const int i = threadIdx.x + r * blockDim.x;
    if (i >= band_w) break;
    const int n = lo + i;
    row[i] = (n < hi) ? sum[r] - comp[r] : 0.0f;
  }
}

// ---------------------------------------------------------------- band values by moments
// The same sums with a few instructions per patch instead of thirty per (patch, sample)
// pair: for an integer offset t from the nearest sample the pulse is a polynomial in
// the fraction, v(t - x/2) = sum_p c_p(t) x^p for x = 2f in [-1, 1], so a sample needs of
// the patches whose nearest sample is b (a bin) only their moments sum_j w_j x_j^p:
//   S[n] = sum_b sum_p c_p(n - b) mom[b][p].
// The truncation |tau| <= cut splits a bin only at t = +-tb, the one integer within half
// a sample of it; the truncated sums of those two offsets are two more moments.  There x
// is compared with the edge itself: t - f against the cut, rounded, lets single patches
// in or out (1.7e-6 of the slab at a cut of three deviations, here 2.5e-8).
//
// Per chunk of patches: arrivals; a stable counting sort by bin (warps own index ranges,
// equal bins within 32 patches are ranked by match_any); threads sum segments of kSeg
// patches of a bin (Kahan), and the segments are added in order as double words.
// Everything is a fixed-order sum, and every product that matters is a double-word one,
// so the result is nearer to the exact sum than adding the patches' FP32 values.
//
// What bounds it: issue slots, about evenly in the arrivals, the segments and the last
// sums (each pair took 30 slots, and half of the lanes' samples are out of a patch's
// reach).  Model build, 2000 patches, 61x61 taps, and the slab's error against FP64,
// from k_slab_values: 192 depths 19.9 -> 8.2 ms, 8.2e-8 -> 3.0e-8; 300 depths 31.4 ->
// 12.9 ms, 9.9e-8 -> 3.5e-8; 384 depths 40.0 -> 16.5 ms, 9.7e-8 -> 3.6e-8; 48 depths,
// 11x11 taps 0.66 -> 0.42 ms.
constexpr int kMom = 12;       // monomials
constexpr int kMomAll = kMom + 2;
constexpr int kMomFull = 6;    // the first of them in double words in the last sum
constexpr int kMomChunk = 1024;
constexpr int kMomThreads = 128;
constexpr int kSeg = 16;

struct MomShape {
  int tb;      // edge offset
  float edge;  // least x with |tb - x / 2| <= cut
  int B0, nb;  // first bin's sample - lo, and most bins
};
size_t mom_smem(const MomShape &s) {
  const size_t segs = kMomChunk / kSeg + s.nb;
  return sizeof(float2) * ((size_t)(2 * s.tb + 1) * kMom + kMomChunk + (segs + s.nb) * kMomAll) +
         sizeof(int) * (size_t)(4 * s.nb + 2 * (s.nb + 1) + segs);
}

__device__ __forceinline__ void kahan(float &s, float &c, float v) {
  const float y = __fsub_rn(v, c), u = __fadd_rn(s, y);
  c = __fsub_rn(__fsub_rn(u, s), y);
  s = u;
}

__global__ void __launch_bounds__(kMomThreads, 4)
    k_slab_moments(Geo g, const PatchDW *__restrict__ pdw, int M, const int *orb_b, const int *orb_a, int nz,
                   const int *band_lo, const int *band_hi, int band_w, MomShape ms, const float2 *__restrict__ coef_g,
                   float *__restrict__ band) {
  extern __shared__ float2 smm[];
  const int tb = ms.tb, nbm = ms.nb, segm = kMomChunk / kSeg + nbm;
  float2 *coef = smm;                                // [2 tb + 1][kMom] (high, low)
  float2 *sorted = coef + (2 * tb + 1) * kMom;       // [kMomChunk] (x, w)
  float2 *part = sorted + kMomChunk;                 // [segm][kMomAll] (sum, compensation)
  float2 *mom = part + segm * kMomAll;               // [nbm][kMomAll] (high, low)
  int *place = reinterpret_cast<int *>(mom + nbm * kMomAll);  // [4][nbm] counts, then places
  int *start = place + 4 * nbm;                      // [nbm + 1] a bin's first patch in `sorted`
  int *seg0 = start + nbm + 1;                       // [nbm + 1] and first segment
  int *seg_bin = seg0 + nbm + 1;                     // [segm]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int o = blockIdx.x, k = blockIdx.y;
  const int b = orb_b[o], a = orb_a[o];
  const int lo = band_lo[o * nz + k], hi = band_hi[o * nz + k];
  const int nb = max(1, min(nbm, hi - lo - 2 * ms.B0 + 1));  // bins in use
  for (int i = tid; i < (2 * tb + 1) * kMom; i += kMomThreads) coef[i] = coef_g[i];
  for (int i = tid; i < nbm * kMomAll; i += kMomThreads) mom[i] = make_float2(0.0f, 0.0f);
  const double rxd = a * g.dx, ryd = b * g.dy, rzd = g.z0 + k * g.dz;
  const DW rx = to_dw(rxd), ry = to_dw(ryd), rz = to_dw(rzd), r2 = to_dw(rxd * rxd + ryd * ryd + rzd * rzd);
  const DW Fw = to_dw(g.F), F2w = to_dw(2.0 * g.F), FFw = to_dw(g.F * g.F), ks = to_dw(g.ks), G = to_dw(g.G);
  for (int j0 = 0; j0 < M; j0 += kMomChunk) {
    const int cnt = min(kMomChunk, M - j0);
    __syncthreads();
    for (int i = tid; i < 4 * nbm; i += kMomThreads) place[i] = 0;
    __syncthreads();
    // arrivals, and each patch's place among its warp's patches of its bin
    constexpr int kIter = kMomChunk / kMomThreads;
    int at[kIter];     // bin | place << 16, -1: none
    float2 xw[kIter];
#pragma unroll
    for (int i = 0; i < kIter; ++i) {
      const int j = (warp * kIter + i) * 32 + lane;
      int bin = -1;
      xw[i] = make_float2(0.0f, 0.0f);
      if (j < cnt) {
        const PatchDW p = pdw[j0 + j];
        const DW rn = dw_add(dw_add(dw_mul(rx, DW{p.xh, p.xl}), dw_mul(ry, DW{p.yh, p.yl})), dw_mul(rz, DW{p.zh, p.zl}));
        const DW num = dw_add(dw_mul(F2w, rn), r2);
        const DW d = dw_sqrt(dw_add(FFw, num));
        const DW dd = dw_div(num, dw_add(d, Fw));  // d - F, metres
        const DW D = dw_add(dw_mul(ks, dd), G);    // arrival, samples
        const float nr = rintf(D.h);
        const float f = __fadd_rn(__fsub_rn(D.h, nr), D.l);  // D.h - nr is exact
        bin = __float2int_rn(nr) - lo - ms.B0;
        if (bin < 0 || bin >= nb) bin = -1;  // meets no sample of the band
        xw[i] = make_float2(2.0f * f, __fdiv_rn(p.w, dw_add(Fw, dd).h));  // (mm^2 / 1e3) / metres = mm^2 / mm
      }
      const unsigned same = __match_any_sync(0xffffffffu, bin);
      const int rank = __popc(same & ((1u << lane) - 1u));
      at[i] = bin < 0 ? -1 : bin | (place[warp * nbm + bin] + rank) << 16;
      __syncwarp();
      if (bin >= 0 && rank == 0) place[warp * nbm + bin] += __popc(same);
      __syncwarp();
    }
    __syncthreads();
    if (warp == 0) {  // first places and segments of the bins
      int c0 = 0, s0 = 0;
      for (int i0 = 0; i0 < nb; i0 += 32) {
        const int i = i0 + lane;
        int n[4] = {0, 0, 0, 0}, total = 0;
        if (i < nb) {
#pragma unroll
          for (int w = 0; w < 4; ++w) total += n[w] = place[w * nbm + i];
        }
        const int segs = (total + kSeg - 1) / kSeg;
        int c = total, s = segs;  // inclusive sums
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int c2 = __shfl_up_sync(0xffffffffu, c, off), s2 = __shfl_up_sync(0xffffffffu, s, off);
          if (lane >= off) {
            c += c2;
            s += s2;
          }
        }
        if (i < nb) {
          int at0 = c0 + c - total;
          start[i] = at0;
          seg0[i] = s0 + s - segs;
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            place[w * nbm + i] = at0;
            at0 += n[w];
          }
          for (int q = 0; q < segs; ++q) seg_bin[s0 + s - segs + q] = i;
        }
        c0 += __shfl_sync(0xffffffffu, c, 31);
        s0 += __shfl_sync(0xffffffffu, s, 31);
      }
      if (lane == 0) {
        start[nb] = c0;
        seg0[nb] = s0;
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kIter; ++i)
      if (at[i] >= 0) sorted[place[warp * nbm + (at[i] & 0xffff)] + (at[i] >> 16)] = xw[i];
    __syncthreads();
    for (int s = tid; s < seg0[nb]; s += kMomThreads) {
      const int bin = seg_bin[s], i0 = start[bin] + (s - seg0[bin]) * kSeg, i1 = min(i0 + kSeg, start[bin + 1]);
      float sum[kMomAll], comp[kMomAll];
#pragma unroll
      for (int p = 0; p < kMomAll; ++p) sum[p] = comp[p] = 0.0f;
      for (int i = i0; i < i1; ++i) {
        const float2 q = sorted[i];
        float pw = q.y, ep = 0.0f, em = 0.0f;
#pragma unroll
        for (int p = 0; p < kMom; ++p) {
          kahan(sum[p], comp[p], pw);
          ep = fmaf(coef[2 * tb * kMom + p].x, pw, ep);
          em = fmaf(coef[p].x, pw, em);
          pw *= q.x;
        }
        if (q.x >= ms.edge) kahan(sum[kMom], comp[kMom], ep);
        if (q.x <= -ms.edge) kahan(sum[kMom + 1], comp[kMom + 1], em);
      }
#pragma unroll
      for (int p = 0; p < kMomAll; ++p) part[s * kMomAll + p] = make_float2(sum[p], -comp[p]);
    }
    __syncthreads();
    for (int i = tid; i < nb * kMomAll; i += kMomThreads) {
      const int bin = i / kMomAll, p = i % kMomAll;
      DW v{mom[i].x, mom[i].y};
      for (int s = seg0[bin]; s < seg0[bin + 1]; ++s) {
        const float2 u = part[s * kMomAll + p];
        v = dw_add(v, fast_two_sum(u.x, u.y));
      }
      mom[i] = make_float2(v.h, v.l);
    }
  }
  __syncthreads();
  float *row = band + ((size_t)o * nz + k) * band_w;
  for (int i = tid; i < band_w; i += kMomThreads) {
    if (lo + i >= hi) {
      row[i] = 0.0f;
      continue;
    }
    const int c = i - ms.B0;  // this sample's bin
    float acc = 0.0f, err = 0.0f;
    auto add = [&](float h, float l) {
      const DW s = two_sum(acc, h);
      acc = s.h;
      err += s.l + l;
    };
    for (int bin = max(0, c - tb + 1); bin <= min(nb - 1, c + tb - 1); ++bin) {
      const float2 *m = mom + bin * kMomAll, *w = coef + (c - bin + tb) * kMom;
      float rest = 0.0f;
#pragma unroll
      for (int p = kMom - 1; p >= kMomFull; --p) rest = fmaf(w[p].x, m[p].x, rest);
#pragma unroll
      for (int p = kMomFull - 1; p >= 0; --p) {
        const DW pr = two_prod(w[p].x, m[p].x);
        rest += fmaf(w[p].y, m[p].x, fmaf(w[p].x, m[p].y, pr.l));
        add(pr.h, 0.0f);
      }
      err += rest;
    }
    if (c - tb >= 0 && c - tb < nb) add(mom[(c - tb) * kMomAll + kMom].x, mom[(c - tb) * kMomAll + kMom].y);
    if (c + tb >= 0 && c + tb < nb) add(mom[(c + tb) * kMomAll + kMom + 1].x, mom[(c + tb) * kMomAll + kMom + 1].y);
    row[i] = acc + err;
  }
}

// The pulse's polynomials c_p(t), t = -tb .. tb, as (high, low) pairs: interpolation at
// Chebyshev points in FP64.  False when they miss the pulse by more than 1e-9 of its
// largest value (a carrier or an envelope that varies too fast within a sample).
bool pulse_polynomials(double sigma, double omega, int tb, std::vector<float2> *out) {
  auto pulse = [&](double tau) {
    return -std::exp(-tau * tau / (2.0 * sigma * sigma)) *
           (tau / (sigma * sigma) * std::cos(omega * tau) + omega * std::sin(omega * tau));
  };
  double T[kMom][kMom] = {};  // monomial coefficients of the Chebyshev polynomials
  T[0][0] = T[1][1] = 1.0;
  for (int j = 2; j < kMom; ++j)
    for (int p = 0; p < kMom; ++p) T[j][p] = (p ? 2.0 * T[j - 1][p - 1] : 0.0) - T[j - 2][p];
  double node[4 * kMom];  // cos(pi i / (2 kMom)): the points are at odd i
  for (int i = 0; i < 4 * kMom; ++i) node[i] = std::cos(M_PI * i / (2 * kMom));
  out->resize((size_t)(2 * tb + 1) * kMom);
  double top = 0.0, miss = 0.0;
  for (int t = 0; t <= tb; ++t) {  // v is odd: c_p(-t) = (-1)^(p + 1) c_p(t)
    double c[kMom] = {}, v[kMom];
    for (int i = 0; i < kMom; ++i) v[i] = pulse(t - 0.5 * node[2 * i + 1]);
    for (int j = 0; j < kMom; ++j) {
      double aj = 0.0;
      for (int i = 0; i < kMom; ++i) aj += v[i] * node[j * (2 * i + 1) % (4 * kMom)];
      aj *= (j ? 2.0 : 1.0) / kMom;
      for (int p = 0; p < kMom; ++p) c[p] += aj * T[j][p];
    }
    for (int i = 0; i <= kMom; i += 2) {  // between the points, where the error peaks
      const double x = node[2 * i], want = pulse(t - 0.5 * x);
      double got = 0.0;
      for (int p = kMom - 1; p >= 0; --p) got = got * x + c[p];
      top = std::max(top, std::fabs(want));
      miss = std::max(miss, std::fabs(got - want));
    }
    for (int p = 0; p < kMom; ++p) {
      const float h = (float)c[p], l = (float)(c[p] - (double)h);
      (*out)[(size_t)(tb - t) * kMom + p] = p % 2 ? make_float2(h, l) : make_float2(-h, -l);
      (*out)[(size_t)(tb + t) * kMom + p] = make_float2(h, l);
    }
  }
  return miss <= 1e-9 * top;
}

// FP32 operators' slab rows (DirectRows) of one direction: row e of (orbit o, tile T)
// holds, for input element e (forward: depth, adjoint: sample), the tile's outputs.
__global__ void k_pack_rows(const float *band, const int *band_lo, const int *band_hi, int band_w, int nz, int dir,
                            int tiles, const uint2 *range, float *out) {
  const int ot = blockIdx.x, o = ot / tiles, T = ot % tiles;
  const int lo = (int)(range[ot].x & 0xffffu), hi = lo + (int)(range[ot].x >> 16);
  if (lo >= hi) return;
  const int e0 = lo / kRowChunk * kRowChunk, e1 = (hi + kRowChunk - 1) / kRowChunk * kRowChunk;
  out += (size_t)range[ot].y * kRowChunk * kOutTile;
  for (int i = threadIdx.x; i < (e1 - e0) * kOutTile; i += blockDim.x) {
    const int e = e0 + i / kOutTile, q = T * kOutTile + i % kOutTile;
    const int k = dir == 0 ? e : q, n = dir == 0 ? q : e;
    float v = 0.0f;
    if (k < nz) {
      const int bl = band_lo[o * nz + k], bh = band_hi[o * nz + k];
      if (n >= bl && n < bh) v = band[((size_t)o * nz + k) * band_w + (n - bl)];
    }
    out[i] = v;
  }
}

__global__ void k_slab_column(const float *band, const int *band_lo, int band_w, int nz, int nt, int o, int k,
                              float *out) {
  const int lo = band_lo[o * nz + k];
  const float *row = band + ((size_t)o * nz + k) * band_w;
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < nt; n += gridDim.x * blockDim.x) {
    const int i = n - lo;
    out[n] = (i >= 0 && i < band_w) ? row[i] : 0.0f;
  }
}

}  // namespace

int oam::disc_margin(const oam_model *m) {
  if (m->disc != OAM_DISC_TRILINEAR) return 0;
  const oam_grid &g = m->grid;
  return (int)std::ceil(g.fs_hz * (g.dx_m + g.dy_m + g.dz_m) / m->sensor.c_mps) + 2;
}

// Time origin, window check and bands [lo, hi) per (orbit, depth) from the
// range of d - F over the patches; each band is widened by `widen` samples on
// both sides (0 for a model build; the footprint planner widens to cover
// rounding of its host-side distances).  Also the slab's nonzero count and
// the operator's algorithmic flops.
oam_status oam::plan_bands(oam_model *m, const std::vector<double2> &h_range, int widen) {
  const oam_grid &gr = m->grid;
  const int nz = gr.nz, nt = gr.nt, O = m->n_orb;
  double dmin = INFINITY, dmax = -INFINITY;
  for (const double2 &r : h_range) {
    dmin = std::min(dmin, r.x);
    dmax = std::max(dmax, r.y);
  }
  const double fs = gr.fs_hz, c = m->sensor.c_mps, F = m->sensor.focal_m, ks = fs / c;
  const double reach = m->cut + disc_margin(m);  // samples an arrival reaches on either side
  const double t0 = std::isnan(gr.t0_s) ? (std::floor(fs * (F + dmin) / c - reach) - 2.0) / fs : gr.t0_s;
  m->t0 = t0;
  const double G = fs * (F / c - t0);
  if (ks * dmin + G - reach < 0 || ks * dmax + G + reach >= nt) return OAM_ERR_WINDOW;
  m->G = G;
  widen += disc_margin(m);

  // bands [lo, hi) per (orbit, depth)
  m->h_band_lo.resize((size_t)O * nz);
  m->h_band_hi.resize((size_t)O * nz);
  int wmax = 1;
  m->n_lo = nt;
  m->n_hi = 0;
  for (size_t i = 0; i < h_range.size(); ++i) {
    int lo = (int)std::ceil(ks * h_range[i].x + G - m->cut) - widen;
    int hi = (int)std::floor(ks * h_range[i].y + G + m->cut) + 1 + widen;
    lo = std::max(lo, 0);
    hi = std::min(hi, nt);
    if (hi < lo) hi = lo;
    m->h_band_lo[i] = lo;
    m->h_band_hi[i] = hi;
    wmax = std::max(wmax, hi - lo);
    if (hi > lo) {
      m->n_lo = std::min(m->n_lo, lo);
      m->n_hi = std::max(m->n_hi, hi);
    }
  }
  m->band_w = (wmax + 3) & ~3;
  if (m->band_w > 512) return OAM_ERR_UNSUPPORTED;

  // algorithmic work: entries in bands, and multiply-adds over in-grid voxel/position pairs
  std::vector<long long> orb_sum(O, 0);
  for (int o = 0; o < O; ++o)
    for (int k = 0; k < nz; ++k) orb_sum[o] += m->h_band_hi[(size_t)o * nz + k] - m->h_band_lo[(size_t)o * nz + k];
  long long nnz = 0;
  double fl = 0;
  for (int b = -m->R; b <= m->R; ++b)
    for (int a = -m->R; a <= m->R; ++a) {
      long long sum = orb_sum[m->h_tap_orbit[(b + m->R) * m->W + (a + m->R)]];
      nnz += sum;
      long long pairs = (long long)std::max(0, gr.py - std::abs(b)) * std::max(0, gr.px - std::abs(a));
      fl += 2.0 * (double)pairs * (double)sum;
    }
  m->nnz = nnz;
  m->flops = fl;
  return OAM_OK;
}

// Row and column offsets that couple two positions of the scan.
static int row_offsets(const oam_model *m) { return std::min(m->R, m->grid.py - 1) + 1; }
static int col_offsets(const oam_model *m) { return std::min(m->R, m->grid.px - 1) + 1; }
// The split form keeps FP32 rows for windows of up to nine folded taps (uses_direct).
static bool needs_rows(const oam_model *m) {
  return m->precision == OAM_PREC_FP32 ||
         (m->precision == OAM_PREC_BF16X3 && row_offsets(m) * col_offsets(m) <= 9);
}

// FP32 operators' slab rows of one direction (0 forward, 1 adjoint): per (orbit, output
// tile) the input range and first chunk, as DirectRows packs them.  Returns the chunks.
static long long plan_rows(const oam_model *m, int dir, int *tiles, std::vector<uint2> *range) {
  const int nz = m->grid.nz, O = m->n_orb, NT = ((dir == 0 ? m->grid.nt : nz) + kOutTile - 1) / kOutTile;
  *tiles = NT;
  range->assign((size_t)O * NT, make_uint2(0, 0));
  long long chunks = 0;
  std::vector<int> lo(NT), hi(NT);
  std::vector<char> used(O, 0);
  for (int b = 0; b < row_offsets(m); ++b)
    for (int a = 0; a < col_offsets(m); ++a) used[m->h_tap_orbit[(b + m->R) * m->W + (a + m->R)]] = 1;
  for (int o = 0; o < O; ++o) {
    if (!used[o]) continue;
    lo.assign(NT, 1 << 30);
    hi.assign(NT, 0);
    for (int k = 0; k < nz; ++k) {
      const int bl = m->h_band_lo[(size_t)o * nz + k], bh = m->h_band_hi[(size_t)o * nz + k];
      if (bh <= bl) continue;
      if (dir == 0) {
        for (int T = bl / kOutTile; T <= (bh - 1) / kOutTile; ++T) {
          lo[T] = std::min(lo[T], k);
          hi[T] = std::max(hi[T], k + 1);
        }
      } else {
        lo[k / kOutTile] = std::min(lo[k / kOutTile], bl);
        hi[k / kOutTile] = std::max(hi[k / kOutTile], bh);
      }
    }
    for (int T = 0; T < NT; ++T) {
      if (hi[T] <= lo[T]) continue;
      (*range)[(size_t)o * NT + T] = make_uint2((unsigned)lo[T] | (unsigned)(hi[T] - lo[T]) << 16, (unsigned)chunks);
      chunks += (hi[T] + kRowChunk - 1) / kRowChunk - lo[T] / kRowChunk;
    }
  }
  return chunks;
}

// Build one direction's slab rows.
static oam_status build_rows(oam_model *m, int dir, DirectRows *L, const int *d_band_hi, cudaStream_t st) {
  std::vector<uint2> range, taps;
  const long long chunks = plan_rows(m, dir, &L->tiles, &range);
  if (chunks > 0xffffffffLL) return OAM_ERR_UNSUPPORTED;
  const int R = m->R, W = m->W, NA = R + 1;
  taps.assign((size_t)L->tiles * NA * (NA + 1), make_uint2(0, 0));
  for (int T = 0; T < L->tiles; ++T)
    for (int b = 0; b < row_offsets(m); ++b) {
      uint2 *row = &taps[((size_t)T * NA + b) * (NA + 1)];
      unsigned lo = 0xffffffffu, hi = 0;
      for (int a = 0; a < col_offsets(m); ++a) {
        row[a] = range[(size_t)m->h_tap_orbit[(b + R) * W + (a + R)] * L->tiles + T];
        if (!(row[a].x >> 16)) continue;
        L->items += ((row[a].x & 0xffffu) + (row[a].x >> 16) + kRowChunk - 1) / kRowChunk -
                    (row[a].x & 0xffffu) / kRowChunk;
        lo = std::min(lo, row[a].x & 0xffffu);
        hi = std::max(hi, (row[a].x & 0xffffu) + (row[a].x >> 16));
      }
      if (hi > lo) row[NA].x = lo | (hi - lo) << 16;
    }
  oam_status rc;
  uint2 *d_range = nullptr;
  if ((rc = dev_alloc(m, &L->d_taps, taps.size())) ||
      (rc = dev_alloc(m, &L->d_rows, (size_t)chunks * kRowChunk * kOutTile)))
    return rc;
  OAM_CUDA_TRY(cudaMallocAsync((void **)&d_range, sizeof(uint2) * range.size(), st));
  OAM_CUDA_TRY(cudaMemcpyAsync(d_range, range.data(), sizeof(uint2) * range.size(), cudaMemcpyHostToDevice, st));
  OAM_CUDA_TRY(cudaMemcpyAsync(L->d_taps, taps.data(), sizeof(uint2) * taps.size(), cudaMemcpyHostToDevice, st));
  k_pack_rows<<<m->n_orb * L->tiles, 256, 0, st>>>(m->d_band, m->d_band_lo, d_band_hi, m->band_w, m->grid.nz, dir,
                                                   L->tiles, d_range, L->d_rows);
  OAM_LAUNCHED();
  OAM_CUDA_TRY(cudaFreeAsync(d_range, st));
  OAM_CUDA_TRY(cudaStreamSynchronize(st));  // host tables above go out of scope
  return OAM_OK;
}

// Device bytes build_slab allocates for a model whose bands are planned.
size_t oam::slab_plan_bytes(const oam_model *m) {
  const size_t O = m->n_orb, nz = m->grid.nz;
  size_t b = alloc_bytes<int>((size_t)m->W * m->W) + alloc_bytes<int>(O * nz) + alloc_bytes<float>(O * nz * m->band_w);
  if (!needs_rows(m)) return b;
  for (int dir = 0; dir < 2; ++dir) {
    std::vector<uint2> range;
    int tiles = 0;
    const long long chunks = plan_rows(m, dir, &tiles, &range);
    b += alloc_bytes<uint2>((size_t)tiles * (m->R + 1) * (m->R + 2)) +
         alloc_bytes<float>((size_t)chunks * kRowChunk * kOutTile);
  }
  return b;
}

oam_status oam::build_slab(oam_model *m, cudaStream_t st) {
  const oam_grid &gr = m->grid;
  const int nz = gr.nz, nt = gr.nt, O = m->n_orb;
  oam_status rc;
  int *d_orb_b = nullptr, *d_orb_a = nullptr;
  double2 *d_range = nullptr;
  if ((rc = dev_alloc(m, &m->d_tap_orbit, m->W * m->W))) return rc;
  OAM_CUDA_TRY(cudaMemcpyAsync(m->d_tap_orbit, m->h_tap_orbit.data(), sizeof(int) * m->W * m->W,
                               cudaMemcpyHostToDevice, st));
  OAM_CUDA_TRY(cudaMallocAsync((void **)&d_orb_b, sizeof(int) * O, st));
  OAM_CUDA_TRY(cudaMallocAsync((void **)&d_orb_a, sizeof(int) * O, st));
  OAM_CUDA_TRY(cudaMallocAsync((void **)&d_range, sizeof(double2) * O * nz, st));
  OAM_CUDA_TRY(cudaMemcpyAsync(d_orb_b, m->h_orb_b.data(), sizeof(int) * O, cudaMemcpyHostToDevice, st));
  OAM_CUDA_TRY(cudaMemcpyAsync(d_orb_a, m->h_orb_a.data(), sizeof(int) * O, cudaMemcpyHostToDevice, st));

  Geo g{};
  g.F = m->sensor.focal_m;
  g.dx = gr.dx_m;
  g.dy = gr.dy_m;
  g.dz = gr.dz_m;
  g.z0 = gr.z0_rel_m;
  g.ks = gr.fs_hz / m->sensor.c_mps;
  g.cut = m->cut;
  g.inv2s2 = (float)(1.0 / (2.0 * m->sigma_s * m->sigma_s));
  g.env2 = (float)(1.0 / (2.0 * m->sigma_s * m->sigma_s * std::log(2.0)));
  g.invs2 = (float)(1.0 / (m->sigma_s * m->sigma_s));
  g.omega = (float)m->omega;
  g.cyc = (float)(m->omega / M_PI);

  PatchDW *d_pdw = nullptr;  // double-word patches, freed with the other temporaries
  OAM_CUDA_TRY(cudaMallocAsync((void **)&d_pdw, sizeof(PatchDW) * m->M, st));
  k_patch_dw<<<(m->M + 255) / 256, 256, 0, st>>>(m->d_patch, m->M, d_pdw);
  OAM_LAUNCHED();
  k_delta_range<<<dim3(O, nz), 256, 0, st>>>(g, m->d_patch, d_pdw, m->M, d_orb_b, d_orb_a, nz, d_range);
  OAM_LAUNCHED();
  std::vector<double2> h_range((size_t)O * nz);
  OAM_CUDA_TRY(cudaMemcpyAsync(h_range.data(), d_range, sizeof(double2) * O * nz, cudaMemcpyDeviceToHost, st));
  OAM_CUDA_TRY(cudaStreamSynchronize(st));

  rc = plan_bands(m, h_range, 0);
  if (rc) {
    cudaFreeAsync(d_orb_b, st);
    cudaFreeAsync(d_orb_a, st);
    cudaFreeAsync(d_range, st);
    cudaFreeAsync(d_pdw, st);
    return rc;
  }
  g.G = m->G;

  int *d_band_hi = nullptr;
  if ((rc = dev_alloc(m, &m->d_band_lo, (size_t)O * nz))) return rc;
  OAM_CUDA_TRY(cudaMallocAsync((void **)&d_band_hi, sizeof(int) * O * nz, st));
  OAM_CUDA_TRY(cudaMemcpyAsync(m->d_band_lo, m->h_band_lo.data(), sizeof(int) * O * nz, cudaMemcpyHostToDevice, st));
  OAM_CUDA_TRY(cudaMemcpyAsync(d_band_hi, m->h_band_hi.data(), sizeof(int) * O * nz, cudaMemcpyHostToDevice, st));
  if ((rc = dev_alloc(m, &m->d_band, (size_t)O * nz * m->band_w))) return rc;
  if (m->disc == OAM_DISC_TRILINEAR) {
    Geo33 g3{};
    g3.F = m->sensor.focal_m * 1e3;
    g3.dx = gr.dx_m * 1e3;
    g3.dy = gr.dy_m * 1e3;
    g3.dz = gr.dz_m * 1e3;
    g3.z0 = gr.z0_rel_m * 1e3;
    g3.c = m->sensor.c_mps * 1e3;
    g3.fs = gr.fs_hz;
    g3.t0 = m->t0;
    g3.sigma = m->sigma_s;
    g3.omega = m->omega;
    g3.T = (int)std::floor(m->cut);
    g3.len = (int)std::ceil(2.0 * gr.fs_hz * (gr.dx_m + gr.dy_m + gr.dz_m) / m->sensor.c_mps) + 4;
    const int threads = std::max(128, ((m->band_w + 3) / 4 + 31) & ~31);
    const size_t sm = sizeof(double) * (2 * g3.T + 1 + (size_t)k33Chunk * g3.len) + sizeof(int) * (k33Chunk + 2) +
                      sizeof(double) * k33Chunk;
    if (threads > 1024 || sm > 200 * 1024) return OAM_ERR_UNSUPPORTED;
    if (sm > 48 * 1024)  // one limit for every model: builds from several threads would lower each other's
      OAM_CUDA_TRY(
          cudaFuncSetAttribute(k_slab33_values, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    k_slab33_values<<<dim3(O, nz), threads, sm, st>>>(g3, m->d_patch, m->M, d_orb_b, d_orb_a, nz, nt, m->d_band_lo,
                                                      d_band_hi, m->band_w, m->d_band);
  } else {
    // k_slab_values where the pulse varies too fast within a sample for the polynomials, is
    // shorter than two samples a side, or its bins exceed the shared memory of two blocks
    // per SM; and for few patches, which do not repay the moments' last sums (build of 192
    // depths, 61x61 taps, ms, moments against values: 64 patches 4.5, 3.5; 256 5.6, 4.9; 512
    // 5.9, 6.9; 48 depths, 11x11 taps, 256 patches 0.32, 0.30, 512 0.31, 0.35)
    constexpr int kMomPatches = 352;
    MomShape ms{};
    ms.tb = (int)std::floor(m->cut - 0.5) + 1;
    const double edge = 2.0 * (ms.tb - m->cut);
    ms.edge = (float)edge;
    if ((double)ms.edge < edge) ms.edge = std::nextafter(ms.edge, INFINITY);
    ms.B0 = std::max(0, (int)std::floor(m->cut) - 1);
    ms.nb = std::max(1, m->band_w - 2 * ms.B0 + 1);
    std::vector<float2> coef;
    if (m->M >= kMomPatches && m->cut >= 2.0 && m->cut <= 64.0 && mom_smem(ms) <= 100 * 1024 &&
        pulse_polynomials(m->sigma_s, m->omega, ms.tb, &coef)) {
      float2 *d_coef = nullptr;
      OAM_CUDA_TRY(cudaMallocAsync((void **)&d_coef, sizeof(float2) * coef.size(), st));
      OAM_CUDA_TRY(cudaMemcpyAsync(d_coef, coef.data(), sizeof(float2) * coef.size(), cudaMemcpyHostToDevice, st));
      OAM_CUDA_TRY(cudaFuncSetAttribute(k_slab_moments, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024));
      k_slab_moments<<<dim3(O, nz), kMomThreads, mom_smem(ms), st>>>(
          g, d_pdw, m->M, d_orb_b, d_orb_a, nz, m->d_band_lo, d_band_hi, m->band_w, ms, d_coef, m->d_band);
      cudaFreeAsync(d_coef, st);
    } else {
      const int threads = m->band_w <= 128 ? 128 : 256;
      const int T0 = (int)std::floor(m->cut + 0.5) + 1;  // rotation table half-length
      k_slab_values<<<dim3(O, nz), threads, sizeof(float2) * (2 * T0 + 1), st>>>(
          g, d_pdw, m->M, d_orb_b, d_orb_a, nz, m->d_band_lo, d_band_hi, m->band_w, T0, m->d_band);
    }
  }
  OAM_LAUNCHED();

  if (needs_rows(m) && ((rc = build_rows(m, 0, &m->rows_fwd, d_band_hi, st)) ||
                                        (rc = build_rows(m, 1, &m->rows_adj, d_band_hi, st))))
    return rc;
  cudaFreeAsync(d_orb_b, st);
  cudaFreeAsync(d_orb_a, st);
  cudaFreeAsync(d_range, st);
  cudaFreeAsync(d_pdw, st);
  cudaFreeAsync(d_band_hi, st);
  return OAM_OK;
}

oam_status oam::slab_column(const oam_model *m, int b, int a, int k, float *d_out, cudaStream_t st) {
  const int o = m->h_tap_orbit[(b + m->R) * m->W + (a + m->R)];
  k_slab_column<<<(m->grid.nt + 255) / 256, 256, 0, st>>>(m->d_band, m->d_band_lo, m->band_w, m->grid.nz,
                                                          m->grid.nt, o, k, d_out);
  OAM_LAUNCHED();
  return OAM_OK;
}
