// Plain FP32 forward and adjoint operators on CUDA cores.
//
// Both are lateral correlations of the single-position slab with the volume or
// the signals ("two coordinate systems": the absolute index of a voxel and its
// offset relative to each scan position; Methods, Efficient reconstruction
// based on scanning symmetries).  Voxels and samples outside the grids are zero.
//
// One kernel serves both: out[pos][n] += F[pos][k] S[k][n], K = depths and N =
// samples for the forward operator, the reverse for the adjoint.  The slab is
// mirror-symmetric (S[b][a] = S[+-b][+-a]; Results, axial symmetry), so the four
// mirrored taps share their slab rows and their inputs are summed first:
//   P[pos][k] = X[y + b][x][k] + X[y - b][x][k]          (once per row offset b)
//   F[pos][k] = P[x + a][k] + P[x - a][k]                (once per tap)
// which cuts the products 3.9x at 61x61 taps.  A block serves an output tile of kTile
// and a tile of positions; it walks the row offsets and the 16-deep K chunks whose band
// meets the output tile, with P in shared memory, and the taps a of each chunk.  A
// thread keeps 8 positions x 4 outputs in registers as packed pairs of positions.
//   k_corr_one    one tap: a banded product per position, nothing folded.
//   k_corr_warps  32 positions; the block's eight warps share out the taps, each with
//                 its own F and slab rows, so nothing but P is exchanged between warps,
//                 and up to eight blocks of a cluster share out the row offsets: the
//                 short chain for small problems.
//   k_corr_block  128 positions; four warps take each tap together, 32 positions each,
//                 sharing its slab rows (a quarter of the L2 reads): large problems.
//
// What bounds them: k_corr_block the shared memory (84 % of its rate, with the FP32 pipe
// at 64 %: three 16-byte reads per 16 packed products, and the folding's two reads and a
// write per input), for 1.5x the band's products in 32-output tiles; other maps of lanes
// to positions and outputs read more (55 and 51 ms against 50 below).  k_corr_warps the
// chain of staging, folding and products per chunk.  One application, GB300, from a
// kernel without folding: 200x200x300 forward, 61x61 taps, 360 -> 50 ms; 32x32x48, 11x11
// taps, 283 -> 29 us (42 without clusters); 70x37x52 adjoint, 15x15 taps, 888 -> 94 us
// (132).
//
// Each output sums up to win^2 x band products (about 3e5 at 61x61 taps).  One
// FP32 accumulator for all of them loses about sqrt(n) units in the last place,
// so the kernels sum in three levels: the products of at most 8 taps of a chunk, then
// those of a row offset (in registers or shared memory), then the row offsets, in shared
// memory or the output.  The order does not depend on the position, so a shifted input gives the
// shifted output to the bit.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "f32x2.cuh"
#include "internal.cuh"

using namespace oam;

namespace {

constexpr int kWarps = 8;        // warps per block
constexpr int kThreads = 32 * kWarps;
constexpr int kPos = 32;         // positions per block
constexpr int kChunk = kRowChunk;  // K elements per chunk (16)
constexpr int kTile = kOutTile;  // outputs per block (32)
constexpr int kFlush = 8;        // a warp's taps per first-level sum
constexpr int kMaxStrip = 352;   // staged positions a block takes on run-on tiles
constexpr int kTableR = 31;      // largest half window whose tap table is copied to shared memory

__device__ __forceinline__ void copy16_async(void *dst, const void *src, bool real) {  // zeros unless real
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(real ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory");
}

struct CorrShape {
  int px, py, R;
  int len, out_len;  // input and output row lengths
  int sp;            // positions per tile-grid row: px (tiles run on over rows) or a multiple of the tile
  int strip;         // staged positions per block: tile + (rows wrapped + 2) R
  int group;         // chunks staged together (1, 2, 4 or 8)
  const uint2 *taps;  // [output tile][R + 1][R + 2] (DirectRows)
  const float *rows;  // slab rows
};

// K range [lo, hi) of a table entry.
__device__ __forceinline__ int k_lo(uint2 t) { return (int)(t.x & 0xffffu); }
__device__ __forceinline__ int k_hi(uint2 t) { return (int)(t.x & 0xffffu) + (int)(t.x >> 16); }

// Float of K quarter kq of staged position r: 64-byte rows, the 16-byte quarters
// exchanged so that eight neighbouring positions' reads fall in distinct banks.
__device__ __forceinline__ int p_at(int r, int kq) { return r * kChunk + 4 * (kq ^ ((r >> 1) & 3)); }

// Row and column (-1: padding) of the staged positions of a tile that starts at (y0, x0).
template <int kN>
__device__ __forceinline__ void stage_where(const CorrShape &s, int y0, int x0, int2 *where) {
  const int wp = s.px + s.R;
  for (int r = threadIdx.x; r < s.strip; r += kN) {
    const long long q = (long long)y0 * wp + x0 - s.R + r;
    const int y = q < 0 ? -1 : (int)(q / wp), x = q < 0 ? -1 : (int)(q % wp);
    where[r] = make_int2(y, x < s.px ? x : -1);
  }
}

// F of tap a for the position staged at pm, K quarter by quarter: F[k][position m] at d.
template <int kM>
__device__ __forceinline__ void fold_tap(const float *P, int pm, int a, float *d, int kq) {
  float4 f = *reinterpret_cast<const float4 *>(P + p_at(pm + a, kq));
  if (a > 0) {
    const float4 h = *reinterpret_cast<const float4 *>(P + p_at(pm - a, kq));
    f = make_float4(f.x + h.x, f.y + h.y, f.z + h.z, f.w + h.w);
  }
  d += 4 * kq * kM;
  d[0] = f.x;
  d[kM] = f.y;
  d[2 * kM] = f.z;
  d[3 * kM] = f.w;
}

// a1[position pair][output] += F[ka .. kb)[8 positions] S[ka .. kb)[4 outputs].
template <int kM>
__device__ __forceinline__ void multiply(const float *F, const float *S, int ka, int kb, uint64_t (&a1)[4][4]) {
  for (int kk = ka; kk < kb; kk += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 sv = *reinterpret_cast<const float4 *>(S + (kk + u) * kTile);
      const uint64_t s2[4] = {f2_pack(sv.x, sv.x), f2_pack(sv.y, sv.y), f2_pack(sv.z, sv.z), f2_pack(sv.w, sv.w)};
      const ulonglong2 f0 = *reinterpret_cast<const ulonglong2 *>(F + (kk + u) * kM);
      const ulonglong2 f1 = *reinterpret_cast<const ulonglong2 *>(F + (kk + u) * kM + 4);
      const uint64_t f2[4] = {f0.x, f0.y, f1.x, f1.y};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) a1[i][j] = f2_fma(f2[i], s2[j], a1[i][j]);
    }
  }
}

// ---------------------------------------------------------------- k_corr_one
constexpr int kOneThreads = 128;
constexpr int kOneK = 128;          // K elements staged at once
constexpr int kOneRow = kOneK + 4;  // floats per staged position: eight of them meet distinct banks

// A window of one tap is a banded product per position: the block's 32 positions and the
// tile's slab rows are staged 128 K elements at a time, the four warps take every fourth
// four of them and add their sums in shared memory at the end.
// What bounds it: the staging's latency, under four blocks an SM; the kernels below pay a
// chain of chunks with barriers for folding that one tap does not have.  us a call, from
// those: 48x48x101 forward 16.5 -> 8.0, 64x64x128 27 -> 8.0 (adjoint 21 -> 7.9),
// 128x128x64 16.5 -> 14.4 (37 -> 10.2), 200x200x300 125 -> 85 (97 -> 68).
template <bool kVec>
__global__ void __launch_bounds__(kOneThreads, 4)
    k_corr_one(const CorrShape s, const float *__restrict__ in, float *__restrict__ out) {
  __shared__ __align__(16) float X[kPos * kOneRow];
  __shared__ __align__(16) float S[kOneK * kTile];
  static_assert(kPos * kOneRow >= 3 * kPos * kTile, "three warps' sums in the inputs' place");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockIdx.y;
  const long long o0 = (long long)blockIdx.x * kPos, positions = (long long)s.py * s.px;
  const uint2 t = s.taps[(size_t)T * 2];  // one tap a row
  const int lo = (int)(t.x >> 16) ? k_lo(t) / kChunk * kChunk : 0, hi = (int)(t.x >> 16) ? k_hi(t) : 0;
  if (hi == 0 && s.out_len % 4 == 0) {  // no slab row meets the tile: zeros
    for (int i = tid; i < kPos * (kTile / 4); i += kOneThreads) {
      const int r = i / (kTile / 4), n = T * kTile + 4 * (i % (kTile / 4));
      if (o0 + r < positions && n < s.out_len)
        *reinterpret_cast<float4 *>(out + (o0 + r) * s.out_len + n) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    return;
  }
  const float *rows = s.rows + (size_t)t.y * kChunk * kTile;
  const int ng = lane & 7, pg = lane >> 3;  // outputs 4 ng .. +3 of the tile, positions pg, pg + 4, .. pg + 28
  uint64_t sum[8][2], acc[8][2];            // [position][output pair]
#pragma unroll
  for (int i = 0; i < 8; ++i) sum[i][0] = sum[i][1] = 0;
  for (int k0 = lo; k0 < hi; k0 += kOneK) {
    const int n = min(kOneK, hi - k0), n4 = (n + 3) / 4;
    __syncthreads();
    for (int i = tid; i < kPos * (kOneK / 4); i += kOneThreads) {
      const int r = i / (kOneK / 4), k = 4 * (i % (kOneK / 4));
      if (k >= n) continue;
      const bool ok = o0 + r < positions;
      const float *src = in + (ok ? (o0 + r) * s.len + k0 + k : 0);
      float *dst = X + r * kOneRow + k;
      if (kVec) {
        copy16_async(dst, src, ok);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[q] = ok && k0 + k + q < s.len ? src[q] : 0.0f;
      }
    }
    for (int i = tid; i < 4 * n4 * (kTile / 4); i += kOneThreads)  // whole chunks are stored
      copy16_async(S + 4 * i, rows + (size_t)(k0 - lo) * kTile + 4 * i, true);
    copies_commit();
    copies_wait<0>();
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = 0;
    for (int q = warp; q < n4; q += kOneThreads / 32) {
      ulonglong2 w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) w[u] = *reinterpret_cast<const ulonglong2 *>(S + (4 * q + u) * kTile + 4 * ng);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 f = *reinterpret_cast<const float4 *>(X + (pg + 4 * i) * kOneRow + 4 * q);
        const uint64_t f2[4] = {f2_pack(f.x, f.x), f2_pack(f.y, f.y), f2_pack(f.z, f.z), f2_pack(f.w, f.w)};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          acc[i][0] = f2_fma(f2[u], w[u].x, acc[i][0]);
          acc[i][1] = f2_fma(f2[u], w[u].y, acc[i][1]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      sum[i][0] = f2_add(sum[i][0], acc[i][0]);
      sum[i][1] = f2_add(sum[i][1], acc[i][1]);
    }
  }
  __syncthreads();
  if (warp) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      *reinterpret_cast<ulonglong2 *>(X + ((warp - 1) * kPos + pg + 4 * i) * kTile + 4 * ng) =
          make_ulonglong2(sum[i][0], sum[i][1]);
  }
  __syncthreads();
  if (warp) return;
  const int n = T * kTile + 4 * ng;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
#pragma unroll
    for (int w = 0; w < 3; ++w) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(X + (w * kPos + pg + 4 * i) * kTile + 4 * ng);
      sum[i][0] = f2_add(sum[i][0], v.x);
      sum[i][1] = f2_add(sum[i][1], v.y);
    }
    if (o0 + pg + 4 * i >= positions) continue;
    float *dst = out + (o0 + pg + 4 * i) * s.out_len + n;
    const float2 a = f2_unpack(sum[i][0]), b = f2_unpack(sum[i][1]);
    if (s.out_len % 4 == 0) {
      if (n < s.out_len) *reinterpret_cast<float4 *>(dst) = make_float4(a.x, a.y, b.x, b.y);
    } else {
      if (n < s.out_len) dst[0] = a.x;
      if (n + 1 < s.out_len) dst[1] = a.y;
      if (n + 2 < s.out_len) dst[2] = b.x;
      if (n + 3 < s.out_len) dst[3] = b.y;
    }
  }
}

// ---------------------------------------------------------------- k_corr_warps
// A window of few taps leaves warps without one, so the block stages a group of G chunks
// and warp w takes chunk w / (kWarps / G) of it and the taps a = w (mod kWarps / G): the
// fewer taps, the more chunks at once.  us from one chunk at a time: 3x3 taps, 48x48x101
// 27 -> 23 (adjoint 24 -> 17), 64x64x128 47 -> 37 (41 -> 27); 7x7 taps 84 -> 76 (86 -> 76).
int chunk_group(int R) { return R == 1 ? 4 : R <= 3 ? 2 : 1; }

// Shared memory: raw rows of the two row offsets, double-buffered (the first of a pair
// holds P once added) [2][2][group][strip][kChunk]; per warp F [kChunk][kPos] and two slots of
// slab rows [kChunk][kTile]; the tap table (R <= kTableR); per staged position its row
// and column; the tile's sums [2][kThreads] pairs.
size_t warps_smem(int strip, int R, int group) {
  return sizeof(float) * ((size_t)4 * group * strip * kChunk + kWarps * kChunk * (kPos + 2 * kTile) + kPos * kTile) +
         (R <= kTableR ? sizeof(uint2) * (R + 1) * (R + 2) : 0) + sizeof(int2) * strip;
}

// The blocks of a cluster (grid z) share out a tile's row offsets, b = z (mod Z), and
// add their sums in rank order at the end.
// kVec: input rows are whole float4 from a 16-byte boundary.  kGroups: groups of chunks.
template <bool kVec, bool kGroups>
__global__ void __launch_bounds__(kThreads, 2)
    k_corr_warps(const CorrShape s, const float *__restrict__ in, float *__restrict__ out) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int G = kGroups ? s.group : 1;
  const int R = s.R, NA = R + 1, wp = s.px + R, p_size = G * s.strip * kChunk;
  float *Pb = reinterpret_cast<float *>(smem);  // [buffer][side][p_size]
  float *Fb = Pb + 4 * p_size;                  // [warp][kChunk][kPos]; the warps' sums at the end of a row offset
  float *Sb = Fb + kWarps * kChunk * kPos;      // [warp][slot][kChunk][kTile]
  // the tile's sums: of output pairs [half][position x group of four], over this block's row offsets
  float2 *sum3 = reinterpret_cast<float2 *>(Sb + 2 * kWarps * kChunk * kTile);
  int2 *where = reinterpret_cast<int2 *>(sum3 + 2 * kThreads);  // staged position: row y, column x (-1: padding)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int T = blockIdx.y, tile = blockIdx.x, Z = gridDim.z;
  static_assert(kPos * 8 == kThreads, "a thread per position and group of four outputs");
  sum3[tid] = sum3[kThreads + tid] = make_float2(0.0f, 0.0f);
  const int y0 = tile * kPos / s.sp, x0 = tile * kPos % s.sp;
  const int y1 = min((tile * kPos + kPos - 1) / s.sp, s.py - 1);  // rows of the tile
  const uint2 *tab = s.taps + (size_t)T * NA * (NA + 1);
  if (R <= kTableR) {
    uint2 *t = reinterpret_cast<uint2 *>(where + s.strip);
    for (int i = tid; i < NA * (NA + 1); i += kThreads) t[i] = tab[i];
    tab = t;
  }
  stage_where<kThreads>(s, y0, x0, where);
  __syncthreads();
  float *F = Fb + warp * kChunk * kPos, *S = Sb + warp * 2 * kChunk * kTile;
  // staged index of the position this lane folds
  const int pm = ((tile * kPos + lane) / s.sp - y0) * wp + ((tile * kPos + lane) % s.sp - x0) + R;
  const int ng = lane & 7, pg = lane >> 3;  // outputs 4 ng .. +3 of the tile, positions 8 pg .. +7

  // this warp's chunk of a group, and its taps
  const int share = kWarps / G, own = kGroups ? warp / share : 0;
  unsigned own_taps = 0x01010101u << warp;
  if (kGroups) {
    own_taps = 0;
    for (int a = warp % share; a < 32; a += share) own_taps |= 1u << a;
  }

  // Walk of the (row offset b, group of chunks from c) with work: c0 .. c1 - 1 are b's chunks.
  int b = (int)blockIdx.z - Z, c = 0, c1 = 0;
  auto advance = [&](int &b, int &c, int &c1) {
    if ((c += G) < c1) return;
    while ((b += Z) <= R) {
      if (y0 + b >= s.py && y1 - b < 0) continue;  // neither row offset meets the grid
      const uint2 t = tab[b * (NA + 1) + NA];      // the union of its taps' ranges
      if (t.x >> 16) {
        c = k_lo(t) / kChunk;
        c1 = (k_hi(t) + kChunk - 1) / kChunk;
        return;
      }
    }
  };
  // This warp's taps whose range meets its chunk of the group from c of row offset b, one bit each.
  auto my_taps = [&](int b, int c, unsigned long long &m0, unsigned long long &m1) {
    c += own;
    auto word = [&](int i) {
      const int a = 32 * i + lane;
      const uint2 t = a < NA ? tab[b * (NA + 1) + a] : make_uint2(0, 0);
      return __ballot_sync(0xffffffffu, k_lo(t) < (c + 1) * kChunk && k_hi(t) > c * kChunk && (t.x >> 16)) &
             own_taps;
    };
    m0 = m1 = 0;
    m0 = word(0);
    if (NA > 32) m0 |= (unsigned long long)word(1) << 32;
    if (NA > 64) m1 = word(2);
    if (NA > 96) m1 |= (unsigned long long)word(3) << 32;
  };
  auto pop = [&](unsigned long long &m0, unsigned long long &m1) {  // lowest tap, NA when none is left
    int a = NA;
    if (m0) {
      a = __ffsll((long long)m0) - 1;
      m0 &= m0 - 1;
    } else if (m1) {
      a = 63 + __ffsll((long long)m1);
      m1 &= m1 - 1;
    }
    return a;
  };
  // Request the raw rows of (b, c) into buffer pb.
  auto request_rows = [&](int b, int c, int pb) {
    const int quarters = G * s.strip * (kChunk / 4), lg = kGroups ? 31 - __clz(G) : 0;
    for (int side = 0; side < (b ? 2 : 1); ++side)
      for (int i = tid; i < quarters; i += kThreads) {
        // a position's chunks follow one another, as they do in its input row
        const int r = i / (kChunk / 4) >> lg, h = kGroups ? i / (kChunk / 4) & (G - 1) : 0, kq = i % (kChunk / 4);
        const int k = (c + h) * kChunk + 4 * kq;
        const int2 w = where[r];
        const int y = side ? w.x - b : w.x + b;
        const bool ok = w.y >= 0 && y >= 0 && y < s.py;
        const float *src = in + (ok ? ((size_t)y * s.px + w.y) * s.len + k : 0);
        float *dst = Pb + (2 * pb + side) * p_size + h * s.strip * kChunk + p_at(r, kq);
        if (kVec) {
          copy16_async(dst, k < s.len ? src : in, ok && k < s.len);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) dst[q] = ok && k + q < s.len ? src[q] : 0.0f;
        }
      }
  };
  // Request the slab rows of tap a in this warp's chunk of the group into its slot.
  auto request_slab = [&](int b, int c, int a, int slot) {
    if (a >= NA) return;
    c += own;
    const uint2 t = tab[b * (NA + 1) + a];
    const float *src = s.rows + ((size_t)t.y + (c - k_lo(t) / kChunk)) * (kChunk * kTile);
    float *dst = S + slot * kChunk * kTile;
#pragma unroll
    for (int j = 0; j < kChunk * kTile / 128; ++j) copy16_async(dst + 128 * j + 4 * lane, src + 128 * j + 4 * lane, true);
  };

  uint64_t a1[4][4], a2[4][4];  // [position pair][output]
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) a1[i][j] = a2[i][j] = 0;
  // Add the warps' sums of a row offset to the tile's: two of a lane's four outputs at
  // a time through the F buffers, a thread per pair.
  auto flush = [&] {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      __syncthreads();
      // [warp][position][2 outputs of each group of four]
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 u = f2_unpack(a2[i][2 * half]), v = f2_unpack(a2[i][2 * half + 1]);
        *reinterpret_cast<float2 *>(F + (8 * pg + 2 * i) * 16 + 2 * ng) = make_float2(u.x, v.x);
        *reinterpret_cast<float2 *>(F + (8 * pg + 2 * i + 1) * 16 + 2 * ng) = make_float2(u.y, v.y);
        a2[i][2 * half] = a2[i][2 * half + 1] = 0;
      }
      __syncthreads();
      float2 v = *reinterpret_cast<const float2 *>(Fb + 2 * tid);
#pragma unroll
      for (int w = 1; w < kWarps; ++w) {
        const float2 u = *reinterpret_cast<const float2 *>(Fb + w * kChunk * kPos + 2 * tid);
        v.x += u.x;
        v.y += u.y;
      }
      float2 &o = sum3[half * kThreads + tid];
      o = make_float2(o.x + v.x, o.y + v.y);
    }
    __syncthreads();
  };

  int pb = 0, slot = 0;
  unsigned long long m0 = 0, m1 = 0;
  int a = NA;  // this warp's tap
  advance(b, c, c1);
  if (b <= R) {
    request_rows(b, c, 0);
    my_taps(b, c, m0, m1);
    a = pop(m0, m1);
    request_slab(b, c, a, 0);
    copies_commit();
  }
  while (b <= R) {
    const int k0 = (c + own) * kChunk;
    float *P = Pb + 2 * pb * p_size;
    copies_wait<0>();
    __syncthreads();
    if (b > 0) {
      float4 *p0 = reinterpret_cast<float4 *>(P);
      const float4 *p1 = reinterpret_cast<const float4 *>(P + p_size);
      for (int i = tid; i < p_size / 4; i += kThreads) {
        const float4 u = p0[i], v = p1[i];
        p0[i] = make_float4(u.x + v.x, u.y + v.y, u.z + v.z, u.w + v.w);
      }
      __syncthreads();
    }
    // the next chunk and this warp's taps of it
    int bn = b, cn = c, c1n = c1, chain = 0;
    advance(bn, cn, c1n);
    unsigned long long n0 = 0, n1 = 0;
    if (bn <= R) my_taps(bn, cn, n0, n1);
    bool ahead = false;  // the next chunk's rows are requested
    for (int step = 0; a < NA; ++step) {
      // request the tap after this one, here or in the next chunk
      __syncwarp();  // the other slot's tap is done
      int an = pop(m0, m1);
      const bool last = an >= NA;
      if (last) {
        an = bn <= R ? pop(n0, n1) : NA;
        request_slab(bn, cn, an, slot ^ 1);
      } else {
        request_slab(b, c, an, slot ^ 1);
      }
      copies_commit();
      if (step == 0) {
        if (bn <= R) request_rows(bn, cn, pb ^ 1);
        copies_commit();
        ahead = true;
      }
      // F of this tap
#pragma unroll
      for (int kq = 0; kq < kChunk / 4; ++kq) fold_tap<kPos>(P + own * s.strip * kChunk, pm, a, F + lane, kq);
      // this tap's slab rows are older than the last two copies (steps 0 and 1: the
      // next tap's and the next chunk's) or than the last one
      if (step < 2) copies_wait<2>();
      else copies_wait<1>();
      __syncwarp();
      const uint2 t = tab[b * (NA + 1) + a];
      const int ka = max(k_lo(t) - k0, 0) & ~3, kb = min(k_hi(t) - k0, kChunk);
      multiply<kPos>(F + 8 * pg, S + slot * kChunk * kTile + 4 * ng, ka, kb, a1);
      if (++chain == kFlush || last) {
        chain = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            a2[i][j] = f2_add(a2[i][j], a1[i][j]);
            a1[i][j] = 0;
          }
      }
      slot ^= 1;
      a = an;
      if (last) break;
    }
    if (!ahead) {  // no tap of this warp here: it still stages its share of the next rows
      if (bn <= R) request_rows(bn, cn, pb ^ 1);
      a = bn <= R ? pop(n0, n1) : NA;
      request_slab(bn, cn, a, slot);
      copies_commit();
    }
    if (bn != b) flush();
    b = bn;
    c = cn;
    c1 = c1n;
    m0 = n0;
    m1 = n1;
    pb ^= 1;
  }
  // Write the tile: rank z takes the z-th share of the pairs.
  auto cluster = cooperative_groups::this_cluster();
  cluster.sync();
  const int part = 2 * kThreads / Z;
  for (int j = tid; j < part; j += kThreads) {
    const int i = blockIdx.z * part + j, half = i / kThreads, e = i % kThreads;
    float2 v = *cluster.map_shared_rank(sum3 + i, 0);
    for (int z = 1; z < Z; ++z) {
      const float2 u = *cluster.map_shared_rank(sum3 + i, z);
      v.x += u.x;
      v.y += u.y;
    }
    const int o = tile * kPos + e / 8, y = o / s.sp, x = o % s.sp, n = T * kTile + 4 * (e % 8) + 2 * half;
    if (y >= s.py || x >= s.px) continue;
    float *dst = out + ((size_t)y * s.px + x) * s.out_len + n;
    if (n < s.out_len) dst[0] = v.x;
    if (n + 1 < s.out_len) dst[1] = v.y;
  }
  cluster.sync();  // every rank has read this block's sums
}

// ---------------------------------------------------------------- k_corr_block
constexpr int kBlockPos = 128;  // positions per block, one thread each for the folding
constexpr int kBlockStrip = 400;  // staged positions a block takes on run-on tiles

// Shared memory: P [strip][kChunk], F [2][kChunk][kBlockPos], slab rows
// [2][kChunk][kTile], second-level sums [16][threads] pairs, a row offset's taps, per
// staged position its row and column.
size_t block_smem(int strip, int R) {
  return sizeof(float) * ((size_t)strip * kChunk + 2 * kChunk * (kBlockPos + kTile)) +
         sizeof(uint64_t) * 16 * kBlockPos + sizeof(uint2) * (R + 2) + sizeof(int2) * strip;
}

// kVec: as above.
template <bool kVec>
__global__ void __launch_bounds__(kBlockPos, 4)
    k_corr_block(const CorrShape s, const float *__restrict__ in, float *__restrict__ out) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int R = s.R, NA = R + 1, wp = s.px + R;
  float *P = reinterpret_cast<float *>(smem);
  float *F = P + (size_t)s.strip * kChunk;
  float *S = F + 2 * kChunk * kBlockPos;
  uint64_t *sum2 = reinterpret_cast<uint64_t *>(S + 2 * kChunk * kTile) + threadIdx.x;  // this thread's, kBlockPos apart
  uint2 *tap = reinterpret_cast<uint2 *>(S + 2 * kChunk * kTile + 32 * kBlockPos);      // [R + 2]
  int2 *where = reinterpret_cast<int2 *>(tap + NA + 1);
  const int tid = threadIdx.x, T = blockIdx.y, tile = blockIdx.x;
  const int y0 = tile * kBlockPos / s.sp, x0 = tile * kBlockPos % s.sp;
  const int y1 = min((tile * kBlockPos + kBlockPos - 1) / s.sp, s.py - 1);  // rows of the tile
  stage_where<kBlockPos>(s, y0, x0, where);
  // staged index of the position this thread folds
  const int pm = ((tile * kBlockPos + tid) / s.sp - y0) * wp + ((tile * kBlockPos + tid) % s.sp - x0) + R;
  const int ng = tid & 7, pg = tid >> 3;  // outputs 4 ng .. +3 of the tile, positions 8 pg .. +7
  const int n = T * kTile + 4 * ng;
  uint64_t a1[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      a1[i][j] = 0;
      sum2[(4 * i + j) * kBlockPos] = 0;
    }
  // add a row offset's sums to the output
  auto flush = [&](bool first) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[j] = f2_unpack(sum2[(4 * i + j) * kBlockPos]);
        sum2[(4 * i + j) * kBlockPos] = 0;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int o = tile * kBlockPos + 8 * pg + 2 * i + h, y = o / s.sp, x = o % s.sp;
        if (y >= s.py || x >= s.px) continue;
        float *dst = out + ((size_t)y * s.px + x) * s.out_len + n;
        float w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = h ? v[j].y : v[j].x;
        if (s.out_len % 4 == 0) {
          if (n >= s.out_len) continue;
          float4 u = first ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<const float4 *>(dst);
          *reinterpret_cast<float4 *>(dst) =
              first ? make_float4(w[0], w[1], w[2], w[3]) : make_float4(u.x + w[0], u.y + w[1], u.z + w[2], u.w + w[3]);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (n + j < s.out_len) dst[j] = first ? w[j] : dst[j] + w[j];
        }
      }
    }
  };
  bool first = true;
  for (int b = 0; b <= R; ++b) {
    if (y0 + b >= s.py && y1 - b < 0) continue;  // neither row offset meets the grid
    __syncthreads();
    for (int a = tid; a <= NA; a += kBlockPos) tap[a] = s.taps[((size_t)T * NA + b) * (NA + 1) + a];
    __syncthreads();
    const uint2 all = tap[NA];
    if (!(all.x >> 16)) continue;
    for (int c = k_lo(all) / kChunk; c * kChunk < k_hi(all); ++c) {
      const int k0 = c * kChunk;
      // the chunk's taps, one bit each (the same in every warp)
      unsigned long long m0 = 0, m1 = 0;
      auto word = [&](int i) {
        const int a = 32 * i + (tid & 31);
        const uint2 t = a < NA ? tap[a] : make_uint2(0, 0);
        return (unsigned long long)__ballot_sync(0xffffffffu,
                                                 k_lo(t) < k0 + kChunk && k_hi(t) > k0 && (t.x >> 16));
      };
      m0 = word(0);
      if (NA > 32) m0 |= word(1) << 32;
      if (NA > 64) m1 = word(2);
      if (NA > 96) m1 |= word(3) << 32;
      auto request = [&](int buf) {  // the next tap's slab rows; returns it (NA: none is left)
        int a = NA;
        if (m0) {
          a = __ffsll((long long)m0) - 1;
          m0 &= m0 - 1;
        } else if (m1) {
          a = 63 + __ffsll((long long)m1);
          m1 &= m1 - 1;
        }
        if (a < NA) {
          const float *src = s.rows + ((size_t)tap[a].y + (c - k_lo(tap[a]) / kChunk)) * (kChunk * kTile);
          static_assert(kChunk * kTile == 4 * kBlockPos, "one 16-byte copy per thread");
          copy16_async(S + buf * kChunk * kTile + 4 * tid, src + 4 * tid, true);
        }
        copies_commit();
        return a;
      };
      __syncthreads();  // the previous chunk's operands are read
      int buf = 0, chain = 0, a = request(0);
      for (int i = tid; i < s.strip * (kChunk / 4); i += kBlockPos) {
        const int r = i / (kChunk / 4), kq = i % (kChunk / 4), k = k0 + 4 * kq;
        const int2 w = where[r];
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int side = 0; side < (b ? 2 : 1); ++side) {
          const int y = side ? w.x - b : w.x + b;
          if (w.y < 0 || y < 0 || y >= s.py) continue;
          const float *src = in + ((size_t)y * s.px + w.y) * s.len + k;
          float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
          if (kVec) {
            if (k < s.len) u = *reinterpret_cast<const float4 *>(src);
          } else {
            if (k < s.len) u.x = src[0];
            if (k + 1 < s.len) u.y = src[1];
            if (k + 2 < s.len) u.z = src[2];
            if (k + 3 < s.len) u.w = src[3];
          }
          v = make_float4(v.x + u.x, v.y + u.y, v.z + u.z, v.w + u.w);
        }
        *reinterpret_cast<float4 *>(P + p_at(r, kq)) = v;
      }
      __syncthreads();
      auto fold = [&](int a, int buf) {
#pragma unroll
        for (int kq = 0; kq < kChunk / 4; ++kq) fold_tap<kBlockPos>(P, pm, a, F + buf * kChunk * kBlockPos + tid, kq);
      };
      if (a < NA) fold(a, 0);
      while (a < NA) {
        copies_wait<0>();
        __syncthreads();  // this tap's operands are in place, the other buffer is read
        const int next = request(buf ^ 1);
        if (next < NA) fold(next, buf ^ 1);
        multiply<kBlockPos>(F + buf * kChunk * kBlockPos + 8 * pg, S + buf * kChunk * kTile + 4 * ng,
                            max(k_lo(tap[a]) - k0, 0) & ~3, min(k_hi(tap[a]) - k0, kChunk), a1);
        if (++chain == kFlush || next >= NA) {
          chain = 0;
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              sum2[(4 * i + j) * kBlockPos] = f2_add(sum2[(4 * i + j) * kBlockPos], a1[i][j]);
              a1[i][j] = 0;
            }
        }
        a = next;
        buf ^= 1;
      }
    }
    flush(first);
    first = false;
  }
  if (first) flush(true);  // no slab row meets the tile: zeros
}

oam_status run(const oam_model *m, bool fwd, const float *in, float *out, cudaStream_t st) {
  const oam_grid &g = m->grid;
  const DirectRows &L = fwd ? m->rows_fwd : m->rows_adj;
  CorrShape s{};
  s.px = g.px;
  s.py = g.py;
  s.R = m->R;
  s.len = fwd ? g.nz : g.nt;
  s.out_len = fwd ? g.nt : g.nz;
  s.taps = L.d_taps;
  s.rows = L.d_rows;
  const bool vec = s.len % 4 == 0;
  if (m->R == 0) {
    ProfScope prof(m, st, fwd);
    const dim3 grid((unsigned)(((long long)g.px * g.py + kPos - 1) / kPos), L.tiles);
    if (vec) k_corr_one<true><<<grid, kOneThreads, 0, st>>>(s, in, out);
    else k_corr_one<false><<<grid, kOneThreads, 0, st>>>(s, in, out);
    OAM_LAUNCHED();
    return OAM_OK;
  }
  // k_corr_block from three of its blocks with work on the fullest SM on: alone or in twos
  // they are bound by their chains of taps, which the eight warps cut eightfold.  us,
  // block against warps, with one: 48x48x64 31x31 taps 950, 259; two: 80x80x64 21x21
  // taps 516, 362, 64x64x128 61x61 taps 4202, 2976, 96x64x64 11x11 taps 171, 141,
  // 128x128x64 11x11 taps adjoint 312, 369; three: 128x96x100 15x15 taps adjoint 667,
  // 705; five: 96x96x128 31x31 taps 1498, 1818, 128x128x64 11x11 taps 218, 358.
  const long long busy = fwd ? (m->n_hi - m->n_lo + kTile - 1) / kTile : L.tiles;
  const int sms = std::max(1, m->sm_count);
  // Inputs of one chunk leave the warps nothing to share but their set-up (from one
  // block per SM on: 128x128x4 forward, 3x3 taps 15, 49; 9x9 taps 42, 70).
  const long long blocks = ((long long)g.px * g.py + kBlockPos - 1) / kBlockPos * busy;
  const bool block = blocks > (s.len <= kChunk ? 1LL : 2LL) * sms;
  // Tiles run on over scan rows (no idle positions) unless the padding between
  // many short rows makes the strip too long; then every tile stays in its row.
  const int tile = block ? kBlockPos : kPos;
  const int wrap = tile + ((s.px + tile - 2) / s.px + 2) * s.R;
  const bool run_on = wrap <= (block ? kBlockStrip : kMaxStrip);
  s.sp = run_on ? s.px : (s.px + tile - 1) / tile * tile;
  s.strip = run_on ? wrap : tile + 2 * s.R;
  const long long tiles = ((long long)s.py * s.sp + tile - 1) / tile;
  s.group = chunk_group(s.R);
  const size_t sm = block ? block_smem(s.strip, s.R) : warps_smem(s.strip, s.R, s.group);
  // Blocks that share out a tile's row offsets: the count that finishes first, in units of
  // a row offset, 0.6 more for a block's start and end, times the waves at the blocks an
  // SM holds (the idle part of the last wave counts half).  us with 1, 2, 4, 8: 32x32x48
  // 11x11 taps forward 43 30 34 44, adjoint 79 44 38 42; 70x37x52 15x15 taps adjoint
  // 132 116 94 98; 96x64x64 11x11 taps forward 171 191 272 532.
  int Z = 1;
  if (!block) {
    const double slots = (sm <= 112 * 1024 ? 2.0 : 1.0) * sms;
    double best = 0;
    for (int z = 1; z <= std::min(8, s.R + 1); z *= 2) {
      const double waves = (double)(tiles * busy * z) / slots;
      const double cost = (waves <= 1 ? 1.0 : 0.5 * (waves + std::ceil(waves))) * ((s.R + z) / z + 0.6);
      if (z == 1 || cost <= best) {
        best = cost;
        Z = z;
      }
    }
  }
  void (*const kernels[2][2][2])(const CorrShape, const float *, float *) = {
      {{k_corr_warps<false, false>, k_corr_warps<false, true>}, {k_corr_warps<true, false>, k_corr_warps<true, true>}},
      {{k_corr_block<false>, k_corr_block<false>}, {k_corr_block<true>, k_corr_block<true>}}};
  auto fn = kernels[block][vec][s.group > 1];
  // one limit for all launches: calls from several threads would lower each other's
  // between setting it and the launch
  OAM_CUDA_TRY(cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  ProfScope prof(m, st, fwd);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)tiles, L.tiles, Z);  // tile neighbours share slab rows
  cfg.blockDim = dim3(block ? kBlockPos : kThreads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = Z;
  cfg.attrs = &attr;
  cfg.numAttrs = Z > 1;
  OAM_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, s, in, out));
  OAM_LAUNCHED();
  return OAM_OK;
}

}  // namespace

// The split form takes three launches and two transforms, so small sums are faster here.  us
// of that form and of these kernels, with the triples of all position tiles: one tap 64x64x128
// 25, 8; 200x200x300 141, 85.  3x3 taps 600x1x128 37, 12 (0.7e3), 32x32x48 21, 12 (1e3),
// 48x48x101 23, 23 (4.6e3), 128x128x4 32, 15 (4.1e3), adjoint 28, 23 (6.1e3); 64x64x128
// 27, 37 (9.7e3), adjoint 25, 27.  5x5 taps 32x32x48 23, 16 (2.3e3), 48x48x101 23, 37 (1.0e4).
// One row of 17 taps 600x1x128 36, 23 (3.4e3), of 31 taps 45, 70.  Above nine folded taps it
// gains little (32x32x48, 7x7 taps 23, 19; 9x9 taps 21, 27), so those keep no rows.
bool oam::uses_direct(const oam_model *m, bool fwd) {
  if (m->precision != OAM_PREC_BF16X3) return m->precision == OAM_PREC_FP32;
  const DirectRows &L = fwd ? m->rows_fwd : m->rows_adj;
  if (!L.d_rows) return false;
  const long long tiles = ((long long)m->grid.px * m->grid.py + kPos - 1) / kPos;
  return m->R == 0 || tiles * L.items <= 6500;
}

oam_status oam::forward_fp32(const oam_model *m, const float *H, float *s, cudaStream_t st) {
  return run(m, true, H, s, st);
}

oam_status oam::adjoint_fp32(const oam_model *m, const float *s, float *H, cudaStream_t st) {
  return run(m, false, s, H, st);
}
