// Split-BF16 forward and adjoint operators on the 5th-generation tensor cores
// (tcgen05 MMA, accumulators in tensor memory, operands staged by the TMA
// engine).  Both are the lateral correlations of Eq. 4 ("two coordinate
// systems", Methods, Efficient reconstruction based on scanning symmetries).
//
// Along the scan's y axis the correlation is diagonal in the lateral frequency:
// with the lines of the input zero-padded to P points (mix_lines.cu), and the
// slab's transform over its row offset real because the slab is even in it
// (Results, axial symmetry),
//   S_v[a][k][n] = sum_b S[b][a][k][n] cos(2 pi v b / P),
// each of the P/2 + 1 frequencies v is a correlation along x alone, the same for
// the real and the imaginary part of the transformed lines:
//
//   forward  D_v[row][n] += sum_{a, k}  X_v[row + a][k] * S_v[a][k][n]
//   adjoint  D_v[row][k] += sum_{a, n}  X_v[row + a][n] * S_v[a][k][n]
//
// One implicit GEMM per block of 128 rows (positions x of a frequency's real and
// imaginary part): M = 128 rows (one tensor-memory lane each), N = the slab band
// of one 16-deep K chunk (time samples for A, depths for A^T), K = (tap a,
// 16-chunk).  The P/2 + 1 frequencies of two rows each stand for py + R padded
// scan rows, and a row meets R + 1 folded taps instead of (R + 1)^2: 24x fewer
// products than the correlation over both axes at a 61x61 window, for a slab
// (P/2 + 1) / (R + 1) = 4 times the size at 200 lines and two line transforms.
// Measured on a GB300 against that form (one application): 200x200x300 forward
// 5.78 -> 0.46 ms (k_corr_line 0.34), adjoint 5.71 -> 0.46 ms, 96x96x192 forward 0.86 ->
// 0.10 ms.
//
// Mirror folding.  S_v[a] = S_v[-a], so the two mirrored taps share one slab tile
// and their operand rows are summed before the product:
//   F[row][k] = X_v[row + a][k] + X_v[row - a][k]
// (one row for a = 0).  A block stages the rows of 32 K elements at a time (TMA,
// 128-byte swizzle); the fold warps build F from two shifted rows, split it into
// FP16 hi/lo in tensor memory, and one warp walks the items while an elected
// lane issues the MMAs with A read from tensor memory.
//
// The packed input holds, per frequency, R zero positions, then each row of px
// positions followed by R zeros (stride Wp = px + R), so a lateral offset a is a
// shift by a positions of a staged strip.  A block's 128 positions are
// consecutive in one of two grids (the position tiling, a tile parameter): the
// padded grid (o = row*Wp + x; padding positions compute and are dropped; strips
// of 128 + 2R positions) or the scan grid (o = row*px + x, every lane an output;
// lane m reads strip position m + R*(rows wrapped before m) + R + a, and a strip
// holds 128 + (w + 2) R positions for tiles that wrap w rows).
//
// Each product uses two-term 16-bit splits v = hi + lo of the slab and of the
// folded iterate: D += F_hi S_hi + F_hi S_lo + F_lo S_hi, accumulated in FP32 in
// tensor memory.  The terms are FP16 (22 significant bits together, BF16 terms
// hold 16) of operands scaled by powers of two: the slab by one for the model,
// the iterate by one for each frequency and row, from the magnitudes that the line
// transform finds on the lines of the row's window.  The taps of a tile go to up to four blocks, whose partial sums the
// inverse line transform adds in index order.  (Adding them in clusters through
// distributed shared memory was slower: 9000 cycles a block for two blocks' sums, and
// clusters of four leave SMs idle.)
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>

#include "f32x2.cuh"
#include "internal.cuh"
#include "tc_ptx.cuh"

using namespace oam;

namespace oam {

constexpr int kStageK = 32;        // K elements per stage (two 16-deep MMA chunks)
constexpr int kTileM = 128;        // positions per block
constexpr int kFoldWarpChoices[] = {4, 8, 16};  // warps that build the folded operand (then run the epilogue)
constexpr int kDefaultFoldWarps = 8;
constexpr int kMaxItems = 8;       // item ring depth (slab tile + folded operand)
constexpr int kFoldCols = 32;      // tensor-memory columns per folded operand: 2 chunks x (hi, lo) x 8
constexpr int kSmemLimit = 227 * 1024;
constexpr int kStageRow = 36;      // floats per row of a fold warp's 32 x 32 epilogue stage

// One ring item: the slab tiles of one (|a|, stage), hi then lo of each of
// its two 16-deep chunks; 8 bytes, so a block's item tables stay small.  The
// same for every frequency, whose tiles lie v_stride bytes apart.
struct __align__(8) TcItem {
  uint32_t off16;  // byte offset of the item's tiles in a frequency's data, in 16-byte units
  uint8_t c16[2];  // accumulator column / 16 of each tile
  uint8_t n16[2];  // MMA N / 16 of each tile (0 = no tile)
  __host__ __device__ uint32_t col(int c) const { return 16u * c16[c]; }
  __host__ __device__ uint32_t n(int c) const { return 16u * n16[c]; }
  __host__ __device__ uint32_t bytes() const { return 64u * (n(0) + n(1)); }  // hi + lo of both tiles
};

struct TcTile {
  int a, chunk, col, n;
  long long off;  // byte offset of the hi part in a frequency's data; lo follows after n*32 bytes
};

struct TcLayout {
  int dir = 0;            // 0 forward, 1 adjoint
  int stages = 0;         // K stages of kStageK
  int acc_cols = 0;       // accumulator width (multiple of 16)
  int out_lo = 0;         // output index of accumulator column 0
  int in_lo = 0;          // input index of packed element 0
  int in_elems = 0;       // packed elements per position (32 * stages)
  int slot_bytes = 0;     // shared-memory slot per item
  int ring_pref = 0;      // item-ring depth chosen by oam_model_autotune (0 = deepest that fits)
  int tiling = 0;         // position tiling: 0 auto, 1 padded grid, 2 scan grid
  int parts = 1;          // blocks that share a tile's taps
  bool wide = false;      // some tile is wider than one MMA
  double cols = 0;        // MMA columns x 16 summed over a = 0 .. R and the stages
  int fold_warps = kDefaultFoldWarps;  // fold-warp count chosen by oam_model_autotune (4, 8 or 16)
  TcItem *d_items = nullptr;  // [R + 1][stages]
  uint8_t *d_data = nullptr;  // [P/2 + 1][v_stride]
  size_t v_stride = 0;        // bytes of one frequency's tiles
  float *d_pack = nullptr;    // packed input [(P/2 + 1) rows][in_elems]
  std::vector<int2> reach;    // [stages] accumulator columns [x, y) that a stage's elements reach
  int2 *d_reach = nullptr;
  CUtensorMap tmap;       // FP32 packed input [qtot][in_elems], box 32 x (128 + 2R), 128-byte swizzle
  CUtensorMap tmap_scan;  // the same with the scan-grid strip positions (when they fit one box)
};

// The line transforms' plan, common to both directions.
struct TcLine {
  int P = 0, Q = 0;           // transform size, frequencies P/2 + 1
  int halo = 0;               // rows coupled along y: min(R, py - 1)
  int segs = 1, valid = 0;    // segments of a line, output rows of each
  int nr = 0, rows = 0;       // packed rows and positions per frequency
  int words = 0, planes = 0;  // mark words per column, planes (LineShape) of the direction with more
  float2 *d_tw = nullptr;     // [P] roots
  unsigned *d_marks = nullptr;  // [planes][px][words], [Q][px] magnitudes, two flags, [planes][px][words] grown
  unsigned *d_smax = nullptr;   // bound of the transformed slab's magnitude, as float bits
  float *d_part = nullptr;    // partial sums [parts][Q][nr][px][acc_cols]
};

}  // namespace oam

namespace {

struct CorrParams {
  int wp, px, R, stages;
  int sp;          // row stride of the grid the position tiles follow: Wp (padded) or px (scan)
  int nr, rows;    // packed rows and positions per frequency
  const TcItem *items;  // [R + 1][stages]
  const uint8_t *data;
  size_t v_stride;
  int slot_bytes, n_items, strip_rows, strip_bytes, items_bytes;
  int acc_cols, tmem_cols, fold_col0;
  const unsigned *marks;  // [planes][px][words] (LineShape): positions with a non-zero, with a non-finite input
  unsigned *grown;        // [planes][px][words]: positions whose window holds one
  const int *any_bad;     // some position has a non-finite input
  int *spoiled;           // the same, for the inverse transform
  int words, planes;
  const unsigned *vmax;  // [frequencies][px] largest magnitude of the transformed lines, as float bits
  const unsigned *smax;  // the slab's, over its transform (an upper bound)
  float *part;         // partial sums [parts][frequencies][nr][px][acc_cols]
  float *out;          // the operator's output [positions][out_len]: channels outside z0 .. z1 are zeroed here
  int positions, out_len, z0, z1;
  int *status;
  long long budget;
};

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int c0, int c1, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(ptx::smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(ptx::smem_addr(bar))
      : "memory");
}

// Lateral offset |a| of the j-th item of a stage.  Items alternate between
// the small and the large offsets (0, R, 1, R - 1, ...): the band, and with it
// the MMA width N, grows with the offset, so each pair of items costs about
// the same MMA time while its fold work is the same for every pair.
__device__ __forceinline__ int a_of(int j, int R) { return (j & 1) ? R - (j >> 1) : (j >> 1); }


// Staged FP32 rows are 128 bytes with the TMA's 128-byte swizzle: 16-byte
// chunk c of row r sits at chunk c ^ (r & 7).  Read the 8 elements of
// quarter q as four FP32 pairs.
__device__ __forceinline__ void load_row(const float *strip, int row, int q, uint64_t (&v)[4]) {
  const ulonglong2 *r2 = reinterpret_cast<const ulonglong2 *>(strip + row * 32);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const ulonglong2 u = r2[(2 * q + i) ^ (row & 7)];
    v[2 * i] = u.x;
    v[2 * i + 1] = u.y;
  }
}

// Add the 8 elements of quarter q of a staged row.
__device__ __forceinline__ void add_row(const float *strip, int row, int q, uint64_t (&v)[4]) {
  const ulonglong2 *r2 = reinterpret_cast<const ulonglong2 *>(strip + row * 32);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const ulonglong2 u = r2[(2 * q + i) ^ (row & 7)];
    v[2 * i] = f2_add(v[2 * i], u.x);
    v[2 * i + 1] = f2_add(v[2 * i + 1], u.y);
  }
}


// 2^e, -126 <= e <= 127.
__device__ __forceinline__ float pow2(int e) { return __int_as_float((e + 127) << 23); }

// Exponent e of the power of two that brings a magnitude of at most `top` into
// [2^14, 2^15), below FP16's largest 65504 (0 for an all-zero operand).
__device__ __forceinline__ int scale_exp(float top) {
  return top > 0.0f ? min(126, max(-126, 14 - ilogbf(top))) : 0;
}

// Split four FP32 pairs (scaled into FP16's range) into FP16 pairs: hi = v with
// its low 13 fraction bits cleared (an FP16 value), lo = v - hi rounded to
// nearest even; element 2e in the low half of word e.
__device__ __forceinline__ void split_f16(const uint64_t (&v)[4], uint32_t (&hv)[4], uint32_t (&lv)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 u = f2_unpack(v[e]);
    const float x = __uint_as_float(__float_as_uint(u.x) & 0xffffe000u);
    const float y = __uint_as_float(__float_as_uint(u.y) & 0xffffe000u);
    const __half2 h2 = __floats2half2_rn(x, y);
    const float2 rest = f2_unpack(f2_sub(v[e], f2_pack(x, y)));
    const __half2 l2 = __floats2half2_rn(rest.x, rest.y);
    hv[e] = *reinterpret_cast<const uint32_t *>(&h2);
    lv[e] = *reinterpret_cast<const uint32_t *>(&l2);
  }
}

// Fold one item: F = X[m + R + a] + X[m + R - a] (X[m + R] alone for a = 0)
// for this thread's row m and its E of the stage's 32 K elements (8-element
// quarters q0 .. q0 + E/8 - 1), times the power of two `sc`, split into FP16
// hi/lo words in the order the tensor-memory store takes them: E = 8: hi[4],
// lo[4]; E >= 16: per 16-deep chunk, hi[8] then lo[8].
template <int E>
__device__ __forceinline__ void fold_item(const float *X1, int m, int R, int a, int q0, uint64_t sc, uint32_t (&w)[E]) {
  constexpr int NQ = E / 8;
  uint64_t f[NQ][4];
#pragma unroll
  for (int i = 0; i < NQ; ++i) load_row(X1, m + R + a, q0 + i, f[i]);
  if (a > 0) {
#pragma unroll
    for (int i = 0; i < NQ; ++i) add_row(X1, m + R - a, q0 + i, f[i]);
  }
#pragma unroll
  for (int i = 0; i < NQ; ++i) {
#pragma unroll
    for (int e = 0; e < 4; ++e) f[i][e] = f2_mul(f[i][e], sc);
    uint32_t hv[4], lv[4];
    split_f16(f[i], hv, lv);
    const int hb = E == 8 ? 0 : 16 * (i >> 1) + 4 * (i & 1);  // word of the quarter's first hi pair
    const int lb = E == 8 ? 4 : hb + 8;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      w[hb + e] = hv[e];
      w[lb + e] = lv[e];
    }
  }
}

// Store one folded item into its tensor-memory slot (slot column 0 = chunk 0
// hi, 8 = chunk 0 lo, 16 = chunk 1 hi, 24 = chunk 1 lo; a column holds two
// FP16 K elements).
template <int E>
__device__ __forceinline__ void store_item(uint32_t slot_addr, int q0, const uint32_t (&w)[E]) {
  if constexpr (E == 8) {
    const uint32_t col = (uint32_t)(16 * (q0 >> 1) + 4 * (q0 & 1));
    uint32_t h[4] = {w[0], w[1], w[2], w[3]}, l[4] = {w[4], w[5], w[6], w[7]};
    ptx::tmem_st4(slot_addr + col, h);
    ptx::tmem_st4(slot_addr + col + 8u, l);
  } else if constexpr (E == 16) {
    ptx::tmem_st16(slot_addr + (uint32_t)(8 * q0), w);  // q0 = 2 * chunk
  } else {
    ptx::tmem_st32(slot_addr, w);
  }
}

// D (col d) += A (tensor memory, 16 deep) x B (n columns); kWide: n above one MMA's 256.
template <bool kWide>
__device__ __forceinline__ void mma_cols(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t n) {
  if (!kWide || n <= 256u) {
    ptx::mma_f16_ta(d, a, b, idesc | ((n >> 3) << 17), 1);
  } else {  // 256 columns, then the rest: 256 rows of 16 bytes further in the tile
    ptx::mma_f16_ta(d, a, b, idesc | (32u << 17), 1);
    ptx::mma_f16_ta(d + 256u, a, b + 256u, idesc | (((n - 256u) >> 3) << 17), 1);
  }
}

// The marks of column x (mix_lines.cu), or-ed over the columns within R and grown by
// R rows: one warp, lanes over columns, then over the rows of a word.
__device__ __forceinline__ void grow_marks(const CorrParams &p, int x, int lane) {
  const int xa = max(0, x - p.R), xb = min(p.px - 1, x + p.R);
  const int planes = *p.any_bad ? p.planes : 1;
  for (int which = 0; which < planes; ++which) {
    const unsigned *src = p.marks + (size_t)(which * p.px) * p.words;
    unsigned *dst = p.grown + (size_t)(which * p.px + x) * p.words;
    unsigned win[5] = {0, 0, 0, 0, 0};  // words w - 2 .. w + 2 (R <= 64)
    for (int j = -2; j < p.words; ++j) {  // word j + 2 joins; word j is complete
      unsigned m = 0;
      if (j + 2 < p.words)
        for (int xx = xa + lane; xx <= xb; xx += 32) m |= __ldcg(src + (size_t)xx * p.words + j + 2);
#pragma unroll
      for (int i = 0; i < 4; ++i) win[i] = win[i + 1];
      win[4] = __reduce_or_sync(0xffffffffu, m);
      if (j < 0) continue;
      bool any = false;
#pragma unroll
      for (int i = 0; i < 5; ++i) {  // rows lane - R .. lane + R of word j
        const int lo = max(lane - p.R - 32 * (i - 2), 0), hi = min(lane + p.R - 32 * (i - 2), 31);
        if (lo <= hi) any = any || (win[i] & (0xffffffffu << lo) & (0xffffffffu >> (31 - hi))) != 0;
      }
      const unsigned out = __ballot_sync(0xffffffffu, any);
      if (lane == 0) dst[j] = out;
    }
  }
}

// Zeros in the output's channels outside z0 .. z1 (whole groups of four) for this
// block's share of the positions: the store traffic runs under the products.
__device__ __forceinline__ void zero_outside(const CorrParams &p, int lane) {
  const int lo4 = p.z0 / 4, n4 = lo4 + (p.out_len - p.z1) / 4;
  if (n4 <= 0) return;
  const int blocks = gridDim.x * gridDim.y * gridDim.z, blk = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  const int per = (p.positions + blocks - 1) / blocks;
  for (int o = blk * per; o < min(p.positions, (blk + 1) * per); ++o) {
    float4 *row = reinterpret_cast<float4 *>(p.out + (size_t)o * p.out_len);
    for (int i = lane; i < n4; i += 32) row[i < lo4 ? i : p.z1 / 4 + i - lo4] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// Block (position tile, tap part, frequency).  What bounds it: shared memory.  A pair of
// items reads 64 KB of strip rows (512 cycles at 128 bytes each), the tensor cores read
// its tiles three times (336) and the copy engine writes them (224 cycles): 1072, and
// 1100 measured at 320 accumulator columns.
template <int FW, bool kWide>
__global__ void __launch_bounds__(96 + 32 * FW, 1)
    k_corr_line(const __grid_constant__ CUtensorMap tmap, const CorrParams p) {
  constexpr int kFoldWarps = FW;
  constexpr int kThreads = 96 + 32 * FW;
  constexpr int G = FW / 4;   // K groups per tensor-memory lane quarter
  constexpr int E = 32 / G;   // stage K elements folded per thread and item
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // 128-byte-swizzled TMA destinations need 1024-byte alignment
  uint8_t *smem = smem_raw + ((1024u - (ptx::smem_addr(smem_raw) & 1023u)) & 1023u);
  // item ring: slab tile in shared memory + folded operand in tensor memory;
  // items go in pairs (the two taps of one fold pass), one set of barriers per pair
  const int K = p.n_items, KP = K / 2;
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
  uint64_t *strip_full = bars, *strip_empty = bars + 3;  // one pair per strip buffer
  uint64_t *acc_ready = bars + 6, *acc_full = bars + 7;
  uint64_t *slab_full = bars + 8, *fold_full = bars + 8 + KP, *item_empty = bars + 8 + 2 * KP;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + 512);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + 516);
  volatile int *never = reinterpret_cast<volatile int *>(smem + 520);  // stays 0: waits that ignore abort
  uint8_t *line_exp = smem + 640;  // [strip_rows <= 256] biased exponents of the strip's lines (0: padding)
  TcItem *sitems = reinterpret_cast<TcItem *>(smem + 1024);           // [stages][nj]: this part's items
  uint8_t *strips = smem + 1024 + p.items_bytes;                       // [3][strip_bytes]: stage st in buffer st % 3
  uint8_t *slots = strips + 3 * p.strip_bytes;                         // [K][slot_bytes]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile = blockIdx.x, parts = gridDim.y, freq = blockIdx.z;
  const int R = p.R, NA = R + 1, NP = (NA + 1) / 2;  // a = 0 .. R in pairs
  const int j0 = 2 * ((int)blockIdx.y * NP / parts), j1 = min(NA, 2 * (((int)blockIdx.y + 1) * NP / parts)), nj = j1 - j0;
  const int r0 = tile * kTileM / p.sp, x0 = tile * kTileM % p.sp;  // the tile's first position
  const int qt = freq * p.rows + r0 * p.wp + x0;                    // strip start: R positions before it
  const uint8_t *data = p.data + (size_t)freq * p.v_stride;
  const int L = p.strip_rows;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 3; ++i) {
      ptx::mbar_init(&strip_full[i], 1);
      ptx::mbar_init(&strip_empty[i], kFoldWarps);
    }
    ptx::mbar_init(acc_ready, kFoldWarps);
    ptx::mbar_init(acc_full, 1);
    for (int i = 0; i < KP; ++i) {
      ptx::mbar_init(&slab_full[i], 1);
      ptx::mbar_init(&fold_full[i], kFoldWarps);
      ptx::mbar_init(&item_empty[i], 1);
    }
    *abort_flag = 0;
    *never = 0;
    ptx::mbar_fence_init();
    // the first strips travel while the block sets up
    for (int st = 0; st < min(2, p.stages); ++st) {
      ptx::mbar_arrive_expect_tx(&strip_full[st], (uint32_t)(L * 128));
      tma_load_2d(strips + (size_t)st * p.strip_bytes, &tmap, kStageK * st, qt, &strip_full[st]);
    }
  }
  for (int i = threadIdx.x; i < p.stages * nj; i += kThreads)
    sitems[i] = p.items[a_of(j0 + i % nj, R) * p.stages + i / nj];
  for (int i = threadIdx.x; i < L; i += kThreads) {
    const int q = r0 * p.wp + x0 - R + i, x = q < 0 ? p.px : q % p.wp;
    line_exp[i] = x < p.px ? (uint8_t)(__ldg(p.vmax + (size_t)freq * p.px + x) >> 23) : 0;
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, p.tmem_cols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  auto fail = [&](int code) {
    *abort_flag = 1;
    atomicOr(p.status, code);
  };

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int it_slab = 0, loads = min(2, p.stages);  // item pairs and strips requested (two before the block's barrier)
      int k = 0;
      uint32_t lap = 0;  // parity of the item ring's current lap
      bool ok = true;
      // Stage st's strip goes to buffer st % 3 once the fold warps have released
      // stage st - 3; it is requested two stages ahead of its use.
      auto load_strip = [&](int st) {
        const int s = st % 3;
        if (!ptx::mbar_wait(&strip_empty[s], ((st / 3) & 1) ^ 1, abort_flag, p.budget)) return false;
        ptx::mbar_arrive_expect_tx(&strip_full[s], (uint32_t)(L * 128));
        tma_load_2d(strips + (size_t)s * p.strip_bytes, &tmap, kStageK * st, qt, &strip_full[s]);
        ++loads;
        return true;
      };
      for (int st = 0; st < p.stages && ok; ++st) {
        const TcItem *row_items = sitems + st * nj;
        for (int j = 0; j < nj; j += 2) {  // pair slot k holds items j (slot 2k) and j + 1 (slot 2k + 1) of the stage
          const TcItem ia = row_items[j], ib = j + 1 < nj ? row_items[j + 1] : TcItem{};
          if (!ptx::mbar_wait(&item_empty[k], lap ^ 1, abort_flag, p.budget)) {
            fail(2);
            ok = false;
            break;
          }
          ptx::mbar_arrive_expect_tx(&slab_full[k], ia.bytes() + ib.bytes());
          if (ia.bytes() > 0)
            ptx::bulk_g2s(slots + (size_t)(2 * k) * p.slot_bytes, data + (size_t)ia.off16 * 16, ia.bytes(),
                          &slab_full[k]);
          if (ib.bytes() > 0)
            ptx::bulk_g2s(slots + (size_t)(2 * k + 1) * p.slot_bytes, data + (size_t)ib.off16 * 16, ib.bytes(),
                          &slab_full[k]);
          ++it_slab;
          if (++k == KP) {
            k = 0;
            lap ^= 1;
          }
          if (j == 0 && st + 2 < p.stages && !load_strip(st + 2)) {
            fail(1);
            ok = false;
            break;
          }
        }
      }
      if (!ok) {
        // let copies already issued land before the block exits
        for (int i = std::max(0, it_slab - KP); i < it_slab; ++i)
          ptx::mbar_wait(&slab_full[i % KP], (i / KP) & 1, never, p.budget);
        for (int st = std::max(0, loads - 3); st < loads; ++st)
          ptx::mbar_wait(&strip_full[st % 3], (st / 3) & 1, never, p.budget);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // The whole warp walks the item ring, so every MMA operand is computed
    // warp-uniformly; one elected lane issues the MMAs and commits.  (A loop
    // run by a single lane issues at about half the rate.)
    bool ok = __all_sync(0xffffffffu, ptx::mbar_wait(acc_ready, 0, abort_flag, p.budget));
    if (!ok && lane == 0) fail(4);
    ptx::tc_fence_after();
    const bool leader = ptx::elect_one();
    int k = 0;
    uint32_t lap = 0;
    // B descriptor template (start-address field in 16-byte units; fields never carry)
    const uint64_t slot_desc = ptx::smem_desc(ptx::smem_addr(slots), 0, 128);
    const uint32_t idesc = ptx::idesc_f16_f32(kTileM, 0);
    for (int st = 0; st < p.stages && ok; ++st) {
      const TcItem *row_items = sitems + st * nj;
      for (int j = 0; j < nj; j += 2) {
        bool w = ptx::mbar_wait(&slab_full[k], lap, abort_flag, p.budget);
        if (w) w = ptx::mbar_wait(&fold_full[k], lap, abort_flag, p.budget);
        if (!__all_sync(0xffffffffu, w)) {
          if (lane == 0) fail(8);
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        for (int h = 0; h < 2 && j + h < nj; ++h) {
          const TcItem item = row_items[j + h];
          const uint32_t slot = (uint32_t)(2 * k + h);
          const uint32_t a_base = tmem + (uint32_t)p.fold_col0 + 32u * slot;
          const uint64_t dB = slot_desc + (uint64_t)((slot * (uint32_t)p.slot_bytes) >> 4);
          const uint32_t n0 = item.n(0), n1 = item.n(1);
          const uint64_t b0h = dB + ((uint64_t)n0 << 16), b0l = b0h + 2u * n0;  // lbo = 16 n bytes; lo 32 n bytes on
          const uint64_t dB1 = dB + 4u * n0;                                   // second tile 64 n0 bytes later
          const uint64_t b1h = dB1 + ((uint64_t)n1 << 16), b1l = b1h + 2u * n1;
          const uint32_t d0 = tmem + item.col(0), d1 = tmem + item.col(1);
          if (leader) {
            // the two chunks accumulate into different columns: interleave them
            if (n0) mma_cols<kWide>(d0, a_base, b0h, idesc, n0);
            if (n1) mma_cols<kWide>(d1, a_base + 16u, b1h, idesc, n1);
            if (n0) mma_cols<kWide>(d0, a_base + 8u, b0h, idesc, n0);
            if (n1) mma_cols<kWide>(d1, a_base + 24u, b1h, idesc, n1);
            if (n0) mma_cols<kWide>(d0, a_base, b0l, idesc, n0);
            if (n1) mma_cols<kWide>(d1, a_base + 16u, b1l, idesc, n1);
          }
        }
        if (leader) ptx::mma_commit(&item_empty[k]);  // the pair's slots are free once its MMAs complete
        __syncwarp();
        if (++k == KP) {
          k = 0;
          lap ^= 1;
        }
      }
    }
    if (leader) ptx::mma_commit(acc_full);
    __syncwarp();
  } else if (warp == 2 + kFoldWarps) {
    // ------------------------------------------------------------ marks, zeros
    zero_outside(p, lane);
    if (lane == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) *p.spoiled = *p.any_bad;
    if (blockIdx.y == 0)
      for (int x = freq * gridDim.x + tile; x < p.px; x += gridDim.z * gridDim.x) grow_marks(p, x, lane);
  } else {
    // ------------------------------------------------------------ fold warps, then epilogue
    const int fw = warp - 2;        // 0 .. kFoldWarps-1
    const int quarter = warp & 3;   // tensor-memory lanes 32*quarter .. +31
    const int kq = fw >> 2;         // K group of the stage this warp folds (E elements)
    const uint32_t lane_base = (uint32_t)(32 * quarter) << 16;
    const int nb = (p.acc_cols + 31) / 32;  // 32-column blocks of the accumulator
    const int blk_begin = kq * nb / G, blk_end = (kq + 1) * nb / G;
    for (int j = blk_begin; j < blk_end; ++j) ptx::tmem_st32_zero(tmem + lane_base + (uint32_t)(32 * j));
    ptx::tmem_wait_st();
    ptx::tc_fence_before();
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(acc_ready);

    bool ok = true;
    const int m = 32 * quarter + lane;  // row (tensor-memory lane) this thread folds
    const int o = tile * kTileM + m;    // its position in the tile grid
    const int row = o / p.sp, x = o % p.sp;
    const int pm = (row - r0) * p.wp + (x - x0);  // its packed offset from the tile's first
    const int q0 = kq * (E / 8);        // first 8-element quarter of the stage
    // The row's own scale, from the largest magnitude of the lines in its window: one of the
    // whole scan would leave FP16's range to columns 1e-6 below its strongest.
    int top = 0;
#pragma unroll 8
    for (int i = pm; i <= pm + 2 * R; ++i) top = max(top, (int)line_exp[i]);
    const int ef = min(126, 140 - top);  // the fold doubles: into [2^14, 2^15), below FP16's largest 65504
    const uint64_t sc = f2_pack(pow2(ef), pow2(ef));
    int k = 0;
    uint32_t lap = 0;
    for (int st = 0; st < p.stages && ok; ++st) {
      const int s = st % 3;
      ok = __all_sync(0xffffffffu, ptx::mbar_wait(&strip_full[s], (st / 3) & 1, abort_flag, p.budget));
      if (!ok) {
        if (lane == 0) fail(32);
        break;
      }
      const float *X1 = reinterpret_cast<const float *>(strips + (size_t)s * p.strip_bytes);
      // two items per pass, in pair slot k: one wait, fence and barrier step for both
      for (int j = 0; j < nj; j += 2) {
        const bool two = j + 1 < nj;
        uint32_t w0[E], w1[E];  // folded in registers while the pair slot may still be in use
        fold_item<E>(X1, pm, R, a_of(j0 + j, R), q0, sc, w0);
        if (two) fold_item<E>(X1, pm, R, a_of(j0 + j + 1, R), q0, sc, w1);
        ok = ptx::mbar_wait(&item_empty[k], lap ^ 1, abort_flag, p.budget);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
          if (lane == 0) fail(64);
          break;
        }
        const uint32_t fa = tmem + lane_base + (uint32_t)p.fold_col0 + 64u * (uint32_t)k;
        store_item<E>(fa, q0, w0);
        if (two) store_item<E>(fa + 32u, q0, w1);
        ptx::tmem_wait_st();
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&fold_full[k]);
        if (++k == KP) {
          k = 0;
          lap ^= 1;
        }
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&strip_empty[s]);
    }

    // Epilogue: this warp's lane quarter and column share of the accumulator.  A lane
    // holds one row; 32-column blocks go through the (now free) strips, rows of 36 floats
    // so that neither side meets a bank twice, and leave as four whole 128-byte pieces a
    // store.  6900 cycles a block at 320 columns: the blocks of a wave write together, and
    // 24 bytes a cycle from each of 152 SMs are the memory's rate.
    bool done = ptx::mbar_wait(acc_full, 0, abort_flag, 4 * p.budget);
    done = __all_sync(0xffffffffu, done && ok);
    ptx::tc_fence_after();
    if (done) {
      const float us = pow2(-scale_exp(__uint_as_float(*p.smax))), uf = pow2(-ef);
      const int pos = row < p.nr && x < p.px ? row * p.px + x : -1;  // this lane's row in the output
      float *base = p.part + ((size_t)blockIdx.y * gridDim.z + freq) * p.nr * p.px * p.acc_cols + 4 * (lane & 7);
      float *dst[8];  // rows 4 i + lane / 8 of the quarter
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int q = __shfl_sync(0xffffffffu, pos, 4 * i + (lane >> 3));
        dst[i] = q >= 0 ? base + (size_t)q * p.acc_cols : nullptr;
      }
      float *stage = reinterpret_cast<float *>(strips) + fw * 32 * kStageRow;
      for (int j = blk_begin; j < blk_end; ++j) {
        uint32_t r[32];
        ptx::tmem_ld32(tmem + lane_base + (uint32_t)(32 * j), r);
        ptx::tmem_wait_ld();
        auto val = [&](int i) { return __uint_as_float(r[i]) * us * uf; };  // exact unless it leaves FP32's range
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 8; ++q)
          *reinterpret_cast<float4 *>(stage + lane * kStageRow + 4 * q) =
              make_float4(val(4 * q), val(4 * q + 1), val(4 * q + 2), val(4 * q + 3));
        __syncwarp();
        if (32 * j + 4 * (lane & 7) < p.acc_cols) {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (dst[i])
              *reinterpret_cast<float4 *>(dst[i] + 32 * j) =
                  *reinterpret_cast<const float4 *>(stage + (4 * i + (lane >> 3)) * kStageRow + 4 * (lane & 7));
        }
      }
    }
    ptx::tc_fence_before();
  }
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, p.tmem_cols);
  }
}

// ---------------------------------------------------------------- packers
// Slab tiles of every frequency: hi then lo, each [2 chunks of 8][n rows][8] FP16
// (K-major core matrices).  S_v[a][k][n] = sum_{b=0}^{halo} w_b cos(2 pi v b / P)
// S[b][a][k][n], w_0 = 1, w_{>0} = 2 (the +-b pair; row offsets beyond the halo
// meet no row).  Block (tile, kPackThreads of its elements), a thread per element:
// the slab values of its element in shared memory, then every frequency in turn.
constexpr int kPackThreads = 128;

// Upper bound of the transformed slab's magnitude: its largest entry times the
// window (the weights of a row offset's cosine sum to at most W).
__global__ void k_slab_max(const float *__restrict__ band, size_t n, float terms, unsigned *smax) {
  float top = 0.0f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    top = fmaxf(top, fabsf(band[i]));
  const unsigned t = __reduce_max_sync(0xffffffffu, __float_as_uint(top * terms));
  if ((threadIdx.x & 31) == 0) atomicMax(smax, t);
}

__global__ void __launch_bounds__(kPackThreads) k_pack_tiles(const float *__restrict__ band, const int *band_lo,
                                                             const int *band_hi, int band_w, int nz, int dir, int t_lo,
                                                             const int *tap_orbit, int R, int halo, int P,
                                                             const float2 *__restrict__ tw, const unsigned *smax,
                                                             const TcTile *tiles, size_t v_stride, uint8_t *data) {
  extern __shared__ float smp[];
  float *cosT = smp, *sv = smp + P;  // [P], [halo + 1][kPackThreads]
  const TcTile t = tiles[blockIdx.x];
  if ((int)blockIdx.y * kPackThreads >= 16 * t.n) return;
  const int tid = threadIdx.x, i = blockIdx.y * kPackThreads + tid;
  for (int j = tid; j < P; j += kPackThreads) cosT[j] = tw[j].x;
  __syncthreads();
  if (i >= 16 * t.n) return;
  const int row = (i >> 3) % t.n, kk = (i / (8 * t.n)) * 8 + (i & 7);  // row: along N, kk: along K (0..15)
  const int k = dir == 0 ? 16 * t.chunk + kk : t.col + row;
  const int n = dir == 0 ? t_lo + t.col + row : t_lo + 16 * t.chunk + kk;
  const int W = 2 * R + 1;
  for (int b = 0; b <= halo; ++b) {
    float v = 0.0f;
    if (k < nz) {
      const int o = tap_orbit[(b + R) * W + (t.a + R)];
      const int lo = band_lo[o * nz + k], hi = band_hi[o * nz + k];
      if (n >= lo && n < hi) v = band[((size_t)o * nz + k) * band_w + (n - lo)];
    }
    sv[b * kPackThreads + tid] = b == 0 ? v : 2.0f * v;
  }
  const float sc = pow2(scale_exp(__uint_as_float(*smax)));
  __half *dst = reinterpret_cast<__half *>(data + t.off) + i;
  auto put = [&](int f, float v) {
    v *= sc;
    const __half h = __float2half_rn(v);
    __half *d = dst + (size_t)f * (v_stride / sizeof(__half));
    d[0] = h;
    d[16 * t.n] = __float2half_rn(v - __half2float(h));
  };
  // Frequencies f and P / 2 - f (P is a multiple of 4) differ in the sign of the odd row
  // offsets' terms; four pairs at a time share a slab value.
  for (int f0 = 0; f0 <= P / 4; f0 += 4) {
    float even[4] = {}, odd[4] = {};
    int j[4] = {}, step[4];  // j = f b mod P
#pragma unroll
    for (int q = 0; q < 4; ++q) step[q] = f0 + q;
    auto term = [&](int b, float (&sum)[4]) {
      const float v = sv[b * kPackThreads + tid];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        sum[q] = fmaf(cosT[j[q]], v, sum[q]);
        j[q] += step[q];
        if (j[q] >= P) j[q] -= P;
      }
    };
    for (int b = 0; b <= halo; b += 2) {
      term(b, even);
      if (b < halo) term(b + 1, odd);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int f = f0 + q;
      if (f > P / 4) break;
      put(f, even[q] + odd[q]);
      if (f < P / 4) put(P / 2 - f, even[q] - odd[q]);
    }
  }
}

// Positions of a staged strip on the scan grid: 128 positions wrap at most
// (px + 126) / px rows, each adding R rows of padding to the span, plus
// R rows of halo on either side.
int strip_rows_for(int px, int R) { return kTileM + ((px + kTileM - 2) / px + 2) * R; }

int pow2_cols(int n) {
  int c = 32;
  while (c < n) c <<= 1;
  return c;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

oam_status encode_tmap(CUtensorMap *map, float *base, long long qtot, int elems, int rows) {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !p) {
      cudaGetLastError();
      return OAM_ERR_CUDA;
    }
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  const cuuint64_t dims[2] = {(cuuint64_t)elems, (cuuint64_t)qtot};
  const cuuint64_t strides[1] = {(cuuint64_t)elems * sizeof(float)};
  const cuuint32_t box[2] = {(cuuint32_t)kStageK, (cuuint32_t)rows};
  const cuuint32_t estr[2] = {1, 1};
  if (fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
         CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
      CUDA_SUCCESS)
    return OAM_ERR_CUDA;
  return OAM_OK;
}

// Longest line one transform takes.
constexpr int kLineMax = 512;

// The line transforms' plan: the smallest size that holds a line and its halo, or
// overlapping segments of the largest.
oam_status plan_line(const oam_model *m, TcLine *T) {
  const int py = m->grid.py;
  T->halo = std::min(m->R, py - 1);
  T->segs = 1;
  T->valid = py;
  T->P = py + T->halo <= kLineMax ? mix_size_for(py + T->halo) : kLineMax;
  if (py + T->halo > kLineMax) {
    T->valid = kLineMax - 2 * T->halo;
    T->segs = (py + T->valid - 1) / T->valid;
  }
  T->Q = T->P / 2 + 1;
  T->nr = 2 * T->segs;
  const long long rows = m->R + (long long)T->nr * (m->grid.px + m->R);
  if (rows * T->Q > 0x7fffffffLL) return OAM_ERR_UNSUPPORTED;
  T->rows = (int)rows;
  T->words = (py + 31) / 32;
  return OAM_OK;
}

// Sample (forward) or depth (adjoint) range [x, y) of the slab of every orbit in each
// 16-deep K chunk, from accumulator column 0: [orbit][chunks] (x >= y: none), in one pass
// over the bands.
std::vector<int2> chunk_ranges(const oam_model *m, int dir, int chunks, int t_lo) {
  const int nz = m->grid.nz;
  std::vector<int2> r((size_t)m->n_orb * chunks, make_int2(1 << 30, -1));
  for (int o = 0; o < m->n_orb; ++o) {
    int2 *row = r.data() + (size_t)o * chunks;
    for (int k = 0; k < nz; ++k) {
      const int bl = m->h_band_lo[(size_t)o * nz + k] - t_lo, bh = m->h_band_hi[(size_t)o * nz + k] - t_lo;
      if (bh <= bl) continue;
      const int lo = dir == 0 ? bl : k, hi = dir == 0 ? bh : k + 1;
      const int c0 = dir == 0 ? k / 16 : bl / 16, c1 = dir == 0 ? k / 16 : (bh - 1) / 16;
      for (int c = c0; c <= c1; ++c) row[c] = make_int2(std::min(row[c].x, lo), std::max(row[c].y, hi));
    }
  }
  return r;
}

// Columns [col, col + n) of a tile over a range, whole 16-column groups.
void tile_cols(int lo, int hi, int *col, int *n) {
  *col = lo & ~15;
  *n = ((hi - *col) + 15) & ~15;
}

// Blocks that share a tile's taps.  At least one per 5 1/3 pairs of taps: the tensor
// cores truncate when they add to an accumulator, and the frequencies' sums cancel
// over depth, so the fewer products one accumulator takes the less that costs
// (200x200x300, 16 pairs, forward with 1, 2, 3, 4 parts: 4.7e-6, 2.3e-6, 1.5e-6,
// 1.2e-6 against FP64, and 3.4e-6 for three BF16 products per tap with no transform;
// 164x228x154, 11 pairs: 4.4e-6, 2.1e-6, 1.5e-6, 1.2e-6 and 1.9e-6).  Beyond
// that, as many as finish first, in units of one pair of items (~0.55 us): a block's
// pairs and about 18 for its set-up and epilogue, times the waves of one block per SM,
// and a part's sums written and read once more (40 us for 62 MB).
int choose_parts(const TcLine *T, int px, int R, int stages, int acc_cols) {
  constexpr int kSms = 152;  // of every device: the footprint query has none to ask
  const int NP = (R + 2) / 2;
  const long long tiles0 = ((long long)T->nr * px + kTileM - 1) / kTileM * T->Q;
  const double part_units = (double)T->Q * T->nr * px * acc_cols * 4.0 / (1.55e12 * 0.55e-6);
  double best = 0;
  int parts = 0;
  for (int q = std::min(4, (3 * NP + 15) / 16); q <= std::min(4, NP); ++q) {
    const double cost = (double)((tiles0 * q + kSms - 1) / kSms) * ((double)((NP + q - 1) / q) * stages + 18) +
                        (q - 1) * part_units;
    if (!parts || cost < best) {
      best = cost;
      parts = q;
    }
  }
  return parts;
}

// K stages and accumulator columns of one direction for the support [n_lo, n_hi).
void dir_sizes(int dir, int nz, int n_lo, int n_hi, int *stages, int *acc_cols) {
  const int support = n_hi - (n_lo & ~15);
  *stages = ((dir == 0 ? nz : support) + kStageK - 1) / kStageK;
  *acc_cols = ((dir == 0 ? support : nz) + 15) & ~15;
}

// One direction's item and tile tables from the band form (host only): per (|a|,
// stage) the union of the row offsets' bands.
oam_status plan_dir(const oam_model *m, const TcLine *T, TcLayout *L, int dir, std::vector<TcItem> &items,
                    std::vector<TcTile> &tiles) {
  const int nz = m->grid.nz, R = m->R, W = m->W;
  const int t_lo = m->n_lo & ~15;
  L->dir = dir;
  dir_sizes(dir, nz, m->n_lo, m->n_hi, &L->stages, &L->acc_cols);
  L->out_lo = dir == 0 ? t_lo : 0;
  L->in_lo = dir == 0 ? 0 : t_lo;
  L->in_elems = kStageK * L->stages;
  if (pow2_cols(L->acc_cols) > 512) return OAM_ERR_UNSUPPORTED;

  items.assign((size_t)(R + 1) * L->stages, TcItem{});
  L->reach.assign(L->stages, make_int2(L->acc_cols, 0));
  const int chunks = 2 * L->stages;
  const std::vector<int2> ranges = chunk_ranges(m, dir, chunks, t_lo);
  tiles.clear();
  long long off = 0;
  int max_item = 16;
  L->wide = false;
  L->cols = 0;
  for (int a = 0; a <= R; ++a) {
    for (int s = 0; s < L->stages; ++s) {
      TcItem it{};
      it.off16 = (uint32_t)(off / 16);
      for (int c = 0; c < 2; ++c) {
        const int chunk = 2 * s + c;
        int lo = 1 << 30, hi = -1;
        for (int b = 0; b <= R; ++b) {
          const int2 r = ranges[(size_t)m->h_tap_orbit[(b + R) * W + (a + R)] * chunks + chunk];
          const int bl = r.x, bh = r.y;
          int col, n;
          if (bh <= bl) continue;
          // a single offset's band wider than 256 columns is not taken
          tile_cols(bl, bh, &col, &n);
          if (n > 256 || col + n > L->acc_cols) return OAM_ERR_UNSUPPORTED;
          if (b > T->halo) continue;
          lo = std::min(lo, bl);
          hi = std::max(hi, bh);
        }
        if (hi <= lo) continue;
        int col, n;
        tile_cols(lo, hi, &col, &n);
        L->reach[s] = make_int2(std::min(L->reach[s].x, col), std::max(L->reach[s].y, col + n));
        it.c16[c] = (uint8_t)(col / 16);
        it.n16[c] = (uint8_t)(n / 16);
        L->wide = L->wide || n > 256;
        L->cols += 16.0 * n;
        tiles.push_back(TcTile{a, chunk, col, n, off});
        off += 64LL * n;  // hi + lo: 2 x (n rows x 16 elements x 2 bytes)
      }
      max_item = std::max(max_item, (int)it.bytes());
      items[(size_t)a * L->stages + s] = it;
    }
  }
  L->slot_bytes = (max_item + 127) & ~127;
  L->v_stride = (size_t)std::max<long long>(off, 16);
  L->parts = choose_parts(T, m->grid.px, R, L->stages, L->acc_cols);
  return OAM_OK;
}

// Build one direction's item and tile tables from the band form, then pack.
oam_status build_dir(oam_model *m, TcLayout *L, int dir, cudaStream_t st, int *d_band_hi) {
  const TcLine *T = m->tc_line;
  std::vector<TcItem> items;
  std::vector<TcTile> tiles;
  oam_status rc = plan_dir(m, T, L, dir, items, tiles);
  if (rc) return rc;
  const int nz = m->grid.nz, t_lo = m->n_lo & ~15;
  const size_t qtot = (size_t)T->rows * T->Q;
  if ((rc = dev_alloc(m, &L->d_items, items.size()))) return rc;
  if ((rc = dev_alloc(m, &L->d_data, L->v_stride * T->Q))) return rc;
  if ((rc = dev_alloc(m, &L->d_pack, qtot * L->in_elems))) return rc;
  if ((rc = dev_alloc(m, &L->d_reach, L->reach.size()))) return rc;
  OAM_CUDA_TRY(cudaMemcpyAsync(L->d_reach, L->reach.data(), sizeof(int2) * L->reach.size(), cudaMemcpyHostToDevice, st));
  OAM_CUDA_TRY(cudaMemcpyAsync(L->d_items, items.data(), sizeof(TcItem) * items.size(), cudaMemcpyHostToDevice, st));
  // padding positions and channels stay zero: the line transform writes the others
  OAM_CUDA_TRY(cudaMemsetAsync(L->d_pack, 0, sizeof(float) * qtot * L->in_elems, st));
  if (!tiles.empty()) {
    int n_max = 0;
    for (const TcTile &t : tiles) n_max = std::max(n_max, t.n);
    TcTile *d_tiles = nullptr;
    OAM_CUDA_TRY(cudaMallocAsync((void **)&d_tiles, sizeof(TcTile) * tiles.size(), st));
    OAM_CUDA_TRY(cudaMemcpyAsync(d_tiles, tiles.data(), sizeof(TcTile) * tiles.size(), cudaMemcpyHostToDevice, st));
    const dim3 grid((unsigned)tiles.size(), (unsigned)((16 * n_max + kPackThreads - 1) / kPackThreads));
    const size_t sm = sizeof(float) * ((size_t)T->P + (size_t)(T->halo + 1) * kPackThreads);  // at most 35 KB
    k_pack_tiles<<<grid, kPackThreads, sm, st>>>(m->d_band, m->d_band_lo, d_band_hi, m->band_w, nz, dir, t_lo,
                                                 m->d_tap_orbit, m->R, T->halo, T->P, T->d_tw, T->d_smax,
                                                 d_tiles, L->v_stride, L->d_data);
    OAM_LAUNCHED();
    OAM_CUDA_TRY(cudaFreeAsync(d_tiles, st));
  }
  OAM_CUDA_TRY(cudaStreamSynchronize(st));  // host tables above go out of scope
  for (int scan = 0; scan < 2; ++scan) {
    const int rows = scan ? strip_rows_for(m->grid.px, m->R) : kTileM + 2 * m->R;
    if (rows > 256) continue;
    rc = encode_tmap(scan ? &L->tmap_scan : &L->tmap, L->d_pack, (long long)qtot, L->in_elems, rows);
    if (rc) return rc;
  }
  return OAM_OK;
}

struct Launch {
  CorrParams p;
  size_t smem;
  int tiling;   // 1 padded grid, 2 scan grid
  int n_tiles;  // position tiles of a frequency (the grid's x)
};

oam_status plan_launch(const oam_model *m, const TcLine *T, const TcLayout *L, Launch *out) {
  const int R = m->R, px = m->grid.px;
  CorrParams p{};
  p.wp = px + R;
  p.px = px;
  p.R = R;
  p.stages = L->stages;
  p.nr = T->nr;
  p.rows = T->rows;
  p.items = L->d_items;
  p.data = L->d_data;
  p.v_stride = L->v_stride;
  p.slot_bytes = L->slot_bytes;
  p.items_bytes = (int)((sizeof(TcItem) * L->stages * (R + 1) + 1023) & ~size_t(1023));
  p.fold_col0 = (L->acc_cols + 31) & ~31;
  const int tmem_items = (512 - p.fold_col0) / kFoldCols;
  auto strip_bytes = [](int rows) { return (rows * 128 + 1023) & ~1023; };  // 128-byte rows, 1024-byte aligned
  auto fixed_for = [&](int rows) { return 1024 /* alignment slack */ + 1024 + p.items_bytes + 3 * strip_bytes(rows); };
  auto ring_for = [&](int rows) {  // deepest ring (whole pairs) that shared and tensor memory hold
    const int n = std::min(kMaxItems, std::min(tmem_items, (kSmemLimit - fixed_for(rows)) / L->slot_bytes));
    return n < 0 ? 0 : n & ~1;
  };
  const int rows_pad = kTileM + 2 * R, rows_scan = strip_rows_for(px, R);
  int tiling = L->tiling;
  if (tiling == 0)  // the scan grid unless its longer strips cost ring depth
    tiling = rows_scan <= 256 && ring_for(rows_scan) >= ring_for(rows_pad) ? 2 : 1;
  if (tiling == 2 && rows_scan > 256) return OAM_ERR_UNSUPPORTED;
  p.sp = tiling == 2 ? px : p.wp;
  p.strip_rows = tiling == 2 ? rows_scan : rows_pad;
  p.strip_bytes = strip_bytes(p.strip_rows);
  const int fixed = fixed_for(p.strip_rows);
  p.n_items = ring_for(p.strip_rows);
  if (L->ring_pref >= 2) p.n_items = std::min(p.n_items, L->ring_pref);
  p.n_items &= ~1;  // items go in pairs (one fold pass each)
  if (p.n_items < 2) return OAM_ERR_UNSUPPORTED;
  p.acc_cols = L->acc_cols;
  p.tmem_cols = pow2_cols(p.fold_col0 + kFoldCols * p.n_items);
  p.part = T->d_part;
  p.status = m->d_status;
  p.budget = 4000000000LL;  // ~2 s at 2 GHz
  // the strips and slots, or where they are smaller the fold warps' epilogue stages
  out->smem = (size_t)fixed + (size_t)p.n_items * p.slot_bytes;
  out->smem = std::max(out->smem, (size_t)2048 + p.items_bytes + sizeof(float) * 32 * kStageRow * L->fold_warps);
  out->p = p;
  out->tiling = tiling;
  out->n_tiles = (int)(((long long)T->nr * p.sp + kTileM - 1) / kTileM);
  if (out->smem > (size_t)kSmemLimit) return OAM_ERR_UNSUPPORTED;
  return OAM_OK;
}

template <int FW, bool kWide>
oam_status launch_corr(const Launch &lp, const TcLayout *L, dim3 grid, cudaStream_t st) {
  OAM_CUDA_TRY(
      cudaFuncSetAttribute(k_corr_line<FW, kWide>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit));
  k_corr_line<FW, kWide><<<grid, 96 + 32 * FW, lp.smem, st>>>(lp.tiling == 2 ? L->tmap_scan : L->tmap, lp.p);
  OAM_LAUNCHED();
  return OAM_OK;
}

template <bool kWide>
oam_status launch_corr_fw(const Launch &lp, const TcLayout *L, dim3 grid, cudaStream_t st) {
  if (L->fold_warps == 4) return launch_corr<4, kWide>(lp, L, grid, st);
  if (L->fold_warps == 16) return launch_corr<16, kWide>(lp, L, grid, st);
  return launch_corr<8, kWide>(lp, L, grid, st);
}

// Which kernel zeroes the output's channels outside the accumulator, by the time that it
// adds (us).  A spare warp of each correlation block takes 0.08 a position and 0.035 a
// store, of which the block's products hide most: 200x200x300, 61 taps 76 under 340.  The
// inverse's own blocks write 3.2 TB/s but hide nothing: 35 there.  With few blocks or few
// taps the spare warps are last: 64x64x128, 3 taps, 33 blocks, 20.7 against 9.5 for the
// kernel without them; 32x32x48, 1 tap 13.0 against 7.1; 200x200x300, 1 tap 75 against 42.
bool zeros_in_inverse(const oam_model *m, const TcLine *T, const TcLayout *L, const Launch &lp, int out_len) {
  const int outside4 = (lp.p.z0 + out_len - lp.p.z1) / 4, sms = std::max(1, m->sm_count);
  if (outside4 <= 0) return false;
  const long long blocks = (long long)lp.n_tiles * L->parts * T->Q, positions = (long long)m->grid.px * m->grid.py;
  const int pairs = ((m->R + 2) / 2 + L->parts - 1) / L->parts;
  const double products = 0.55 * (pairs * L->stages + 8) * (double)((blocks + sms - 1) / sms);
  const double spare = (double)positions / (double)std::min<long long>(blocks, sms) * (0.08 + 0.035 * ((outside4 + 31) / 32));
  return spare - 0.8 * products > (double)positions * outside4 * 16 / 3.2e6;
}

size_t mark_words(const oam_model *m, const TcLine *T) {
  return (size_t)m->grid.px * ((size_t)2 * T->planes * T->words + T->Q) + 2;
}

oam_status run_corr(const oam_model *m, const TcLayout *L, const float *in, int in_len, float *out, int out_len,
                    cudaStream_t st) {
  const TcLine *T = m->tc_line;
  if (!T || !T->d_part || !L || !L->d_pack) return OAM_ERR_UNSUPPORTED;
  Launch lp;
  oam_status rc = plan_launch(m, T, L, &lp);
  if (rc) return rc;
  LineShape s{};
  s.px = m->grid.px;
  s.py = m->grid.py;
  s.R = m->R;
  s.halo = T->halo;
  s.segs = T->segs;
  s.valid = T->valid;
  s.len = in_len;
  s.in_lo = L->in_lo;
  s.elems = L->in_elems;
  s.wp = lp.p.wp;
  s.rows = T->rows;
  s.nr = T->nr;
  s.out_len = out_len;
  s.out_lo = L->out_lo;
  s.acc = L->acc_cols;
  s.words = T->words;
  s.marks = T->d_marks;
  s.planes = 1 + L->stages;
  unsigned *tail = T->d_marks + (size_t)T->planes * s.px * s.words;
  s.vmax = tail;
  tail += (size_t)s.px * T->Q;
  s.any_bad = reinterpret_cast<int *>(tail);
  lp.p.spoiled = s.any_bad + 1;
  s.spoiled = lp.p.spoiled;
  s.grown = tail + 2;
  s.reach = L->d_reach;
  lp.p.marks = s.marks;
  lp.p.grown = tail + 2;
  lp.p.any_bad = s.any_bad;
  lp.p.words = s.words;
  lp.p.planes = s.planes;
  s.parts = L->parts;
  lp.p.out = out;
  lp.p.positions = s.px * s.py;
  lp.p.out_len = out_len;
  line_channels(s, &lp.p.z0, &lp.p.z1);
  s.zeros = zeros_in_inverse(m, T, L, lp, out_len);
  if (s.zeros) lp.p.z0 = 0, lp.p.z1 = out_len;  // none are left to the correlation
  lp.p.vmax = s.vmax;
  lp.p.smax = T->d_smax;
  ProfScope prof(m, st, L->dir == 0);
  const dim3 grid(lp.n_tiles, L->parts, T->Q);
  rc = line_r2c(T->P, st, s, in, T->d_tw, L->d_pack);
  if (!rc) rc = L->wide ? launch_corr_fw<true>(lp, L, grid, st) : launch_corr_fw<false>(lp, L, grid, st);
  if (!rc) rc = line_c2r(T->P, st, s, T->d_part, T->d_tw, out);
  // the inverse clears the marks and magnitudes; without it they would reach the next application
  if (rc) cudaMemsetAsync(T->d_marks, 0, sizeof(unsigned) * mark_words(m, T), st);
  return rc;
}

size_t part_floats(const oam_model *m, const TcLine *T, int parts, int acc_cols) {
  return (size_t)parts * T->Q * T->nr * m->grid.px * acc_cols;
}
size_t part_floats(const oam_model *m, const TcLine *T, const TcLayout *L) {
  return part_floats(m, T, L->parts, L->acc_cols);
}

}  // namespace

// Device bytes tc_build allocates, from the planned bands (host only; no
// device call).  Fails like tc_build on shapes the kernels do not take.
oam_status oam::tc_plan_bytes(const oam_model *m, size_t *bytes) {
  if (kTileM + 2 * m->R > 256) return OAM_ERR_UNSUPPORTED;  // padded-grid strip positions per TMA box
  TcLine T;
  TcLayout Ls[2];
  std::vector<TcItem> items;
  std::vector<TcTile> tiles;
  oam_status rc = plan_line(m, &T);
  if (rc) return rc;
  size_t b = 0, part = 0;
  for (int dir = 0; dir < 2; ++dir) {
    TcLayout *L = &Ls[dir];
    if ((rc = plan_dir(m, &T, L, dir, items, tiles))) return rc;
    Launch lp;
    if ((rc = plan_launch(m, &T, L, &lp))) return rc;
    T.planes = std::max(T.planes, 1 + L->stages);
    b += alloc_bytes<TcItem>(items.size()) + alloc_bytes<int2>(L->stages) + alloc_bytes<uint8_t>(L->v_stride * T.Q) +
         alloc_bytes<float>((size_t)T.rows * T.Q * L->in_elems);
    // The bands planned here are up to kSlack samples wider at either end than those of
    // the build, and a narrower support can take more parts: the most that any of them takes.
    constexpr int kSlack = 4;
    for (int lo = m->n_lo; lo <= m->n_lo + kSlack; ++lo)
      for (int hi = std::max(lo, m->n_hi - kSlack); hi <= m->n_hi; ++hi) {
        int stages, acc;
        dir_sizes(dir, m->grid.nz, lo, hi, &stages, &acc);
        part = std::max(part, part_floats(m, &T, choose_parts(&T, m->grid.px, m->R, stages, acc), acc));
      }
  }
  *bytes = b + alloc_bytes<float>(part) + alloc_bytes<float2>(T.P) + alloc_bytes<unsigned>(mark_words(m, &T)) + alloc_bytes<unsigned>(1);
  return OAM_OK;
}

oam_status oam::tc_build(oam_model *m, cudaStream_t st) {
  if (kTileM + 2 * m->R > 256) return OAM_ERR_UNSUPPORTED;  // padded-grid strip positions per TMA box
  TcLine *T = m->tc_line = new TcLine();
  oam_status rc = plan_line(m, T);
  if (rc) return rc;
  const std::vector<float2> roots = mix_roots(T->P);
  if ((rc = dev_alloc(m, &T->d_tw, roots.size())) || (rc = dev_alloc(m, &T->d_smax, 1))) return rc;
  OAM_CUDA_TRY(cudaMemcpyAsync(T->d_tw, roots.data(), sizeof(float2) * roots.size(), cudaMemcpyHostToDevice, st));
  OAM_CUDA_TRY(cudaMemsetAsync(T->d_smax, 0, sizeof(unsigned), st));
  const size_t nb = (size_t)m->n_orb * m->grid.nz;
  k_slab_max<<<4 * std::max(1, m->sm_count), 256, 0, st>>>(m->d_band, nb * m->band_w, (float)m->W, T->d_smax);
  OAM_LAUNCHED();
  int *d_band_hi = nullptr;
  OAM_CUDA_TRY(cudaMallocAsync((void **)&d_band_hi, sizeof(int) * nb, st));
  OAM_CUDA_TRY(cudaMemcpyAsync(d_band_hi, m->h_band_hi.data(), sizeof(int) * nb, cudaMemcpyHostToDevice, st));
  m->tc_fwd = new TcLayout();
  m->tc_adj = new TcLayout();
  rc = build_dir(m, m->tc_fwd, 0, st, d_band_hi);
  if (!rc) rc = build_dir(m, m->tc_adj, 1, st, d_band_hi);
  cudaFreeAsync(d_band_hi, st);
  if (rc) return rc;
  for (TcLayout *L : {m->tc_fwd, m->tc_adj}) {
    Launch lp;
    if ((rc = plan_launch(m, T, L, &lp))) return rc;
    T->planes = std::max(T->planes, 1 + L->stages);
  }
  if ((rc = dev_alloc(m, &T->d_marks, mark_words(m, T)))) return rc;
  OAM_CUDA_TRY(cudaMemsetAsync(T->d_marks, 0, sizeof(unsigned) * mark_words(m, T), st));
  return dev_alloc(m, &T->d_part, std::max(part_floats(m, T, m->tc_fwd), part_floats(m, T, m->tc_adj)));
}

void oam::tc_free(oam_model *m, cudaStream_t st) {
  for (TcLayout *L : {m->tc_fwd, m->tc_adj}) {
    if (!L) continue;
    for (void *p : {(void *)L->d_items, (void *)L->d_data, (void *)L->d_pack, (void *)L->d_reach})
      if (p) cudaFreeAsync(p, st);
    delete L;
  }
  m->tc_fwd = m->tc_adj = nullptr;
  if (TcLine *T = m->tc_line) {
    for (void *p : {(void *)T->d_tw, (void *)T->d_marks, (void *)T->d_smax, (void *)T->d_part})
      if (p) cudaFreeAsync(p, st);
    delete T;
  }
  m->tc_line = nullptr;
}

// Executed MMA flops of one application: 3 products x 2 x M x (16 x N) over the
// (frequency, position tile, a >= 0) work items.
double oam::tc_exec_flops(const oam_model *m, int dir) {
  const TcLayout *L = dir == 0 ? m->tc_fwd : m->tc_adj;
  Launch lp;
  if (!L || uses_direct(m, dir == 0) || plan_launch(m, m->tc_line, L, &lp)) return 0.0;
  return 3.0 * 2.0 * kTileM * (double)lp.n_tiles * m->tc_line->Q * L->cols;
}

oam_status oam::forward_tc(const oam_model *m, const float *H, float *s, cudaStream_t st) {
  return run_corr(m, m->tc_fwd, H, m->grid.nz, s, m->grid.nt, st);
}

oam_status oam::adjoint_tc(const oam_model *m, const float *s, float *H, cudaStream_t st) {
  return run_corr(m, m->tc_adj, s, m->grid.nt, H, m->grid.nz, st);
}

// ---------------------------------------------------------------- autotuner
// Per direction, time every (position tiling, fold-warp count, ring depth) on
// the model's own shapes (CUDA events on `st`) and keep the fastest.
oam_status oam::tc_autotune(oam_model *m, int reps, cudaStream_t st, int *best_fwd, int *best_adj, int *warps_fwd,
                            int *warps_adj) {
  if (!m->tc_fwd) return OAM_ERR_UNSUPPORTED;
  const size_t nv = vol_elems(m), ns = sig_elems(m);
  float *buf = nullptr;
  if (cudaMalloc((void **)&buf, (nv + ns) * sizeof(float)) != cudaSuccess) {
    cudaGetLastError();
    return OAM_ERR_OOM;
  }
  oam_status rc = OAM_OK;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  cudaMemsetAsync(buf, 0, (nv + ns) * sizeof(float), st);
  for (int dir = 0; dir < 2 && !rc; ++dir) {
    TcLayout *L = dir == 0 ? m->tc_fwd : m->tc_adj;
    float best_ms = 1e30f;
    int best = 0, best_w = kDefaultFoldWarps, best_t = 0;
    for (int tiling = 1; tiling <= 2 && !rc; ++tiling) {
      L->tiling = tiling;
      L->ring_pref = 0;
      Launch lp;
      if (plan_launch(m, m->tc_line, L, &lp)) continue;  // this tiling does not fit the model
      const int deepest = lp.p.n_items;
      for (int fw : kFoldWarpChoices) {
        L->fold_warps = fw;
        for (int depth = 2; depth <= deepest; depth += 2) {
          L->ring_pref = depth;
          for (int r = 0; r <= reps && !rc; ++r) {  // first run warms up
            if (r == 1) cudaEventRecord(e0, st);
            rc = dir == 0 ? run_corr(m, L, buf, m->grid.nz, buf + nv, m->grid.nt, st)
                          : run_corr(m, L, buf + nv, m->grid.nt, buf, m->grid.nz, st);
          }
          cudaEventRecord(e1, st);
          if (cudaEventSynchronize(e1) != cudaSuccess) rc = OAM_ERR_CUDA;
          if (rc) break;
          float ms = 0;
          cudaEventElapsedTime(&ms, e0, e1);
          if (ms < best_ms) {
            best_ms = ms;
            best = depth;
            best_w = fw;
            best_t = tiling;
          }
        }
        if (rc) break;
      }
    }
    L->tiling = best_t;
    L->ring_pref = best;
    L->fold_warps = best_w;
    (dir == 0 ? *best_fwd : *best_adj) = best;
    (dir == 0 ? *warps_fwd : *warps_adj) = best_w;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(buf);
  return rc;
}

oam_status oam::tc_set_tiles(oam_model *m, int dir, int fold_warps, int ring) {
  TcLayout *L = dir == 0 ? m->tc_fwd : m->tc_adj;
  if (!L) return OAM_ERR_UNSUPPORTED;
  bool okw = false;
  for (int fw : kFoldWarpChoices) okw = okw || fw == fold_warps;
  if (!okw || ring < 0 || (ring & 1)) return OAM_ERR_INVALID_ARG;
  const int keep_ring = L->ring_pref, keep_w = L->fold_warps;
  L->ring_pref = ring;
  L->fold_warps = fold_warps;
  Launch lp;
  oam_status rc = plan_launch(m, m->tc_line, L, &lp);
  if (rc || (ring >= 2 && lp.p.n_items != ring)) {
    L->ring_pref = keep_ring;
    L->fold_warps = keep_w;
    return rc ? rc : OAM_ERR_INVALID_ARG;
  }
  return OAM_OK;
}

oam_status oam::tc_set_tiling(oam_model *m, int dir, int tiling) {
  TcLayout *L = dir == 0 ? m->tc_fwd : m->tc_adj;
  if (!L) return OAM_ERR_UNSUPPORTED;
  if (tiling < 0 || tiling > 2) return OAM_ERR_INVALID_ARG;
  const int keep = L->tiling;
  L->tiling = tiling;
  Launch lp;
  const oam_status rc = plan_launch(m, m->tc_line, L, &lp);
  if (rc) L->tiling = keep;
  return rc;
}

int oam::tc_get_tiling(const oam_model *m, int dir) {
  const TcLayout *L = dir == 0 ? m->tc_fwd : m->tc_adj;
  Launch lp;
  return L && plan_launch(m, m->tc_line, L, &lp) == OAM_OK ? lp.tiling : 0;
}

void oam::tc_get_tiles(const oam_model *m, int dir, int *fold_warps, int *ring) {
  const TcLayout *L = dir == 0 ? m->tc_fwd : m->tc_adj;
  if (!L) {
    *fold_warps = *ring = 0;
    return;
  }
  Launch lp;
  *fold_warps = L->fold_warps;
  *ring = plan_launch(m, m->tc_line, L, &lp) == OAM_OK ? lp.p.n_items : 0;
}
