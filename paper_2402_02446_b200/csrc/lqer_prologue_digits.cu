// Activation prologue of larger batches with ranks above 64, or of several layers on one activation (paper Section 4.1: X_q in MXINT8, blocks [1,16]; Section 3.1:
// the small high-precision product T = X_q A_k), in three launches:
//   quantise_kernel  X -> Xcat[:, 0:K64] (the exact bf16 values of X_q), one exponent byte per 16-block, and per row the
//                    range of its exponents; A_q -> digit planes (below);
//   project_kernel   T = X_q A_q as ONE integer contraction on the tcgen05 int8 tensor cores, into 64-bit sums;
//   finish_kernel    T re-quantised along the rank, appended to Xcat.
//
// The projection has to be exact (T is re-quantised, and its rounding decisions must be those of a 64-bit sum), but the
// blocks of a row have exponents of their own, so the int32 products of different blocks cannot simply be added up.  Here
// a row is written in fixed-point formats instead: in a window of nine exponents [E - 8, E], a value m * 2^(e-6) is the
// integer m * 2^(8-(E-e)), at most 127 * 2^8 in magnitude, times 2^(E-14): sixteen bits, i.e. two signed base-256 digits.  A
// column of A_q takes the same form over its blocks.  T is then three integer contractions (high x high, the two mixed ones
// into one accumulator, low x low) over the WHOLE of K, exact in int32 for up to 32768 K per CTA, and one 64-bit combination
// per element of T.  Partial sums of different K ranges are integers with a common scale, so they are added with 64-bit
// integer atomics, in any order: exact and reproducible.
// Rows whose blocks spread over more than nine exponents have up to three windows, stacked downwards from the row's largest
// exponent or upwards from its smallest, whichever leaves most blocks to the first.  Each further one is another pass of the
// same contraction, over those panels of 128 K in which the CTA's rows have a block in it, whose sums enter the row's 64-bit
// sums nine bits higher or lower: 63 bits in all.  2048 rows of 4096 columns at rank 256 take 110 us with their GEMM with
// one window, 116 with two massive channels (x1000), 124 with 41 outlier channels (x500), 143 with 25 binades everywhere;
// launch_prologue (below), which no spread touches, 167.  Adding up such blocks one by one, as is done with what no window
// holds, took 253, 326 and 941.
// What lies below three windows, and blocks of A_q outside the window of their column (the one that holds most of them), is
// zero in the digit planes; a bit per block says so, and finish_kernel adds the marked blocks in fp64, one by one.  The same
// call: five blocks of every row 35 binades down 162 us, twelve blocks of every column of A_q 12 binades down 191.  It is not
// made for more: block exponents drawn from 51 binades, a third of them marked, take 811.
// Scaling every block's products in fp64 instead, as the other prologues do, is bound by 14.7 block products per clock and
// SM: 115 us for 2048 rows of 4096 columns at rank 256.
#include <algorithm>

#include "lqer_tc_ptx.cuh"

namespace lqer {
namespace pdg {
using namespace tc;

constexpr int kWindow = 8;                        // a window holds the exponents [E - 8, E]
constexpr int kMaxWindows = 3;                    // of a row, kWindow + 1 apart: 32512^2 * 32768 * 2^18 < 2^63
constexpr int kColsPerWarp = 2;                   // columns of A_q one warp turns into digits,
constexpr int kColShares = 4;                     // in one of so many shares of K
constexpr int ROWS = 128;
constexpr int PANEL = 128;                        // K per stage: one 128-byte swizzled row of int8
constexpr int MAX_NT = 128;                       // T columns per CTA: three int32 accumulators of 128 columns in tensor memory
constexpr int STAGES = 3;
constexpr int X_PLANE = ROWS * PANEL;             // 16384
constexpr int A_PLANE = MAX_NT * PANEL;           // 16384
constexpr int STAGE_BYTES = 2 * X_PLANE + 2 * A_PLANE;
constexpr int CONV_WARPS = 16;
constexpr int WORKERS = CONV_WARPS * 32;          // threads of the converter warps; they do phase 1 too
constexpr int NUM_THREADS = (2 + CONV_WARPS) * 32;
constexpr int kParts = CONV_WARPS;                // shares of a row in phase 1, at most
constexpr int MASK_WORDS = 32768 / PANEL / 32;    // a bit for each panel of a CTA's range of K
constexpr int OFF_MASKS = STAGES * STAGE_BYTES + 128, OFF_INFO = STAGES * STAGE_BYTES + 256;
constexpr int SMEM_BYTES = OFF_INFO + ROWS * 4 + 1024;
static_assert((kMaxWindows - 1) * MASK_WORDS * 4 <= 128, "panel masks");
constexpr int kQuantThreads = 256;
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");
constexpr int kFinishRows = 16;
constexpr int TMEM_COLS = 512;

struct LayerA {                                   // one layer's A section and its place among the unit's T columns
  const uint8_t* asec;
  int8_t* Tm;                                     // optional exports
  uint8_t* Te;
  int k_pad, col0;
};
struct Unit {                                     // one X and the layers that multiply it
  const void* X;
  uint16_t* xcat;                                 // [M, ld]: X_q values, then T columns
  uint8_t* ebytes;                                // [M, ep] exponent bytes of X_q's blocks; 0: a block of zeros
  uint32_t* rowparts;                             // [M][kParts]: largest | smallest << 8 | mean << 16 exponent byte of each share
  int* rowinfo;                                   // [M]: E + 1024 of the lowest window, bit 16: the row has blocks below it
  int* colinfo;                                   // [ktot]: E + 1024 of A_q's columns, bit 16: it has blocks outside its window
  uint32_t* rowfar;                               // [M][far_words]: a bit per block below the row's windows (rows with bit 16 only)
  uint32_t* colout;                               // [ktot][far_words]: a bit per block outside the column's window (the same)
  uint8_t* planes;                                // digit planes of A_q: [column tile][panel][hi, lo][columns][128], swizzled
  unsigned long long* tacc;                       // [row tile][ktot][128] sums (splits > 1)
  LayerA layer[kDigitMaxLayers];
  int n_layers, ktot;
  int K, K64, ld, ep, panels;
  int row_tiles, col_tiles, splits;
  int windows, far_words;
  int first_a, first_rows;                        // quantise_kernel: this unit's first warp of each kind
  int first_item, first_finish;                   // project_kernel, finish_kernel: its first CTA
  size_t xcat_extent;                             // bytes, for the checked build
};
struct Params {
  Unit U[kDigitMaxUnits];
  int n, M, x_type;
  int warps_per_row;                              // a power of two up to kParts
  int rows_begin, n_warps;                        // warps of quantise_kernel: A_q of all units, then (from rows_begin) their rows
  int a_bits, lr_bits, exp_min, exp_max, w_exp_min;
  DeviceStatus* status;
  long long wait_limit;
  int stall;                                      // test hook: the last panel's A digits are withheld
};

// Checked build: whether n elements from p[at] on lie in an array of `total` of them (all of a unit's arrays are scratch).
template <class T>
__device__ __forceinline__ bool inside(const Params& p, const T*, size_t at, size_t n, size_t total, int site) {
  return LQER_IN_BOUNDS(p.status, at * sizeof(T), n * sizeof(T), total * sizeof(T), site);
}
__device__ __forceinline__ const Unit& unit_of(const Params& p, int index, int Unit::* first) {
  int u = 0;
  for (int i = 1; i < p.n; ++i)
    if (index >= p.U[i].*first) u = i;
  return p.U[u];
}
__device__ __forceinline__ void tile_columns(int ktot, int col_tiles, int ct, int& c0, int& nt) {
  const unsigned nb = (unsigned)ktot >> 4;                             // at most 128
  c0 = (int)((unsigned)ct * nb / (unsigned)col_tiles) << 4;
  nt = ((int)((unsigned)(ct + 1) * nb / (unsigned)col_tiles) << 4) - c0;
}
__device__ __forceinline__ bool outside(int eb, int E) { return eb - 127 > E || eb - 127 < E - kWindow; }

// The window [E - 8, E] that holds most of the blocks counted in hist[exponent byte], for one warp.
__device__ __forceinline__ int best_window(const int* hist, int lane) {
  int best = -1, at = 0;
  for (int eb = 1 + lane; eb < 256; eb += 32) {   // the lowest top that holds the most
    int n = 0;
    for (int d = 0; d <= kWindow; ++d) n += eb - d >= 1 ? hist[eb - d] : 0;
    if (n > best) { best = n; at = eb; }
  }
  for (int s = 16; s > 0; s >>= 1) {
    const int ob = __shfl_xor_sync(0xFFFFFFFFu, best, s), oa = __shfl_xor_sync(0xFFFFFFFFu, at, s);
    if (ob > best || (ob == best && oa < at)) { best = ob; at = oa; }
  }
  return at - 127;
}

// Two base-256 digits of four integers xi = v * scale (|xi| <= 32512): xi = hi * 256 + lo, both signed bytes.
// The sum v * scale + (1.5 * 2^23 + 128) is exact and carries xi + 128 in its low 16 bits.
__device__ __forceinline__ void digits_of(float v0, float v1, float v2, float v3, float scale, uint32_t& hi, uint32_t& lo) {
  const float kMagic = 12583040.0f;
  const uint32_t u0 = __float_as_uint(fmaf(v0, scale, kMagic)), u1 = __float_as_uint(fmaf(v1, scale, kMagic));
  const uint32_t u2 = __float_as_uint(fmaf(v2, scale, kMagic)), u3 = __float_as_uint(fmaf(v3, scale, kMagic));
  const uint32_t a = __byte_perm(u0, u1, 0x5410), b = __byte_perm(u2, u3, 0x5410);
  hi = __byte_perm(a, b, 0x7531);
  lo = __byte_perm(a, b, 0x6420) ^ 0x80808080u;
}

// One signed byte of a word as a float without a conversion instruction (they run at an eighth of the rate): offset by 128
// it is the low byte of the float 1.5 * 2^23 + 128 + value.
__device__ __forceinline__ float byte_value(uint32_t w, uint32_t select) {
  return __uint_as_float(__byte_perm(w ^ 0x80808080u, 0x4B400000u, select)) - 12583040.0f;
}

// The window of a column whose non-zero blocks' exponent bytes reach from mn to mx: E, and bit 16 if some lie outside.  byte_of(b): block b's exponent byte, 0 for a block of zeros.  One warp; hist: 256 ints of its own.
template <class F>
__device__ __forceinline__ int window_of(int mx, int mn, int blocks, int* hist, int lane, F&& byte_of) {
  if (mx - mn <= kWindow || mx == 0) return mx - 127 + 1024;
  for (int i = lane; i < 256; i += 32) hist[i] = 0;
  __syncwarp();
  for (int b = lane; b < blocks; b += 32) {
    const int eb = byte_of(b);
    if (eb != 0) atomicAdd(&hist[eb], 1);
  }
  __syncwarp();
  const int E = best_window(hist, lane);
  __syncwarp();
  return (E + 1024) | 1 << 16;
}

// One warp: a share of K of two columns of a layer's A_q -> windows (every share works them out) and digit planes.
__device__ __forceinline__ void a_digits(const Params& p, const Unit& u, int part, int lane, int* hist) {
  const int share = part % kColShares;
  part /= kColShares;
  int l = 0;
  for (; l + 1 < u.n_layers && part >= u.layer[l].k_pad / kColsPerWarp; ++l) part -= u.layer[l].k_pad / kColsPerWarp;
  const LayerA& la = u.layer[l];
  if (part >= la.k_pad / kColsPerWarp) return;
  const int c = part * kColsPerWarp, kb = u.K / 16, kp = la.k_pad;
  const uint4* mant = reinterpret_cast<const uint4*>(la.asec);
  const uint8_t* aexp = la.asec + (size_t)kb * kp * 16;
  auto zero = [&](int b, int j) {
    const uint4 v = mant[(size_t)b * kp + c + j];
    return (v.x | v.y | v.z | v.w) == 0u;
  };
  int mx[2] = {0, 0}, mn[2] = {255, 255};
  for (int b0 = lane; b0 < kb; b0 += 8 * 32) {
    uint32_t e2[8];                                                    // eight loads in flight before the first is looked at
#pragma unroll
    for (int i = 0; i < 8; ++i) e2[i] = b0 + 32 * i < kb ? *reinterpret_cast<const uint16_t*>(aexp + (size_t)(b0 + 32 * i) * kp + c) : 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int eb = (int)((e2[i] >> (8 * j)) & 0xFFu);
        // (only the lowest exponent may be a block of zeros)
        if (eb != 0 && (eb - 127 > p.w_exp_min || !zero(b0 + 32 * i, j))) { mx[j] = max(mx[j], eb); mn[j] = min(mn[j], eb); }
      }
  }
  int info[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    mx[j] = __reduce_max_sync(0xFFFFFFFFu, mx[j]);
    mn[j] = __reduce_min_sync(0xFFFFFFFFu, mn[j]);
    info[j] = window_of(mx[j], mn[j], kb, hist, lane, [&](int b) { return zero(b, j) ? 0 : (int)aexp[(size_t)b * kp + c + j]; });
  }
  const int col = la.col0 + c;
  if (share == 0) {
    if (lane == 0 && inside(p, u.colinfo, col, 2, u.ktot, 333)) { u.colinfo[col] = info[0]; u.colinfo[col + 1] = info[1]; }
    for (int j = 0; j < 2; ++j)
      if ((info[j] >> 16) != 0)
        for (int b0 = 0; b0 < kb; b0 += 32) {
          const int b = b0 + lane;
          const unsigned out = __ballot_sync(0xFFFFFFFFu, b < kb && outside(aexp[(size_t)b * kp + c + j], (info[j] & 0xFFFF) - 1024) && !zero(b, j));
          const size_t at = (size_t)(col + j) * u.far_words + (b0 >> 5);
          if (lane == 0 && inside(p, u.colout, at, 1, (size_t)u.ktot * u.far_words, 334)) u.colout[at] = out;
        }
  }
  int c0 = 0, nt = 0;
  for (int ct = 0; ct < u.col_tiles; ++ct) {                           // (tiles are whole 16-blocks: both columns lie in one)
    tile_columns(u.ktot, u.col_tiles, ct, c0, nt);
    if (col < c0 + nt) break;
  }
  uint8_t* img = u.planes + (size_t)u.panels * 2 * PANEL * c0;
  const int n = col - c0;
  for (int b0 = share * 32 + lane; b0 < u.ep; b0 += 2 * 32 * kColShares) {
    uint4 v[2][2];
    int d[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int b = b0 + 32 * kColShares * i;
        v[i][j] = make_uint4(0u, 0u, 0u, 0u);
        d[i][j] = -1;
        if (b < kb) {
          v[i][j] = mant[(size_t)b * kp + c + j];
          d[i][j] = (info[j] & 0xFFFF) - 1024 - ((int)aexp[(size_t)b * kp + c + j] - 127);
        }
      }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int b = b0 + 32 * kColShares * i;
      if (b >= u.ep) break;
      uint8_t* tile = img + (size_t)(b >> 3) * (2 * PANEL * nt);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        uint4 hi = make_uint4(0u, 0u, 0u, 0u), lo = hi;
        if (d[i][j] >= 0 && d[i][j] <= kWindow) {
          const float scale = pow2f(kWindow - d[i][j]);
          const uint32_t w[4] = {v[i][j].x, v[i][j].y, v[i][j].z, v[i][j].w};
          uint32_t h[4], o[4];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            digits_of(byte_value(w[q], 0x7640), byte_value(w[q], 0x7641), byte_value(w[q], 0x7642), byte_value(w[q], 0x7643), scale, h[q], o[q]);
          hi = make_uint4(h[0], h[1], h[2], h[3]);
          lo = make_uint4(o[0], o[1], o[2], o[3]);
        }
        uint8_t* at = tile + (n + j) * PANEL + (((b & 7) ^ ((n + j) & 7)) << 4);
        if (!inside(p, u.planes, at - u.planes, nt * PANEL + 16, (size_t)u.panels * 2 * PANEL * u.ktot, 335)) continue;
        *reinterpret_cast<uint4*>(at) = hi;
        *reinterpret_cast<uint4*>(at + nt * PANEL) = lo;
      }
    }
  }
}

__device__ __forceinline__ void load16(const void* X, int x_type, int M, int K, int row, int col, const QuantConsts& qc, int a_bits,
                                       float (&v)[16]) {
  const size_t idx = (size_t)row * K + col;
  if (x_type == kXBF16) {
    const uint4* src = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(X) + idx);
    const uint4 a = __ldg(src), b = __ldg(src + 1);
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) { v[2 * i] = __uint_as_float(w[i] << 16); v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u); }
  } else if (x_type == kXMXINT8) {
    const uint8_t* xb = static_cast<const uint8_t*>(X);
    const uint4 a = __ldg(reinterpret_cast<const uint4*>(xb + idx));
    const uint32_t eb = __ldg(xb + (size_t)M * K + (size_t)row * (K / 16) + (col >> 4));
    const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 q = mxint_quad_values(w[i], eb, a_bits, qc.emin, qc.emax);
      v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
    }
  } else {
    const float4* src = reinterpret_cast<const float4*>(static_cast<const float*>(X) + idx);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 q = __ldg(src + i);
      v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
    }
  }
}

// One warp: share `part` of a row.  A lane owns a whole 16-block; kBatch blocks of a lane are loaded together.
constexpr int kBatch = 2;
__device__ __forceinline__ void quantise_row(const Params& p, const Unit& u, int row, int part, int lane) {
  if (u.splits > 1) {
    // the sums start at zero: any share of them will do (the last row takes those of the last row tile's missing rows too)
    const int rows_here = row == p.M - 1 ? u.row_tiles * ROWS - row : 1;
    unsigned long long* acc = u.tacc + (size_t)row * u.ktot;
    if (inside(p, u.tacc, (size_t)row * u.ktot, (size_t)rows_here * u.ktot, (size_t)u.row_tiles * u.ktot * ROWS, 336))
    for (int i = part * 32 + lane; i < rows_here * u.ktot; i += p.warps_per_row * 32) acc[i] = 0ull;
  }
  const QuantConsts qc = quant_consts(p.a_bits, p.exp_min, p.exp_max);
  const int kb = u.K / 16, xb = u.K64 / 16, stride = p.warps_per_row * 32;
  int mx = 0, mn = 255, sum = 0, n = 0;
  uint8_t* erow = u.ebytes + (size_t)row * u.ep;
  uint16_t* xrow = u.xcat + (size_t)row * u.ld;
  float v[kBatch][16];
#pragma unroll
  for (int h = 0; h < kBatch; ++h) {
    const int b = part * 32 + lane + h * stride;
    if (b < kb) load16(u.X, p.x_type, p.M, u.K, row, b * 16, qc, p.a_bits, v[h]);
  }
  for (int b0 = part * 32 + lane; b0 < u.ep; b0 += kBatch * stride) {
#pragma unroll
    for (int h = 0; h < kBatch; ++h) {
      const int b = b0 + h * stride;
      if (b >= u.ep) break;
      uint4 m8 = make_uint4(0u, 0u, 0u, 0u), x0 = m8, x1 = m8;
      int e = 0, eb = 0;
      if (b < kb) {
        quantize_block16(v[h], qc, e, m8, x0, x1);
        // (a block of narrower mantissas is a block of 8-bit ones with trailing zeros: the windows count in those)
        if ((m8.x | m8.y | m8.z | m8.w) != 0u) { eb = e + 127; mx = max(mx, eb); mn = min(mn, eb); sum += eb; ++n; }
      }
      const int bn = b + kBatch * stride;                              // the next block is on its way while this one is stored
      if (bn < kb) load16(u.X, p.x_type, p.M, u.K, row, bn * 16, qc, p.a_bits, v[h]);
      if (b < xb && LQER_IN_BOUNDS(p.status, ((size_t)row * u.ld + b * 16) * 2, 32, u.xcat_extent, 331)) {
        *reinterpret_cast<uint4*>(xrow + b * 16) = x0;
        *reinterpret_cast<uint4*>(xrow + b * 16 + 8) = x1;
      }
      if (inside(p, u.ebytes, (size_t)row * u.ep + b, 1, (size_t)p.M * u.ep, 337)) erow[b] = (uint8_t)eb;
    }
  }
  mx = __reduce_max_sync(0xFFFFFFFFu, mx);
  mn = __reduce_min_sync(0xFFFFFFFFu, mn);
  sum = __reduce_add_sync(0xFFFFFFFFu, sum);
  n = __reduce_add_sync(0xFFFFFFFFu, n);
  if (lane == 0 && inside(p, u.rowparts, (size_t)row * kParts + part, 1, (size_t)p.M * kParts, 338))
    u.rowparts[(size_t)row * kParts + part] = (uint32_t)(mx | mn << 8 | (n > 0 ? sum / n : 0) << 16);
}

// Bound by reading X and writing Xcat; no warp waits for another.
__global__ void __launch_bounds__(kQuantThreads, 3) quantise_kernel(const __grid_constant__ Params p) {
  __shared__ int s_hist[kQuantThreads / 32][256];
  pdl_wait();
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = (int)blockIdx.x * (kQuantThreads / 32) + warp;
  if (w >= p.n_warps) return;
  if (w < p.rows_begin) {
    const Unit& u = unit_of(p, w, &Unit::first_a);
    a_digits(p, u, w - u.first_a, lane, s_hist[warp]);
  } else {
    const Unit& u = unit_of(p, w, &Unit::first_rows);
    const int share = w - u.first_rows;
    quantise_row(p, u, share / p.warps_per_row, share % p.warps_per_row, lane);
  }
}

__device__ __forceinline__ void umma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}
// int8 x int8 -> int32, both operands K-major, M = m, N = n.
__host__ __device__ constexpr uint32_t make_idesc_i8(int m, int n) {
  return (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
// The terms of T[row, col] that the digit planes leave out, in fp64: the marked blocks of the row and of the column.
__device__ __noinline__ double outside_terms(const Params& p, const Unit& u, int row, int col, int rinfo, int cinfo) {
  if (row >= p.M) return 0.0;
  int l = 0;
  while (l + 1 < u.n_layers && col >= u.layer[l + 1].col0) ++l;
  const LayerA& la = u.layer[l];
  const int kb = u.K / 16, c = col - la.col0;
  const uint8_t* aexp = la.asec + (size_t)kb * la.k_pad * 16;
  const bool row_far = (rinfo >> 16) != 0, col_out = (cinfo >> 16) != 0;
  double t = 0.0;
  for (int w = 0; w < u.far_words; ++w) {
    uint32_t marked = (row_far ? u.rowfar[(size_t)row * u.far_words + w] : 0u) | (col_out ? u.colout[(size_t)col * u.far_words + w] : 0u);
    for (; marked != 0; marked &= marked - 1) {
      const int b = 32 * w + __ffs(marked) - 1;
      const uint2* xv = reinterpret_cast<const uint2*>(u.xcat + (size_t)row * u.ld + b * 16);
      const uint32_t* av = reinterpret_cast<const uint32_t*>(la.asec + ((size_t)b * la.k_pad + c) * 16);
      float s = 0.0f;                                                  // sixteen products with one scale: exact
#pragma unroll 1                                                       // (few registers: finish_kernel wants two CTAs per SM)
      for (int i = 0; i < 4; ++i) {
        const uint2 x = xv[i];
        const uint32_t a = av[i];
        s = fmaf(__uint_as_float(x.x << 16), byte_value(a, 0x7640), s);
        s = fmaf(__uint_as_float(x.x & 0xFFFF0000u), byte_value(a, 0x7641), s);
        s = fmaf(__uint_as_float(x.y << 16), byte_value(a, 0x7642), s);
        s = fmaf(__uint_as_float(x.y & 0xFFFF0000u), byte_value(a, 0x7643), s);
      }
      t += (double)s * pow2d((int)aexp[(size_t)b * la.k_pad + c] - 127 - (p.lr_bits - 2));
    }
  }
  return t;
}

// kFinishRows rows of a tile's columns: the 64-bit sums -> T -> T_q.  Sixteen lanes hold a 16-block of T.
__global__ void __launch_bounds__(WORKERS) finish_kernel(const __grid_constant__ Params p) {
  pdl_launch_dependents();
  const Unit& u = unit_of(p, blockIdx.x, &Unit::first_finish);
  int item = (int)blockIdx.x - u.first_finish;
  const int rg = item % (ROWS / kFinishRows); item /= ROWS / kFinishRows;
  const int ct = item % u.col_tiles, rt = item / u.col_tiles;
  int c0, nt;
  tile_columns(u.ktot, u.col_tiles, ct, c0, nt);
  const int tid = threadIdx.x, j16 = tid & 15;
  pdl_wait();
  if (rt * ROWS + rg * kFinishRows >= p.M) return;
  const LayerA& la = u.layer[0];                                       // exports: a unit of one layer only
  const int items = kFinishRows * (nt >> 4);
  const unsigned half = 0xFFFFu << (tid & 16);
  auto row_of = [&](int k) { return rt * ROWS + rg * kFinishRows + k % kFinishRows; };
  auto col_of = [&](int k) { return c0 + (k / kFinishRows) * 16 + j16; };
  auto load = [&](int k, long long& s, int& ri) {
    const int r = row_of(k) - rt * ROWS;
    const bool in = k < items && row_of(k) < p.M;
    s = in ? (long long)__ldcg(u.tacc + ((size_t)rt * u.ktot + col_of(k)) * ROWS + r) : 0;
    ri = in ? __ldcg(u.rowinfo + row_of(k)) : 1024;
  };
  auto p2_of = [&](int ri, int ci) { return (ri & 0xFFFF) + (ci & 0xFFFF) - 2048 - 14 - kWindow - (p.lr_bits - 2); };   // T = s * 2^p2
  auto put = [&](int row, int col, int m, int e) {
    const size_t at = (size_t)row * u.ld + u.K64 + col;
    if (row < p.M && LQER_IN_BOUNDS(p.status, at * 2, 2, u.xcat_extent, 332)) {
      u.xcat[at] = (uint16_t)bf16_bits_of(m, e - (p.a_bits - 2));
      if (la.Tm != nullptr) la.Tm[(size_t)row * la.k_pad + col] = (int8_t)m;
      if (la.Te != nullptr && j16 == 0) la.Te[(size_t)row * (la.k_pad / 16) + col / 16] = (uint8_t)(e + 127);
    }
  };
  bool again = false;                                                  // a 16-block with marked blocks in its terms was left out
#pragma unroll 1
  for (int o = tid >> 4; o < items; o += 4 * (WORKERS / 16)) {
    long long s[4];
    int ri[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) load(o + i * (WORKERS / 16), s[i], ri[i]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = o + i * (WORKERS / 16);
      if (k >= items) break;                                           // the same for all lanes of a warp but its half
      const int ci = u.colinfo[col_of(k)], p2 = p2_of(ri[i], ci);
      if (__any_sync(half, ((ri[i] | ci) >> 16) != 0)) { again = true; continue; }
      // the decisions of a 64-bit sum in integers (64-bit integers become doubles and doubles integers at a few per clock only)
      const unsigned long long mag = (unsigned long long)(s[i] < 0 ? -s[i] : s[i]);
      const int top = mag == 0 ? -(1 << 20) : 63 - __clzll((long long)mag) + p2;                  // floor(log2 |T|)
      const int bt = __reduce_max_sync(half, top);
      const int e = min(max(bt, p.exp_min), p.exp_max);
      const int qmax = (1 << (p.a_bits - 1)) - 1, sh = e - (p.a_bits - 2) - p2;                   // |T| in steps = mag * 2^-sh
      int m;
      if (top > e) {
        m = qmax;
      } else if (sh <= 0) {
        m = mag == 0 ? 0 : (int)(mag << min(-sh, 63));
      } else if (sh > 63) {
        m = 0;
      } else {                                                                                    // half to even
        const unsigned long long q = mag >> sh, rest = mag & ((1ull << sh) - 1ull), tie = 1ull << (sh - 1);
        m = (int)q + (rest > tie || (rest == tie && (q & 1ull)) ? 1 : 0);
      }
      m = min(m, qmax);
      put(row_of(k), col_of(k), s[i] < 0 ? -m : m, e);
    }
  }
  if (!again) return;
  // (a loop of its own: with the call among the four above, the common case took 3 us longer for its registers)
#pragma unroll 1
  for (int k = tid >> 4; k < items; k += WORKERS / 16) {
    long long s;
    int ri;
    load(k, s, ri);
    const int row = row_of(k), col = col_of(k), ci = u.colinfo[col];
    const bool marked = ((ri | ci) >> 16) != 0;
    if (!__any_sync(half, marked)) continue;
    double t = (double)s * pow2d(p2_of(ri, ci));
    if (marked) t += outside_terms(p, u, row, col, ri, ci);
    double amax = fabs(t);
#pragma unroll 1
    for (int d = 1; d < 16; d <<= 1) amax = fmax(amax, __shfl_xor_sync(half, amax, d));
    const int e = block_exponent(amax, p.exp_min, p.exp_max);
    put(row, col, quant_mantissa(t, e, p.a_bits), e);
  }
}

__global__ void __launch_bounds__(NUM_THREADS, 1) project_kernel(const __grid_constant__ Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 1);
  volatile WaitState* ws = reinterpret_cast<volatile WaitState*>(tmem_slot + 2);
  uint32_t* s_mask = reinterpret_cast<uint32_t*>(smem + OFF_MASKS);           // [window - 1][MASK_WORDS]: panels with a block in it
  int* s_windows = reinterpret_cast<int*>(smem + OFF_INFO);                   // [ROWS]: a row's windows beyond the first; bit 8: stacked upwards
  const uint32_t bar0 = smem_u32(bars);
  auto full = [&](int s) { return bar0 + 8u * s; };
  auto empty = [&](int s) { return bar0 + 8u * (STAGES + s); };
  const uint32_t done = bar0 + 8u * (2 * STAGES);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full(s), CONV_WARPS + 1); mbar_init(empty(s), 1); }
    mbar_init(done, 1);
    ws->abort = 0;
    ws->limit = p.wait_limit;
    for (int i = 0; i < (kMaxWindows - 1) * MASK_WORDS; ++i) s_mask[i] = 0u;
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), TMEM_COLS);
  const Unit& u = unit_of(p, blockIdx.x, &Unit::first_item);
  int item = (int)blockIdx.x - u.first_item;
  const int sp = item % u.splits; item /= u.splits;
  const int ct = item % u.col_tiles, rt = item / u.col_tiles;
  int c0, nt;
  tile_columns(u.ktot, u.col_tiles, ct, c0, nt);
  const int pn0 = (int)((long long)sp * u.panels / u.splits), pn1 = (int)((long long)(sp + 1) * u.panels / u.splits);
  const int np = pn1 - pn0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_launch_dependents();
  pdl_wait();

  // the panel (of this CTA's np) after panel q in pass w: all of them in the first pass
  auto next_panel = [&](int q, int w) {
    ++q;
    if (w == 0) return q;
    while (q < np) {
      const uint32_t rest = s_mask[(w - 1) * MASK_WORDS + (q >> 5)] >> (q & 31);
      if (rest != 0) return q + __ffs(rest) - 1;
      q = (q | 31) + 1;
    }
    return np;
  };
  int i = 0;                                                        // panels this role has been through, in all passes
  bool ok = true;

  // what the converters keep from pass to pass
  const int cw = warp - 2;
  const int r = cw * 8 + (lane >> 2), q4 = lane & 3;                // row of the tile; blocks 2 q4, 2 q4 + 1 of a panel
  const int row = rt * ROWS + r;
  const bool live = warp >= 2 && row < p.M;
  const uint16_t* xrow = u.xcat + (size_t)(live ? row : 0) * u.ld + q4 * 32;
  const uint8_t* erow = u.ebytes + (size_t)(live ? row : 0) * u.ep + q4 * 2;
  int first = 0, dir = -1;                                          // the row's first window's E + 127; the others lie nine down or up
  auto load_panel = [&](int q, uint4 (&x)[4], uint32_t& eb) {
    eb = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = make_uint4(0u, 0u, 0u, 0u);
    if (live && q < np) {
      const int pn = pn0 + q;
      eb = *reinterpret_cast<const uint16_t*>(erow + pn * 8);
      const uint4* src = reinterpret_cast<const uint4*>(xrow + pn * PANEL);
      if (pn * PANEL + q4 * 32 < u.K64) { x[0] = src[0]; x[1] = src[1]; x[2] = src[2]; x[3] = src[3]; }
    }
  };
  for (int w = 0, passes = 0; w < u.windows; ++w) {
    if (w > 0 && next_panel(-1, w) >= np) continue;               // the masks are final: every thread decides the same
    if (warp == 0) {
      // ------------------------------------------------------------ A digits: one bulk copy per plane pair
      if (lane == 0 && ok) {
        const uint8_t* img = u.planes + (size_t)u.panels * 2 * PANEL * c0;
        const uint32_t bytes = (uint32_t)(2 * PANEL * nt);
        for (int q = next_panel(-1, w); q < np; q = next_panel(q, w), ++i) {
          const int st = i % STAGES;
          if (p.stall != 0 && pn0 + q == u.panels - 1) { ok = false; break; }
          if (!mbar_wait<true>(empty(st), (uint32_t)((i / STAGES) & 1) ^ 1u, ws)) { ok = false; break; }
          if (!inside(p, u.planes, img - u.planes + (size_t)(pn0 + q) * bytes, bytes, (size_t)u.panels * 2 * PANEL * u.ktot, 342)) { ok = false; break; }
          mbar_expect_tx(full(st), bytes);
          bulk_load(smem_u32(smem + st * STAGE_BYTES + 2 * X_PLANE), img + (size_t)(pn0 + q) * bytes, bytes, full(st));
        }
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------ MMA issuer: the whole warp loops, one lane issues
      const uint32_t idesc = make_idesc_i8(ROWS, nt);
      const uint64_t xd0 = make_desc(smem_u32(smem)), ad0 = make_desc(smem_u32(smem + 2 * X_PLANE));
      uint32_t add = 0u;
      for (int q = next_panel(-1, w); q < np && ok; q = next_panel(q, w), ++i) {
        const int st = i % STAGES;
        const uint64_t xh = xd0 + (uint64_t)(st * (STAGE_BYTES >> 4)), xl = xh + (X_PLANE >> 4);
        const uint64_t ah = ad0 + (uint64_t)(st * (STAGE_BYTES >> 4)), al = ah + (uint64_t)((nt * PANEL) >> 4);
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(full(st), (uint32_t)((i / STAGES) & 1), ws)) != 0;
        if (!ok) break;
        tc_fence_after();
        if (elect_one()) {
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {                         // 32 K = 32 bytes per instruction
            const uint32_t acc = ks > 0 ? 1u : add;
            umma_i8(tmem, xh + 2 * ks, ah + 2 * ks, idesc, acc);
            umma_i8(tmem + MAX_NT, xh + 2 * ks, al + 2 * ks, idesc, acc);
            umma_i8(tmem + MAX_NT, xl + 2 * ks, ah + 2 * ks, idesc, 1u);
            umma_i8(tmem + 2 * MAX_NT, xl + 2 * ks, al + 2 * ks, idesc, acc);
          }
          umma_commit(empty(st));
        }
        add = 1u;
        __syncwarp();
      }
      if (ok && elect_one()) umma_commit(done);
    } else {
      // ------------------------------------------------------------ X_q values -> digit planes of the stage
      uint4 x[2][4];
      uint32_t eb[2];
      auto fetch = [&](int q, int h) { load_panel(q, x[h], eb[h]); };
      int q0 = next_panel(-1, w), q1 = next_panel(q0, w);          // the panels in x[0] and x[1]
      fetch(q0, 0);
      fetch(q1, 1);
      if (w == 0) {
        // the row's exponents from its shares (the row's four lanes look at four of them each)
        int top = 0, low = 255, mean = 0, n = 0;
        for (int k = q4; live && k < p.warps_per_row; k += 4) {
          const uint32_t v = u.rowparts[(size_t)row * kParts + k];
          if ((v & 0xFFu) == 0) continue;                          // a share of zeros
          top = max(top, (int)(v & 0xFFu)); low = min(low, (int)((v >> 8) & 0xFFu)); mean += (int)(v >> 16); ++n;
        }
#pragma unroll
        for (int k = 1; k < 4; k <<= 1) {
          top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, k)); low = min(low, __shfl_xor_sync(0xFFFFFFFFu, low, k));
          mean += __shfl_xor_sync(0xFFFFFFFFu, mean, k); n += __shfl_xor_sync(0xFFFFFFFFu, n, k);
        }
        const int all = top != 0 ? (top - low) / (kWindow + 1) : 0;   // windows beyond the first that the row would fill
        const int more = min(all, u.windows - 1);
        const bool up = all > 0 && all == more && mean <= n * (low + kWindow);
        first = up ? low + kWindow : top;
        dir = up ? 1 : -1;
        if (q4 == 0) {
          s_windows[r] = more | (up ? 256 : 0);
          if (live && sp == 0 && inside(p, u.rowinfo, row, 1, p.M, 339))
            u.rowinfo[row] = ((up ? first : first - more * (kWindow + 1)) - 127 + 1024) | (all > more ? 1 << 16 : 0);
        }
        unsigned far = sp == 0 && ct == 0 ? __ballot_sync(0xFFFFFFFFu, live && all > more) : 0u;
        while (far != 0) {                                             // a row at a time, all lanes
          const int src = __ffs(far) - 1;
          far &= ~(0xFu << (src & ~3));
          const int frow = __shfl_sync(0xFFFFFFFFu, row, src), ftop = __shfl_sync(0xFFFFFFFFu, top, src);
          for (int b0 = 0; b0 < u.K / 16; b0 += 32) {
            const int e = b0 + lane < u.K / 16 ? (int)u.ebytes[(size_t)frow * u.ep + b0 + lane] : 0;
            const unsigned low = __ballot_sync(0xFFFFFFFFu, e != 0 && ftop - e >= u.windows * (kWindow + 1));
            const size_t at = (size_t)frow * u.far_words + (b0 >> 5);
            if (lane == 0 && inside(p, u.rowfar, at, 1, (size_t)p.M * u.far_words, 340)) u.rowfar[at] = low;
          }
        }
      }
      const int eref = first + dir * w * (kWindow + 1);            // the window's E + 127 (beyond the row's last one: no block lies in it)
      const float base = pow2f(14 - min(max(eref - 127, -56), 55 + kWindow));
      auto put = [&](int q, int h2) {
        const int st = i % STAGES;
        if (__all_sync(0xFFFFFFFFu, mbar_wait(empty(st), (uint32_t)((i / STAGES) & 1) ^ 1u, ws)) == 0) { ok = false; return; }
        uint8_t* hi_p = smem + st * STAGE_BYTES;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int e = (int)((eb[h2] >> (8 * h)) & 0xFFu), d = eref - e;
          const float scale = e != 0 && (unsigned)d <= (unsigned)kWindow ? base : 0.0f;
          if (w == 0 && e != 0 && (unsigned)d > (unsigned)kWindow) {   // a later pass's, or finish_kernel's
            const int at = (dir > 0 ? kWindow - d : d) / (kWindow + 1);
            if (at < u.windows) atomicOr(s_mask + (at - 1) * MASK_WORDS + (q >> 5), 1u << (q & 31));
          }
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint4& v = x[h2][2 * h + (k >> 1)];
            const uint32_t a = (k & 1) ? v.z : v.x, b = (k & 1) ? v.w : v.y;
            digits_of(__uint_as_float(a << 16), __uint_as_float(a & 0xFFFF0000u), __uint_as_float(b << 16), __uint_as_float(b & 0xFFFF0000u),
                      scale, hi[k], lo[k]);
          }
          const uint32_t dst = (uint32_t)(r * PANEL + (((2 * q4 + h) ^ (r & 7)) << 4));
          *reinterpret_cast<uint4*>(hi_p + dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(hi_p + X_PLANE + dst) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(full(st));
        ++i;
      };
      while (q0 < np && ok) {
        put(q0, 0);
        q0 = next_panel(q1, w);
        fetch(q0, 0);
        if (ok && q1 < np) {
          put(q1, 1);
          q1 = next_panel(q0, w);
          fetch(q1, 1);
        }
      }
      // ------------------------------------------------------------ the sums: 64-bit combination, to memory
      if (ok) ok = __all_sync(0xFFFFFFFFu, mbar_wait(done, (uint32_t)(passes & 1), ws)) != 0;
      asm volatile("bar.sync 2, %0;" ::"n"(WORKERS) : "memory");  // s_windows is another warp's
      tc_fence_after();
      // 16 columns of a tensor memory lane's row at a time
      if (ok) {
        const int tr = (warp & 3) * 32 + lane;                     // a warp reads the lanes of its number mod 4
        const int more = s_windows[tr] & 0xFF, above = (s_windows[tr] >> 8) != 0 ? w : more - w;   // windows of the row under this one
        const long long unit = 1LL << (w <= more ? above * (kWindow + 1) : 0);
        unsigned long long* acc = u.tacc + ((size_t)rt * u.ktot + c0) * ROWS + tr;
        for (int cb = (cw >> 2) * 16; cb < nt; cb += 64) {
          uint32_t hh[16], mid[16], ll[16];
          const uint32_t base_t = tmem + ((uint32_t)((warp & 3) * 32) << 16) + cb;
          tmem_ld16(base_t, hh);
          tmem_ld16(base_t + MAX_NT, mid);
          tmem_ld16(base_t + 2 * MAX_NT, ll);
          tmem_ld_wait();
          if (w <= more) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const long long v = ((long long)(int)hh[j] * 65536 + (long long)(int)mid[j] * 256 + (long long)(int)ll[j]) * unit;
              unsigned long long* at = acc + (size_t)(cb + j) * ROWS;
              if (!inside(p, u.tacc, at - u.tacc, 1, (size_t)u.row_tiles * u.ktot * ROWS, 341)) continue;
              if (u.splits > 1) atomicAdd(at, (unsigned long long)v);
              else *at = (unsigned long long)v + (w > 0 ? *at : 0ull);
            }
          }
        }
        __threadfence();
      }
    }
    ++passes;
    tc_fence_before();
    __syncwarp();
    // every role is through this pass (or has given up): the masks are final, the accumulators and the ring are free
    asm volatile("bar.sync 1, %0;" ::"n"(NUM_THREADS) : "memory");
    tc_fence_after();
  }

  if (ws->abort != 0) {
    const long long t0 = clock64();
    while (clock64() - t0 < 400000) { }                     // copies in flight land before the CTA's shared memory goes
    if (tid == 0) report_error(p.status, LQER_ERR_TIMEOUT, 330, blockIdx.x);
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace pdg

// Scratch of a unit whose layers' rank paddings sum to ktot (behind its Xcat): exponent bytes, windows, digit planes of A_q,
// counters and 64-bit sums.
static size_t digit_unit_scratch(int K64, int ktot, int M) {
  using namespace pdg;
  const size_t panels = (size_t)(K64 + PANEL - 1) / PANEL, rt = (size_t)(M + ROWS - 1) / ROWS;
  const size_t words = (size_t)(K64 / 16 + 31) / 32;
  return align256((size_t)M * panels * 8) + align256((size_t)M * kParts * 4) + align256((size_t)M * 4) + align256((size_t)ktot * 4) +
         align256((size_t)M * words * 4) + align256((size_t)ktot * words * 4) + align256(panels * 2 * PANEL * ktot) +
         align256(rt * ktot * ROWS * 8);
}
size_t prologue_digits_scratch_bytes(const PackedMeta& m, int M) { return digit_unit_scratch(m.K64, m.k_pad, M); }
// The unit of each call: calls that multiply the same X share one (an X that is not known yet is nobody else's).
static int digit_units(const DigitCall* calls, int n, int* unit_at) {
  int units = 0, first[kDigitMaxLayers];
  for (int g = 0; g < n; ++g) {
    int q = 0;
    while (q < units && !(calls[g].X != nullptr && calls[first[q]].X == calls[g].X && calls[first[q]].meta->K == calls[g].meta->K)) ++q;
    if (q == units) first[units++] = g;
    unit_at[g] = q;
  }
  return units;
}
size_t prologue_digits_group_bytes(const DigitCall* calls, int n, int M) {
  using namespace pdg;
  int unit_at[kDigitMaxLayers], ktot[kDigitMaxUnits] = {}, K64[kDigitMaxUnits] = {};
  const int units = digit_units(calls, n, unit_at);
  for (int g = 0; g < n; ++g) { ktot[unit_at[g]] += calls[g].meta->k_pad; K64[unit_at[g]] = calls[g].meta->K64; }
  size_t bytes = 0;
  for (int q = 0; q < units; ++q) bytes += align256((size_t)M * (K64[q] + ktot[q]) * 2) + digit_unit_scratch(K64[q], ktot[q], M);
  return bytes;
}

cudaError_t launch_prologue_digits(const DigitCall* calls, int n, int M, int x_type, void* scratch, GemmActs* places, int8_t* Tm,
                                   uint8_t* Te, DeviceStatus* st, cudaStream_t s) {
  using namespace pdg;
  if (n < 1 || n > kDigitMaxLayers) return cudaErrorInvalidValue;
  static OncePerDevice once;
  cudaError_t err = once.run([] { return cudaFuncSetAttribute(project_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES); });
  if (err != cudaSuccess) return err;
  const PackedMeta& m0 = *calls[0].meta;
  Params p;
  p.n = 0; p.M = M; p.x_type = x_type;
  p.a_bits = m0.a_bits; p.lr_bits = m0.lr_bits; p.exp_min = m0.exp_min; p.exp_max = m0.exp_max; p.w_exp_min = m0.w_exp_min;
  p.status = st;
  p.wait_limit = wait_limit_cycles();
  // layers that multiply the same X share its quantised values
  int unit_at[kDigitMaxLayers];
  digit_units(calls, n, unit_at);
  for (int g = 0; g < n; ++g) {
    const PackedMeta& m = *calls[g].meta;
    if (m.k_pad == 0) return cudaErrorInvalidValue;
    Unit& u = p.U[unit_at[g]];
    if (unit_at[g] == p.n) {
      ++p.n;
      u.X = calls[g].X; u.K = m.K; u.K64 = m.K64;
      u.panels = (m.K64 + PANEL - 1) / PANEL;
      u.ep = u.panels * 8;
      u.row_tiles = (M + ROWS - 1) / ROWS;
      u.far_words = (m.K64 / 16 + 31) / 32;
      u.windows = m.K64 <= 32768 ? kMaxWindows : 2;          // 63 bits: 2^20 K leave room for two
      u.n_layers = 0; u.ktot = 0;
    }
    LayerA& la = u.layer[u.n_layers++];
    la.asec = static_cast<const uint8_t*>(calls[g].packed) + m.off_a;
    la.Tm = n == 1 ? Tm : nullptr; la.Te = n == 1 ? Te : nullptr;
    la.k_pad = m.k_pad; la.col0 = u.ktot;
    places[g].t_col = m.K64 + u.ktot;
    u.ktot += m.k_pad;
  }
  uint8_t* at = static_cast<uint8_t*>(scratch);
  int items = 0, longest = 0;
  for (int q = 0; q < p.n; ++q) {
    Unit& u = p.U[q];
    u.ld = u.K64 + u.ktot;
    u.col_tiles = (u.ktot + MAX_NT - 1) / MAX_NT;
    u.splits = (u.K64 + 32767) / 32768;                     // int32 sums: at most 32768 K per CTA
    items += u.row_tiles * u.col_tiles * u.splits;
    longest = std::max(longest, u.ep);
    u.xcat = reinterpret_cast<uint16_t*>(at);
    u.xcat_extent = (size_t)M * u.ld * 2;
    at += align256(u.xcat_extent);
    u.ebytes = at; at += align256((size_t)M * u.ep);
    u.rowparts = reinterpret_cast<uint32_t*>(at); at += align256((size_t)M * kParts * 4);
    u.rowinfo = reinterpret_cast<int*>(at); at += align256((size_t)M * 4);
    u.colinfo = reinterpret_cast<int*>(at); at += align256((size_t)u.ktot * 4);
    u.rowfar = reinterpret_cast<uint32_t*>(at); at += align256((size_t)M * u.far_words * 4);
    u.colout = reinterpret_cast<uint32_t*>(at); at += align256((size_t)u.ktot * u.far_words * 4);
    u.planes = at; at += align256((size_t)u.panels * 2 * PANEL * u.ktot);
    u.tacc = reinterpret_cast<unsigned long long*>(at); at += align256((size_t)u.row_tiles * u.ktot * ROWS * 8);
  }
  for (int g = 0; g < n; ++g) {
    places[g].xcat = p.U[unit_at[g]].xcat;
    places[g].ld = p.U[unit_at[g]].ld;
  }
  // K ranges: CTAs for one round over the SMs, and at least two panels a range
  const int sms = std::max(sm_count(), 1);
  for (;;) {
    int pick = -1;
    double len = 2.0;
    for (int q = 0; q < p.n; ++q) {
      const Unit& u = p.U[q];
      const double l = (double)u.panels / u.splits;
      if (l > len && items + u.row_tiles * u.col_tiles <= sms) { len = l; pick = q; }
    }
    if (pick < 0) break;
    ++p.U[pick].splits;
    items += p.U[pick].row_tiles * p.U[pick].col_tiles;
  }
  // A row to a warp where the rows fill the SMs (32 warps each), to several warps otherwise, down to one block per lane.
  p.warps_per_row = 1;
  while (p.warps_per_row < kParts && (long long)p.n * M * p.warps_per_row < (long long)32 * sms && longest > 32 * kBatch * p.warps_per_row)
    p.warps_per_row *= 2;
  int warps = 0, finish = 0;
  items = 0;
  for (int q = 0; q < p.n; ++q) { p.U[q].first_a = warps; warps += p.U[q].ktot / kColsPerWarp * kColShares; }
  p.rows_begin = warps;
  for (int q = 0; q < p.n; ++q) {
    Unit& u = p.U[q];
    u.first_rows = warps; warps += M * p.warps_per_row;
    u.first_item = items; items += u.row_tiles * u.col_tiles * u.splits;
    u.first_finish = finish; finish += u.row_tiles * u.col_tiles * (ROWS / kFinishRows);
  }
  p.n_warps = warps;
  for (int q = p.n; q < kDigitMaxUnits; ++q) p.U[q] = p.U[0];
  p.stall = take_stall(kFamPrologue) ? 1 : 0;
  LaunchScope scope(kFamPrologue, s, 3);
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3((warps + kQuantThreads / 32 - 1) / (kQuantThreads / 32));
  cfg.blockDim = dim3(kQuantThreads);
  if ((err = cudaLaunchKernelEx(&cfg, quantise_kernel, p)) != cudaSuccess) return err;
  cfg.gridDim = dim3(items);
  cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  if ((err = cudaLaunchKernelEx(&cfg, project_kernel, p)) != cudaSuccess) return err;
  cfg.gridDim = dim3(finish);
  cfg.blockDim = dim3(WORKERS);
  cfg.dynamicSmemBytes = 0;
  return cudaLaunchKernelEx(&cfg, finish_kernel, p);
}

}  // namespace lqer
