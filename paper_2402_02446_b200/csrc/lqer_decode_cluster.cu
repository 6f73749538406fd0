// The layer for 3 to 16 tokens in one launch (paper Section 3.1 / 3.2: Y = X_q W_q + q(X_q A_q) B_q; Section 2.1: few
// tokens per step make it memory bound on its weights).
//
// A cluster of CS CTAs owns a range of weight tiles (128 columns); its CTAs share the contraction: CTA q takes the slabs
// [q k_slabs / CS, (q + 1) k_slabs / CS).  So a CTA quantises only its part of X.  What the parts have to exchange:
//   - Y: consumer warps multiply 32 columns of a tile each, every third stage, and send their sums to the CTAs that own the columns
//     (st.async, counted in bytes on that CTA's mbarrier), whose epilogue warps add them in order, add the rank term and write Y once,
//     while the consumers are in the next tile.
//   - T = X_q A_q: the first clusters of a layer form it, one or a few rank blocks each.  Each CTA multiplies its part (int8
//     mma.sync per 16-block, exact, scaled and summed in fp64) and stores its partial sums into the CTA of its cluster that owns
//     the row; the owner adds them in order, re-quantises along the rank, writes T_q to scratch in global memory and counts its
//     blocks in.  Every epilogue warp waits for the count before its first rank term, and where a CTA's wait in vain, another of its warps
//     forms T_q by itself (form_t_alone).  The layer's last warp to have read T_q zeroes the counters for the next call.  Where a
//     cluster has few weights to multiply, it forms all of T itself, and the owners of the rows store T_q into its CTAs' shared memory.
// So a cluster waits for other clusters of its launch, which need not be there yet: launches on several streams get their places one by
// one, and the clusters that form a layer's T cannot leave before all of it is there.  With form_t_alone nobody waits for a cluster that has no
// place, and launches cannot hold each other up, however many there are.  (With one cluster for all of a layer's T nobody would either:
// 4096 / 11008, 4 rows, rank 32 64 -> 68 us a layer, rank 128 68 -> 89, 3 rows, rank 256 78 -> 128; placed as a whole by a cooperative launch
// 64 -> 72, 68 -> 75, 78 -> 86 and 3 us a launch on the host.)
//
// The packed weights come by bulk copies, a stage (two slabs of a tile, 9 KB) at a time: a producer warp keeps a ring of stages full, from
// before griddepcontrol.wait on, for weights depend on no earlier kernel.  Twelve consumer warps read a stage's mantissas with ldmatrix (the
// 16 bytes that the tile stores for a column and block pair are a row of it, so every lane of a group of four gets one word without
// bank conflicts), convert them to bf16 in registers and feed them to mma.sync.m16n8k16, weights on the 16-row side.
// What bounds it: 540 cycles a stage up to eight rows, some 650 beyond (the ALU pipe's shifts and masks, two cycles each, and the MMAs,
// 8.6 each), i.e. 4.6 and 3.8 TB/s; and some 7 us around the stages, of which the chain X -> X_q -> T -> T_q -> rank term is 4.5.
// A CTA has an SM to itself: with two launches resident side by side, each with half of an SM, clusters came to lie two to an SM on some
// and on others not at all; a run of (tile, step) to each CTA of 148 without clusters, the sums exchanged through global memory, took
// 94 us where this takes 64 (decoder layer of 4096 / 11008, 4 rows); copies of 0.5 to 2 KB, padded against bank conflicts, 118.
#include <algorithm>
#include <mutex>

#include "lqer_cluster_plan.h"
#include "lqer_gemm_small.cuh"
#include "lqer_mma_frag.cuh"

namespace lqer {
namespace dcl {
using namespace mf;
using sg::bf16_rn;
using tc::smem_u32;

struct Layer {
  const void* X;
  void* Y;
  const uint8_t* wsec;
  const uint8_t* bsec;
  const uint8_t* asec;
  size_t y_extent, w_extent;
  int K, N, k_pad, k_slabs, r_blocks, tiles;
  int cluster_begin, clusters;
  uint8_t* tq;                              // T_q on its way between clusters: eight planes (token_offset)
  int* tcount;                              // arrivals, departures: zero between calls
  int t_blocks;                             // rank blocks of T that each of the layer's first clusters forms
  int t_clusters, t_tiles;                  // ... and how many those are, if they get fewer tiles than the others: so many each
  int t_expect;                             // arrivals that make T_q whole (one more under the test hooks)
};
struct Params {
  Layer L[kMaxLayers];
  int n, M;
  DeviceStatus* status;
  int x_type, y_type;
  int a_bits, lr_bits, exp_min, exp_max;
  int steps_max;                            // steps of a CTA, at most: the extent of the activation planes
  int slots;                                // ring slots
  int off_red, red_bytes, off_xq, off_xe, off_tpart, off_trecv, off_tq, off_ring;   // offsets in shared memory (the planes of X_q come first)
  long long wait_limit;
  long long lag;                            // checked build, test hook: see lqer_debug_converter_lag
  int stall;                                // test hook: the sums of the first tile and a cluster's own T_q wait for bytes that never come (see also t_expect)
};

__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_cta(uint32_t addr, uint32_t cta) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Stores into another CTA's shared memory that count themselves in on its mbarrier.
__device__ __forceinline__ void st_async(uint32_t addr, double a, double b, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(addr), "d"(a), "d"(b), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async(uint32_t addr, float a, float b, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr), "f"(a), "f"(b), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async(uint32_t addr, uint32_t a, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(a), "r"(bar) : "memory");
}
__device__ __forceinline__ void arrive_remote(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait of a whole warp for a phase that other CTAs of the cluster complete (one answer for all lanes).
__device__ __forceinline__ bool wait_cluster(uint32_t bar, uint32_t parity, volatile tc::WaitState* ws) {
  const long long t0 = clock64();
  for (int spins = 0;; ++spins) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (__all_sync(0xFFFFFFFFu, ok != 0)) return true;
    if ((spins & 63) == 63) {
      bool give_up = ws->abort != 0;
      if (clock64() - t0 > ws->limit) { ws->abort = 1; give_up = true; }
      if (__any_sync(0xFFFFFFFFu, give_up)) return false;
    }
  }
}
__device__ __forceinline__ bool count_reached(const int* count, int expect) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
  return __all_sync(0xFFFFFFFFu, v >= expect) != 0;
}
// The same for a counter in global memory that other clusters of the launch raise, or for a warp of the CTA that has done their work.
enum TState { kAwaited = 0, kHere, kFormed };    // T_q as a CTA knows it: not there, counted in by its clusters, formed by the CTA's own warp
__device__ __forceinline__ bool wait_count(const int* count, int expect, volatile int* t_state, volatile tc::WaitState* ws) {
  const long long t0 = clock64();
  while (!count_reached(count, expect)) {
    if (__any_sync(0xFFFFFFFFu, *t_state == kFormed)) { __threadfence(); break; }
    bool give_up = ws->abort != 0;
    if (clock64() - t0 > ws->limit) { ws->abort = 1; give_up = true; }
    if (__any_sync(0xFFFFFFFFu, give_up)) return false;
    __nanosleep(64);
  }
  if (*t_state == kAwaited) *t_state = kHere;
  return true;
}
template <bool kBackoff = false>
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile tc::WaitState* ws) {
  return __all_sync(0xFFFFFFFFu, tc::mbar_wait<kBackoff>(bar, parity, ws)) != 0;
}
__device__ __forceinline__ void worker_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(kWorkers) : "memory"); }
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix2(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}

// A stage in shared memory: two slabs of a packed weight tile, as they lie in the packed buffer.
template <int WB>
struct Stage {
  static constexpr int kMant = slab_mantissa_bytes(WB);
  static constexpr int kTile = slab_bytes(WB);
  static constexpr int kBytes = 2 * kTile;
};
// Four consecutive columns of a row of Y (a lane of a quad of lanes that hold a 16-block of the row), all lanes calling.
__device__ __forceinline__ void write_y4(const Params& p, const Layer& ly, int row, int col, float4 v, bool live) {
  if (p.y_type == kYMXINT8) {
    uint32_t m8;
    uint2 unused;
    int e;
    quantize_quad(v, p.a_bits, p.exp_min, p.exp_max, e, m8, unused);
    const size_t idx = (size_t)row * ly.N + col;
    uint8_t* yq = static_cast<uint8_t*>(ly.Y);
    if (live && LQER_IN_BOUNDS(p.status, (size_t)p.M * ly.N + idx / 16, 1, ly.y_extent, 732)) {
      *reinterpret_cast<uint32_t*>(yq + idx) = m8;
      if ((col & 15) == 0) yq[(size_t)p.M * ly.N + idx / 16] = (uint8_t)(e + 127);
    }
  } else if (live) {
    const size_t idx = (size_t)row * ly.N + col;
    if (p.y_type == kYBF16) {
      if (LQER_IN_BOUNDS(p.status, idx * 2, 8, ly.y_extent, 731))
        *reinterpret_cast<uint2*>(static_cast<uint16_t*>(ly.Y) + idx) =
            make_uint2(bf16_rn(v.x) | (bf16_rn(v.y) << 16), bf16_rn(v.z) | (bf16_rn(v.w) << 16));
    } else if (LQER_IN_BOUNDS(p.status, idx * 4, 16, ly.y_extent, 731)) {
      *reinterpret_cast<float4*>(static_cast<float*>(ly.Y) + idx) = v;
    }
  }
}

// Block `kb` (16 elements from column 16 kb) of a row of X in any of the three types.
__device__ __forceinline__ void load_x_block(float (&v)[16], const void* X, int x_type, int M, int K, int row, int kb, int bits, int emin, int emax) {
  const size_t idx = (size_t)row * K + (size_t)kb * 16;
  if (x_type == kXBF16) {
    const uint4* src = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(X) + idx);
    const uint4 a = __ldg(src), b = __ldg(src + 1);
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) { v[2 * i] = __uint_as_float(w[i] << 16); v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u); }
  } else if (x_type == kXMXINT8) {
    const uint8_t* xb = static_cast<const uint8_t*>(X);
    const uint4 m = __ldg(reinterpret_cast<const uint4*>(xb + idx));
    const uint32_t eb = __ldg(xb + (size_t)M * K + idx / 16);
    const uint32_t w[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 q = mxint_quad_values(w[i], eb, bits, emin, emax);
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

// Activations as the MMA's narrow operand (n = 8 tokens to a tile, MT tiles).  MMA i of a step of 128 K takes four K from each lane t, in the
// order in which the lanes get the weights: word t of every block pair (4-bit mantissas: K 32 (i >> 1) + 8 t + 4 (i & 1) of the step),
// or word t of every slab (2-bit ones: K 64 (i >> 2) + 16 t + 4 (i & 3)).  Four planes, of the MMAs 2 m and 2 m + 1 of every step: [step][MMA where MT
// == 2][token, lane t][16 bytes], the 16 bytes being both MMAs' words of one tile, or one MMA's of two.
// The sixteen K of a block (f0, f1: eight pairs of bf16 values) to their places.
template <int WB, int MT>
__device__ __forceinline__ void store_block(uint8_t* planes, uint32_t plane, int row, int block, const uint4& f0, const uint4& f1) {
  const int b = block & 3, slab = block >> 2;
  uint8_t* at = planes + plane_offset((slab & 1) * 2 + (WB == 4 ? b >> 1 : 0), plane) + (uint32_t)((slab >> 1) * (512 * MT) + (row >> 3) * 4) +
                ((row & 7) * 4 + (WB == 4 ? (b & 1) * 2 : b)) * 16;
  const uint32_t next = WB == 4 ? 16u : plane;               // the block's second half: the next lane's, or the next pair of MMAs
  if (MT == 1) {
    *reinterpret_cast<uint4*>(at) = f0;
    *reinterpret_cast<uint4*>(at + next) = f1;
  } else {
    const uint32_t w[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int h = 0; h < 2; ++h) *reinterpret_cast<uint32_t*>(at + (k >> 1) * next + (k & 1) * 512 + h * 8) = w[2 * k + h];
  }
}
// T_q: eight planes of [rank slab of 64][16 positions][MT pairs of words]; plane i of a lane's 32 ranks holds its ranks 4 i .. 4 i + 3.
// Byte offset of (token, slab, rank c of the slab, a multiple of 4) within its plane.
template <int MT>
__device__ __forceinline__ uint32_t token_offset(int row, int slab, int c) {
  return (uint32_t)(slab * (128 * MT) + (2 * (row & 7) + (c >> 5)) * (8 * MT) + (row >> 3) * 4);
}
__device__ __forceinline__ void mma_w(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// 128 K of NP units: columns g and g + 8 of a unit are rows g and g + 8 of the MMA.  word(o, m): eight converted weights of column octet o,
// for the MMAs 2 m and 2 m + 1; load(m, b0, b1): those MMAs' activations (two words for each tile of tokens).
// The MMAs of a step add up in chains of four (MT == 1; eight otherwise), and the chains' sums are added to acc by fp32 additions: the
// accumulators of mma.sync cut off what does not fit, and one chain over 1700 K was up to 14 times as far off as kernels that
// add by rounded fp32 operations (2-norm against 64 bits for 13824 K of one sign, block exponents over a dozen binades: 4 rows 8.5e-7,
// column-owner kernel 6.2e-8, with these chains 5.1e-8; 16 rows 8.5e-7, tensor-memory GEMM 8.9e-8, with these 5.0e-8).
template <int MT, int NP, class Word, class Load>
__device__ __forceinline__ void multiply_step(float (&acc)[NP][MT][4], Word&& word, Load&& load) {
  constexpr int kChain = MT == 1 ? 2 : 4;            // m per chain
  float d[NP][MT][4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (m % kChain == 0) {
#pragma unroll
      for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) d[p][i][q] = 0.f;
    }
    uint32_t b[2][2 * MT];
    load(m, b[0], b[1]);
    uint4 w[2 * NP];
#pragma unroll
    for (int o = 0; o < 2 * NP; ++o) w[o] = word(o, m);
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
      for (int i = 0; i < MT; ++i) mma_w(d[p][i], w[2 * p].x, w[2 * p + 1].x, w[2 * p].y, w[2 * p + 1].y, b[0][2 * i], b[0][2 * i + 1]);
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
      for (int i = 0; i < MT; ++i) mma_w(d[p][i], w[2 * p].z, w[2 * p + 1].z, w[2 * p].w, w[2 * p + 1].w, b[1][2 * i], b[1][2 * i + 1]);
    if (m % kChain == kChain - 1) {
#pragma unroll
      for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[p][i][q] += d[p][i][q];
    }
  }
}
// Eight signed bytes as bf16 values times sc, exact, by the integers' bits (conversion instructions run at an eighth of the rate): byte + 128 is the low
// byte of the float 1.5 * 2^23 + 128 + byte.
__device__ __forceinline__ uint4 convert_i8x8(uint32_t w0, uint32_t w1, float sc) {
  const float back = -12583040.0f * sc;
  auto value = [&](uint32_t u, uint32_t select) { return fmaf(__uint_as_float(__byte_perm(u, 0x4B400000u, select)), sc, back); };
  auto pair = [&](uint32_t u, uint32_t lo, uint32_t hi) { return __byte_perm(__float_as_uint(value(u, lo)), __float_as_uint(value(u, hi)), 0x7632); };
  w0 ^= 0x80808080u;
  w1 ^= 0x80808080u;
  return make_uint4(pair(w0, 0x7640, 0x7641), pair(w0, 0x7642, 0x7643), pair(w1, 0x7640, 0x7641), pair(w1, 0x7642, 0x7643));
}
// int -> fp64 by the integer's bits (2^52 + 2^31 + v), where the conversion instruction runs at a sixteenth of the rate.
__device__ __forceinline__ double int_to_double(int v) { return __hiloint2double(0x43300000, v ^ 0x80000000) - 4503601774854144.0; }

// A 16-block of T in as many neighbouring lanes, as MXINT8 along the rank: the lane's value in bf16 and its neighbour's.
__device__ __forceinline__ uint32_t quantize_t(const Params& p, double v) {
  double amax = (v != v) ? 0.0 : fabs(v);
#pragma unroll
  for (int d = 1; d < 16; d <<= 1) amax = fmax(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, d));
  const int e = block_exponent(amax, p.exp_min, p.exp_max);
  const uint32_t bits = (uint32_t)bf16_bits_of(quant_mantissa(v, e, p.a_bits), e - (p.a_bits - 2)) & 0xFFFFu;
  return bits | (__shfl_down_sync(0xFFFFFFFFu, bits, 1) << 16);
}
// Warps that share the tiles of T of a cluster with `cols` ranks.
__device__ __forceinline__ int warps_per_tile(int cols) { return cols == 0 || cols / 8 >= kWorkerWarps ? 1 : kWorkerWarps / (cols / 8); }
// The byte of T_q in scratch that ranks j and j + 1 (j even) of a row begin at.
template <int MT>
__device__ __forceinline__ uint32_t tq_offset(int row, int j, uint32_t rplane) {
  return (uint32_t)((j & 31) >> 2) * rplane + token_offset<MT>(row, j >> 6, j & 63) + (uint32_t)((j & 2) * 2 * MT);
}
constexpr int kHelpWait = 200000;               // cycles (T takes some 10 us where its clusters run)
// All of a layer's T_q by one warp, unless the clusters that are to form it do so meanwhile: the same sums in the same order, hence the
// same bytes whoever writes them.  A lane has a rank of a row and walks K (0.5 us a block of 16): half a millisecond for 4 rows, rank 32 and
// K = 4096, where waiting takes as long as other launches hold the places.
template <int MT>
__device__ __forceinline__ void form_t_alone(const Params& p, const Layer& ly, int CS, uint32_t rplane, const volatile int* t_state) {
  const int lane = threadIdx.x & 31, total = p.M * ly.k_pad, kblocks = ly.K / 16;
  const QuantConsts qc = quant_consts(p.a_bits, p.exp_min, p.exp_max);
  const int bias = -127 - (p.a_bits - 2) - (p.lr_bits - 2);
#pragma unroll 1
  for (int o = lane; o - lane < total; o += 32) {
    if (__any_sync(0xFFFFFFFFu, *t_state != kAwaited) || count_reached(ly.tcount, ly.t_expect)) return;
    const bool live = o < total;
    const int row = live ? o / ly.k_pad : 0, j = o % ly.k_pad, rb_lo = j / 16 / ly.t_blocks * ly.t_blocks;
    const int share = warps_per_tile(16 * (min(rb_lo + ly.t_blocks, ly.r_blocks) - rb_lo));
    double v = 0.0;
#pragma unroll 1
    for (int c = 0; c < CS; ++c) {
      const int lo = c * ly.k_slabs / CS * 4, hi = min((c + 1) * ly.k_slabs / CS * 4, kblocks);
      double sum = 0.0;
#pragma unroll 1
      for (int first = lo; first < lo + share; ++first) {
        double acc = 0.0;
#pragma unroll 1
        for (int b = first; b < hi; b += share) {
          float x[16];
          int e;
          uint4 m8, f0, f1;
          load_x_block(x, ly.X, p.x_type, p.M, ly.K, row, b, p.a_bits, p.exp_min, p.exp_max);
          quantize_block16(x, qc, e, m8, f0, f1);
          const uint4 a = __ldg(reinterpret_cast<const uint4*>(ly.asec + ((size_t)b * ly.k_pad + j) * 16));
          const int ea = __ldg(ly.asec + (size_t)kblocks * ly.k_pad * 16 + (size_t)b * ly.k_pad + j);
          int dot = __dp4a((int)m8.x, (int)a.x, 0);
          dot = __dp4a((int)m8.y, (int)a.y, dot);
          dot = __dp4a((int)m8.z, (int)a.z, dot);
          dot = __dp4a((int)m8.w, (int)a.w, dot);
          acc = fma(int_to_double(dot), pow2d(e + bias + ea), acc);
        }
        sum += acc;
      }
      v += sum;
    }
    const uint32_t bits = quantize_t(p, live ? v : 0.0), at = tq_offset<MT>(row, j, rplane);
    if (live && (lane & 1) == 0 && LQER_IN_BOUNDS(p.status, at, 4, 8 * rplane, 735)) *reinterpret_cast<uint32_t*>(ly.tq + at) = bits;
  }
  __threadfence();
  __syncwarp();
}

// WB: mantissa bits of W_q (4 or 2).  MT: tiles of eight tokens (1 or 2).  LOCAL: every cluster forms all of T for itself.
template <int WB, int MT, bool LOCAL>
__global__ void __launch_bounds__(kThreads, 1) decode_cluster_kernel(const __grid_constant__ Params p, int CS) {
  using St = Stage<WB>;
  constexpr int kTile = St::kTile, kMant = St::kMant;
  constexpr int TS = token_stride(MT);
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) uint64_t s_bars[3 + 2 * kRed + 2 * kMaxSlots];
  __shared__ tc::WaitState s_ws;
  __shared__ volatile int s_t_state;                   // of TState

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int rank = (int)cta_rank(), cluster = (int)blockIdx.x / CS;
  int layer = 0;
#pragma unroll
  for (int i = 1; i < kMaxLayers; ++i)
    if (i < p.n && cluster >= p.L[i].cluster_begin) layer = i;
  const Layer& ly = p.L[layer];
  const int M = p.M, K = ly.K, k_pad = ly.k_pad;
  const int cl = cluster - ly.cluster_begin;
  // this cluster's tiles: t_tiles for each of those that form T, equal shares of the rest for the others
  const int f_all = ly.t_clusters * ly.t_tiles, others = ly.clusters - ly.t_clusters, rest = ly.tiles - f_all, nth = cl - ly.t_clusters;
  const int tile_lo = nth < 0 ? cl * ly.t_tiles : f_all + (int)((uint32_t)nth * (uint32_t)rest / (uint32_t)others);
  const int chunks = nth < 0 ? ly.t_tiles : f_all + (int)((uint32_t)(nth + 1) * (uint32_t)rest / (uint32_t)others) - tile_lo;
  const int s_lo = rank * ly.k_slabs / CS, s_hi = (rank + 1) * ly.k_slabs / CS, n_slabs = s_hi - s_lo;
  const int steps = (n_slabs + 1) / 2;                               // of two slabs (128 K)
  const uint32_t plane = plane_bytes(p.steps_max, MT);
  const uint32_t sm = smem_u32(smem);
  const uint32_t bar0 = smem_u32(s_bars);
  const uint32_t t_full = bar0, t_seen = bar0 + 8;
  const uint32_t t_ready = bar0 + 16;
  auto red_full = [&](int b) { return bar0 + 24 + 8u * b; };
  auto red_free = [&](int b) { return bar0 + 24 + 8u * (kRed + b); };
  auto full = [&](int s) { return bar0 + 24 + 8u * (2 * kRed + s); };
  auto empty = [&](int s) { return bar0 + 24 + 8u * (2 * kRed + kMaxSlots + s); };
  // unit j of a tile is CTA j mod CS's (columns beyond N are multiplied like the others: a packed tile has all of them)
  const int n_own = kUnits / CS;
  const uint32_t chunk_bytes = (uint32_t)(n_own * kUnit * 8 * ((M + 1) / 2) * CS * kPhases);
  // This cluster's share of T: rank blocks [rb_lo, rb_hi), i.e. NT tiles of 8 columns; where there are fewer tiles than warps,
  // WPN warps share one and split its blocks of K.
  const int rb_lo = LOCAL ? 0 : min(cl * ly.t_blocks, ly.r_blocks), rb_hi = min(rb_lo + ly.t_blocks, ly.r_blocks);
  const int t_cols = 16 * (rb_hi - rb_lo), NT = t_cols / 8, WPN = warps_per_tile(t_cols);
  const int RP = 8 * MT / CS;                                        // rows whose T a CTA owns
  const int own_rows = max(0, min(M - rank * RP, RP));
  const uint32_t rplane = (uint32_t)((k_pad + 127) / 128) * (256u * MT);   // a plane of T_q: rank slabs, an even number of them

  if (warp == kWorkerWarps) {
    // ------------------------------------------------------------------ producer
    // (the one slab of an odd last step is taken twice: its second half meets activations that are zeros)
    const int x_hi = chunks * steps;
    auto fill = [&](int x, int slot) -> bool {
      const int tile = x / steps, slab = s_lo + 2 * (x - tile * steps);
      const size_t src = ((size_t)(tile_lo + tile) * ly.k_slabs + slab) * kTile;
      const uint32_t dst = sm + p.off_ring + slot * St::kBytes;
      const uint32_t bytes = slab + 1 < s_hi ? 2 * kTile : kTile;
      if (!LQER_IN_BOUNDS(p.status, src, bytes, ly.w_extent, 733)) return false;
      tc::mbar_expect_tx(full(slot), 2 * kTile);
      tc::bulk_load(dst, ly.wsec + src, bytes, full(slot));
      if (bytes == kTile) tc::bulk_load(dst + kTile, ly.wsec + src, bytes, full(slot));
      return true;
    };
    int x = 0;
    bool go = true;
    if (lane == 0) {
      tc::mbar_init(t_full, 1);
      tc::mbar_init(t_seen, CS * kEpilogue);
      tc::mbar_init(t_ready, 1);
      for (int i = 0; i < kRed; ++i) { tc::mbar_init(red_full(i), 1); tc::mbar_init(red_free(i), CS * kEpilogue); }
      for (int i = 0; i < p.slots; ++i) { tc::mbar_init(full(i), 1); tc::mbar_init(empty(i), kColumnWarps); }
      s_ws.abort = 0;
      s_ws.limit = p.wait_limit;
      s_t_state = kAwaited;
      tc::fence_barrier_init();
      tc::fence_proxy_async_smem();
      if (NT > 0 && own_rows > 0) tc::mbar_expect_tx(t_full, (uint32_t)(own_rows * t_cols * 8 * CS));
      if (LOCAL) tc::mbar_expect_tx(t_ready, (uint32_t)(M * k_pad * 2) + (p.stall ? 16u : 0u));
      for (int i = 0; i < min(chunks, kRed); ++i) tc::mbar_expect_tx(red_full(i), chunk_bytes + (p.stall && i == 0 ? 16u : 0u));
    }
    __syncwarp();
    tc::pdl_launch_dependents();
    cluster_arrive();
    // (a copy takes its issuing thread some 50 ns: the others do not wait for all of the ring)
    const int first = min(min(p.slots, x_hi), kPhases);
    if (lane == 0)
      for (; x < first && go; ++x) go = fill(x, x);
    __syncwarp();
    cluster_wait();
    __syncthreads();
    if (lane == 0) {
      for (; x < p.slots && x < x_hi && go; ++x) go = fill(x, x);
      RingWalk<kPhases> walk(x);
      int held = -1, held_slot = 0;                    // checked build, test hook: a stage whose copy comes late (see lqer_debug_converter_lag)
      for (; x < x_hi && go; ++x) {
        const int slot = walk.turn[0].slot;
        if (!tc::mbar_wait<true>(empty(slot), walk.turn[0].parity, &s_ws)) break;
        if (kDebugBounds && p.lag > 0 && held < 0 && x % 5 == 4 && x + p.slots - kPhases < x_hi) { held = x; held_slot = slot; }
        else go = fill(x, slot);
        walk.next(p.slots);
        if (kDebugBounds && held >= 0 && x >= held + p.slots - kPhases) {    // (until here no stage waits for this one)
          const long long t0 = clock64();
          while (clock64() - t0 < p.lag) { }
          go = go && fill(held, held_slot);
          held = -1;
        }
      }
      if (!go) s_ws.abort = 1;
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    if (s_ws.abort != 0) {                             // given up: copies in flight land before the CTA's shared memory goes
      const long long t0 = clock64();
      while (clock64() - t0 < 400000) { }
    }
    return;
  }
  tc::pdl_launch_dependents();
  cluster_arrive();
  if (warp > kWorkerWarps) {
    // ------------------------------------------------------------------ T where its clusters do not come
    cluster_wait();
    __syncthreads();
    tc::pdl_wait();
    if (!LOCAL && k_pad > 0) {
      const long long t0 = clock64();
      while (__all_sync(0xFFFFFFFFu, s_t_state == kAwaited && *(volatile int*)&s_ws.abort == 0)) {
        if (__any_sync(0xFFFFFFFFu, clock64() - t0 > kHelpWait)) {
          form_t_alone<MT>(p, ly, CS, rplane, &s_t_state);
          s_t_state = kFormed;
          break;
        }
        __nanosleep(500);
      }
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    return;
  }

  // ---- A_q of this CTA's blocks and this cluster's ranks: the first words into registers, the others towards L2
  const int kblocks = K / 16, kb0 = s_lo * 4, nreal = min(n_slabs * 4, kblocks - kb0);
  const int nt_first = NT >= kWorkerWarps ? warp : NT > 0 ? warp % NT : 0, sub = NT >= kWorkerWarps || NT == 0 ? 0 : warp / NT;
  const bool t_active = NT > 0 && (NT >= kWorkerWarps || warp < NT * WPN);
  constexpr int UB = 6;                                                // words of each of the two in flight (with eight the registers spill)
  uint32_t aw[2][UB], ae[2][UB];
  auto load_a = [&](int bq, int nt, uint32_t (&w)[UB], uint32_t (&e)[UB]) {
    const uint8_t* am = ly.asec + ((size_t)(kb0 + bq) * k_pad + rb_lo * 16 + nt * 8 + g) * 16 + t * 4;
    const uint8_t* ax = ly.asec + (size_t)kblocks * k_pad * 16 + (size_t)(kb0 + bq) * k_pad + rb_lo * 16 + nt * 8 + t * 2;
#pragma unroll
    for (int u = 0; u < UB; ++u) {
      w[u] = 0u; e[u] = 0u;
      if (bq + u * WPN < nreal) {
        w[u] = __ldg(reinterpret_cast<const uint32_t*>(am));
        e[u] = (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(ax));
      }
      am += (size_t)WPN * k_pad * 16;
      ax += (size_t)WPN * k_pad;
    }
  };
  if (t_active) {
    load_a(sub, nt_first, aw[0], ae[0]);
    load_a(sub + UB * WPN, nt_first, aw[1], ae[1]);
  }
  if (NT > 0)
    for (int i = tid; i < nreal * NT; i += kWorkers) {                 // 128 bytes of mantissas each, and the exponents beside them
      const size_t at = (size_t)(kb0 + i / NT) * k_pad + rb_lo * 16 + (i % NT) * 8;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(ly.asec + at * 16));
      if (i % 4 == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(ly.asec + (size_t)kblocks * k_pad * 16 + at));
    }
  // B_q of this CTA's units, towards L2
  if (k_pad > 0 && warp >= kConsumers)
    for (int i = tid - kConsumers * 32; i < chunks * n_own * ly.r_blocks; i += kEpilogue * 32) {
      const int rb = i % ly.r_blocks, u = i / ly.r_blocks, col = (rank + (u % n_own) * CS) * kUnit;
      const uint8_t* bt = ly.bsec + (size_t)(tile_lo + u / n_own) * ly.r_blocks * kTileN * 17;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(bt + ((size_t)rb * kTileN + col) * 16));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(bt + ((size_t)rb * kTileN + col + 8) * 16));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(bt + (size_t)ly.r_blocks * kTileN * 16 + rb * kTileN + col));
    }
  // ---- zeros where no activation is written: rows beyond M, the second half of an odd last step, ranks beyond k_pad
  for (int o = tid * 16; o < (int)plane_offset(4, plane); o += kWorkers * 16) *reinterpret_cast<uint4*>(smem + o) = make_uint4(0u, 0u, 0u, 0u);
  uint8_t* xq = smem + p.off_xq;
  int8_t* xe = reinterpret_cast<int8_t*>(smem + p.off_xe);
  const int xq_stride = p.steps_max * 128 + 16, xe_stride = p.steps_max * 8;
  cluster_wait();                                    // every CTA's barriers are set up
  __syncthreads();
  tc::pdl_wait();                                    // X and Y may be in use by the kernel before

  // ---- X -> MXINT8, a lane per 16-block: bf16 pairs for W_q, mantissas and exponents for A_q
  {
    const QuantConsts qc = quant_consts(p.a_bits, p.exp_min, p.exp_max);
    const int n_blk = M * nreal;
    float v[2][16];                                  // a block is on its way while the one before is quantised
    const int row_step = kWorkers / nreal, blk_step = kWorkers % nreal;
    int row = tid / nreal, blk = tid % nreal, i = tid;
    auto next = [&](int& r, int& b) {
      r += row_step;
      b += blk_step;
      if (b >= nreal) { b -= nreal; ++r; }
    };
    if (i < n_blk) load_x_block(v[0], ly.X, p.x_type, M, K, row, kb0 + blk, p.a_bits, p.exp_min, p.exp_max);
    while (i < n_blk) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (i >= n_blk) break;
        const int r = row, c = blk;
        next(row, blk);
        i += kWorkers;
        if (i < n_blk) load_x_block(v[h ^ 1], ly.X, p.x_type, M, K, row, kb0 + blk, p.a_bits, p.exp_min, p.exp_max);
        int e;
        uint4 m8, f0, f1;
        quantize_block16(v[h], qc, e, m8, f0, f1);
        if (NT > 0) {
          *reinterpret_cast<uint4*>(xq + r * xq_stride + c * 16) = m8;
          xe[r * xe_stride + c] = (int8_t)e;
        }
        store_block<WB, MT>(smem, plane, r, c, f0, f1);
      }
    }
  }
  worker_barrier();

  // ---- T over this CTA's blocks, a share of them and a tile of ranks to a warp
  if (t_active) {
    const int bias = -127 - (p.a_bits - 2) - (p.lr_bits - 2);        // exponent bytes carry +127
    double* tpart = reinterpret_cast<double*>(smem + p.off_tpart);
    // rows beyond M are read (whatever lies there) but never sent
    for (int nt = nt_first; nt < NT; nt += kWorkerWarps) {
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      if (nt != nt_first) {
        load_a(sub, nt, aw[0], ae[0]);
        load_a(sub + UB * WPN, nt, aw[1], ae[1]);
      }
      for (int b0 = sub; b0 < nreal; b0 += 2 * UB * WPN) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int bq = b0 + h * UB * WPN;
          if (bq >= nreal) break;
          // (blocks beyond the last have zeros for A_q: without a branch the chains of UB blocks run side by side)
#pragma unroll
          for (int u = 0; u < UB; ++u) {
            const int b = min(bq + u * WPN, nreal - 1);
            const uint32_t a0 = *reinterpret_cast<const uint32_t*>(xq + g * xq_stride + b * 16 + t * 4);
            const uint32_t a1 = MT == 2 ? *reinterpret_cast<const uint32_t*>(xq + (g + 8) * xq_stride + b * 16 + t * 4) : 0u;
            int c[4];
            mma_s8(c, a0, a1, aw[h][u]);
            const int ea_lo = (int)(ae[h][u] & 0xFFu), ea_hi = (int)(ae[h][u] >> 8);
            const int ex0 = xe[g * xe_stride + b] + bias;
            acc[0] = fma(int_to_double(c[0]), pow2d(ex0 + ea_lo), acc[0]);
            acc[1] = fma(int_to_double(c[1]), pow2d(ex0 + ea_hi), acc[1]);
            if (MT == 2) {
              const int ex1 = xe[(g + 8) * xe_stride + b] + bias;
              acc[2] = fma(int_to_double(c[2]), pow2d(ex1 + ea_lo), acc[2]);
              acc[3] = fma(int_to_double(c[3]), pow2d(ex1 + ea_hi), acc[3]);
            }
          }
          if (bq + 2 * UB * WPN < nreal) load_a(bq + 2 * UB * WPN, nt, aw[h], ae[h]);
        }
      }
#pragma unroll
      for (int h = 0; h < MT; ++h)
        *reinterpret_cast<double2*>(tpart + (sub * (8 * MT) + g + 8 * h) * t_cols + nt * 8 + t * 2) = make_double2(acc[2 * h], acc[2 * h + 1]);
    }
  }
  if (NT > 0) {
    // the sum of the CTA's shares, to the CTA that owns the row
    worker_barrier();
    const double* tpart = reinterpret_cast<const double*>(smem + p.off_tpart);
    const int pairs = t_cols / 2;
    for (int o = tid; o < M * pairs; o += kWorkers) {
      const int row = o / pairs, owner = row / RP;
      const double* src = tpart + row * t_cols + (o % pairs) * 2;
      double a = 0.0, b = 0.0;
#pragma unroll 4
      for (int c = 0; c < WPN; ++c) {
        const double2 d = *reinterpret_cast<const double2*>(src + c * (8 * MT) * t_cols);
        a += d.x; b += d.y;
      }
      st_async(map_cta(sm + p.off_trecv + (uint32_t)((rank * RP + row % RP) * t_cols + (o % pairs) * 2) * 8u, owner), a, b, map_cta(t_full, owner));
    }
  }
  bool ok = true;

  if (warp < kConsumers) {
    // ------------------------------------------------------------------ consumers
    const ConvConsts kc = conv_consts<WB>();
    const int cw = warp % kColumnWarps, phase = warp / kColumnWarps, col = cw * 2 * kUnit;
    const uint8_t* x_lane = smem + lane * 16;
    // addresses of the rows of 16 bytes that ldmatrix distributes: lanes 8 i .. 8 i + 7 give the eight columns of piece i
    const uint32_t w_row = sm + p.off_ring + (col + (lane & 7)) * 16 + (WB == 4 ? (lane >> 4) * kTile + ((lane >> 3) & 1) * 2048 : ((lane >> 3) & 1) * kTile);
    const uint8_t* e_lane = smem + p.off_ring + kMant + (col + g) * 4;
    int x = phase;
    RingCursor at(phase);
#pragma unroll 1
    for (int r = 0, begin = 0, b = 0, turn = 0; r < chunks; ++r, begin += steps) {     // b, turn: r mod and by kRed
      float acc[2][MT][4];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[u][i][c] = 0.f;
#pragma unroll 1
      for (; x < begin + steps; x += kPhases) {
        const int slot = at.slot;
        if (!warp_wait(full(slot), at.parity, &s_ws)) { ok = false; break; }
        uint32_t w[4][4], e[4][2];
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          if (WB == 4) ldmatrix4(w[o], w_row + slot * St::kBytes + o * 128);
          else ldmatrix2(w[o], w_row + slot * St::kBytes + o * 128);
#pragma unroll
          for (int h = 0; h < 2; ++h) e[o][h] = *reinterpret_cast<const uint32_t*>(e_lane + slot * St::kBytes + o * 32 + h * kTile);
        }
        const uint8_t* xs = x_lane + (x - begin) * (512 * MT);
        multiply_step<MT, 2>(acc, [&](int o, int m) -> uint4 {
          uint32_t s2, c2;
          if (WB == 4) {
            w_scale_pair(e[o][m >> 1], 2 * (m & 1) + (t >> 1), s2, c2);
            return convert_nibbles(w[o][m], s2, c2, kc);
          } else {
            w_scale_pair2(e[o][m >> 1], t, s2, c2);
            return convert_crumbs(w[o][m >> 1], m & 1, s2, c2, kc);
          }
        }, [&](int m, uint32_t (&b0)[2 * MT], uint32_t (&b1)[2 * MT]) {
          uint4 v = *reinterpret_cast<const uint4*>(xs + plane_offset(m, plane));
          if (MT == 1) {
            b0[0] = v.x; b0[1] = v.y; b1[0] = v.z; b1[1] = v.w;
          } else {
            b0[0] = v.x; b0[2 * MT - 2] = v.y; b0[1] = v.z; b0[2 * MT - 1] = v.w;
            v = *reinterpret_cast<const uint4*>(xs + plane_offset(m, plane) + 512);
            b1[0] = v.x; b1[2 * MT - 2] = v.y; b1[1] = v.z; b1[2 * MT - 1] = v.w;
          }
        });
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(empty(slot));
        at.next(kPhases, p.slots);
      }
      if (ok && r == 0 && NT > 0) ok = wait_cluster(t_seen, 0, &s_ws);       // the sums lie where T was formed
      if (ok && r >= kRed) ok = wait_cluster(red_free(b), (uint32_t)(turn - 1) & 1u, &s_ws);
      if (!ok) break;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int j = 2 * cw + u;
        const uint32_t base = map_cta(sm + p.off_red + b * p.red_bytes + (uint32_t)((((j / CS) * CS + rank) * kPhases + phase) * kUnit * TS * 4), (uint32_t)(j % CS));
        const uint32_t bar = map_cta(red_full(b), (uint32_t)(j % CS));
#pragma unroll
        for (int i = 0; i < MT; ++i)
          if (8 * i + 2 * t < M) {
            st_async(base + (uint32_t)((g * TS + 8 * i + 2 * t) * 4), acc[u][i][0], acc[u][i][1], bar);
            st_async(base + (uint32_t)(((g + 8) * TS + 8 * i + 2 * t) * 4), acc[u][i][2], acc[u][i][3], bar);
          }
      }
      if (++b == kRed) { b = 0; ++turn; }
    }
  } else {
    // ------------------------------------------------------------------ epilogue
    const int ew_ = warp - kConsumers, etid = tid - kConsumers * 32;
    // the rows of T this CTA owns: sum in order, MXINT8 along the rank, out to scratch for all clusters of the layer
    auto reduce_t = [&]() -> bool {
      const int total = own_rows * t_cols;
      if (ew_ * 32 >= total) return true;
      if (!wait_cluster(t_full, 0, &s_ws)) return false;
      const double* tp = reinterpret_cast<const double*>(smem + p.off_trecv);
      int done = 0;                                    // 16-blocks
      for (int o = etid; o - lane < total; o += kEpilogue * 32) {
        const bool live = o < total;
        done += min(32, total - (o - lane)) >> 4;
        double v = 0.0;
        if (live) {
#pragma unroll 8
          for (int c = 0; c < CS; ++c) v += tp[c * RP * t_cols + o];
        }
        const uint32_t bits = quantize_t(p, v);
        if (live && (lane & 1) == 0) {
          const int row = rank * RP + o / t_cols, j = rb_lo * 16 + o % t_cols;
          const uint32_t at = tq_offset<MT>(row, j, rplane);
          if (LOCAL) {
            for (int c = 0; c < CS; ++c) st_async(map_cta(sm + p.off_tq + at, c), bits, map_cta(t_ready, c));
          } else if (LQER_IN_BOUNDS(p.status, at, 4, 8 * rplane, 734)) {
            *reinterpret_cast<uint32_t*>(ly.tq + at) = bits;
          }
        }
      }
      __syncwarp();
      // (one lane's release covers what the warp wrote before)
      if (lane == 0 && !LOCAL) asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(ly.tcount), "r"(done) : "memory");
      return true;
    };
    if (NT > 0) {
      ok = reduce_t();
      __syncwarp();
      if (lane < CS) arrive_remote(map_cta(t_seen, lane));
    }
    const uint32_t r_off = (uint32_t)((t >> 1) * (128 * MT) + (2 * g + (t & 1)) * (8 * MT));   // the lane's position within a step of a plane of T_q
    bool have_t = false;
    // Units of this warp to come; after the last one's rank term it counts itself out.  The layer's last warp to do so zeroes the counters for
    // the next call (all of T_q is there then: some warp has waited for it).
    int left = 0, out = 0;
    for (int r = 0; r < chunks; ++r)
      for (int q = (ew_ - r * n_own) & (kEpilogue - 1); q < n_own; q += kEpilogue) ++left;
    auto count_out = [&]() {
      if (k_pad > 0 && !LOCAL && left == 0 && lane == 0) out = atomicAdd(ly.tcount + 1, 1);
    };
    count_out();
#pragma unroll 1
    for (int r = 0, b = 0, turn = 0; r < chunks && ok; ++r) {
      bool here = false;                               // the tile's sums have come
      // the units of one tile after the other go to the epilogue warps in turn
      for (int q = (ew_ - r * n_own) & (kEpilogue - 1); q < n_own; q += kEpilogue) {
        const int unit = rank + q * CS, col = (tile_lo + r) * kTileN + unit * kUnit;
        float term[1][MT][4];
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) term[0][i][c] = 0.f;
        const uint8_t* bt = ly.bsec + (size_t)(tile_lo + r) * ly.r_blocks * kTileN * 17;
#pragma unroll 1
        for (int j = 0; j * 128 < k_pad; ++j) {
          uint4 w[2][2];
          float sc[2][2];
#pragma unroll
          for (int o = 0; o < 2; ++o) {
            const int nl = unit * kUnit + o * 8 + g;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int rb = 8 * j + 2 * t + u;
              const bool in = rb < ly.r_blocks;
              w[o][u] = in ? ld_stream16(bt + ((size_t)rb * kTileN + nl) * 16) : make_uint4(0u, 0u, 0u, 0u);
              sc[o][u] = in ? pow2f((int)bt[(size_t)ly.r_blocks * kTileN * 16 + rb * kTileN + nl] - 127 - (p.lr_bits - 2)) : 1.0f;
            }
          }
          if (!have_t) {
            ok = LOCAL ? wait_cluster(t_ready, 0, &s_ws) : wait_count(ly.tcount, ly.t_expect, &s_t_state, &s_ws);
            have_t = true;
            if (!ok) break;
          }
          // all of the lane's T_q of these ranks at once
          const int blocks = ly.r_blocks - (8 * j + 2 * t);
          const uint32_t x_at = j * (256 * MT) + r_off;
          uint32_t x[8][2 * MT];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const bool in = (i >> 2) < blocks;
            if (MT == 1) {
              const uint2 a = !in ? make_uint2(0u, 0u) : LOCAL ? *reinterpret_cast<const uint2*>(smem + p.off_tq + x_at + i * rplane)
                                                                    : __ldcg(reinterpret_cast<const uint2*>(ly.tq + x_at + i * rplane));
              x[i][0] = a.x; x[i][1] = a.y;
            } else {
              const uint4 a = !in ? make_uint4(0u, 0u, 0u, 0u) : LOCAL ? *reinterpret_cast<const uint4*>(smem + p.off_tq + x_at + i * rplane)
                                                                            : __ldcg(reinterpret_cast<const uint4*>(ly.tq + x_at + i * rplane));
              x[i][0] = a.x; x[i][2 * MT - 2] = a.y; x[i][1] = a.z; x[i][2 * MT - 1] = a.w;
            }
          }
          multiply_step<MT, 1>(term, [&](int o, int m) {
            const uint4& a = w[o][m >> 1];
            return convert_i8x8(m & 1 ? a.z : a.x, m & 1 ? a.w : a.y, sc[o][m >> 1]);
          }, [&](int m, uint32_t (&b0)[2 * MT], uint32_t (&b1)[2 * MT]) {
#pragma unroll
            for (int i = 0; i < 2 * MT; ++i) { b0[i] = x[2 * m][i]; b1[i] = x[2 * m + 1][i]; }
          });
        }
        if (!ok) break;
        --left;
        count_out();
        if (!here) { ok = wait_cluster(red_full(b), (uint32_t)turn & 1u, &s_ws); here = true; }
        if (!ok) break;
        float* buf = reinterpret_cast<float*>(smem + p.off_red + b * p.red_bytes) + q * CS * kPhases * kUnit * TS;
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 6
          for (int c = 0; c < CS * kPhases; ++c) {
            const float2 a0 = *reinterpret_cast<const float2*>(buf + (c * kUnit + g) * TS + 8 * i + 2 * t);
            const float2 a1 = *reinterpret_cast<const float2*>(buf + (c * kUnit + g + 8) * TS + 8 * i + 2 * t);
            v[0] += a0.x; v[1] += a0.y; v[2] += a1.x; v[3] += a1.y;
          }
          *reinterpret_cast<float2*>(buf + g * TS + 8 * i + 2 * t) = make_float2(v[0] + term[0][i][0], v[1] + term[0][i][1]);
          *reinterpret_cast<float2*>(buf + (g + 8) * TS + 8 * i + 2 * t) = make_float2(v[2] + term[0][i][2], v[3] + term[0][i][3]);
        }
        __syncwarp();
        // a quad of lanes holds a row's sixteen columns
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          const int row = (lane >> 2) + 8 * i, c = (lane & 3) * 4;
          const float* src = buf + c * TS + row;
          write_y4(p, ly, row, col + c, make_float4(src[0], src[TS], src[2 * TS], src[3 * TS]), row < M && col + c < ly.N);
        }
      }
      if (ok && !here) ok = wait_cluster(red_full(b), (uint32_t)turn & 1u, &s_ws);
      if (!ok) break;
      if (r + kRed < chunks) {
        // (its bytes cannot come before this warp's arrivals below)
        if (etid == 0) tc::mbar_expect_tx(red_full(b), chunk_bytes);
        __syncwarp();
        if (lane < CS) arrive_remote(map_cta(red_free(b), lane));
      }
      if (++b == kRed) { b = 0; ++turn; }
    }
    if (ok && k_pad > 0 && !LOCAL && lane == 0 && out == ly.clusters * CS * kEpilogue - 1) {
      ly.tcount[0] = 0;
      ly.tcount[1] = 0;
    }
  }
  __syncwarp();
  cluster_arrive();                                  // this warp's last store into another CTA lies behind it
  cluster_wait();                                    // no CTA leaves while another may still store into its shared memory
  if (tid == 0 && s_ws.abort != 0) report_error(p.status, LQER_ERR_TIMEOUT, 730, blockIdx.x);
}

static cudaLaunchConfig_t launch_config(int CS, int clusters, size_t smem, cudaLaunchAttribute* attr, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * CS);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CS; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}
// Clusters of CS CTAs that the device holds at a time (-1 if the query fails).
template <int WB, int MT, bool LOCAL>
static int resident_clusters(int CS) {
  static std::mutex mu;
  static int known[64][4] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  std::lock_guard<std::mutex> lock(mu);
  int& n = known[dev][CS == 8 ? 3 : CS == 4 ? 2 : CS == 2 ? 1 : 0];
  if (n == 0) {
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = launch_config(CS, 1, kSmemMax, attr, nullptr);
    if (cudaFuncSetAttribute(decode_cluster_kernel<WB, MT, LOCAL>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, decode_cluster_kernel<WB, MT, LOCAL>, &cfg) != cudaSuccess) {
      n = 0;
      return -1;
    }
  }
  return n;
}
template <int WB, int MT, bool LOCAL>
static cudaError_t launch(const Params& p, int clusters, int CS, size_t smem, cudaStream_t s) {
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = launch_config(CS, clusters, smem, attr, s);
  LaunchScope scope(kFamDecode, s);
  return cudaLaunchKernelEx(&cfg, decode_cluster_kernel<WB, MT, LOCAL>, p, CS);
}
struct Entry {
  int (*resident)(int);
  cudaError_t (*go)(const Params&, int, int, size_t, cudaStream_t);
};
template <int WB, int MT>
static Entry entry(bool local) {
  return local ? Entry{resident_clusters<WB, MT, true>, launch<WB, MT, true>} : Entry{resident_clusters<WB, MT, false>, launch<WB, MT, false>};
}
static Entry entry_of(int wb, int mt, bool local) {
  if (wb == 4) return mt == 1 ? entry<4, 1>(local) : entry<4, 2>(local);
  return mt == 1 ? entry<2, 1>(local) : entry<2, 2>(local);
}

static bool plan(const PackedMeta* metas, int n, int M, Plan& q) {
  static thread_local PlanCache cache;
  Shape sh = {};
  if (cudaGetDevice(&sh.dev) != cudaSuccess) return false;
  sh.n = n; sh.M = M; sh.w_bits = metas[0].w_bits;
  for (int i = 0; i < n; ++i) { sh.k_slabs[i] = metas[i].k_slabs; sh.tiles[i] = metas[i].n_tiles; sh.r_blocks[i] = metas[i].r_blocks; }
  const int mt = M > 8 ? 2 : 1;
  return cache.find(sh, [&](int CS) { return std::min(entry_of(sh.w_bits, mt, false).resident(CS), entry_of(sh.w_bits, mt, true).resident(CS)); }, q);
}
}  // namespace dcl

// Whether n layers with one M go out as one launch of this kernel: at 3 to 16 rows, up to four layers, wherever X_q fits.  Measured on one
// B200, us a call in a chain of such calls over weights beyond L2, the same sums through two CTAs to an SM with a ring of each lane's own
// pieces (before) / this kernel; for 16 rows the kernels that share a prologue, which took the larger of these calls / this kernel:
//   4096 x 4096, rank 32 alone   4 rows 11.2 / 10.5   8 rows 11.4 / 10.7   16 rows 14.7 / 13.1
//   three of them                4 rows 20.8 / 15.3   8 rows 21.3 / 15.6   16 rows 28.1 / 20.7
//   two of 4096 x 11008          4 rows 30.3 / 25.6   8 rows 30.8 / 26.1   16 rows 33.1 / 30.6
//   11008 x 4096 alone           4 rows 17.2 / 13.9   8 rows 18.4 / 14.9   16 rows 28.9 / 22.4
//   two of 5120 x 13824, rank 64 4 rows 43.8 / 31.7   8 rows 44.5 / 32.9   16 rows 45.8 / 41.7
//   the same, rank 256           3 rows 48.9 / 34.4   8 rows 53.2 / 36.1   16 rows 52.7 / 46.9
//   2048 x 2048, rank 32 alone   4 rows 8.9 / 7.2;  rank 64, 16 rows 10.7 / 10.6
// and a whole layer of hidden 1024 to 2048 at 16 rows: 1024, rank 0 26.2 / 29.0, rank 32 42.3 / 42.8; 1984, rank 0 41.5 / 42.1; 2048, rank 64
// 62.5 / 51.6.  (Short contractions of 9 and more rows without a rank are where the smaller CTAs were as fast or faster.)
// One and two rows keep the column-owner kernel, whose launches several layers share bit for bit.
int decode_cluster_max_layers() { return dcl::kMaxLayers; }
bool decode_cluster_takes(const PackedMeta* metas, int n, int M) {
  using namespace dcl;
  if (n < 1 || n > kMaxLayers || M < 3 || M > kRows) return false;
  Plan q;
  return plan(metas, n, M, q);
}

cudaError_t launch_decode_cluster(const lqer_call_t* calls, const PackedMeta* metas, int n, void* scratch, int* counts, DeviceStatus* st,
                                  int x_type, int y_type, cudaStream_t s) {
  using namespace dcl;
  if (n < 1 || n > kMaxLayers) return cudaErrorInvalidValue;
  const int M = calls[0].M;
  Plan q;
  if (!plan(metas, n, M, q)) return cudaErrorInvalidConfiguration;
  Params p;
  p.n = n; p.M = M; p.status = st; p.x_type = x_type; p.y_type = y_type;
  p.a_bits = metas[0].a_bits; p.lr_bits = metas[0].lr_bits; p.exp_min = metas[0].exp_min; p.exp_max = metas[0].exp_max;
  p.wait_limit = wait_limit_cycles();
  p.stall = take_stall(kFamDecode) ? 1 : 0;
  p.lag = debug_converter_lag();
  p.steps_max = q.steps_max;
  p.slots = q.slots;
  p.off_red = q.off_red; p.red_bytes = q.red_bytes;
  p.off_xq = q.off_xq; p.off_xe = q.off_xe; p.off_tpart = q.off_tpart; p.off_trecv = q.off_trecv; p.off_tq = q.off_tq; p.off_ring = q.off_ring;
  int begin = 0;
  size_t t_off = 0;
  for (int i = 0; i < kMaxLayers; ++i) {
    const int g = i < n ? i : 0;
    const PackedMeta& m = metas[g];
    if (m.a_bits != p.a_bits || m.lr_bits != p.lr_bits || m.exp_min != p.exp_min || m.exp_max != p.exp_max || m.w_bits != metas[0].w_bits)
      return cudaErrorInvalidValue;
    Layer& ly = p.L[i];
    const uint8_t* base = static_cast<const uint8_t*>(calls[g].packed);
    ly.X = calls[g].X; ly.Y = calls[g].Y;
    ly.wsec = base + m.off_w; ly.bsec = base + m.off_b; ly.asec = base + m.off_a;
    ly.y_extent = y_bytes(y_type, (size_t)M, (size_t)m.N);
    if (kDebugBounds) ly.y_extent -= std::min(ly.y_extent, debug_y_shrink());
    ly.w_extent = m.off_b - m.off_w;
    ly.K = m.K; ly.N = m.N; ly.k_pad = m.k_pad; ly.k_slabs = m.k_slabs; ly.r_blocks = m.r_blocks; ly.tiles = m.n_tiles;
    ly.cluster_begin = begin;
    ly.clusters = q.clusters[g];
    ly.tq = static_cast<uint8_t*>(scratch) + t_off;
    ly.tcount = counts + 2 * g;
    // the warps of an owner count their 16-blocks of T in
    ly.t_expect = M * m.r_blocks + (p.stall != 0 || (kDebugBounds && p.lag > 0) ? 1 : 0);
    ly.t_blocks = q.t_blocks[g]; ly.t_clusters = q.t_clusters[g]; ly.t_tiles = q.t_tiles[g];
    if (i < n) t_off += decode_cluster_scratch_bytes(m);
    if (i < n) begin += q.clusters[g];
  }
  return entry_of(metas[0].w_bits, M > 8 ? 2 : 1, q.local).go(p, q.total, q.CS, q.smem, s);
}

}  // namespace lqer
