// The layer for M <= 16 tokens in one launch (paper Section 3.1 / 3.2: Y = X_q W_q + q(X_q A_q) B_q; Section 2.1: few
// tokens per step make it memory bound on its weights).
//
// A cluster of CS CTAs (8 where the contraction has 16 slabs of 64) owns a range of output columns; its CTAs share the
// contraction: CTA q takes the slabs [q k_slabs / CS, (q + 1) k_slabs / CS).  So a CTA quantises only its part of X.  What the
// parts have to exchange:
//   - Y: the warps of a CTA own column octets, a round of them at a time, over the CTA's slabs.  Warp w's sums of a round go
//     to CTA w mod CS (st.async, counted in bytes on that CTA's mbarrier), which adds them in CTA order and writes Y once.
//   - T = X_q A_q: the first clusters of a layer form it, one or a few rank blocks each.  Each CTA multiplies its part (int8
//     mma.sync per 16-block, exact, scaled and summed in fp64) and stores its partial sums into the CTA of its cluster that owns
//     the row; the owner adds them in CTA order, re-quantises along the rank, writes T_q to scratch in global memory and counts its
//     blocks in.  Every cluster of the layer waits for the count (bounded) before its first rank term, the last thing of its
//     first round; the last warp to have read T_q zeroes the counters for the next call.
// So a cluster waits for other clusters of its launch.  The launch has no more of them than the device holds at a time, those
// that form T come first, and launch_decode_cluster says what keeps launches on several streams from holding each other up.
//
// The weights take the register-operand form (lqer_mma_frag.cuh): a lane loads the 16 bytes which the packed tile stores
// for one column and block pair, here through its own slots of a ring in shared memory (cp.async; a lane reads back only
// what it copied itself, so the ring needs no barrier), converts them to bf16 in registers and feeds them to
// mma.sync.m16n8k16.  The ring is filled before griddepcontrol.wait, for weights depend on no earlier kernel.
#include <algorithm>
#include <mutex>

#include "lqer_gemm_small.cuh"
#include "lqer_mma_frag.cuh"

namespace lqer {
namespace dcl {
using namespace mf;
using sg::bf16_rn;
using tc::smem_u32;

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kMaxLayers = 4;                // layers of a launch, at most
constexpr int kOcts = 4;                    // column octets a warp owns in a round, at most
constexpr int kRows = 16;

struct Layer {
  const void* X;
  void* Y;
  const uint8_t* wsec;
  const uint8_t* bsec;
  const uint8_t* asec;
  size_t y_extent, w_extent;
  int K, N, k_pad, k_slabs, r_blocks;
  int cluster_begin, clusters;
  uint8_t* tq;                              // T_q on its way between clusters: eight planes (the layout of the activations)
  int* tcount;                              // arrivals, departures: zero between calls
  int t_blocks;                             // rank blocks of T that each of the layer's first clusters forms
  int t_expect;                             // arrivals that make T_q whole (one more under the test hook)
};
struct Params {
  Layer L[kMaxLayers];
  int n, M;
  DeviceStatus* status;
  int x_type, y_type;
  int a_bits, lr_bits, exp_min, exp_max;
  int slabs_max;                            // slabs of a CTA, rounded up to even: the extent of the activation planes
  int off_red[2], off_xq, off_xe, off_tpart, off_ring;   // offsets in shared memory (the planes of X_q come first)
  long long wait_limit;
  int stall;                                // test hook: the sums of the first round wait for bytes that never come (see also t_expect)
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
// The same for a counter in global memory that other clusters of the launch raise.
__device__ __forceinline__ bool wait_count(const int* count, int expect, volatile tc::WaitState* ws) {
  const long long t0 = clock64();
  for (;;) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
    if (__all_sync(0xFFFFFFFFu, v >= expect)) return true;
    bool give_up = ws->abort != 0;
    if (clock64() - t0 > ws->limit) { ws->abort = 1; give_up = true; }
    if (__any_sync(0xFFFFFFFFu, give_up)) return false;
    __nanosleep(64);
  }
}
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void cp16(uint32_t dst, const void* src) { asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp8(uint32_t dst, const void* src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp4(uint32_t dst, const void* src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory"); }

template <int WB>
__host__ __device__ constexpr int stage_bytes() { return kOcts * 32 * (WB == 4 ? 16 : 8) + kOcts * 32 * 4; }

// Words from column to column of a warp's sums in the buffer of the CTA that adds them: tokens, two more against bank conflicts.
__host__ __device__ constexpr int token_stride(int mt) { return 8 * mt + 2; }

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

// Activations as the MMA's narrow operand (n = 8 tokens to a tile, MT tiles): eight planes of [slab][16 positions][MT pairs of
// words]; plane i of a lane's 32 K holds its K 4 i .. 4 i + 3.  Byte offset of (token, slab, column c of the slab, a multiple of 4)
// within its plane; the second pair of K lies 4 MT bytes on.
template <int MT>
__device__ __forceinline__ uint32_t token_offset(int row, int slab, int c) {
  return (uint32_t)(slab * (128 * MT) + (2 * (row & 7) + (c >> 5)) * (8 * MT) + (row >> 3) * 4);
}
__device__ __forceinline__ void mma_w(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// 128 K of NP pairs of column octets: the octets of a pair are rows g and g + 8 of the MMA.  word(o, m): eight converted weights.
// RANK: the activations (T_q) come from global memory, and only the first `blocks` 16-blocks of the lane's two exist.
// The MMAs of a step add up in chains of four (MT == 1; eight otherwise, for want of registers), and the chains' sums are added to
// acc by fp32 additions: the accumulators of mma.sync cut off what does not fit, and one chain over a CTA's whole part of K was up to
// 14 times as far off as the kernels that took these calls before (2-norm against 64 bits for 13824 K of one sign, block
// exponents over a dozen binades: 4 rows 8.5e-7, column-owner kernel 6.2e-8, now 5.1e-8; 16 rows 8.5e-7, tensor-memory GEMM 8.9e-8,
// now 5.0e-8).  Chains of eight for MT == 1 are at 1.0 to 1.7 times the column-owner kernel where the signs are mixed, of four at
// 0.8 to 1.2.  us a call with one chain / these: 4096 x 4096, 4 rows 11.4 / 11.5, 16 rows 15.4 / 15.4.  The one or two rank steps of MT == 2
// continue acc itself (with chains of their own, 16 rows of rank 256 took 24.6 us instead of 22.0: spilled registers).
template <int MT, int NP, bool RANK = false, class Word>
__device__ __forceinline__ void multiply_step(float (&acc)[kOcts / 2][MT][4], const uint8_t* x, uint32_t plane, Word&& word, int blocks = 2) {
  constexpr bool kChains = !(RANK && MT == 2);
  constexpr int kChain = MT == 1 ? 2 : 4;            // m per chain
  float d[NP][MT][4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (kChains && m % kChain == 0) {
#pragma unroll
      for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) d[p][i][q] = 0.f;
    }
    uint4 w[2 * NP];
#pragma unroll
    for (int o = 0; o < 2 * NP; ++o) w[o] = word(o, m);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint8_t* at = x + (2 * m + h) * plane;
      uint32_t b[2 * MT];
      if (MT == 1) {
        uint2 v = make_uint2(0u, 0u);
        if (!RANK) v = *reinterpret_cast<const uint2*>(at);
        else if ((m >> 1) < blocks) v = __ldcg(reinterpret_cast<const uint2*>(at));
        b[0] = v.x; b[1] = v.y;
      } else {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (!RANK) v = *reinterpret_cast<const uint4*>(at);
        else if ((m >> 1) < blocks) v = __ldcg(reinterpret_cast<const uint4*>(at));
        b[0] = v.x; b[2 * MT - 2] = v.y; b[1] = v.z; b[2 * MT - 1] = v.w;
      }
#pragma unroll
      for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int i = 0; i < MT; ++i)
          mma_w(kChains ? d[p][i] : acc[p][i], h ? w[2 * p].z : w[2 * p].x, h ? w[2 * p + 1].z : w[2 * p + 1].x, h ? w[2 * p].w : w[2 * p].y,
                h ? w[2 * p + 1].w : w[2 * p + 1].y, b[2 * i], b[2 * i + 1]);
    }
    if (kChains && m % kChain == kChain - 1) {
#pragma unroll
      for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[p][i][q] += d[p][i][q];
    }
  }
}
// int -> fp64 by the integer's bits (2^52 + 2^31 + v), where the conversion instruction runs at a sixteenth of the rate.
__device__ __forceinline__ double int_to_double(int v) { return __hiloint2double(0x43300000, v ^ 0x80000000) - 4503601774854144.0; }

// WB: mantissa bits of W_q (4 or 2).  MT: tiles of eight tokens (1 or 2).  YQ: Y is MXINT8 (a warp then owns whole 16-column
// blocks).  D: ring slots per warp.
template <int WB, int MT, bool YQ, int D>
__global__ void __launch_bounds__(kThreads, 2) decode_cluster_kernel(const __grid_constant__ Params p, int CS) {
  constexpr int kTile = WB == 4 ? kWTileBytes : 2048 + kTileN * 4;   // bytes of a packed weight tile
  constexpr int kMant = WB == 4 ? kWTileNibbleBytes : 2048;          // of which mantissas
  constexpr int kPiece = WB == 4 ? 16 : 8;                           // a lane's mantissas in one octet of a step
  constexpr int kStage = stage_bytes<WB>();
  constexpr int TS = token_stride(MT);
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) uint64_t s_bars[6];
  __shared__ tc::WaitState s_ws;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int rank = (int)cta_rank(), cluster = (int)blockIdx.x / CS;
  int layer = 0;
#pragma unroll
  for (int i = 1; i < kMaxLayers; ++i)
    if (i < p.n && cluster >= p.L[i].cluster_begin) layer = i;
  const Layer& ly = p.L[layer];
  const int M = p.M, K = ly.K, k_pad = ly.k_pad;
  const int cl = cluster - ly.cluster_begin;
  constexpr int kUnit = YQ ? 2 : 1;                                  // octets that stay together
  const int n_units = ly.N / (8 * kUnit);
  const int oc_lo = kUnit * (int)((long long)cl * n_units / ly.clusters), oc_hi = kUnit * (int)((long long)(cl + 1) * n_units / ly.clusters);
  const int n_oct = oc_hi - oc_lo, rounds = (n_oct + kWarps * kOcts - 1) / (kWarps * kOcts);
  // octets of warp w in round r: [first, first + count); all rounds but the last are full
  auto octets = [&](int r, int w, int& count) {
    const int left = min(n_oct - r * (kWarps * kOcts), kWarps * kOcts) / kUnit;
    const int a = w * left / kWarps, b = (w + 1) * left / kWarps;
    count = kUnit * (b - a);
    return oc_lo + r * (kWarps * kOcts) + kUnit * a;
  };
  const int s_lo = rank * ly.k_slabs / CS, s_hi = (rank + 1) * ly.k_slabs / CS, n_slabs = s_hi - s_lo;
  const int ksteps = (n_slabs + 1) / 2;                              // steps of two slabs (128 K)
  const uint32_t plane = (uint32_t)p.slabs_max * (128u * MT);
  const uint32_t sm = smem_u32(smem);
  const uint32_t bar0 = smem_u32(s_bars);
  const uint32_t t_full = bar0, t_seen = bar0 + 8;
  auto red_full = [&](int b) { return bar0 + 16 + 8u * b; };
  auto red_free = [&](int b) { return bar0 + 32 + 8u * b; };
  const int slots_w = kWarps / CS;                                   // warps of a CTA whose sums go to the same CTA
  // This cluster's share of T: rank blocks [rb_lo, rb_hi), i.e. NT tiles of 8 columns; where there are fewer tiles than warps,
  // WPN warps share one and split its blocks of K.
  const int rb_lo = min(cl * ly.t_blocks, ly.r_blocks), rb_hi = min(rb_lo + ly.t_blocks, ly.r_blocks);
  const int t_cols = 16 * (rb_hi - rb_lo), NT = t_cols / 8, WPN = NT == 0 || NT >= kWarps ? 1 : kWarps / NT;
  const int RP = kRows / CS;                                         // rows whose T a CTA owns
  const int own_rows = max(0, min(M - rank * RP, RP));
  const uint32_t rplane = (uint32_t)((k_pad + 127) / 128) * (256u * MT);   // a plane of T_q: rank slabs, an even number of them

  // bytes of round r that come to this CTA
  auto round_bytes = [&](int r) {
    int total = 0;
    for (int s = 0; s < slots_w; ++s) {
      int c;
      octets(r, rank + s * CS, c);
      total += c;
    }
    return (uint32_t)(total * 64 * ((M + 1) / 2) * CS);
  };
  if (tid == 0) {
    tc::mbar_init(t_full, 1);
    tc::mbar_init(t_seen, CS * kWarps);
    for (int i = 0; i < 2; ++i) { tc::mbar_init(red_full(i), 1); tc::mbar_init(red_free(i), CS * kWarps); }
    s_ws.abort = 0;
    s_ws.limit = p.wait_limit;
    tc::fence_barrier_init();
    if (NT > 0 && own_rows > 0) tc::mbar_expect_tx(t_full, (uint32_t)(own_rows * t_cols * 8 * CS * WPN));
    // (a round that brings nothing is not armed: its phase would pass before every warp has seen the one before)
    if (round_bytes(0) > 0) tc::mbar_expect_tx(red_full(0), round_bytes(0) + (p.stall ? 16u : 0u));
    if (rounds > 1 && round_bytes(1) > 0) tc::mbar_expect_tx(red_full(1), round_bytes(1));
  }
  tc::pdl_launch_dependents();
  cluster_arrive();

  // ---- weights: this lane's pieces of the steps to come, through its own slots of the ring
  const uint32_t ring = sm + p.off_ring + warp * (D * kStage);
  int pf_round = 0, pf_step = 0, pf_count = 0, pf_slot = 0;
  uint32_t pf_w[kOcts], pf_e[kOcts];
  auto pf_columns = [&]() {
    const int first = octets(pf_round, warp, pf_count);
#pragma unroll
    for (int o = 0; o < kOcts; ++o) {
      const int oc = first + o;
      const uint32_t tile = (uint32_t)(oc >> 4) * (uint32_t)ly.k_slabs * (uint32_t)kTile, nl = (uint32_t)((oc & 15) * 8 + g);
      pf_w[o] = tile + nl * 16u + (WB == 4 ? (uint32_t)(t & 1) * 2048u : (uint32_t)(t & 1) * 8u);
      pf_e[o] = tile + (uint32_t)kMant + nl * 4u;
    }
  };
  auto prefetch_step = [&]() {
    if (pf_round < rounds) {
      // the second slab of an odd last step: the lane takes the last one again, its activations are zeros there
      const uint32_t slab = (uint32_t)min(s_lo + 2 * pf_step + (t >> 1), s_hi - 1) * (uint32_t)kTile;
      const uint32_t dst = ring + pf_slot * kStage;
#pragma unroll
      for (int o = 0; o < kOcts; ++o)
        if (o < pf_count && LQER_IN_BOUNDS(p.status, pf_e[o] + slab, 4, ly.w_extent, 733)) {
          if (WB == 4) cp16(dst + (o * 32 + lane) * kPiece, ly.wsec + (pf_w[o] + slab));
          else cp8(dst + (o * 32 + lane) * kPiece, ly.wsec + (pf_w[o] + slab));
          cp4(dst + kOcts * 32 * kPiece + (o * 32 + lane) * 4, ly.wsec + (pf_e[o] + slab));
        }
      if (++pf_step == ksteps) {
        pf_step = 0;
        if (++pf_round < rounds) pf_columns();
      }
    }
    if (++pf_slot == D) pf_slot = 0;
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  pf_columns();
#pragma unroll 1
  for (int i = 0; i < D; ++i) prefetch_step();

  // ---- A_q of this CTA's blocks and this cluster's ranks: the first words into registers
  const int kblocks = K / 16, kb0 = s_lo * 4, nreal = min(n_slabs * 4, kblocks - kb0);
  const int nt_first = NT >= kWarps ? warp : NT > 0 ? warp % NT : 0, sub = NT >= kWarps || NT == 0 ? 0 : warp / NT;
  const bool t_active = NT > 0 && (NT >= kWarps || warp < NT * WPN);
  constexpr int UB = 16;
  uint32_t bw[UB], ew[UB];
  auto load_a = [&](int bq, int nt) {
    const uint8_t* am = ly.asec + ((size_t)(kb0 + bq) * k_pad + rb_lo * 16 + nt * 8 + g) * 16 + t * 4;
    const uint8_t* ae = ly.asec + (size_t)kblocks * k_pad * 16 + (size_t)(kb0 + bq) * k_pad + rb_lo * 16 + nt * 8 + t * 2;
#pragma unroll
    for (int u = 0; u < UB; ++u) {
      bw[u] = 0u; ew[u] = 0u;
      if (bq + u * WPN < nreal) {
        bw[u] = __ldg(reinterpret_cast<const uint32_t*>(am));
        ew[u] = (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(ae));
      }
      am += (size_t)WPN * k_pad * 16;
      ae += (size_t)WPN * k_pad;
    }
  };
  if (t_active) load_a(sub, nt_first);
  // B_q of the octets whose rank term falls to this CTA, towards L2
  if (k_pad > 0 && warp % CS == rank)
    for (int r = 0; r < rounds; ++r) {
      int c;
      const int first = octets(r, warp, c);
      for (int rb = lane >> 2; rb < ly.r_blocks; rb += 8)
        if ((lane & 3) < c) {
          const int oc = first + (lane & 3);
          const uint8_t* bt = ly.bsec + (size_t)(oc >> 4) * ly.r_blocks * kTileN * 17;
          asm volatile("prefetch.global.L2 [%0];" ::"l"(bt + ((size_t)rb * kTileN + (oc & 15) * 8) * 16));
          asm volatile("prefetch.global.L2 [%0];" ::"l"(bt + (size_t)ly.r_blocks * kTileN * 16 + rb * kTileN));
        }
    }
  // ---- zeros where no activation is written: rows beyond M, the second half of an odd last step, ranks beyond k_pad
  for (int o = tid * 16; o < (int)(8 * plane); o += kThreads * 16) *reinterpret_cast<uint4*>(smem + o) = make_uint4(0u, 0u, 0u, 0u);
  uint8_t* xq = smem + p.off_xq;
  int8_t* xe = reinterpret_cast<int8_t*>(smem + p.off_xe);
  const int xq_stride = p.slabs_max * 64 + 16, xe_stride = p.slabs_max * 4;
  cluster_wait();                                    // every CTA's barriers are set up
  __syncthreads();
  tc::pdl_wait();                                    // X and Y may be in use by the kernel before

  // ---- X -> MXINT8, a lane per 16-block: bf16 pairs for W_q, mantissas and exponents for A_q
  {
    const QuantConsts qc = quant_consts(p.a_bits, p.exp_min, p.exp_max);
    const int n_items = M * nreal;
    int row = tid / nreal, b = tid % nreal;
    const int row_step = kThreads / nreal, b_step = kThreads % nreal;
    auto next = [&](int& r, int& c) {
      r += row_step;
      c += b_step;
      if (c >= nreal) { c -= nreal; ++r; }
    };
    float v[2][16];
    if (tid < n_items) load_x_block(v[0], ly.X, p.x_type, M, K, row, kb0 + b, p.a_bits, p.exp_min, p.exp_max);
    for (int i = tid; i < n_items; i += 2 * kThreads) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (i + h * kThreads >= n_items) break;
        const int r = row, c = b;
        next(row, b);
        if (i + (h + 1) * kThreads < n_items) load_x_block(v[h ^ 1], ly.X, p.x_type, M, K, row, kb0 + b, p.a_bits, p.exp_min, p.exp_max);
        int e;
        uint4 m8, f0, f1;
        quantize_block16(v[h], qc, e, m8, f0, f1);
        if (NT > 0) {
          *reinterpret_cast<uint4*>(xq + r * xq_stride + c * 16) = m8;
          xe[r * xe_stride + c] = (int8_t)e;
        }
        uint8_t* dst = smem + token_offset<MT>(r, c >> 2, (c & 3) * 16) + ((c & 1) * 4) * plane;
        const uint32_t w[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (MT == 1) {
            *reinterpret_cast<uint2*>(dst + q * plane) = make_uint2(w[2 * q], w[2 * q + 1]);
          } else {
            *reinterpret_cast<uint32_t*>(dst + q * plane) = w[2 * q];
            *reinterpret_cast<uint32_t*>(dst + q * plane + 8) = w[2 * q + 1];
          }
        }
      }
    }
  }
  __syncthreads();

  // ---- T over this CTA's blocks, to the CTAs that own the rows
  if (t_active) {
    const int bias = -127 - (p.a_bits - 2) - (p.lr_bits - 2);        // exponent bytes carry +127
    // rows beyond M are read (whatever lies there) but never stored
    for (int nt = nt_first; nt < NT; nt += kWarps) {
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      for (int bq = sub; bq < nreal; bq += UB * WPN) {
        if (bq != sub || nt != nt_first) load_a(bq, nt);
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          const int b = bq + u * WPN;
          if (b < nreal) {
            const uint32_t a0 = *reinterpret_cast<const uint32_t*>(xq + g * xq_stride + b * 16 + t * 4);
            const uint32_t a1 = MT == 2 ? *reinterpret_cast<const uint32_t*>(xq + (g + 8) * xq_stride + b * 16 + t * 4) : 0u;
            int c[4];
            mma_s8(c, a0, a1, bw[u]);
            const int ea_lo = (int)(ew[u] & 0xFFu), ea_hi = (int)(ew[u] >> 8);
            const int ex0 = xe[g * xe_stride + b] + bias;
            acc[0] = fma(int_to_double(c[0]), pow2d(ex0 + ea_lo), acc[0]);
            acc[1] = fma(int_to_double(c[1]), pow2d(ex0 + ea_hi), acc[1]);
            if (MT == 2) {
              const int ex1 = xe[(g + 8) * xe_stride + b] + bias;
              acc[2] = fma(int_to_double(c[2]), pow2d(ex1 + ea_lo), acc[2]);
              acc[3] = fma(int_to_double(c[3]), pow2d(ex1 + ea_hi), acc[3]);
            }
          }
        }
      }
#pragma unroll
      for (int h = 0; h < MT; ++h) {
        const int row = g + 8 * h, owner = row / RP;
        if (row < M) {
          const uint32_t at = sm + p.off_tpart + (uint32_t)(((rank * WPN + sub) * RP + row % RP) * t_cols + nt * 8 + t * 2) * 8u;
          st_async(map_cta(at, owner), acc[2 * h], acc[2 * h + 1], map_cta(t_full, owner));
        }
      }
    }
  }
  // the rows this CTA owns: sum in CTA order, MXINT8 along the rank, out to scratch for all clusters of the layer
  auto reduce_t = [&]() -> bool {
    const int total = own_rows * t_cols;
    if (warp * 32 >= total) return true;
    if (!wait_cluster(t_full, 0, &s_ws)) return false;
    const double* tp = reinterpret_cast<const double*>(smem + p.off_tpart);
    int done = 0;                                    // 16-blocks
    for (int o = tid; o - lane < total; o += kThreads) {
      const bool live = o < total;
      done += min(32, total - (o - lane)) >> 4;
      double v = 0.0;
      if (live) {
#pragma unroll 8
        for (int c = 0; c < CS * WPN; ++c) v += tp[(size_t)c * RP * t_cols + o];
      }
      double amax = (v != v) ? 0.0 : fabs(v);
#pragma unroll
      for (int d = 1; d < 16; d <<= 1) amax = fmax(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, d));
      const int e = block_exponent(amax, p.exp_min, p.exp_max);
      const uint32_t bits = (uint32_t)bf16_bits_of(quant_mantissa(v, e, p.a_bits), e - (p.a_bits - 2)) & 0xFFFFu;
      const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, bits, 1);
      if (live && (lane & 1) == 0) {
        const int row = rank * RP + o / t_cols, j = rb_lo * 16 + o % t_cols;
        const uint32_t at = (uint32_t)((j & 31) >> 2) * rplane + token_offset<MT>(row, j >> 6, j & 63) + (uint32_t)((j & 2) * 2 * MT);
        if (LQER_IN_BOUNDS(p.status, at, 4, 8 * rplane, 734)) *reinterpret_cast<uint32_t*>(ly.tq + at) = bits | (next << 16);
      }
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) atomicAdd(ly.tcount, done);
    return true;
  };

  // ---- the rounds
  const ConvConsts kc = conv_consts<WB>();
  const uint32_t x_off = (uint32_t)((t >> 1) * (128 * MT) + (2 * g + (t & 1)) * (8 * MT));   // the lane's position within a step of a plane
  const int eb0 = 2 * (t & 1);
  bool ok = true;
  if (NT > 0) {
    ok = reduce_t();
    __syncwarp();
    if (rounds > 1 && lane < CS) arrive_remote(map_cta(t_seen, lane));
  }
  int slot = 0;
  auto reduce_round = [&](int r) -> bool {
    const int b = r & 1;
    if (round_bytes(r) == 0) return true;                      // nothing comes, as in a short last round
    if (!wait_cluster(red_full(b), (r >> 1) & 1, &s_ws)) return false;
    if (tid == 0 && r + 2 < rounds && round_bytes(r + 2) > 0) tc::mbar_expect_tx(red_full(b), round_bytes(r + 2));
    const float* buf = reinterpret_cast<const float*>(smem + p.off_red[b]);
    for (int s = 0; s < slots_w; ++s) {
      int c;
      const int first = octets(r, rank + s * CS, c);
      for (int i = tid; i - lane < M * 8; i += kThreads) {     // (row, quad of columns)
        const int row = i >> 3, quad = i & 7;
        const bool live = row < M && quad < 2 * c;
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        if (live)
          for (int q = 0; q < CS; ++q) {
            const float* src = buf + ((s * CS + q) * 32 + quad * 4) * TS + row;
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] += src[j * TS];
          }
        write_y4(p, ly, row, first * 8 + quad * 4, make_float4(v[0], v[1], v[2], v[3]), live);
      }
    }
    if (r + 2 < rounds) {
      __syncwarp();
      if (lane < CS) arrive_remote(map_cta(red_free(b), lane));
    }
    return true;
  };
#pragma unroll 1
  for (int r = 0; r < rounds; ++r) {
    int count;
    const int first = octets(r, warp, count);
    float acc[kOcts / 2][MT][4];
#pragma unroll
    for (int o = 0; o < kOcts / 2; ++o)
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[o][i][q] = 0.f;
#pragma unroll 1
    for (int j = 0; j < ksteps; ++j) {
      cp_wait<D - 1>();
      const uint8_t* st = smem + (ring - sm) + slot * kStage + lane * kPiece;
      const uint8_t* se = smem + (ring - sm) + slot * kStage + kOcts * 32 * kPiece + lane * 4;
      const uint8_t* x = smem + j * (256 * MT) + x_off;
      // eight weights of octet o: word m of the lane's four (2-bit mantissas: half a word)
      auto load_w = [&](uint4& w, uint32_t& e, int o) {
        if (WB == 4) {
          w = *reinterpret_cast<const uint4*>(st + o * 32 * kPiece);
        } else {
          const uint2 v = *reinterpret_cast<const uint2*>(st + o * 32 * kPiece);
          w = make_uint4(v.x, v.y, 0u, 0u);
        }
        e = *reinterpret_cast<const uint32_t*>(se + o * 128);
      };
      auto convert = [&](const uint4& w, uint32_t e, int m) -> uint4 {
        uint32_t s2, c2;
        if (WB == 4) {
          w_scale_pair(e, eb0 + (m >> 1), s2, c2);
          return convert_nibbles(m == 0 ? w.x : m == 1 ? w.y : m == 2 ? w.z : w.w, s2, c2, kc);
        } else {
          w_scale_pair2(e, eb0 + (m >> 1), s2, c2);
          return convert_crumbs(m < 2 ? w.x : w.y, m & 1, s2, c2, kc);
        }
      };
      if (count > 2) {
        uint4 w[4];
        uint32_t e[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) load_w(w[o], e[o], min(o, count - 1));
        multiply_step<MT, 2>(acc, x, plane, [&](int o, int m) { return convert(w[o], e[o], m); });
      } else if (count > 0) {
        uint4 w[2];
        uint32_t e[2];
#pragma unroll
        for (int o = 0; o < 2; ++o) load_w(w[o], e[o], min(o, count - 1));
        multiply_step<MT, 1>(acc, x, plane, [&](int o, int m) { return convert(w[o], e[o], m); });
      }
      prefetch_step();
      if (++slot == D) slot = 0;
    }
    // the rank term of warp w's octets is CTA w mod CS's
    if (k_pad > 0 && warp % CS == rank) {
      for (int j = 0; j * 128 < k_pad && ok; ++j) {
        uint4 w[4][2];
        float sc[4][2];
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const int oc = first + max(min(o, count - 1), 0), nl = (oc & 15) * 8 + g;
          const uint8_t* bt = ly.bsec + (size_t)(oc >> 4) * ly.r_blocks * kTileN * 17;
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int rb = 8 * j + 2 * t + u;
            const bool in = rb < ly.r_blocks;
            w[o][u] = in ? ld_stream16(bt + ((size_t)rb * kTileN + nl) * 16) : make_uint4(0u, 0u, 0u, 0u);
            sc[o][u] = in ? pow2f((int)bt[(size_t)ly.r_blocks * kTileN * 16 + rb * kTileN + nl] - 127 - (p.lr_bits - 2)) : 1.0f;
          }
        }
        if (r == 0 && j == 0) ok = wait_count(ly.tcount, ly.t_expect, &s_ws);
        multiply_step<MT, 2, true>(acc, ly.tq + j * (256 * MT) + x_off, rplane, [&](int o, int m) {
          const uint4& v = w[o][m >> 1];
          return tc::convert_i8x8(m & 1 ? v.z : v.x, m & 1 ? v.w : v.y, sc[o][m >> 1]);
        }, ly.r_blocks - (8 * j + 2 * t));
      }
      // the last of the layer's warps to have read T_q zeroes the counters for the next call
      if (r == rounds - 1 && lane == 0 && ok && atomicAdd(ly.tcount + 1, 1) == ly.clusters * kWarps - 1) {
        ly.tcount[0] = 0;
        ly.tcount[1] = 0;
      }
    }
    if (r > 0) ok = ok && reduce_round(r - 1);
    if (r == 1 && NT > 0) ok = ok && wait_cluster(t_seen, 0, &s_ws);   // the sums of the odd rounds lie where T was formed
    if (r > 1) ok = ok && wait_cluster(red_free(r & 1), ((r >> 1) - 1) & 1, &s_ws);
    if (!ok) break;
    {
      const uint32_t dst_cta = (uint32_t)(warp % CS);
      const uint32_t base = map_cta(sm + p.off_red[r & 1] + (uint32_t)(((warp / CS) * CS + rank) * 32 * TS * 4), dst_cta);
      const uint32_t bar = map_cta(red_full(r & 1), dst_cta);
#pragma unroll
      for (int o = 0; o < kOcts; ++o)
        if (o < count) {
#pragma unroll
          for (int i = 0; i < MT; ++i)
            if (8 * i + 2 * t < M)
              st_async(base + (uint32_t)(((o * 8 + g) * TS + 8 * i + 2 * t) * 4), acc[o >> 1][i][2 * (o & 1)], acc[o >> 1][i][2 * (o & 1) + 1], bar);
        }
    }
  }
  cluster_arrive();                                  // this warp's last store into another CTA lies behind it
  if (ok) ok = reduce_round(rounds - 1);
  cp_wait<0>();
  cluster_wait();                                    // no CTA leaves while another may still store into its shared memory
  if (tid == 0 && s_ws.abort != 0) report_error(p.status, LQER_ERR_TIMEOUT, 730, blockIdx.x);
}


// Clusters of CS CTAs that the device holds at a time, with one or two CTAs to an SM (0 if the query fails).
constexpr int kSmemTwo = 112 * 1024, kSmemOne = 220 * 1024;
static cudaLaunchConfig_t launch_config(int CS, int clusters, size_t smem, bool cooperative, cudaLaunchAttribute* attr, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * CS);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CS; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  attr[2].id = cudaLaunchAttributeCooperative;
  attr[2].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cooperative ? 3 : 2;
  return cfg;
}
template <int WB, int MT, bool YQ, int D>
static int resident_clusters(int CS, bool two) {
  static std::mutex mu;
  static int known[64][4][2] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lock(mu);
  int& n = known[dev][CS == 8 ? 3 : CS == 4 ? 2 : CS == 2 ? 1 : 0][two ? 1 : 0];
  if (n == 0) {
    cudaLaunchAttribute attr[3];
    const cudaLaunchConfig_t cfg = launch_config(CS, 1, two ? kSmemTwo : kSmemOne, false, attr, nullptr);
    if (cudaFuncSetAttribute(decode_cluster_kernel<WB, MT, YQ, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemOne) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, decode_cluster_kernel<WB, MT, YQ, D>, &cfg) != cudaSuccess)
      n = 0;
  }
  return n;
}
template <int WB, int MT, bool YQ, int D>
static cudaError_t launch(const Params& p, int clusters, int CS, size_t smem, bool cooperative, cudaStream_t s) {
  cudaLaunchAttribute attr[3];
  const cudaLaunchConfig_t cfg = launch_config(CS, clusters, smem, cooperative, attr, s);
  LaunchScope scope(kFamDecode, s);
  return cudaLaunchKernelEx(&cfg, decode_cluster_kernel<WB, MT, YQ, D>, p, CS);
}
// The instance of the kernel for a call.
template <int WB, int MT, bool YQ>
struct Instance {
  static int resident(int CS, bool two) { return two ? resident_clusters<WB, MT, YQ, 2>(CS, true) : resident_clusters<WB, MT, YQ, 4>(CS, false); }
  static cudaError_t go(const Params& p, int clusters, int CS, bool two, size_t smem, bool cooperative, cudaStream_t s) {
    return two ? launch<WB, MT, YQ, 2>(p, clusters, CS, smem, cooperative, s) : launch<WB, MT, YQ, 4>(p, clusters, CS, smem, cooperative, s);
  }
};
struct Entry {
  int (*resident)(int, bool);
  cudaError_t (*go)(const Params&, int, int, bool, size_t, bool, cudaStream_t);
};
template <int WB, int MT, bool YQ>
static Entry entry() { return Entry{Instance<WB, MT, YQ>::resident, Instance<WB, MT, YQ>::go}; }
static Entry entry_of(int wb, int mt, bool yq) {
  if (wb == 4) return mt == 1 ? (yq ? entry<4, 1, true>() : entry<4, 1, false>()) : (yq ? entry<4, 2, true>() : entry<4, 2, false>());
  return mt == 1 ? (yq ? entry<2, 1, true>() : entry<2, 1, false>()) : (yq ? entry<2, 2, true>() : entry<2, 2, false>());
}

}  // namespace dcl

// The cluster size and the shared memory of a launch over these layers, functions of the shapes alone.
namespace dcl {
struct Plan {
  int CS, slabs_max;
  int off_red[2], off_xq, off_xe, off_tpart, off_ring;
  bool two;                                 // two CTAs to an SM
  size_t smem;
};
static Plan plan(const PackedMeta* metas, int n, int M) {
  int k_slabs_min = metas[0].k_slabs, k_slabs_max = 0, r_blocks_max = 0;
  for (int i = 0; i < n; ++i) {
    k_slabs_min = std::min(k_slabs_min, (int)metas[i].k_slabs);
    k_slabs_max = std::max(k_slabs_max, (int)metas[i].k_slabs);
    r_blocks_max = std::max(r_blocks_max, (int)metas[i].r_blocks);
  }
  Plan q;
  q.CS = 8;
  while (q.CS > 1 && k_slabs_min < 2 * q.CS) q.CS >>= 1;             // at least one step of two slabs to a CTA
  const int MT = M > 8 ? 2 : 1;
  auto al = [](int v) { return (v + 127) / 128 * 128; };
  const int red = al(kWarps * 32 * token_stride(MT) * 4), stage = metas[0].w_bits == 4 ? stage_bytes<4>() : stage_bytes<2>();
  q.slabs_max = ((k_slabs_max + q.CS - 1) / q.CS + 1) / 2 * 2;
  int off = q.slabs_max * 1024 * MT;
  q.off_red[0] = off; off += red;
  // X_q for the projection and the partial sums of T share their room with the sums of the odd rounds
  q.off_red[1] = off;
  q.off_xq = off;
  q.off_xe = q.off_xq + al(8 * MT * (q.slabs_max * 64 + 16));
  q.off_tpart = q.off_xe + al(8 * MT * q.slabs_max * 4);
  q.off_ring = std::max(off + red, q.off_tpart + (r_blocks_max > 0 ? std::max(kWarps, 2 * r_blocks_max) * 1024 : 0));
  q.two = q.off_ring + kWarps * 2 * stage <= kSmemTwo;
  q.smem = (size_t)q.off_ring + (size_t)kWarps * (q.two ? 2 : 4) * stage;
  return q;
}
}  // namespace dcl

// Whether n layers with one M go out as one launch of this kernel (with Y of y_type): at 3 to 16 rows, up to four layers, and
// where it is the faster way.  Measured on one B200, us a call, what ran before / this kernel (rank 32 unless stated):
//   4096 x 4096 alone            4 rows 19.9 / 12.0    8 rows 20.9 / 12.4    16 rows 21.8 / 15.9
//   three of them                4 rows 28.8 / 21.0    8 rows 27.0 / 21.4    16 rows 27.4 / 27.1
//   two of 4096 x 11008          4 rows 38.7 / 30.5    8 rows 32.4 / 31.2    16 rows 32.9 / 38.9
//   two of 5120 x 13824, rank 64 4 rows 50.0 / 43.7    8 rows 45.7 / 44.6    16 rows 46.4 / 54.3
//   three of 2048 x 2048         4 rows 14.3 / 11.9    8 rows 20.0 / 12.3    16 rows 20.6 / 14.4
//   six of 4096 x 4096           4 rows 34.5 / 37.1    8 rows 35.2 / 37.8    16 rows 35.8 / 46.5
// Up to eight rows one MMA multiplies sixteen weight columns with all tokens; from nine on it takes two, and the tensor pipe is
// as busy as the conversion, so larger launches keep the kernels that share a prologue (11008 x 4096 alone, 16 rows: 29.9 / 32.4).
// Three rows with ranks above 128 are level or worse in large launches (a 4064 / 10192 layer at rank 256 122.8 / 134.9, 4096 / 11008 126.6 /
// 129.5; 2048 / 5632 87.3 / 62.3): the same line.
// One and two rows keep the column-owner kernel (2 rows: 4096 x 4096 16.4 / 15.6, two of 4096 x 11008 26.0 / 30.3).
constexpr long long kClusterMaxWeights = 30000000;        // K N over the layers, from nine rows on and at three with ranks above 128
int decode_cluster_max_layers() { return dcl::kMaxLayers; }
bool decode_cluster_takes(const PackedMeta* metas, int n, int M, int y_type) {
  using namespace dcl;
  if (n < 1 || n > kMaxLayers || M < 3 || M > kRows) return false;
  long long weights = 0;
  int k_pad = 0;
  for (int i = 0; i < n; ++i) {
    if (!w_offsets_fit(metas[i])) return false;
    weights += (long long)metas[i].K64 * metas[i].N;
    k_pad = std::max(k_pad, (int)metas[i].k_pad);
  }
  if ((M > 8 || (M == 3 && k_pad > 128)) && weights > kClusterMaxWeights) return false;
  const Plan q = plan(metas, n, M);
  if (q.smem > (size_t)kSmemOne) return false;
  return entry_of(metas[0].w_bits, M > 8 ? 2 : 1, y_type == kYMXINT8).resident(q.CS, q.two) >= n;
}

cudaError_t launch_decode_cluster(const lqer_call_t* calls, const PackedMeta* metas, int n, void* scratch, int* counts, DeviceStatus* st,
                                  int x_type, int y_type, cudaStream_t s) {
  using namespace dcl;
  if (n < 1 || n > kMaxLayers) return cudaErrorInvalidValue;
  const int M = calls[0].M;
  const Plan q = plan(metas, n, M);
  const int CS = q.CS;
  Params p;
  p.n = n; p.M = M; p.status = st; p.x_type = x_type; p.y_type = y_type;
  p.a_bits = metas[0].a_bits; p.lr_bits = metas[0].lr_bits; p.exp_min = metas[0].exp_min; p.exp_max = metas[0].exp_max;
  p.wait_limit = wait_limit_cycles();
  const bool stall = take_stall(kFamDecode);
  p.stall = stall ? 1 : 0;
  p.slabs_max = q.slabs_max;
  p.off_red[0] = q.off_red[0]; p.off_red[1] = q.off_red[1];
  p.off_xq = q.off_xq; p.off_xe = q.off_xe; p.off_tpart = q.off_tpart; p.off_ring = q.off_ring;
  const bool yq = y_type == kYMXINT8;
  const Entry kernel = entry_of(metas[0].w_bits, M > 8 ? 2 : 1, yq);
  // No more clusters than the device holds at a time (they wait for the T_q of others).  With two CTAs to an SM the last few
  // places are left free: 4096 x 4096, 4 rows, 14.3 us with 32 of 33 clusters and 12.0 with 28; larger launches lose more by the
  // longer ranges of columns (two of 4096 x 11008: 35.5 with 28, 30.5 with 32, 34 with 33).
  int budget = kernel.resident(CS, q.two);
  // The clusters that form a layer's T wait for one another, and all others of the layer, placed after them, wait for these.  A launch
  // that runs beside others may get its places one by one, and until all of a layer's T clusters have theirs the ones that do
  // cannot leave.  At most a quarter of the places go to such clusters, so that four launches on as many streams cannot hold
  // each other up for good; where that would cost too much (one CTA to an SM: 13824 x 2048 of rank 256, 4 rows, 40.6 us instead of 21.8)
  // the launch is a cooperative one, which is placed as a whole or not yet (some 1 us more).  With two CTAs to an SM the
  // quarter costs nothing (rank 256, 4 rows: 4096 x 4096 14.4 / 14.3, 2048 x 5632 14.0 / 13.5; up to rank 128 nothing changes).
  const int most = std::max(budget / 4, 1);
  bool cooperative = false;
  constexpr long long kFewWeights = 30000000;
  long long weights = 0;
  for (int i = 0; i < n; ++i) weights += (long long)metas[i].K64 * metas[i].N;
  if (q.two && budget >= 8) budget = weights <= kFewWeights ? budget * 7 / 8 : budget / 4 * 4;
  if (budget < n) return cudaErrorInvalidConfiguration;
  // clusters per layer: each has one, the others go one by one where the time (column octets x steps of K) is longest, as long
  // as every warp of a cluster has an octet
  int clusters[kMaxLayers];
  double per_oct[kMaxLayers];
  int total = 0;
  for (int i = 0; i < n; ++i) {
    clusters[i] = 1;
    per_oct[i] = 0.5 * ((metas[i].k_slabs + CS - 1) / CS) + 1.0;
    ++total;
  }
  while (total < budget) {
    int best = -1;
    double worst = 0.0;
    for (int i = 0; i < n; ++i) {
      const double t = (double)(metas[i].N / 8) / clusters[i] * per_oct[i];
      if (clusters[i] < metas[i].N / (yq ? 16 : 8) / kWarps && t > worst) { worst = t; best = i; }
    }
    if (best < 0) break;
    ++clusters[best];
    ++total;
  }
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
    ly.K = m.K; ly.N = m.N; ly.k_pad = m.k_pad; ly.k_slabs = m.k_slabs; ly.r_blocks = m.r_blocks;
    ly.cluster_begin = begin;
    ly.clusters = clusters[g];
    ly.tq = static_cast<uint8_t*>(scratch) + t_off;
    ly.tcount = counts + 2 * g;
    // the warps of an owner count their 16-blocks of T in
    ly.t_expect = M * m.r_blocks + (stall ? 1 : 0);
    const int formers = q.two ? std::min(clusters[g], most) : clusters[g];
    ly.t_blocks = (m.r_blocks + formers - 1) / formers;
    if (i < n && std::min(formers, (int)m.r_blocks) > most) cooperative = true;
    if (i < n) t_off += decode_cluster_scratch_bytes(m);
    if (i < n) begin += clusters[g];
  }
  return kernel.go(p, total, CS, q.two, q.smem, cooperative, s);
}

}  // namespace lqer
