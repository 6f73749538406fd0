// Small-batch form of the layer's contraction (paper Section 3.1 / 3.2: Y = [X_q | T_q] . [W_q ; B_q];
// Section 2.1: few tokens per step make the layer memory bound on its weights).
//
// The weights are the MMA's 128-row operand and the tokens its narrow one:
//     D[128 weight columns, N tokens] += Wtile[128, 16 K] . Xtile[N, 16 K]^T        (tcgen05.mma, bf16 -> fp32)
// and the weight operand comes from TENSOR MEMORY: a converter thread owns a weight column, turns its packed mantissas
// into their exact bf16 values in registers and stores them to its lane (tcgen05.st), so the converted weights never
// touch shared memory.  An MMA of K = 16 then takes 17 cycles at N = 16, 19 at 32, 32 at 64, 64 at 128 (measured; with
// the operand in shared memory 39 at N = 16, and 128 with the tokens on the 64- or 128-row side against 256 weight
// columns).  A CTA streams packed weight tiles exactly once into a ring of some 200 KB, in batches of four slabs of 64 K:
// one bulk copy for each 128-column half of the tile and a TMA load for each of the four [N, 64] activation tiles (every
// copy costs its issuing thread and the copy engine a hundred cycles and more, so a slab of weights at a time held the ring
// back).
// What bounds it is the stream of weights and, close behind, the instructions that expand them (1.8 per weight).
//
// Work items are (layer, 256-column tile, K chunk).  A layer alone is cut into chunks by its shape, layers that share a launch by
// the shapes of all of them (launch_gemm_small), so a result does not depend on the number of SMs, but its last bits may on the layers
// beside it.  Each chunk is summed from zero in tensor memory and, if a tile has more than one, leaves its fp32 partial in scratch;
// the CTAs whose last chunk is of one tile add its chunks up together, in chunk order, a share of the rows each (finish_tile), and
// none depends on another's help; or a CTA takes several or all chunks of a tile, one after the other (RUN).
// Roles per CTA:
//   warp 0      producer: bulk copies of packed weight tiles (issued before the dependency wait: weights
//               depend on no earlier kernel) and TMA loads of activation tiles (after it)
//   warp 1      tensor memory allocation, MMA issue (the whole warp runs the loop, one elected lane issues)
//   warps 2-5   epilogue (tcgen05.ld, Y or partial sums)
//   warps 6-29  converters in three groups of 256 threads (a weight column each); group g converts the steps
//               with index = g (mod 3)
// Two rings: PK slots hold a batch {four activation tiles, two halves of four packed weight tiles}, with a barrier for the
// weights and one for the activations (the converters need only the former, so they work while the prologue still runs);
// CV slots (tensor memory) hold a step's converted weights: two slabs, one where 128 tokens leave no room.  A step costs the
// MMA warp some 450 cycles beside the MMAs themselves (waits, the commit, the loop): with a slab to a step that was more
// than the eight MMAs of 32 cycles.
#include <algorithm>
#include <type_traits>

#include "lqer_gemm_small.cuh"
#include "lqer_tc_ptx.cuh"

namespace lqer {
namespace sg {
using namespace tc;

constexpr int BK = 64;
constexpr int BATCH = 4;                   // slabs of 64 K (or of 64 ranks) per PK slot
constexpr int CV_COLS = 64;                // tensor memory columns of a converted slab: 32 for each 128-column half
constexpr int W_HALF_BYTES = BATCH * kWTileBytes;
constexpr int CONVERTER_GROUPS = 3;
constexpr int WARPS_PER_GROUP = 8;
constexpr int NUM_THREADS = (6 + CONVERTER_GROUPS * WARPS_PER_GROUP) * 32;
// A PK slot is free once the MMAs that read its activations have finished AND every converter warp is past it.  A group may own
// no step of a batch, but it looks at every batch's barrier by parity, so it must not be a pass ahead of it (it waits for
// each one) nor a pass behind: without its arrival here the slot could be filled again before the group has looked.
constexpr int PK_FREE_ARRIVALS = 1 + CONVERTER_GROUPS * WARPS_PER_GROUP;

__device__ __forceinline__ void epilogue_barrier() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// NT: the most tokens of the class (32, 64, 128); a launch multiplies N = M rounded up to 16 of them.
template <int NT>
struct Cfg {
  static constexpr int X_BYTES = BATCH * NT * 128;
  static constexpr int PK_SLOT_BYTES = X_BYTES + 2 * W_HALF_BYTES;
  static constexpr int PK_SLOTS = NT == 32 ? 4 : NT == 64 ? 3 : 2;
  static constexpr int ACCS = NT == 32 ? 2 : 1;      // accumulators of two halves x NT columns
  static constexpr int CV_COL0 = ACCS * 2 * NT;      // the converted weights behind them
  static constexpr int STEP = NT == 128 ? 1 : 2;     // slabs of a CV slot: what the MMA warp waits for, issues and commits at once
  static constexpr int CV_SLOTS = CONVERTER_GROUPS;  // one for each group
  static constexpr int OFF_BARS = PK_SLOTS * PK_SLOT_BYTES;
  static constexpr int NUM_BARS = 3 * PK_SLOTS + 2 * CV_SLOTS + 4;
  static constexpr int SMEM_BYTES = OFF_BARS + NUM_BARS * 8 + 64 + 1024;
  static constexpr int TMEM_COLS = 512;
  static_assert(CV_COL0 + CV_SLOTS * STEP * CV_COLS <= TMEM_COLS, "tensor memory budget");
  static_assert(BATCH % STEP == 0, "a step lies in one batch");
  static_assert(PK_SLOT_BYTES % 1024 == 0, "swizzled activation tiles");
  static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");
};

// The X descriptor comes in halves: only its low word (the address) changes from MMA to MMA.
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 b;\n setp.ne.b32 p, %5, 0;\n mov.b64 b, {%2, %3};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %4, p;\n}\n"
      ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint4& a, const uint4& b, const uint4& c, const uint4& d) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w), "r"(c.x), "r"(c.y), "r"(c.z),
        "r"(c.w), "r"(d.x), "r"(d.y), "r"(d.z), "r"(d.w) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

struct TensorMaps {
  CUtensorMap m[MAX_LAYERS];   // Xcat of each layer, bf16 [M, K64 + k_pad], box x_rows x 64
};

// A tile's counter: chunks that have arrived, shares of the rows that have been taken, CTAs that have left; and whether one of them
// took a share and left before all chunks had arrived.
constexpr int kTaken = 1 << 8, kLeft = 1 << 20, kGaveUp = (int)0x80000000u;
__device__ __forceinline__ int arrived(int v) { return v & 0xFF; }
__device__ __forceinline__ int taken(int v) { return (v >> 8) & 0xFFF; }
__device__ __forceinline__ int left(int v) { return (v >> 20) & 0x7FF; }
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Rows [lo, hi) of a tile from its chunks' partial sums, by `nthreads` threads (a multiple of 64): four columns to a thread.
__device__ __forceinline__ void finish_rows(const Params& p, const Layer& ly, const Item& c, int lo, int hi, int tid, int nthreads) {
  const int col0 = c.tile * BN, c4 = (tid & 63) * 4, step = nthreads >> 6;
  const bool quad_ok = col0 + c4 < ly.N;                                   // N is a multiple of 8: the quad is whole
  const size_t chunk_stride = (size_t)p.M * BN;
  const float* p0 = ly.partials + (size_t)c.tile * ly.chunks * chunk_stride + c4;
  for (int t0 = lo + (tid >> 6); t0 < hi; t0 += 2 * step) {
    float4 v[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
    for (int cb = 0; cb < ly.chunks; cb += 4) {
      float4 t[2][4];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (cb + k < ly.chunks && t0 + u * step < hi)
            t[u][k] = __ldcg(reinterpret_cast<const float4*>(p0 + (size_t)(cb + k) * chunk_stride + (size_t)(t0 + u * step) * BN));
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (cb + k < ly.chunks && t0 + u * step < hi) { v[u].x += t[u][k].x; v[u].y += t[u][k].y; v[u].z += t[u][k].z; v[u].w += t[u][k].w; }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (t0 + u * step < hi) store_row_quad(p, ly, t0 + u * step, col0, c4, quad_ok, v[u]);
  }
}
// Adds a tile's chunks up, by all threads of a CTA or by its epilogue.  A CTA takes a share of the rows as its last chunk arrives and
// waits for the other chunks, but not for long: if it does so in vain, it says so and leaves.  The CTA whose chunk arrives last
// knows by that which shares are taken and does the others, or all of the rows if one has left (what others do of them at the
// same time is the same).  So none depends on another's progress.  The last one to leave puts the counter back to zero.
// With the CTA of the last chunk alone, the sums of 64 rows and 7 chunks took 9 us, 4 now; 4096 x 4096, 20 / 64 / 128 tokens, the call
// 22.3 / 29.2 / 40.8 us alone and 20.1 / 25 / 29.5 shared, 11008 x 4096 30.5 / 39.1 / 57.9 and 27.9 / 34 / 44.4.
constexpr int kFinishWait = 40000;             // cycles (not the launch's wait limit: giving up is no error)
// old: the counter before this CTA's chunk arrived.
template <bool WHOLE_CTA, int RUN>
__device__ __forceinline__ void finish_tile(const Params& p, const Item& c, int old, int tid, int* flag) {
  const Layer& ly = p.L[c.layer];
  int lo = 0, hi = p.M;
  if (RUN != kAllChunks) {                     // (otherwise all of the chunks were this CTA's)
    int* count = ly.counters + c.tile;
    // shares of some 96 rows of partial sums; where that makes one of them, the CTA of the last chunk is through sooner than the first's
    const int shares = min((p.M * ly.chunks + 95) / 96, RUN == kSomeChunks ? p.takers : ly.chunks);
    const int rows = (p.M + shares - 1) / shares, share = shares > 1 ? taken(old) : ly.chunks;
    const bool last = arrived(old) == ly.chunks - 1;
    bool ok = true;
    if (WHOLE_CTA && !last && share < shares) {  // (an epilogue comes here with the last chunk only)
      if (tid == 0) {
        int v = ld_acquire(count);
        for (const long long t0 = clock64(); arrived(v) != ly.chunks && clock64() - t0 < kFinishWait;) v = ld_acquire(count);
        if (arrived(v) != ly.chunks) {
          v = atomicOr(count, kGaveUp);
          __threadfence();
        }
        *flag = arrived(v) == ly.chunks ? 1 : 0;
      }
      __syncthreads();
      ok = *flag != 0;
    }
    if (tid == 0 && left(atomicAdd(count, kLeft)) + 1 == ly.chunks) *count = 0;
    if (!last || (old >= 0 && shares > 1)) lo = share * rows;
    if (!last) hi = ok ? min(p.M, (share + 1) * rows) : lo;
  }
  __threadfence();
  finish_rows(p, ly, c, lo, hi, tid, WHOLE_CTA ? NUM_THREADS : 128);
}
template <int RUN>
__device__ __noinline__ void finish_by_epilogue(const Params& p, const Item c, int old, int tid) { finish_tile<false, RUN>(p, c, old, tid, nullptr); }

// bf16_rn by the conversion instruction, which has one NaN for all.
__device__ __forceinline__ uint16_t bf16_rn_cvt(uint32_t v) {
  uint16_t h;
  asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(h) : "f"(__uint_as_float(v)));
  return (v & 0x7FFFFFFFu) > 0x7F800000u ? (uint16_t)((v >> 16) | 0x40u) : h;
}
// A finished chunk from its accumulator to Y or to the partial sums, by the epilogue's warps: warp q of them has a quarter of the
// lanes; a lane holds a weight column, its columns are the tokens.  Each warp is alone on its scheduler by then and bound by its own
// instructions, so bf16 is the conversion's (7 us for 64 tokens with bf16_rn, 4 now), and a partial sum's address is a constant away
// from the one before.  (All 28 warps at the end took no less time.  The kernel spills 64 - 76 bytes a thread, mostly around the call of
// finish_by_epilogue; every further live value costs 1 - 2 us.)
template <int NT>
__device__ __forceinline__ void store_chunk(const Params& p, const Item& c, uint32_t tmem_base, int acc, int q) {
  const Layer& ly = p.L[c.layer];
  const int lane = threadIdx.x & 31, M = p.M, Nl = ly.N, y_type = p.y_type;
  const int halves = c.tile * BN + 128 < Nl ? 2 : 1;
  const uint32_t t_base = tmem_base + ((uint32_t)(q * 32) << 16) + acc * 2 * NT;
  if (ly.chunks > 1) {
    float* dst0 = ly.partials + (size_t)(c.tile * ly.chunks + c.chunk) * M * BN + q * 32 + lane;
#pragma unroll 1
    for (int h = 0; h < halves; ++h) {
      float* dst = dst0 + h * 128;
#pragma unroll 1
      for (int t0 = 0; t0 < M; t0 += 16, dst += 16 * BN) {
        uint32_t r[16];
        tmem_ld16(t_base + h * NT + t0, r);
        tmem_ld_wait();
        if (kDebugBounds && !LQER_IN_BOUNDS(p.status, (size_t)(dst - ly.partials) * 4, ((size_t)(min(16, M - t0) - 1) * BN + 1) * 4, ly.partial_extent, 704)) continue;
        if (t0 + 16 <= M) {
#pragma unroll
          for (int t = 0; t < 16; ++t) dst[t * BN] = __uint_as_float(r[t]);
        } else {
#pragma unroll
          for (int t = 0; t < 16; ++t)
            if (t0 + t < M) dst[t * BN] = __uint_as_float(r[t]);
        }
      }
    }
    return;
  }
  [[maybe_unused]] const uint8_t* base = static_cast<const uint8_t*>(ly.Y);
  [[maybe_unused]] const size_t extent = ly.y_extent;
  const int size = y_type == kYBF16 ? 2 : y_type == kYMXINT8 ? 1 : 4;
  const size_t step = (size_t)Nl * size, step_e = (size_t)Nl / 16;
#pragma unroll 1
  for (int h = 0; h < halves; ++h) {
    const int col = c.tile * BN + h * 128 + q * 32 + lane;
    uint8_t* dst = static_cast<uint8_t*>(ly.Y) + (size_t)col * size;
    uint8_t* dst_e = static_cast<uint8_t*>(ly.Y) + (size_t)M * Nl + col / 16;            // MXINT8: the exponent bytes
#pragma unroll 1
    for (int t0 = 0; t0 < M; t0 += 16) {
      uint32_t r[16];
      tmem_ld16(t_base + h * NT + t0, r);
      tmem_ld_wait();
      const int rows = M - t0;
      if (y_type == kYMXINT8) {
        // sixteen lanes hold a 16-block of a token's row (N is a multiple of 16 here)
#pragma unroll
        for (int t = 0; t < 16; ++t, dst += step, dst_e += step_e) {
          const float v = __uint_as_float(r[t]);
          float amax = fmaxf(fabsf(v), 0.0f);            // (a NaN counts as zero)
#pragma unroll
          for (int d = 1; d < 16; d <<= 1) amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, d));
          const int e = block_exponent(amax, p.exp_min, p.exp_max);
          if (t < rows && col < Nl && LQER_IN_BOUNDS(p.status, dst_e - base, 1, extent, 703)) {
            *dst = (uint8_t)quant_mantissa(v, e, p.a_bits);
            if ((lane & 15) == 0) *dst_e = (uint8_t)(e + 127);
          }
        }
      } else if (col < Nl) {
        if (size == 2) {
#pragma unroll
          for (int t = 0; t < 16; ++t, dst += step)
            if (t < rows && LQER_IN_BOUNDS(p.status, dst - base, 2, extent, 701)) *reinterpret_cast<uint16_t*>(dst) = bf16_rn_cvt(r[t]);
        } else {
#pragma unroll
          for (int t = 0; t < 16; ++t, dst += step)
            if (t < rows && LQER_IN_BOUNDS(p.status, dst - base, 4, extent, 704)) *reinterpret_cast<uint32_t*>(dst) = r[t];
        }
      }
      __syncwarp();
    }
  }
}

// The batch that starts with slab s: up to BATCH slabs of weights, or two slabs of B_q (8-bit mantissas: eight blocks of 16
// ranks, 16 KB, then their exponent bytes).
__device__ __forceinline__ int batch_end(int s, int s_hi, int k_slabs) {
  return s < k_slabs ? min(s + BATCH, min(s_hi, k_slabs)) : min(s + 2, s_hi);
}
constexpr int RANK_EXP_OFFSET = 8 * kTileN * 16;
static_assert(RANK_EXP_OFFSET + 8 * kTileN <= W_HALF_BYTES, "two rank slabs");
template <int NT, int RUN>
__global__ void __launch_bounds__(NUM_THREADS, 1)
gemm_small_kernel(const __grid_constant__ TensorMaps tmaps, const __grid_constant__ Params p) {
  using C = Cfg<NT>;
  constexpr int PK_SLOTS = C::PK_SLOTS, CV_SLOTS = C::CV_SLOTS, STEP = C::STEP;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* pk_base = smem;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OFF_BARS);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + C::NUM_BARS);
  int* last_flag = reinterpret_cast<int*>(tmem_slot + 1);
  int* at_end = reinterpret_cast<int*>(tmem_slot + 6);         // item whose chunks the whole CTA helps to add up at the end, or -1; its counter's old value
  volatile WaitState* abort_flag = reinterpret_cast<volatile WaitState*>(tmem_slot + 2);

  const uint32_t bar0 = smem_u32(bars);
  auto w_full = [&](int s) { return bar0 + 8u * s; };                       // packed weights of a PK slot have landed
  auto x_full = [&](int s) { return bar0 + 8u * (PK_SLOTS + s); };          // its activation tiles have landed
  auto pk_free = [&](int s) { return bar0 + 8u * (2 * PK_SLOTS + s); };
  auto cv_ready = [&](int s) { return bar0 + 8u * (3 * PK_SLOTS + s); };
  auto cv_free = [&](int s) { return bar0 + 8u * (3 * PK_SLOTS + CV_SLOTS + s); };
  auto acc_full = [&](int a) { return bar0 + 8u * (3 * PK_SLOTS + 2 * CV_SLOTS + a); };
  auto acc_empty = [&](int a) { return bar0 + 8u * (3 * PK_SLOTS + 2 * CV_SLOTS + 2 + a); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = blockIdx.x, num_ctas = gridDim.x;
  const int num_items = p.num_items;

  if (threadIdx.x == 0) {
    for (int s = 0; s < PK_SLOTS; ++s) { mbar_init(w_full(s), 1); mbar_init(x_full(s), 1); mbar_init(pk_free(s), PK_FREE_ARRIVALS); }
    for (int s = 0; s < CV_SLOTS; ++s) { mbar_init(cv_ready(s), WARPS_PER_GROUP); mbar_init(cv_free(s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(acc_full(a), 1); mbar_init(acc_empty(a), 4); }
    abort_flag->abort = 0;
    abort_flag->limit = p.wait_limit;
    at_end[0] = -1;
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_launch_dependents();               // the next kernel may set up (it waits for this one before it touches memory)

  if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      // Packed weights depend on no earlier kernel: the first PK_SLOTS batches are requested at once, and only
      // then does the producer wait for the kernel before (the prologue that writes Xcat) and request the
      // activation tiles of those batches.  They land on a barrier of their own (x_full, used once per slot); later
      // ones share the weights' barrier, so that the MMA warp has one barrier to watch.
      const uint32_t x_tile = (uint32_t)p.x_rows * 128u;       // bytes of a slab's activations (rows beyond M arrive as zeros)
      auto load_x = [&](const CUtensorMap* map, int s, int e, uint32_t slot, uint32_t bar) {
        for (; s < e; ++s, slot += x_tile) tma_load_2d(slot, map, s * BK, 0, bar);
      };
      int npend = 0;                                           // batches requested without their activations: the first ones
      bool waited = false;
      auto flush = [&]() {
        pdl_wait();
        waited = true;
        for (int i = first_item<RUN>(p, cta), q = 0; q < npend; i = next_item<RUN>(p, i, num_ctas)) {
          const Item it = item_of<RUN>(p, i);
          const int k_slabs = p.L[it.layer].k_slabs;
          for (int s = it.s_lo; s < it.s_hi && q < npend; ++q) {
            const int e = batch_end(s, it.s_hi, k_slabs);
            mbar_expect_tx(x_full(q), (e - s) * x_tile);
            load_x(&tmaps.m[it.layer], s, e, smem_u32(pk_base + q * C::PK_SLOT_BYTES), x_full(q));
            s = e;
          }
        }
      };
      int pk = 0;
      uint32_t ph = 0;
      bool ok = true;
      const uint32_t w_tile = (uint32_t)w_tile_bytes(p.w_bits);
      for (int i = first_item<RUN>(p, cta); i < num_items && ok; i = next_item<RUN>(p, i, num_ctas)) {
        const Item it = item_of<RUN>(p, i);
        const Layer& ly = p.L[it.layer];
        const int k_slabs = ly.k_slabs, r_blocks = ly.r_blocks, b_tile_stride = r_blocks * kTileN * 17;
        const int nt0 = 2 * it.tile;
        const int n_half = nt0 + 1 < ly.n_tiles ? 2 : 1;       // 128-column tiles of this 256-column tile that exist
        for (int s = it.s_lo; s < it.s_hi;) {
          const int e = batch_end(s, it.s_hi, k_slabs);
          if (p.stall != 0 && e == it.s_hi && next_item<RUN>(p, i, num_ctas) >= num_items) { ok = false; break; }
          if (!waited && npend == PK_SLOTS) flush();
          if (!mbar_wait<true>(pk_free(pk), ph ^ 1, abort_flag)) { ok = false; break; }
          const uint32_t slot = smem_u32(pk_base + pk * C::PK_SLOT_BYTES), dst = slot + C::X_BYTES;
          const uint32_t bar = w_full(pk), x_bytes = waited ? (uint32_t)(e - s) * x_tile : 0u;
          if (s < k_slabs) {
            const size_t off = ((size_t)nt0 * k_slabs + s) * w_tile, half = (size_t)k_slabs * w_tile;
            const uint32_t bytes = (uint32_t)(e - s) * w_tile;
            if (!LQER_IN_BOUNDS(p.status, off + (n_half - 1) * half, bytes, ly.w_extent, 705)) { ok = false; break; }
            mbar_expect_tx(bar, n_half * bytes + x_bytes);
            bulk_load(dst, ly.wsec + off, bytes, bar);
            if (n_half > 1) bulk_load(dst + W_HALF_BYTES, ly.wsec + off + half, bytes, bar);
          } else {
            const int rb0 = (s - k_slabs) * 4, nb = min((e - s) * 4, r_blocks - rb0);
            if (!LQER_IN_BOUNDS(p.status, (size_t)(nt0 + n_half - 1) * b_tile_stride + (size_t)r_blocks * kTileN * 16 + rb0 * kTileN,
                                nb * kTileN, ly.b_extent, 706)) { ok = false; break; }
            mbar_expect_tx(bar, n_half * nb * (kTileN * 17) + x_bytes);
            for (int h = 0; h < n_half; ++h) {
              const uint8_t* tile = ly.bsec + (size_t)(nt0 + h) * b_tile_stride;
              bulk_load(dst + h * W_HALF_BYTES, tile + (size_t)rb0 * kTileN * 16, nb * kTileN * 16, bar);
              bulk_load(dst + h * W_HALF_BYTES + RANK_EXP_OFFSET, tile + (size_t)r_blocks * kTileN * 16 + rb0 * kTileN, nb * kTileN, bar);
            }
          }
          if (waited) load_x(&tmaps.m[it.layer], s, e, slot, bar);
          else ++npend;
          if (++pk == PK_SLOTS) { pk = 0; ph ^= 1; }
          s = e;
        }
      }
      if (!waited) flush();
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issue
    // The tensor pipe queues very few MMAs, so what the issuing warp spends between two of them beyond the pipe's
    // own time is idle time of the pipe: the whole warp runs the loop (barrier addresses and descriptors are
    // warp-uniform values) and one elected lane issues.
    const uint32_t idesc = make_idesc(128, (p.M + 15) / 16 * 16);
    // This warp shares its scheduler with six converter warps and gets every sixth or seventh issue slot, so its loop is
    // kept short: counters instead of divisions, 32-bit descriptor arithmetic, and tensor memory addresses from the
    // constant 0 (an allocation of all 512 columns begins there) that the compiler can keep in uniform registers.
    const uint32_t x_tile = (uint32_t)p.x_rows * (128u >> 4);           // in descriptor units of 16 bytes
    const uint64_t desc0 = make_desc(smem_u32(pk_base));
    const uint32_t b_hi = (uint32_t)(desc0 >> 32), b_lo0 = (uint32_t)desc0;
    uint32_t cv = 0, cv_ph = 0, pk = 0, acc = 0, acc_ph = 1;
    bool first_pass = true, ok = true;
    for (int i = first_item<RUN>(p, cta); i < num_items && ok; i = next_item<RUN>(p, i, num_ctas)) {
      const Item it = item_of<RUN>(p, i);
      const int k_slabs = p.L[it.layer].k_slabs, r_blocks = p.L[it.layer].r_blocks;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(acc_empty(acc), acc_ph, abort_flag)) != 0;
      if (!ok) break;
      tc_fence_after();
      const uint32_t d_tmem = acc * 2 * NT;
      uint32_t add = 0u;
      for (int s = it.s_lo; s < it.s_hi && ok;) {
        const int e = batch_end(s, it.s_hi, k_slabs);
        // a converted slab implies its batch had landed, and with it (from the second pass over the ring on) the
        // activation tiles; on the first pass the activation tiles have their own barrier
        if (first_pass) {
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(x_full(pk), 0, abort_flag)) != 0;
          if (!ok) break;
        }
        uint32_t b_lo = b_lo0 + pk * (C::PK_SLOT_BYTES >> 4);
        const int whole_end = s < k_slabs ? e : s;                       // steps up to here are whole slabs of weights
        for (; s < e; s += STEP) {
          const uint32_t w = C::CV_COL0 + cv * (STEP * CV_COLS);
          const uint32_t free_bar = cv_free(cv);
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(cv_ready(cv), cv_ph, abort_flag)) != 0;
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            // 16 K = 8 tensor memory columns; +2 in the address field = 32 bytes.  (Unrolled with constant offsets: a loop over
            // the K steps and the halves issued one MMA per 130 cycles.)
            if (s + STEP <= whole_end) {
              umma_bf16_ts(d_tmem, w, b_lo, b_hi, idesc, add);
              umma_bf16_ts(d_tmem + NT, w + 32, b_lo, b_hi, idesc, add);
#pragma unroll
              for (int j = 1; j < 4 * STEP; ++j) {
                const uint32_t x = b_lo + (j >= 4 ? x_tile : 0u) + 2 * (j & 3);
                umma_bf16_ts(d_tmem, w + (j >> 2) * CV_COLS + (j & 3) * 8, x, b_hi, idesc, 1u);
                umma_bf16_ts(d_tmem + NT, w + (j >> 2) * CV_COLS + (j & 3) * 8 + 32, x, b_hi, idesc, 1u);
              }
            } else {
              for (int t = 0; t < STEP && s + t < e; ++t) {
                const int nk = s + t < k_slabs ? 4 : min(4, r_blocks - (s + t - k_slabs) * 4);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                  if (j < nk) {
                    const uint32_t on = t + j > 0 ? 1u : add, x = b_lo + t * x_tile + 2 * j;
                    umma_bf16_ts(d_tmem, w + t * CV_COLS + j * 8, x, b_hi, idesc, on);
                    umma_bf16_ts(d_tmem + NT, w + t * CV_COLS + j * 8 + 32, x, b_hi, idesc, on);
                  }
              }
            }
            umma_commit(free_bar);
            if (s + STEP >= e) umma_commit(pk_free(pk));
          }
          __syncwarp();
          add = 1u;
          b_lo += STEP * x_tile;
          if (++cv == CV_SLOTS) { cv = 0; cv_ph ^= 1; }
        }
        s = e;
        if (++pk == PK_SLOTS) { pk = 0; first_pass = false; }
      }
      if (ok && elect_one()) umma_commit(acc_full(acc));
      __syncwarp();
      if (++acc == C::ACCS) { acc = 0; acc_ph ^= 1; }
    }
  } else if (warp < 6) {
    // ------------------------------------------------------------------ epilogue
    // A lane of tensor memory holds a weight column, its columns the tokens: a token's 32 values of a warp are neighbours.
    const int q = warp & 3;
    const int et = threadIdx.x - 64;               // 0..127: index among the epilogue threads
    uint32_t tile_it = 0;
    bool ok = true;
    pdl_wait();                                    // Y, the scratch and the counters may be in use by the kernel before
    for (int i = first_item<RUN>(p, cta); i < num_items && ok; i = next_item<RUN>(p, i, num_ctas), ++tile_it) {
      const Item it = item_of<RUN>(p, i);
      const Layer& ly = p.L[it.layer];
      const int acc = tile_it % C::ACCS;
      if (!mbar_wait<true>(acc_full(acc), (tile_it / C::ACCS) & 1, abort_flag)) { ok = false; break; }
      tc_fence_after();
      store_chunk<NT>(p, it, tmem_base, acc, q);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty(acc));
      if (ly.chunks > 1) {
        // count this chunk in; the CTA's last one is seen to by all of its threads at the end (every other role is about to fall
        // idle), another one by the epilogue where it is the tile's last to arrive
        if (RUN == kAllChunks && it.chunk + 1 < ly.chunks) continue;       // (the tile's other chunks are this CTA's too)
        __threadfence();
        epilogue_barrier();
        if (kDebugBounds && p.lag > 0 && it.chunk == 0)  // test hook: a tile's first chunk is counted in long after the others
          for (const long long t0 = clock64(); clock64() - t0 < 4 * p.lag;) { }
        if (next_item<RUN>(p, i, num_ctas) >= num_items) {
          if (et == 0) {
            at_end[0] = i;
            at_end[1] = RUN == kAllChunks ? 0 : atomicAdd(ly.counters + it.tile, 1 + kTaken);
          }
          break;
        }
        if (RUN == kAllChunks) { finish_by_epilogue<RUN>(p, it, 0, et); continue; }
        if (et == 0) {
          const int old = atomicAdd(ly.counters + it.tile, 1);
          *last_flag = old;
          if (arrived(old) != ly.chunks - 1 && left(atomicAdd(ly.counters + it.tile, kLeft)) + 1 == ly.chunks) ly.counters[it.tile] = 0;
        }
        epilogue_barrier();
        const int old = *last_flag;
        epilogue_barrier();                         // everyone has read it
        if (arrived(old) == ly.chunks - 1) finish_by_epilogue<RUN>(p, it, old, et);
      }
    }
  } else {
    // ------------------------------------------------------------------ converters
    const int c = threadIdx.x - 6 * 32;          // 0..767
    const int group = c >> 8, col = c & 255;     // stage group; weight column of the 256-column stage
    const int half = col >> 7;                   // its 128-column packed tile; the column within it is the thread's lane of
    const int nl = (warp & 3) * 32 + lane;       // tensor memory: a warp writes the lanes of its number mod 4
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    // the CTA's items one after the other; their slabs form one sequence of which this group takes every third
    uint32_t it_no = 0, batch_no = 0;
    bool ok = true;
    const int w_tile = w_tile_bytes(p.w_bits);
    for (int item = first_item<RUN>(p, cta); item < num_items && ok; item = next_item<RUN>(p, item, num_ctas)) {
      const Item it = item_of<RUN>(p, item);
      const int k_slabs = p.L[it.layer].k_slabs, r_blocks = p.L[it.layer].r_blocks;
      const bool has_w = 2 * it.tile + half < p.L[it.layer].n_tiles;
      for (int s0 = it.s_lo; s0 < it.s_hi && ok; ++batch_no) {
        const int e = batch_end(s0, it.s_hi, k_slabs), pk = batch_no % PK_SLOTS;
        if (kDebugBounds && p.lag > 0) {                 // test hook: a group without a step in this batch comes late
          bool mine = false;
          for (int st = s0, n = it_no; st < e; st += STEP, ++n) mine = mine || n % CONVERTER_GROUPS == group;
          if (!mine) {
            const long long t0 = clock64();
            while (clock64() - t0 < p.lag) { }
          }
        }
        // also where none of the batch's steps is this group's: see PK_FREE_ARRIVALS
        if (!mbar_wait(w_full(pk), (batch_no / PK_SLOTS) & 1, abort_flag)) { ok = false; break; }
        const uint8_t* pkh = pk_base + pk * C::PK_SLOT_BYTES + C::X_BYTES + half * W_HALF_BYTES;
        for (int st = s0; st < e; st += STEP, ++it_no) {
          if (it_no % CONVERTER_GROUPS != (uint32_t)group) continue;
          if (!mbar_wait(cv_free(group), ((it_no / CV_SLOTS) & 1) ^ 1, abort_flag)) { ok = false; break; }
          tc_fence_after();                            // the MMAs that read the slot before have finished
          if (has_w)                                   // (a missing half multiplies what its lanes happen to hold: nobody reads it)
            for (int s = st; s < min(st + STEP, e); ++s) {
              const uint32_t dst = tmem_base + lane_base + C::CV_COL0 + (group * STEP + s - st) * CV_COLS + half * 32;
              uint4 o[4];
              const uint8_t* pkt = pkh + (s - s0) * w_tile;
              if (s >= k_slabs) {
                // 64 ranks: four blocks of 16
                const int rb0 = (s - s0) * 4, nb = min(4, r_blocks - (s - k_slabs) * 4);
      #pragma unroll
                for (int hp = 0; hp < 2; ++hp) {
      #pragma unroll
                  for (int rb = 0; rb < 2; ++rb) {
                    o[2 * rb] = make_uint4(0u, 0u, 0u, 0u);
                    o[2 * rb + 1] = o[2 * rb];
                    if (2 * hp + rb < nb) {
                      const uint4 w = *reinterpret_cast<const uint4*>(pkh + ((rb0 + 2 * hp + rb) * kTileN + nl) * 16);
                      const float scale = pow2f((int)pkh[RANK_EXP_OFFSET + (rb0 + 2 * hp + rb) * kTileN + nl] - 127 - p.lr_shift);
                      o[2 * rb] = convert_i8x8(w.x, w.y, scale);
                      o[2 * rb + 1] = convert_i8x8(w.z, w.w, scale);
                    }
                  }
                  tmem_st16(dst + 16 * hp, o[0], o[1], o[2], o[3]);
                }
              } else if (p.w_bits == 2) {
                const uint4 wv = *reinterpret_cast<const uint4*>(pkt + nl * 16);
                const uint32_t eb = *reinterpret_cast<const uint32_t*>(pkt + 2048 + nl * 4);
                uint32_t s2, c2;
                w_scales2(eb & 0xFFu, s2, c2);
                convert_word2(wv.x, s2, c2, o[0], o[1]);
                w_scales2((eb >> 8) & 0xFFu, s2, c2);
                convert_word2(wv.y, s2, c2, o[2], o[3]);
                tmem_st16(dst, o[0], o[1], o[2], o[3]);
                w_scales2((eb >> 16) & 0xFFu, s2, c2);
                convert_word2(wv.z, s2, c2, o[0], o[1]);
                w_scales2(eb >> 24, s2, c2);
                convert_word2(wv.w, s2, c2, o[2], o[3]);
                tmem_st16(dst + 16, o[0], o[1], o[2], o[3]);
              } else {
                const uint4 wa = *reinterpret_cast<const uint4*>(pkt + nl * 16);
                const uint4 wb = *reinterpret_cast<const uint4*>(pkt + (kTileN + nl) * 16);
                const uint32_t eb = *reinterpret_cast<const uint32_t*>(pkt + kWTileNibbleBytes + nl * 4);
                uint32_t s2, c2;
                w_scales(eb & 0xFFu, s2, c2);
                o[0] = convert_word(wa.x, s2, c2);
                o[1] = convert_word(wa.y, s2, c2);
                w_scales((eb >> 8) & 0xFFu, s2, c2);
                o[2] = convert_word(wa.z, s2, c2);
                o[3] = convert_word(wa.w, s2, c2);
                tmem_st16(dst, o[0], o[1], o[2], o[3]);
                w_scales((eb >> 16) & 0xFFu, s2, c2);
                o[0] = convert_word(wb.x, s2, c2);
                o[1] = convert_word(wb.y, s2, c2);
                w_scales(eb >> 24, s2, c2);
                o[2] = convert_word(wb.z, s2, c2);
                o[3] = convert_word(wb.w, s2, c2);
                tmem_st16(dst + 16, o[0], o[1], o[2], o[3]);
              }
            }
          tmem_st_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(cv_ready(group));
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(pk_free(pk));
        s0 = e;
      }
    }
  }

  // ------------------------------------------------------------------ teardown
  __syncthreads();                      // every role is done (or has given up): the flags below are final for this CTA
  if (at_end[0] >= 0 && abort_flag->abort == 0) finish_tile<true, RUN>(p, item_of<RUN>(p, at_end[0]), at_end[1], threadIdx.x, last_flag);
  if (abort_flag->abort != 0) {
    const long long t0 = clock64();
    while (clock64() - t0 < 400000) { }
    if (threadIdx.x == 0) report_error(p.status, LQER_ERR_TIMEOUT, 600, blockIdx.x);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeTiledFn>(f);
  }();
  return fn;
}

template <int NT, int RUN>
static cudaError_t launch_nt(const TensorMaps& tmaps, const Params& p, int ctas, cudaStream_t s) {
  using C = Cfg<NT>;
  static OncePerDevice once;
  cudaError_t e = once.run([] {
    return cudaFuncSetAttribute(gemm_small_kernel<NT, RUN>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = C::SMEM_BYTES;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // may set up and prefetch weights while the prologue runs
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  LaunchScope scope(kFamDecode, s);
  return cudaLaunchKernelEx(&cfg, gemm_small_kernel<NT, RUN>, tmaps, p);
}

}  // namespace sg

int gemm_small_max_layers() { return sg::MAX_LAYERS; }

cudaError_t launch_gemm_small(const SmallGemmLayer* layers, int n, int M, int y_type, bool tensor_memory_form, int epoch,
                              DeviceStatus* st, cudaStream_t s) {
  using namespace sg;
  if (n < 1 || n > MAX_LAYERS || M < 1 || M > kSmallMaxM) return cudaErrorInvalidValue;
  // up to 16 tokens: the register-operand kernel, unless the caller asks for this file's
  const bool use_mma = !tensor_memory_form && small_takes_mma(*layers[0].meta, M);
  EncodeTiledFn enc = use_mma ? nullptr : encode_fn();
  if (enc == nullptr && !use_mma) return cudaErrorNotSupported;
  const int x_rows = (M + 15) / 16 * 16;
  TensorMaps tmaps;
  Params p;
  int item_begin = 0;
  // K chunks per tile.  A layer alone is cut as its shape says (small_gemm_chunks: enough work items for every SM).
  // Layers that share a launch bring many tiles between them; they are cut by the time model below, never finer than alone
  // (the scratch is sized for that).  The sums of a tile are then grouped differently, so a layer's result in a shared
  // launch may differ from its result alone in the last bits; it is the same whenever the same layers share a launch.
  const int sms = sm_count();
  if (sms < 1) return cudaErrorInvalidDevice;
  int group_chunks = 1;
  p.run = p.takers = 1;
  if (n > 1) {
    // The cut that makes (rounds of items over the SMs) x (slabs per item + what an item costs beside its slabs) smallest,
    // a function of the shapes alone.  The register-operand kernel runs two CTAs per SM, an item each at a time, and an item costs
    // it about ten slabs' worth of time (activation copy, rank term, partial sums); this file's kernel one, and four.
    // The cut is also how long a chain of sums in tensor memory gets, and these cut off what does not fit: two layers of
    // 4096 x 11008 in one piece instead of three chunks a tile are 7 times as far from 64 bits (one sign, block exponents over a dozen
    // binades: 1.9e-6 and 2.7e-7), although that was the faster way.  So what is known better of an item's costs, below, may
    // make the chunks smaller, not larger.
    const int ctas = use_mma ? 2 * 148 : 148, extra = use_mma ? 10 : 4;
    long best = -1, best_rounds = 0, best_len = 0, tiles = 0;
    const int slabs = layers[0].meta->k_slabs, most = small_gemm_chunks(*layers[0].meta);
    bool alike = !use_mma;                                   // one K and one number of chunks for all layers
    for (int i = 0; i < n; ++i) {
      const PackedMeta& m = *layers[i].meta;
      tiles += small_gemm_col_tiles(m);
      alike = alike && m.k_slabs == slabs && small_gemm_chunks(m) == most;
    }
    for (int c = 1; c <= 16; ++c) {
      long items = 0, len = 0;
      for (int i = 0; i < n; ++i) {
        const PackedMeta& m = *layers[i].meta;
        const int ci = std::min(c, small_gemm_chunks(m));
        items += (long)small_gemm_col_tiles(m) * ci;
        len = std::max(len, (long)(m.k_slabs + ci - 1) / ci);
      }
      const long rounds = (items + ctas - 1) / ctas, cost = rounds * (len + extra);
      if (best < 0 || cost < best) { best = cost; group_chunks = c; best_rounds = rounds; best_len = len; }
    }
    // Several rounds of chunks though the tiles fit the SMs at once: then one or more CTAs may have a tile for themselves and take runs of its chunks.
    // In slabs' time (0.4 us), a round costs 6 c - 16 + 4 M / 7 (c chunks a tile), 16 at least, beside its slabs: partial sums of every chunk, of
    // all CTAs at a time; a run costs 3 + M / 17 for each chunk beside its slabs, and 4 + M / 8 at the end if all chunks are its own, 19 + M / 20
    // if their sums meet in scratch.  us, in rounds / in runs of all, or of half of the chunks: two layers of 4096 x 11008, 3 chunks, 20 rows 41.1 /
    // 45.3, 32 rows 46.8 / 45.2, 64 rows 64.3 / 50.6, 128 rows 103 / 70.0; of 2048 x 11008, 32 rows 40.2 / 32.8; three of 4352 x 4352, 5 chunks,
    // 20 rows 40.2 / 36.9, 64 rows 77.8 / 44.5, 128 rows 137 / 65.7, and in 6 chunks 34.6, 41.9, 63.6.
    if (alike && group_chunks > 1 && best_rounds > 1 && tiles <= ctas) {
      long least = best_rounds * (best_len + std::max(16, 6 * group_chunks - 16 + 4 * M / 7));
      for (int c = group_chunks; c <= most; ++c) {
        const int stages = (slabs + c - 1) / c;
        if ((slabs + stages - 1) / stages != c) continue;
        for (int takers = 1; takers < c && takers * tiles <= ctas; ++takers) {
          const int run = (c + takers - 1) / takers;
          const long cost = run * (stages + 3 + M / 17) + (takers == 1 ? 4 + M / 8 : 19 + M / 20);
          if ((takers - 1) * run < c && cost < least) { least = cost; group_chunks = c; p.run = run; p.takers = takers; }
        }
      }
    }
  }
  for (int i = 0; i < MAX_LAYERS; ++i) {
    const SmallGemmLayer& src = layers[i < n ? i : 0];
    const PackedMeta& m = *src.meta;
    if (m.lr_bits != layers[0].meta->lr_bits || m.w_bits != layers[0].meta->w_bits) return cudaErrorInvalidValue;
    const cuuint64_t dims[2] = {(cuuint64_t)xcat_cols(m), (cuuint64_t)M};
    const cuuint64_t strides[1] = {(cuuint64_t)xcat_cols(m) * 2};
    const cuuint32_t box[2] = {BK, (cuuint32_t)x_rows};
    const cuuint32_t estr[2] = {1, 1};
    if (!use_mma &&
        enc(&tmaps.m[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(src.xcat), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
    const uint8_t* base = static_cast<const uint8_t*>(src.packed);
    Layer& ly = p.L[i];
    ly.wsec = base + m.off_w;
    ly.bsec = base + m.off_b;
    ly.xfrag = static_cast<const uint8_t*>(src.xcat);
    ly.flags = src.flags;
    ly.plane = (m.k_slabs + frag_rank_slabs(m)) * 256;
    ly.Y = src.Y;
    ly.y_extent = y_bytes(y_type, (size_t)M, (size_t)m.N);
    if (kDebugBounds) ly.y_extent -= std::min(ly.y_extent, debug_y_shrink());
    ly.w_extent = m.off_b - m.off_w; ly.b_extent = m.off_a - m.off_b;
    ly.partials = src.partials;
    ly.counters = src.counters;
    ly.N = m.N;
    ly.n_tiles = m.n_tiles; ly.k_slabs = m.k_slabs; ly.r_blocks = m.r_blocks;
    ly.spt = m.k_slabs + (use_mma ? (m.r_blocks + 1) / 2 : frag_rank_slabs(m));
    int want = small_gemm_chunks(m);
    if (n > 1 && group_chunks < want) want = group_chunks;
    ly.chunk_stages = (m.k_slabs + want - 1) / want;
    ly.chunks = (m.k_slabs + ly.chunk_stages - 1) / ly.chunk_stages;
    ly.partial_extent = ly.chunks > 1 ? (size_t)small_gemm_col_tiles(m) * ly.chunks * M * 256 * 4 : 0;
    ly.item_begin = item_begin;
    if (i < n) item_begin += small_gemm_col_tiles(m) * (p.run > 1 ? p.takers * p.run : ly.chunks);
  }
  p.n = n;
  p.chunks = p.L[0].chunks;
  p.num_items = item_begin;
  p.status = st;
  p.M = M;
  p.lr_shift = layers[0].meta->lr_bits - 2;
  p.y_type = y_type;
  p.a_bits = layers[0].meta->a_bits; p.exp_min = layers[0].meta->exp_min; p.exp_max = layers[0].meta->exp_max;
  p.x_rows = x_rows;
  p.w_bits = layers[0].meta->w_bits;
  p.wait_limit = wait_limit_cycles();
  p.lag = debug_converter_lag();
  p.epoch = epoch;
  p.exit_count = reinterpret_cast<int*>(reinterpret_cast<uint8_t*>(st) + kFlagAreaOffset + 2 * MAX_LAYERS * 4);
  p.stall = take_stall(kFamDecode) ? 1 : 0;
  if (use_mma) return launch_gemm_mma(p, s);
  const int ctas = std::min(p.num_items / p.run, sms);
  const auto go = [&](auto run) {
    constexpr int RUN = decltype(run)::value;
    return M <= 32 ? launch_nt<32, RUN>(tmaps, p, ctas, s) : M <= 64 ? launch_nt<64, RUN>(tmaps, p, ctas, s) : launch_nt<128, RUN>(tmaps, p, ctas, s);
  };
  if (p.run == 1) return go(std::integral_constant<int, kNoRuns>());
  return p.takers == 1 ? go(std::integral_constant<int, kAllChunks>()) : go(std::integral_constant<int, kSomeChunks>());
}

}  // namespace lqer
