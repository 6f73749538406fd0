// Register fragments of the mma.sync kernels for few tokens (paper Section 3.1 / 3.2): packed weights become bf16 B
// fragments in registers, exactly, and the activations come in matching A fragments (the fragment order of
// lqer_common.cuh).
#pragma once

#include "lqer_tc_ptx.cuh"

namespace lqer {
namespace mf {

__device__ __forceinline__ uint4 ld_stream16(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t ld_stream4(const void* p) {
  uint32_t v;
  asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
// a: the four registers of the A fragment in order (rows g / g + 8 of the first K pair, then of the second), as one
// 16-byte load delivers them.
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
// bf16 pairs (2^(e-2), 2^(e-2)) and (-136 * 2^(e-2), -136 * 2^(e-2)) of exponent byte `byte` of word e4 (eb = e + 127):
// the bf16 bits are (eb - 2) << 7 and 0x8000 | (eb + 5) << 7 | 8, i.e. eb * 0x80 plus a constant, in both halves.
__device__ __forceinline__ void w_scale_pair(uint32_t e4, int byte, uint32_t& s2, uint32_t& c2) {
  const uint32_t eb = __byte_perm(e4, 0u, 0x4440u + byte);
  s2 = eb * 0x00800080u - 0x01000100u;
  c2 = eb * 0x00800080u + 0x82888288u;
}

// (a & b) | c in one instruction, with the mask and the magic number held in registers (given as immediates the pair
// costs two instructions, because one instruction takes one immediate).
__device__ __forceinline__ uint32_t and_or(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
struct ConvConsts {
  uint32_t mask, magic;        // 0x000F000F (nibbles) or 0x00030003 (crumbs), 0x43004300
};
template <int WB>
__device__ __forceinline__ ConvConsts conv_consts() {
  ConvConsts k;
  if (WB == 4) asm volatile("mov.b32 %0, 0x000F000F;" : "=r"(k.mask));     // opaque to the compiler, so that they stay in registers
  else asm volatile("mov.b32 %0, 0x00030003;" : "=r"(k.mask));
  asm volatile("mov.b32 %0, 0x43004300;" : "=r"(k.magic));
  return k;
}
// Eight offset-binary nibbles of one block word -> eight bf16 (n - 8) * 2^(e-2), exact: 0x4300 | n is the bf16 value
// 128 + n, and (128 + n) * s - 136 * s rounds nothing away.  Register i holds K 2 i, 2 i + 1 of the word's eight.
__device__ __forceinline__ uint4 convert_nibbles(uint32_t w, uint32_t s2, uint32_t c2, const ConvConsts& k) {
  uint4 o;
  o.x = tc::fma_bf16x2(and_or(w, k.mask, k.magic), s2, c2);
  o.y = tc::fma_bf16x2(and_or(w >> 4, k.mask, k.magic), s2, c2);
  o.z = tc::fma_bf16x2(and_or(w >> 8, k.mask, k.magic), s2, c2);
  o.w = tc::fma_bf16x2(and_or(w >> 12, k.mask, k.magic), s2, c2);
  return o;
}
// The 2-bit format (mantissas -1, 0, 1; value m * 2^e): crumbs 4 j .. 4 j + 3 of the low and of the high half of a block
// word (K 8 j .. 8 j + 7 of the block's sixteen) -> eight bf16, exact: (128 + c) * s - 129 * s rounds nothing away.
__device__ __forceinline__ uint4 convert_crumbs(uint32_t w, int j, uint32_t s2, uint32_t c2, const ConvConsts& k) {
  uint4 o;
  o.x = tc::fma_bf16x2(and_or(w >> (8 * j), k.mask, k.magic), s2, c2);
  o.y = tc::fma_bf16x2(and_or(w >> (8 * j + 2), k.mask, k.magic), s2, c2);
  o.z = tc::fma_bf16x2(and_or(w >> (8 * j + 4), k.mask, k.magic), s2, c2);
  o.w = tc::fma_bf16x2(and_or(w >> (8 * j + 6), k.mask, k.magic), s2, c2);
  return o;
}
// bf16 pairs (2^e, 2^e) and (-129 * 2^e, -129 * 2^e) of an exponent byte of word e4: bits eb << 7 and 0x8000 | (eb + 7) << 7 | 1.
__device__ __forceinline__ void w_scale_pair2(uint32_t e4, int byte, uint32_t& s2, uint32_t& c2) {
  const uint32_t eb = __byte_perm(e4, 0u, 0x4440u + byte);
  s2 = eb * 0x00800080u;
  c2 = eb * 0x00800080u + 0x83818381u;
}

// A lane's weights of one step in one column octet: one block pair (32 K) of its column - 16 bytes of nibbles, or 8
// bytes of crumbs in w.x, w.y - and the slab's four exponent bytes of that column.
struct WOct {
  uint4 w;
  uint32_t e;
};
// wp / ep: the lane's column in the packed tile of the lane's slab (mantissas of its block pair; exponent word).
template <int WB>
__device__ __forceinline__ void load_w_oct(WOct& f, const uint8_t* wp, const uint8_t* ep) {
  if (WB == 4) {
    f.w = ld_stream16(wp);
  } else {
    asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(f.w.x), "=r"(f.w.y) : "l"(wp));
  }
  f.e = ld_stream4(ep);
}

// One octet's share of a step of weight slabs: eight MMAs.  a: the step's eight A fragments; eb0: index of the first
// exponent byte of the lane's block pair in an exponent word.
template <int WB>
__device__ __forceinline__ void compute_w_oct(float (&acc)[4], const WOct& f, const uint4 (&a)[8], int eb0, const ConvConsts& k) {
  uint32_t s2, c2;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if ((m & 1) == 0) {
      if (WB == 4) w_scale_pair(f.e, eb0 + (m >> 1), s2, c2);
      else w_scale_pair2(f.e, eb0 + (m >> 1), s2, c2);
    }
    uint4 b;
    if (WB == 4) {
      const uint32_t word = m == 0 ? f.w.x : m == 1 ? f.w.y : m == 2 ? f.w.z : f.w.w;
      b = convert_nibbles(word, s2, c2, k);
    } else {
      b = convert_crumbs(m < 2 ? f.w.x : f.w.y, m & 1, s2, c2, k);
    }
    mma_bf16(acc, a[2 * m], b.x, b.y);
    mma_bf16(acc, a[2 * m + 1], b.z, b.w);
  }
}

// One octet's share of a step of the rank term: 128 rank indices, of which the lane takes two 16-blocks of B_q (rb0,
// rb0 + 1) for its column.  bt: the packed B tile of the warp's 128-column half; nl: the lane's column in it; a: the
// step's eight A fragments.
__device__ __forceinline__ void compute_r_oct(float (&acc)[4], const uint8_t* bt, int r_blocks, int rb0, int nl, int lr_shift,
                                              const uint4 (&a)[8]) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int rb = rb0 + u;
    uint4 w = make_uint4(0u, 0u, 0u, 0u);
    float sc = 1.f;
    if (rb < r_blocks) {
      w = ld_stream16(bt + ((size_t)rb * kTileN + nl) * 16);
      sc = pow2f((int)bt[(size_t)r_blocks * kTileN * 16 + rb * kTileN + nl] - 127 - lr_shift);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int m = 2 * u + h;
      const uint4 b = tc::convert_i8x8(h ? w.z : w.x, h ? w.w : w.y, sc);
      mma_bf16(acc, a[2 * m], b.x, b.y);
      mma_bf16(acc, a[2 * m + 1], b.z, b.w);
    }
  }
}

// Byte offset of (row, column c of slab s) in the fragment order; plane: bytes of one plane.
__device__ __forceinline__ size_t frag_offset(int row, int slab, int c, size_t plane) {
  return (size_t)((c & 31) >> 2) * plane + (size_t)slab * 256 + (2 * (row & 7) + (c >> 5)) * 16 + (((c & 3) >> 1) * 2 + (row >> 3)) * 4 +
         (c & 1) * 2;
}

}  // namespace mf
}  // namespace lqer
