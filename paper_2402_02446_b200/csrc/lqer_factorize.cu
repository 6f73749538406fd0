// Factor preparation on the GPU (paper Section 3.1: E_q = W - W_q, A_k = U_k, B_k = Sigma_k V_k^T; Section 3.2:
// SVD of S E_q, A_k = S^-1 U'_k, B_k = Sigma'_k V'_k^T; Appendix A: the calibration of S), so that the packed
// layer can be produced from the weight and a calibration batch alone.
//
//   s        per channel: mean |X| over the tokens of a sample, maximum over the samples, divided by
//            sqrt(min * max)                                                   (fp64 sums, fixed order)
//   G        = diag(s) (W - dq(q(W)))      fp32 [K, N]   (s = 1 for plain LQER)
//   top-k    singular triplets of G by randomised subspace iteration: Q = orth(G Omega); four rounds of
//            Z = orth(G^T Q), Q = orth(G Z); then Bt = G^T Q = Q_b R (Cholesky factor of Bt^T Bt), the right
//            singular vectors V of the small matrix R (one-sided Jacobi in one CTA), and
//            A = diag(1/s) Q V_k,   B = (Bt V_k)^T = Sigma_k V_k^T.
// The large products read G as fp32 and accumulate in fp64 (on the fp64 tensor pipe); everything of rank size is fp64.
// orth() is Cholesky QR applied twice.  Omega (the random test matrix) is an input, so the caller owns the random numbers.
// None of this is on the inference path; every sum has a fixed order.
#include "lqer_common.cuh"

namespace lqer {
namespace fac {

constexpr int kOversample = 16;
constexpr int kIters = 4;
constexpr int kMaxR = 272;                 // 256 + oversample
constexpr int kGramChunks = 32;            // partial Gram matrices (the workspace has room for 64)

// ---------------------------------------------------------------------------- calibration (Appendix A)
// Partial sums of |X| over a chunk of rows: grid (column blocks of 256, row chunks), one thread per column.
__global__ void __launch_bounds__(256) abs_sum_kernel(const float* __restrict__ X, int rows, int K, int rows_per_chunk,
                                                      double* __restrict__ part) {
  const int c = blockIdx.x * 256 + threadIdx.x;
  if (c >= K) return;
  const int r0 = blockIdx.y * rows_per_chunk, r1 = min(rows, r0 + rows_per_chunk);
  double acc = 0.0;
  for (int r = r0; r < r1; ++r) acc += (double)fabsf(X[(size_t)r * K + c]);
  part[(size_t)blockIdx.y * K + c] = acc;
}
// a_bar[c] = max(a_bar[c], sum of the chunks / rows)   (first sample: plain store)
__global__ void __launch_bounds__(256) abs_mean_max_kernel(const double* __restrict__ part, int chunks, int K, int rows,
                                                           int first, double* __restrict__ a_bar) {
  const int c = blockIdx.x * 256 + threadIdx.x;
  if (c >= K) return;
  double acc = 0.0;
  for (int q = 0; q < chunks; ++q) acc += part[(size_t)q * K + c];
  const double a = acc / (double)rows;
  a_bar[c] = first ? a : fmax(a_bar[c], a);
}
// s = a_bar / sqrt(min * max); one CTA.  status: 1 if a channel is identically zero (S is not invertible).
__global__ void __launch_bounds__(1024) normalise_scale_kernel(const double* __restrict__ a_bar, int K, double* __restrict__ s,
                                                               int* __restrict__ status) {
  __shared__ double s_min[1024], s_max[1024];
  double lo = 1e300, hi = 0.0;
  for (int c = threadIdx.x; c < K; c += 1024) { lo = fmin(lo, a_bar[c]); hi = fmax(hi, a_bar[c]); }
  s_min[threadIdx.x] = lo; s_max[threadIdx.x] = hi;
  __syncthreads();
  for (int w = 512; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      s_min[threadIdx.x] = fmin(s_min[threadIdx.x], s_min[threadIdx.x + w]);
      s_max[threadIdx.x] = fmax(s_max[threadIdx.x], s_max[threadIdx.x + w]);
    }
    __syncthreads();
  }
  lo = s_min[0]; hi = s_max[0];
  if (threadIdx.x == 0) *status = lo > 0.0 ? 0 : 1;
  const double norm = lo > 0.0 ? 1.0 / sqrt(lo * hi) : 0.0;
  for (int c = threadIdx.x; c < K; c += 1024) s[c] = lo > 0.0 ? a_bar[c] * norm : 1.0;
}
__global__ void fill_ones_kernel(double* s, int K) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < K) s[c] = 1.0;
}

// ---------------------------------------------------------------------------- G = diag(s) (W - dq(q(W)))
// One thread = one (column n, 16-block of K), as the packing kernel quantises it.
__global__ void __launch_bounds__(256) scaled_error_kernel(const float* __restrict__ W, int K, int N, int w_bits, int emin, int emax,
                                                           const double* __restrict__ s, float* __restrict__ G) {
  const int n = blockIdx.x * 256 + threadIdx.x;
  const int kb = blockIdx.y;
  if (n >= N) return;
  float v[16];
  float amax = 0.0f;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    v[i] = W[(size_t)(kb * 16 + i) * N + n];
    amax = fmaxf(amax, abs_ignore_nan(v[i]));
  }
  const int e = block_exponent(amax, emin, emax);
  const double step = pow2d(e - (w_bits - 2));
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const double err = (double)v[i] - (double)quant_mantissa(v[i], e, w_bits) * step;
    G[(size_t)(kb * 16 + i) * N + n] = (float)(s[kb * 16 + i] * err);
  }
}

// ---------------------------------------------------------------------------- products with G
__global__ void __launch_bounds__(256) widen_kernel(const float* __restrict__ x, size_t n, double* __restrict__ y) {
  const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (i < n) y[i] = (double)x[i];
}
// C[m, r] = op(G) X, fp64 accumulation.  TRANS = false: op(G) = G [m = K, inner = N], X [N, r].
// TRANS = true: op(G) = G^T [m = N, inner = K], X [K, r].
// Bound by the fp64 multiply-adds (2 K N r flop; 43 us for a 4096 x 4096 G at r = 48 and 37 TFLOP/s): they run as
// mma.sync.m16n8k8 in fp64, whose fragments come straight from global memory.  A CTA owns 16 MT rows of C and up to 48
// columns for the whole inner dimension; its eight warps take inner chunks of 16 (8 for G^T) in turn, each holds a full
// tile of sums, and the eight are added in warp order at the end.  The inner positions of an MMA and the rows of its A
// operand may be any, as long as both operands agree and the store knows: a lane takes neighbouring elements of G, one
// vector load each, instead of the fragment's strided ones.
// Measured (4096 x 4096, r = 48): 101 us (G^T) and 87 us (G) per product, against 1250 - 1320 us for a 64 x 64 tile per CTA
// with 4 x 4 outputs per thread, which left 84 SMs without a tile.
constexpr int kGCols = 48, kGTiles = kGCols / 8, kGWarps = 8;
__device__ __forceinline__ void dmma(double (&c)[4], const double (&a)[4], double b0, double b1) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3]) : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(b0), "d"(b1));
}
template <bool TRANS, int MT>
__global__ void __launch_bounds__(kGWarps * 32) g_times_kernel(const float* __restrict__ G, int K, int N, const double* __restrict__ X, int r,
                                                               double* __restrict__ C) {
  extern __shared__ double s_part[];                         // [warp][16 MT][kGCols]
  constexpr int STEP = TRANS ? 8 : 16;                       // inner positions of a chunk
  const int m_total = TRANS ? N : K, inner = TRANS ? K : N;
  const int m0 = blockIdx.x * 16 * MT, c0 = blockIdx.y * kGCols;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int n_tiles = min(kGTiles, (r - c0 + 7) / 8);
  double acc[MT][kGTiles][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int n = 0; n < kGTiles; ++n)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][n][j] = 0.0;

  // one chunk of both operands: gv[i][...] G's elements of m tile i, xv[h][n] X's rows of the chunk's k positions
  constexpr int KS = STEP / 8;                               // MMAs along the inner dimension
  float gv[MT][KS][4];
  double xv[KS][2][kGTiles];
  auto load = [&](int i0) {
    if (TRANS) {
      // lane g: columns 2 MT g + .. of the CTA's 16 MT; its rows are inner positions i0 + t and i0 + t + 4
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = i0 + t + 4 * h, m = m0 + 2 * MT * g;
        float v[2 * MT];
#pragma unroll
        for (int q = 0; q < 2 * MT; ++q) v[q] = 0.0f;
        if (i < inner && m < m_total) {                      // (N is a multiple of 8)
          const float* src = G + (size_t)i * N + m;
          if (MT == 2) {
            const float4 w = *reinterpret_cast<const float4*>(src);
            v[0] = w.x; v[1] = w.y; v[2 * MT - 2] = w.z; v[2 * MT - 1] = w.w;
          } else {
            const float2 w = *reinterpret_cast<const float2*>(src);
            v[0] = w.x; v[1] = w.y;
          }
        }
#pragma unroll
        for (int i2 = 0; i2 < MT; ++i2) { gv[i2][0][2 * h] = v[2 * i2]; gv[i2][0][2 * h + 1] = v[2 * i2 + 1]; }
      }
    } else {
      // lane t: inner positions i0 + 4 t + {0, 1, 2, 3}: k slots t and t + 4 of two MMAs
#pragma unroll
      for (int i2 = 0; i2 < MT; ++i2)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int m = m0 + 16 * i2 + 8 * h + g, i = i0 + 4 * t;
          float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
          if (m < m_total && i < inner) w = *reinterpret_cast<const float4*>(G + (size_t)m * N + i);
          gv[i2][0][h] = w.x; gv[i2][0][2 + h] = w.y; gv[i2][KS - 1][h] = w.z; gv[i2][KS - 1][2 + h] = w.w;
        }
    }
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = TRANS ? i0 + t + 4 * h : i0 + 4 * t + 2 * ks + h;
#pragma unroll
        for (int n = 0; n < kGTiles; ++n) {
          const int c = c0 + 8 * n + g;
          xv[ks][h][n] = i < inner && c < r ? X[(size_t)i * r + c] : 0.0;
        }
      }
  };
  for (int i0 = warp * STEP; i0 < inner; i0 += kGWarps * STEP) {
    load(i0);
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int i2 = 0; i2 < MT; ++i2) {
        // a fragment: (row g, k t), (g + 8, t), (g, t + 4), (g + 8, t + 4)
        const double a[4] = {(double)gv[i2][ks][0], (double)gv[i2][ks][1], (double)gv[i2][ks][2], (double)gv[i2][ks][3]};
#pragma unroll
        for (int n = 0; n < kGTiles; ++n)
          if (n < n_tiles) dmma(acc[i2][n], a, xv[ks][0][n], xv[ks][1][n]);
      }
  }
  double* mine = s_part + (size_t)warp * 16 * MT * kGCols;
#pragma unroll
  for (int i2 = 0; i2 < MT; ++i2)
#pragma unroll
    for (int n = 0; n < kGTiles; ++n)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        // accumulator row g + 8 (j / 2) of m tile i2, column 2 t + j % 2
        const int row = TRANS ? 2 * MT * g + 2 * i2 + (j >> 1) : 16 * i2 + 8 * (j >> 1) + g;
        mine[row * kGCols + 8 * n + 2 * t + (j & 1)] = acc[i2][n][j];
      }
  __syncthreads();
  for (int o = threadIdx.x; o < 16 * MT * kGCols; o += kGWarps * 32) {
    const int m = m0 + o / kGCols, c = c0 + o % kGCols;
    if (m >= m_total || c >= r) continue;
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < kGWarps; ++w) v += s_part[(size_t)w * 16 * MT * kGCols + o];
    C[(size_t)m * r + c] = v;
  }
}
// 32 rows per CTA where that gives a CTA to most SMs, 16 otherwise.
template <bool TRANS>
static cudaError_t g_times(const float* G, int K, int N, const double* X, int r, double* C, cudaStream_t s) {
  const int m = TRANS ? N : K, cols = (r + kGCols - 1) / kGCols;
  static OncePerDevice once;
  const cudaError_t e = once.run([] {
    const cudaError_t e1 = cudaFuncSetAttribute(g_times_kernel<TRANS, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGWarps * 16 * kGCols * 8);
    return e1 != cudaSuccess ? e1
                             : cudaFuncSetAttribute(g_times_kernel<TRANS, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGWarps * 32 * kGCols * 8);
  });
  if (e != cudaSuccess) return e;
  if ((m + 31) / 32 * cols >= 96)
    g_times_kernel<TRANS, 2><<<dim3((m + 31) / 32, cols), kGWarps * 32, kGWarps * 32 * kGCols * 8, s>>>(G, K, N, X, r, C);
  else
    g_times_kernel<TRANS, 1><<<dim3((m + 15) / 16, cols), kGWarps * 32, kGWarps * 16 * kGCols * 8, s>>>(G, K, N, X, r, C);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------- tall-skinny helpers (fp64)
// Partial Gram matrices: part[chunk][r][r] = Y[rows of the chunk]^T Y[rows of the chunk].  grid (r tiles of 16,
// r tiles of 16, chunks), 256 threads = 16 x 16 outputs.
__global__ void __launch_bounds__(256) gram_partial_kernel(const double* __restrict__ Y, int m, int r, int rows_per_chunk,
                                                           double* __restrict__ part) {
  __shared__ double s_a[32][17], s_b[32][17];
  const int i0 = blockIdx.x * 16, j0 = blockIdx.y * 16;
  const int row_lo = blockIdx.z * rows_per_chunk, row_hi = min(m, row_lo + rows_per_chunk);
  const int ti = threadIdx.x & 15, tj = threadIdx.x >> 4;
  double acc = 0.0;
  for (int q0 = row_lo; q0 < row_hi; q0 += 32) {
    for (int q = threadIdx.x; q < 32 * 16; q += 256) {
      const int c = q & 15, rr = q >> 4;
      const int row = q0 + rr;
      s_a[rr][c] = (row < row_hi && i0 + c < r) ? Y[(size_t)row * r + i0 + c] : 0.0;
      s_b[rr][c] = (row < row_hi && j0 + c < r) ? Y[(size_t)row * r + j0 + c] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int rr = 0; rr < 32; ++rr) acc = fma(s_a[rr][ti], s_b[rr][tj], acc);
    __syncthreads();
  }
  if (i0 + ti < r && j0 + tj < r) part[((size_t)blockIdx.z * r + i0 + ti) * r + j0 + tj] = acc;
}
// C = the sum of the partial Gram matrices (in chunk order) = R^T R (upper-triangular R by Cholesky), then Rinv = R^-1; one
// CTA.  A pivot that is not positive (rank-deficient Y) is replaced by a tiny one so that the run stays finite; status
// records it.
// A chain of 2 r short steps, bound by their latency: a step is one update of a whole triangle by all threads (the trailing
// part of C minus the outer product of a finished row; the rows of R^-1 above a finished one) and ONE barrier - the
// division of a row by its pivot is left to whoever reads the row, and done for good at the end -, with both matrices in
// shared memory where they fit (r <= kSharedR).  67 us at r = 48, the sum of the partial matrices included; dot products
// along rows and columns in global memory took 150 us and the sum 15 us in a kernel of its own.
constexpr int kSharedR = 112;              // two r x r fp64 matrices within 200 KB
__global__ void __launch_bounds__(1024) cholesky_inverse_kernel(const double* __restrict__ part, int chunks, double* __restrict__ Cg, int r,
                                                                double* __restrict__ Rinvg, int* __restrict__ status) {
  extern __shared__ double s_mat[];
  __shared__ double s_inv[kMaxR];                            // 1 / pivot of each row
  const bool shared = r <= kSharedR;
  double* C = shared ? s_mat : Cg;
  double* Rinv = shared ? s_mat + r * r : Rinvg;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int q = threadIdx.x; q < r * r; q += 1024) {
    double acc = 0.0;
#pragma unroll 8
    for (int i = 0; i < chunks; ++i) acc += part[(size_t)i * r * r + q];
    C[q] = acc;
    Rinv[q] = q / r == q % r ? 1.0 : 0.0;
  }
  __syncthreads();
  // row j of the upper triangle of C becomes pivot_j times row j of R; the warp that has row j + 1 works out its pivot
  // (all warps doing it would keep the fp64 pipe busy for longer than the update)
  const auto pivot = [&](double d) {
    if (!(d > 0.0)) { d = 1e-300; atomicMax(status, 2); }
    return 1.0 / sqrt(d);
  };
  if (threadIdx.x == 0) s_inv[0] = pivot(C[0]);
  __syncthreads();
  for (int j = 0; j + 1 < r; ++j) {
    const double inv2 = s_inv[j] * s_inv[j];
    for (int i = j + 1 + ty; i < r; i += 32) {
      const double f = C[j * r + i] * inv2;
      for (int c = (i & ~31) + tx; c < r; c += 32)
        if (c >= i) {
          const double v = fma(-f, C[j * r + c], C[i * r + c]);
          C[i * r + c] = v;
          if (c == j + 1) s_inv[j + 1] = pivot(v);
        }
    }
    __syncthreads();
  }
  // R Rinv = I from the last row up: Z (here in Rinv) with Rinv row i = Z row i / pivot_i
  for (int i = r - 1; i > 0; --i) {
    const double inv = s_inv[i];
    for (int q = ty; q < i; q += 32) {
      const double f = C[q * r + i] * (s_inv[q] * inv);      // R[q, i] / pivot_i
      for (int c = (i & ~31) + tx; c < r; c += 32)
        if (c >= i) Rinv[q * r + c] = fma(-f, Rinv[i * r + c], Rinv[q * r + c]);
    }
    __syncthreads();
  }
  for (int q = threadIdx.x; q < r * r; q += 1024) {
    const int row = q / r, col = q % r;
    const double inv = s_inv[row];
    if (shared || col >= row) Cg[q] = col == row ? 1.0 / inv : C[q] * inv;
    Rinvg[q] = Rinv[q] * inv;
  }
}
static cudaError_t cholesky_inverse(const double* part, int chunks, double* C, int r, double* Rinv, int* status, cudaStream_t s) {
  static OncePerDevice once;
  const cudaError_t e = once.run([] {
    return cudaFuncSetAttribute(cholesky_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kSharedR * kSharedR * 8);
  });
  if (e != cudaSuccess) return e;
  cholesky_inverse_kernel<<<1, 1024, r <= kSharedR ? 2 * r * r * 8 : 0, s>>>(part, chunks, C, r, Rinv, status);
  return cudaGetLastError();
}
// Out[m, c] = rowscale[m] * sum_j Y[m, j] T[j, c] for c < cols (T is [r, ldt]); fp64 in, OutT out, optionally
// written transposed (Out[c, m]).  One CTA = 64 rows; T's used columns are walked in tiles of 64.
template <typename OutT, bool TRANSPOSE_OUT>
__global__ void __launch_bounds__(256) tall_times_small_kernel(const double* __restrict__ Y, int m, int r, const double* __restrict__ T,
                                                               int ldt, int cols, const double* __restrict__ rowscale, int invert_scale,
                                                               OutT* __restrict__ Out) {
  __shared__ double s_y[16][65], s_t[16][65];
  const int m0 = blockIdx.x * 64, c0 = blockIdx.y * 64;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  for (int j0 = 0; j0 < r; j0 += 16) {
    for (int q = threadIdx.x; q < 64 * 16; q += 256) {
      const int jj = q & 15, mi = q >> 4;
      s_y[jj][mi] = (m0 + mi < m && j0 + jj < r) ? Y[(size_t)(m0 + mi) * r + j0 + jj] : 0.0;
      const int cc = q & 63, j2 = q >> 6;
      s_t[j2][cc] = (j0 + j2 < r && c0 + cc < cols) ? T[(size_t)(j0 + j2) * ldt + c0 + cc] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = s_y[jj][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = s_t[jj][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = m0 + ty * 4 + i;
    if (row >= m) continue;
    double sc = 1.0;
    if (rowscale != nullptr) sc = invert_scale ? 1.0 / rowscale[row] : rowscale[row];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = c0 + tx * 4 + j;
      if (c < cols) {
        if (TRANSPOSE_OUT) Out[(size_t)c * m + row] = (OutT)(sc * acc[i][j]);
        else Out[(size_t)row * cols + c] = (OutT)(sc * acc[i][j]);
      }
    }
  }
}

// ---------------------------------------------------------------------------- small SVD (one CTA)
// Right singular vectors and singular values of the r x r upper-triangular R (the Cholesky factor left in the upper
// triangle of C, row-major) by one-sided Jacobi: pairs of columns are rotated until all are mutually orthogonal,
// V collects the rotations.  A warp per pair, the pairs of a step disjoint (round-robin tournament).  Mt, Vt: r x r
// scratch, column-major.  Out: Vs row-major [r][r] with the columns in falling order of singular value, sigma[r].
// Bound by the latency of its steps (r - 1 per sweep, one barrier each): both matrices sit in shared memory where they fit.
__global__ void __launch_bounds__(1024) jacobi_right_kernel(const double* __restrict__ C, int r, double* __restrict__ Mtg,
                                                            double* __restrict__ Vtg, double* __restrict__ Vs, double* __restrict__ sigma,
                                                            int* __restrict__ status) {
  extern __shared__ double s_mat[];
  double* Mt = r <= kSharedR ? s_mat : Mtg;
  double* Vt = r <= kSharedR ? s_mat + r * r : Vtg;
  __shared__ int s_rotated;
  __shared__ double s_norm[kMaxR];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int q = tid; q < r * r; q += 1024) {
    const int col = q / r, row = q % r;
    Mt[q] = row <= col ? C[(size_t)row * r + col] : 0.0;
    Vt[q] = row == col ? 1.0 : 0.0;
  }
  const int n = r + (r & 1);                  // players of the tournament (one dummy if r is odd)
  const double tol = 1e-15;
  int sweeps = 0;
  for (; sweeps < 40; ++sweeps) {
    __syncthreads();
    if (tid == 0) s_rotated = 0;
    __syncthreads();
    for (int t = 0; t < n - 1; ++t) {
      for (int i = warp; i < n / 2; i += 32) {
        int a = i == 0 ? n - 1 : (t + i) % (n - 1);
        int b = i == 0 ? t % (n - 1) : (t + n - 1 - i) % (n - 1);
        if (a >= r || b >= r) continue;
        const int p = min(a, b), q = max(a, b);
        double* mp = Mt + (size_t)p * r;
        double* mq = Mt + (size_t)q * r;
        double alpha = 0.0, beta = 0.0, gamma = 0.0;
        for (int row = lane; row < r; row += 32) {
          const double x = mp[row], y = mq[row];
          alpha = fma(x, x, alpha); beta = fma(y, y, beta); gamma = fma(x, y, gamma);
        }
#pragma unroll
        for (int sft = 16; sft > 0; sft >>= 1) {
          alpha += __shfl_xor_sync(0xFFFFFFFFu, alpha, sft);
          beta += __shfl_xor_sync(0xFFFFFFFFu, beta, sft);
          gamma += __shfl_xor_sync(0xFFFFFFFFu, gamma, sft);
        }
        if (fabs(gamma) > tol * sqrt(alpha * beta)) {
          const double zeta = (beta - alpha) / (2.0 * gamma);
          const double tt = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
          const double c = 1.0 / sqrt(1.0 + tt * tt), s = c * tt;
          double* vp = Vt + (size_t)p * r;
          double* vq = Vt + (size_t)q * r;
          for (int row = lane; row < r; row += 32) {
            const double x = mp[row], y = mq[row];
            mp[row] = c * x - s * y; mq[row] = s * x + c * y;
            const double u = vp[row], w = vq[row];
            vp[row] = c * u - s * w; vq[row] = s * u + c * w;
          }
          if (lane == 0) s_rotated = 1;
        }
      }
      __syncthreads();
    }
    if (s_rotated == 0) break;
  }
  if (tid == 0 && sweeps >= 40) atomicMax(status, 3);
  // singular values = column norms; falling order (ties by index)
  for (int j = warp; j < r; j += 32) {
    double a = 0.0;
    for (int row = lane; row < r; row += 32) a = fma(Mt[(size_t)j * r + row], Mt[(size_t)j * r + row], a);
#pragma unroll
    for (int sft = 16; sft > 0; sft >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, sft);
    if (lane == 0) s_norm[j] = a;
  }
  __syncthreads();
  for (int j = tid; j < r; j += 1024) {
    int rank = 0;
    for (int i = 0; i < r; ++i) rank += (s_norm[i] > s_norm[j] || (s_norm[i] == s_norm[j] && i < j)) ? 1 : 0;
    sigma[rank] = sqrt(s_norm[j]);
    for (int row = 0; row < r; ++row) Vs[(size_t)row * r + rank] = Vt[(size_t)j * r + row];
  }
}

}  // namespace fac

int factor_sketch_rank(int K, int N, int k) {
  int r = k + fac::kOversample;
  if (r > K) r = K;
  if (r > N) r = N;
  return r;
}

// Workspace of launch_factorize, in bytes (every piece 256-byte aligned).
size_t factor_workspace_bytes(int K, int N, int k, int max_calib_rows) {
  const int r = factor_sketch_rank(K, N, k);
  const size_t big = (size_t)(K > N ? K : N);
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  size_t b = 0;
  b += al((size_t)K * N * 4);                     // G
  b += 2 * al((size_t)K * 8);                     // a_bar, s
  b += al((size_t)64 * K * 8);                    // partial column sums of |X| (64 row chunks)
  b += 2 * al(big * r * 8);                       // two tall buffers (ping-pong)
  b += al((size_t)N * r * 8);                     // Bt
  b += al((size_t)64 * r * r * 8);                // partial Gram matrices
  b += 5 * al((size_t)r * r * 8);                 // C, Rinv, Mt, Vt, Vs
  b += al((size_t)r * 8) + 256;                   // sigma, status
  b += al((size_t)K * k * 4) + al((size_t)k * N * 4);   // A, B (fp32) where the caller keeps none
  (void)max_calib_rows;
  return b;
}

static cudaError_t orthonormalise(const double* Yin, double* Yout, int m, int r, double* gram_part, double* C, double* Rinv,
                                  int* status, cudaStream_t s) {
  using namespace fac;
  // Cholesky QR, twice: Y = Q R with Q^T Q = I to rounding once the first pass has tamed the conditioning
  const double* src = Yin;
  double* bufs[2] = {Yout, const_cast<double*>(Yin)};
  for (int pass = 0; pass < 2; ++pass) {
    const int chunks = kGramChunks, rows_per_chunk = (m + chunks - 1) / chunks;
    const int rt = (r + 15) / 16;
    gram_partial_kernel<<<dim3(rt, rt, chunks), 256, 0, s>>>(src, m, r, rows_per_chunk, gram_part);
    const cudaError_t e = cholesky_inverse(gram_part, chunks, C, r, Rinv, status, s);
    if (e != cudaSuccess) return e;
    double* dst = bufs[pass];
    tall_times_small_kernel<double, false><<<dim3((m + 63) / 64, (r + 63) / 64), 256, 0, s>>>(src, m, r, Rinv, r, r, nullptr, 0, dst);
    src = dst;
  }
  // after two passes the result sits in Yin's buffer; copy back to Yout so that the caller's view is uniform
  return cudaMemcpyAsync(Yout, src, (size_t)m * r * 8, cudaMemcpyDeviceToDevice, s);
}

// W [K,N], calibration samples Xs[i] [rows[i], K] (n_samples may be 0: plain LQER, S = I), Omega [N, r] fp32 with
// r = factor_sketch_rank.  Outputs A [K,k], B [k,N] fp32 (device).  status_out (device int, may be null inside ws).
cudaError_t launch_factorize(const float* W, const float* const* Xs, const int* rows, int n_samples, const float* Omega, int K,
                             int N, int k, int w_bits, int emin, int emax, float* A, float* B, void* workspace, int** status_dev,
                             float** A_used, float** B_used, cudaStream_t s) {
  using namespace fac;
  const int r = factor_sketch_rank(K, N, k);
  if (r > kMaxR || k < 1) return cudaErrorInvalidValue;
  const size_t big = (size_t)(K > N ? K : N);
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  uint8_t* p = static_cast<uint8_t*>(workspace);
  float* G = reinterpret_cast<float*>(p); p += al((size_t)K * N * 4);
  double* a_bar = reinterpret_cast<double*>(p); p += al((size_t)K * 8);
  double* sc = reinterpret_cast<double*>(p); p += al((size_t)K * 8);
  double* colpart = reinterpret_cast<double*>(p); p += al((size_t)64 * K * 8);
  double* T0 = reinterpret_cast<double*>(p); p += al(big * r * 8);
  double* T1 = reinterpret_cast<double*>(p); p += al(big * r * 8);
  double* Bt = reinterpret_cast<double*>(p); p += al((size_t)N * r * 8);
  double* gram_part = reinterpret_cast<double*>(p); p += al((size_t)64 * r * r * 8);
  double* C = reinterpret_cast<double*>(p); p += al((size_t)r * r * 8);
  double* Rinv = reinterpret_cast<double*>(p); p += al((size_t)r * r * 8);
  double* Mt = reinterpret_cast<double*>(p); p += al((size_t)r * r * 8);
  double* Vt = reinterpret_cast<double*>(p); p += al((size_t)r * r * 8);
  double* Vs = reinterpret_cast<double*>(p); p += al((size_t)r * r * 8);
  double* sigma = reinterpret_cast<double*>(p); p += al((size_t)r * 8);
  int* status = reinterpret_cast<int*>(p); p += 256;
  if (status_dev != nullptr) *status_dev = status;
  if (A == nullptr) A = reinterpret_cast<float*>(p);
  p += al((size_t)K * k * 4);
  if (B == nullptr) B = reinterpret_cast<float*>(p);
  if (A_used != nullptr) *A_used = A;
  if (B_used != nullptr) *B_used = B;

  LaunchScope scope(kFamPrepare, s, 16 + 12 * kIters);
  cudaMemsetAsync(status, 0, 4, s);
  // ---- S (Appendix A), or the identity
  if (n_samples > 0) {
    for (int i = 0; i < n_samples; ++i) {
      const int chunks = rows[i] < 64 ? 1 : 64, rpc = (rows[i] + chunks - 1) / chunks;
      abs_sum_kernel<<<dim3((K + 255) / 256, chunks), 256, 0, s>>>(Xs[i], rows[i], K, rpc, colpart);
      abs_mean_max_kernel<<<(K + 255) / 256, 256, 0, s>>>(colpart, chunks, K, rows[i], i == 0 ? 1 : 0, a_bar);
    }
    normalise_scale_kernel<<<1, 1024, 0, s>>>(a_bar, K, sc, status);
  } else {
    fill_ones_kernel<<<(K + 255) / 256, 256, 0, s>>>(sc, K);
  }
  // ---- G = S (W - W_q)
  scaled_error_kernel<<<dim3((N + 255) / 256, K / 16), 256, 0, s>>>(W, K, N, w_bits, emin, emax, sc, G);
  // ---- subspace iteration
  widen_kernel<<<(int)(((size_t)N * r + 255) / 256), 256, 0, s>>>(Omega, (size_t)N * r, T1);
  cudaError_t e = g_times<false>(G, K, N, T1, r, T0, s);                                 // Y = G Omega      [K, r]
  if (e != cudaSuccess) return e;
  e = orthonormalise(T0, T1, K, r, gram_part, C, Rinv, status, s);           // Q in T1
  if (e != cudaSuccess) return e;
  for (int it = 0; it < kIters; ++it) {
    if ((e = g_times<true>(G, K, N, T1, r, T0, s)) != cudaSuccess) return e;     // Z = G^T Q        [N, r]
    if ((e = orthonormalise(T0, Bt, N, r, gram_part, C, Rinv, status, s)) != cudaSuccess) return e;   // Z in Bt
    if ((e = g_times<false>(G, K, N, Bt, r, T0, s)) != cudaSuccess) return e;    // Y = G Z          [K, r]
    if ((e = orthonormalise(T0, T1, K, r, gram_part, C, Rinv, status, s)) != cudaSuccess) return e;   // Q in T1
  }
  if ((e = g_times<true>(G, K, N, T1, r, Bt, s)) != cudaSuccess) return e;       // Bt = G^T Q       [N, r]
  // ---- small SVD: Bt^T Bt = R^T R, R = U Sigma V^T  ->  G ~ (Q V) Sigma (...)^T
  {
    const int chunks = kGramChunks, rpc = (N + chunks - 1) / chunks, rt = (r + 15) / 16;
    gram_partial_kernel<<<dim3(rt, rt, chunks), 256, 0, s>>>(Bt, N, r, rpc, gram_part);
    if ((e = cholesky_inverse(gram_part, chunks, C, r, Rinv, status, s)) != cudaSuccess) return e;
    static OncePerDevice once;
    e = once.run([] {
      return cudaFuncSetAttribute(jacobi_right_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kSharedR * kSharedR * 8);
    });
    if (e != cudaSuccess) return e;
    jacobi_right_kernel<<<1, 1024, r <= kSharedR ? 2 * r * r * 8 : 0, s>>>(C, r, Mt, Vt, Vs, sigma, status);
  }
  // ---- A = S^-1 Q V_k  [K, k];  B = (Bt V_k)^T  [k, N]
  tall_times_small_kernel<float, false><<<dim3((K + 63) / 64, (k + 63) / 64), 256, 0, s>>>(T1, K, r, Vs, r, k, sc, 1, A);
  tall_times_small_kernel<float, true><<<dim3((N + 63) / 64, (k + 63) / 64), 256, 0, s>>>(Bt, N, r, Vs, r, k, nullptr, 0, B);
  return cudaGetLastError();
}

}  // namespace lqer
