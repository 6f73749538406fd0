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
// orth() is Cholesky QR, applied twice in the end.  Omega (the random test matrix) is an input, so the caller owns the random numbers.
// None of this is on the inference path; every sum has a fixed order.
#include <utility>

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
// Partial Gram matrices, upper tiles: part[chunk][r][r] = Y[rows of the chunk]^T Y[rows of the chunk].  grid (r tiles of 16,
// r tiles of 16, chunks), 256 threads = 16 x 16 outputs; the next 32 rows are on their way while these are multiplied (7.2 us for
// 4096 x 48 against 10.5).
__global__ void __launch_bounds__(256) gram_partial_kernel(const double* __restrict__ Y, int m, int r, int rows_per_chunk,
                                                           double* __restrict__ part) {
  if (blockIdx.x > blockIdx.y) return;                       // only the upper triangle is read
  __shared__ double s_a[2][32][17], s_b[2][32][17];
  const int i0 = blockIdx.x * 16, j0 = blockIdx.y * 16;
  const int row_lo = blockIdx.z * rows_per_chunk, row_hi = min(m, row_lo + rows_per_chunk);
  const int ti = threadIdx.x & 15, tj = threadIdx.x >> 4;    // the output; also a row and column of the tile being loaded
  double va[2], vb[2];
  auto load = [&](int q0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = q0 + tj + 16 * h;
      va[h] = (row < row_hi && i0 + ti < r) ? Y[(size_t)row * r + i0 + ti] : 0.0;
      vb[h] = (row < row_hi && j0 + ti < r) ? Y[(size_t)row * r + j0 + ti] : 0.0;
    }
  };
  double acc = 0.0;
  load(row_lo);
  int buf = 0;
  for (int q0 = row_lo; q0 < row_hi; q0 += 32, buf ^= 1) {
#pragma unroll
    for (int h = 0; h < 2; ++h) { s_a[buf][tj + 16 * h][ti] = va[h]; s_b[buf][tj + 16 * h][ti] = vb[h]; }
    __syncthreads();
    load(q0 + 32);
#pragma unroll
    for (int rr = 0; rr < 32; ++rr) acc = fma(s_a[buf][rr][ti], s_b[buf][rr][tj], acc);
  }
  if (i0 + ti < r && j0 + tj < r) part[((size_t)blockIdx.z * r + i0 + ti) * r + j0 + tj] = acc;
}
// C = the sum of the partial Gram matrices (in chunk order) = R^T R (upper-triangular R by Cholesky), then Rinv = R^-1; one
// CTA.  A column whose pivot is not positive depends on the ones before it (rank-deficient Y): its row of R and its column of
// R^-1 are zero, so that the column is zero from there on and the run stays finite; status records it.
// Ranks beyond kSharedR: both matrices in global memory, a chain of 2 r short steps bound by their latency.  A step is one
// update of a whole triangle by all threads (the trailing part of C minus the outer product of a finished row; the rows of
// R^-1 above a finished one) and one barrier - the division of a row by its pivot is left to whoever reads the row, and done
// for good at the end.
constexpr int kSharedR = 112;              // two r x r fp64 matrices within 203 KB of shared memory
__global__ void __launch_bounds__(1024) cholesky_inverse_kernel(const double* __restrict__ part, int chunks, double* __restrict__ Cg, int r,
                                                                double* __restrict__ Rinvg, int* __restrict__ status) {
  __shared__ double s_inv[kMaxR];                            // 1 / pivot of each row
  double* C = Cg;
  double* Rinv = Rinvg;
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
    if (!(d > 0.0)) { atomicMax(status, 2); return 0.0; }
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
    if (col >= row) C[q] = col == row && inv > 0.0 ? 1.0 / inv : C[q] * inv;
    Rinv[q] *= inv;
  }
}
// The same for r <= kSharedR, in panels of kPanel rows, so that the chain of dependent steps is as short as it can be: one
// warp factors a diagonal block in registers (a column per lane; a step is one reciprocal square root, two shuffles, a product
// and a multiply-add), a thread per remaining column solves for the panel's rows of R, all threads update what is left, and the
// columns of R^-1, which depend on nothing but R, are formed at the end, eight lanes to a column, without a barrier.
// 3 barriers per panel instead of one per row and another per row of the inverse: 28 us at r = 48 against 67.
constexpr int kPanel = 8, kCholThreads = 512;
__host__ __device__ constexpr int chol_ld(int r) { return (r + kPanel - 1) / kPanel * kPanel + 1; }   // odd: eight rows meet no bank twice
__global__ void __launch_bounds__(kCholThreads) cholesky_inverse_panels_kernel(const double* __restrict__ part, int chunks, double* __restrict__ Cg,
                                                                               int r, double* __restrict__ Rinvg, int* __restrict__ status) {
  extern __shared__ double s_mat[];
  const int rp = (r + kPanel - 1) / kPanel * kPanel, ld = chol_ld(r);
  double* C = s_mat;
  double* Ri = s_mat + rp * ld;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int q = tid; q < rp * rp; q += kCholThreads) {
    const int row = q / rp, col = q % rp;
    double acc = row == col ? 1.0 : 0.0;                     // rows beyond r: the identity
    if (row < r && col < r && row <= col) {
      acc = 0.0;
#pragma unroll 16
      for (int i = 0; i < chunks; ++i) acc += part[(size_t)i * r * r + row * r + col];
    }
    C[row * ld + col] = acc;
    Ri[row * ld + col] = 0.0;
  }
  __syncthreads();
  for (int j0 = 0; j0 < rp; j0 += kPanel) {
    if (warp == 0) {
      const int c = lane & 7;
      double d[kPanel];
#pragma unroll
      for (int i = 0; i < kPanel; ++i) d[i] = i <= c ? C[(j0 + i) * ld + j0 + c] : 0.0;
      double mine = 1.0;                                     // 1 / pivot of this lane's column
      bool low = false;
#pragma unroll
      for (int j = 0; j < kPanel; ++j) {
        double p = __shfl_sync(0xFFFFFFFFu, d[j], j);
        if (!(p > 0.0)) { p = __longlong_as_double(0x7FF0000000000000LL); low = true; }   // infinity: a reciprocal root of zero
        const double inv = rsqrt(p);
        if (c == j) mine = inv;
        d[j] *= inv;
#pragma unroll
        for (int i = j + 1; i < kPanel; ++i) d[i] = fma(-__shfl_sync(0xFFFFFFFFu, d[j], i), d[j], d[i]);
      }
      if (low && lane == 0) atomicMax(status, 2);
      if (lane < kPanel) Ri[(j0 + c) * ld + j0 + c] = mine;  // the reciprocals of the diagonal
      if (lane < kPanel)
#pragma unroll
        for (int i = 0; i < kPanel; ++i)
          if (i <= c) C[(j0 + i) * ld + j0 + c] = d[i];
    }
    __syncthreads();
    const int left = rp - j0 - kPanel;
    if (left == 0) break;
    if (tid < left) {
      const int c = j0 + kPanel + tid;
      double x[kPanel];
#pragma unroll
      for (int j = 0; j < kPanel; ++j) x[j] = C[(j0 + j) * ld + c];
#pragma unroll
      for (int j = 0; j < kPanel; ++j) {
        x[j] *= Ri[(j0 + j) * ld + j0 + j];
#pragma unroll
        for (int i = j + 1; i < kPanel; ++i) x[i] = fma(-C[(j0 + j) * ld + j0 + i], x[j], x[i]);
        C[(j0 + j) * ld + c] = x[j];
      }
    }
    __syncthreads();
    for (int q = tid; q < left * left; q += kCholThreads) {
      const int i = j0 + kPanel + q / left, c = j0 + kPanel + q % left;
      if (c >= i) {
        double v = C[i * ld + c];
#pragma unroll
        for (int j = 0; j < kPanel; ++j) v = fma(-C[(j0 + j) * ld + i], C[(j0 + j) * ld + c], v);
        C[i * ld + c] = v;
      }
    }
    __syncthreads();
  }
  // R Rinv = I: column c from its own row upwards, a panel of rows at a time; lane i of eight has row i of the panel
  for (int c0 = warp * 4; c0 < rp; c0 += kCholThreads / 8) {
    const int c = c0 + (lane >> 3), i = lane & 7;
    for (int I = c / kPanel; I >= 0; --I) {
      // every lane of the warp walks the same panels: the four columns of a warp lie in one panel
      const int row = I * kPanel + i;
      double v = row == c ? 1.0 : 0.0;
      for (int k = (I + 1) * kPanel; k <= c; ++k) v = fma(-C[row * ld + k], Ri[k * ld + c], v);
      // back substitution within the panel
      double x = 0.0;
#pragma unroll
      for (int k = kPanel - 1; k >= 0; --k) {
        const double xk = __shfl_sync(0xFFFFFFFFu, v * Ri[row * ld + row], (lane & 24) + k);
        if (i == k) x = xk;
        if (i < k) v = fma(-C[row * ld + I * kPanel + k], xk, v);
      }
      __syncwarp();
      if (row <= c && row != c) Ri[row * ld + c] = x;
      __syncwarp();
    }
  }
  __syncthreads();
  for (int q = tid; q < r * r; q += kCholThreads) {
    const int row = q / r, col = q % r;
    if (col >= row) Cg[q] = C[row * ld + col];
    Rinvg[q] = Ri[row * ld + col];
  }
}
static cudaError_t cholesky_inverse(const double* part, int chunks, double* C, int r, double* Rinv, int* status, cudaStream_t s) {
  static OncePerDevice once;
  constexpr int kMost = 2 * kSharedR * chol_ld(kSharedR) * 8;
  const cudaError_t e = once.run([] { return cudaFuncSetAttribute(cholesky_inverse_panels_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost); });
  if (e != cudaSuccess) return e;
  if (r <= kSharedR)
    cholesky_inverse_panels_kernel<<<1, kCholThreads, 2 * (chol_ld(r) - 1) * chol_ld(r) * 8, s>>>(part, chunks, C, r, Rinv, status);
  else
    cholesky_inverse_kernel<<<1, 1024, 0, s>>>(part, chunks, C, r, Rinv, status);
  return cudaGetLastError();
}
// Out[m, c] = rowscale[m] * sum_j Y[m, j] T[j, c] for c < cols (T is [r, ldt]); fp64 in, OutT out, optionally
// written transposed (Out[c, m]).  One CTA = 32 rows and up to 64 columns; T's used columns are walked in tiles of 64.  Bound by the
// latency of its loads, so all of a step's operands (48 of the r inner positions) are requested together: 8.6 us for 4096 x 48
// against 15.8 with 64 rows and 16 positions.
constexpr int kTallRows = 32, kTallStep = 48;
template <typename OutT, bool TRANSPOSE_OUT>
__global__ void __launch_bounds__(256) tall_times_small_kernel(const double* __restrict__ Y, int m, int r, const double* __restrict__ T,
                                                               int ldt, int cols, const double* __restrict__ rowscale, int invert_scale,
                                                               OutT* __restrict__ Out) {
  __shared__ double s_y[kTallStep][kTallRows + 1], s_t[kTallStep][64];
  const int m0 = blockIdx.x * kTallRows, c0 = blockIdx.y * 64;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;      // columns tx, tx + 32 of rows 4 ty ..
  double acc[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[i][j] = 0.0;
  for (int j0 = 0; j0 < r; j0 += kTallStep) {
    const int n = min(kTallStep, r - j0);
    for (int q = threadIdx.x; q < kTallRows * kTallStep; q += 256) {
      const int jj = q % kTallStep, mi = q / kTallStep;
      s_y[jj][mi] = (m0 + mi < m && jj < n) ? Y[(size_t)(m0 + mi) * r + j0 + jj] : 0.0;
    }
    for (int q = threadIdx.x; q < kTallStep * 64; q += 256) {
      const int cc = q & 63, jj = q >> 6;
      s_t[jj][cc] = (jj < n && c0 + cc < cols) ? T[(size_t)(j0 + jj) * ldt + c0 + cc] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int jj = 0; jj < kTallStep; ++jj) {
      const double b0 = s_t[jj][tx], b1 = s_t[jj][tx + 32];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const double a = s_y[jj][ty * 4 + i];
        acc[i][0] = fma(a, b0, acc[i][0]);
        acc[i][1] = fma(a, b1, acc[i][1]);
      }
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
    for (int j = 0; j < 2; ++j) {
      const int c = c0 + tx + 32 * j;
      if (c < cols) {
        if (TRANSPOSE_OUT) Out[(size_t)c * m + row] = (OutT)(sc * acc[i][j]);
        else Out[(size_t)row * cols + c] = (OutT)(sc * acc[i][j]);
      }
    }
  }
}

// ---------------------------------------------------------------------------- small SVD (one CTA)
// The rotation that makes two columns orthogonal.
__device__ __forceinline__ void rotation(double alpha, double beta, double gamma, double& c, double& s) {
  const double zeta = (beta - alpha) / (2.0 * gamma), az = fabs(zeta);
  const double t = copysign(1.0 / (az + sqrt(fma(az, az, 1.0))), zeta);
  c = rsqrt(fma(t, t, 1.0));
  s = c * t;
}
// Right singular vectors and singular values of the r x r upper-triangular R (the Cholesky factor left in the upper
// triangle of C, row-major) by one-sided Jacobi: pairs of columns are rotated until all are mutually orthogonal,
// V collects the rotations.  A half warp per pair, the pairs of a step disjoint (round-robin tournament).  Mt, Vt: r x r
// scratch, column-major.  Out: Vs row-major [r][r] with the columns in falling order of singular value, sigma[r].
// Bound by its steps (r - 1 per sweep, one barrier each), in them by the fp64 pipe as much as by latency: half warps
// took 707 us at r = 48 to 408.  Both matrices sit in shared memory where they fit.
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
      for (int i0 = 2 * warp; i0 < n / 2; i0 += 64) {      // a half warp per pair: the scalars cost the fp64 pipe as much as a whole row
        const int i = i0 + (lane >> 4);
        int a = n - 1, b = t;
        if (i > 0) {
          a = t + i; b = t + n - 1 - i;
          if (a >= n - 1) a -= n - 1;
          if (b >= n - 1) b -= n - 1;
        }
        const bool live = i < n / 2 && a < r && b < r;
        const int p = live ? min(a, b) : 0, q = live ? max(a, b) : 0;
        double* mp = Mt + (size_t)p * r;
        double* mq = Mt + (size_t)q * r;
        double alpha = 0.0, beta = 0.0, gamma = 0.0;
        if (live)
          for (int row = lane & 15; row < r; row += 16) {
            const double x = mp[row], y = mq[row];
            alpha = fma(x, x, alpha); beta = fma(y, y, beta); gamma = fma(x, y, gamma);
          }
#pragma unroll
        for (int sft = 8; sft > 0; sft >>= 1) {
          alpha += __shfl_xor_sync(0xFFFFFFFFu, alpha, sft);
          beta += __shfl_xor_sync(0xFFFFFFFFu, beta, sft);
          gamma += __shfl_xor_sync(0xFFFFFFFFu, gamma, sft);
        }
        if (live && gamma * gamma > (tol * alpha) * (tol * beta)) {
          double c, s;
          rotation(alpha, beta, gamma, c, s);
          if (s != 0.0) {
            double* vp = Vt + (size_t)p * r;
            double* vq = Vt + (size_t)q * r;
            for (int row = lane & 15; row < r; row += 16) {
              const double x = mp[row], y = mq[row];
              mp[row] = c * x - s * y; mq[row] = s * x + c * y;
              const double u = vp[row], w = vq[row];
              vp[row] = c * u - s * w; vq[row] = s * u + c * w;
            }
            if ((lane & 15) == 0) s_rotated = 1;
          }
        }
        __syncwarp();
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

// Y = Q R with Q^T Q = I by Cholesky QR, `passes` times, with `other` as the second buffer; *out: where Q lies.  One pass leaves
// Q^T Q - I of the size rounding * cond(Y)^2, which is enough between two products of the iteration (what counts there is the
// space the columns span, and that they are far from dependent); a second one makes it orthonormal to rounding.
static cudaError_t orthonormalise(double* Y, double* other, int m, int r, int passes, double* gram_part, double* C, double* Rinv,
                                  int* status, double** out, cudaStream_t s) {
  using namespace fac;
  const int chunks = kGramChunks, rows_per_chunk = (m + chunks - 1) / chunks, rt = (r + 15) / 16;
  for (int pass = 0; pass < passes; ++pass) {
    gram_partial_kernel<<<dim3(rt, rt, chunks), 256, 0, s>>>(Y, m, r, rows_per_chunk, gram_part);
    const cudaError_t e = cholesky_inverse(gram_part, chunks, C, r, Rinv, status, s);
    if (e != cudaSuccess) return e;
    tall_times_small_kernel<double, false><<<dim3((m + kTallRows - 1) / kTallRows, (r + 63) / 64), 256, 0, s>>>(Y, m, r, Rinv, r, r, nullptr, 0, other);
    std::swap(Y, other);
  }
  *out = Y;
  return cudaGetLastError();
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

  LaunchScope scope(kFamPrepare, s, 18 + 8 * kIters);
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
  double* Q = nullptr;
  double* Z = nullptr;
  cudaError_t e = g_times<false>(G, K, N, T1, r, T0, s);                                 // Y = G Omega      [K, r]
  if (e != cudaSuccess) return e;
  if ((e = orthonormalise(T0, T1, K, r, 1, gram_part, C, Rinv, status, &Q, s)) != cudaSuccess) return e;   // Q in T1
  for (int it = 0; it < kIters; ++it) {
    if ((e = g_times<true>(G, K, N, Q, r, T0, s)) != cudaSuccess) return e;      // Z = G^T Q        [N, r]
    if ((e = orthonormalise(T0, Bt, N, r, 1, gram_part, C, Rinv, status, &Z, s)) != cudaSuccess) return e;   // Z in Bt
    if ((e = g_times<false>(G, K, N, Z, r, T0, s)) != cudaSuccess) return e;     // Y = G Z          [K, r]
    // Q in T1, after the last round in T0
    if ((e = orthonormalise(T0, T1, K, r, it + 1 < kIters ? 1 : 2, gram_part, C, Rinv, status, &Q, s)) != cudaSuccess) return e;
  }
  if ((e = g_times<true>(G, K, N, Q, r, Bt, s)) != cudaSuccess) return e;        // Bt = G^T Q       [N, r]
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
  tall_times_small_kernel<float, false><<<dim3((K + kTallRows - 1) / kTallRows, (k + 63) / 64), 256, 0, s>>>(Q, K, r, Vs, r, k, sc, 1, A);
  tall_times_small_kernel<float, true><<<dim3((N + kTallRows - 1) / kTallRows, (k + 63) / 64), 256, 0, s>>>(Bt, N, r, Vs, r, k, nullptr, 0, B);
  return cudaGetLastError();
}

}  // namespace lqer
