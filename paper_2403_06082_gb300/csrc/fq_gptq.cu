// Frame-domain GPTQ on the GPU (Algorithm 1, steps 2-4): the offline quantizer that turns the
// frame coefficients C = T_out W T_in^T into 2-bit codes while keeping the proxy loss
//     L(D_hat) = ||D C_prev - D_hat C_prev||_F^2 = tr((D - D_hat) H (D - D_hat)^T),
//     H = C_prev C_prev^T,   C_prev = T_in A_prev (calibration tokens in the frame domain)
// small (Sec. 3).  Everything runs in fp64: it is an offline step whose integer decisions
// (which level each coefficient rounds to, with the rounding errors of earlier columns fed into
// later ones) should not depend on the arithmetic's precision.
//
// Steps, in the order of the method:
//   1. optional clip of D to [mu - 2 sigma, mu + 2 sigma], mu and sigma over all of D;
//   2. each row's 2-bit grid, fixed before the iteration: zero = fp16(min), scale =
//      fp16((max - min) / 3) (1 when 0), and the diagonal de-noising gain P / (P + scale^2 / 12);
//   3. the damped Hessian H + damp mean(diag H) I and the upper factor U of its inverse,
//      H^-1 = U^T U.  With J the exchange matrix, J H J = L L^T (lower Cholesky) gives
//      H = (J L J)(J L J)^T, so U = (J L J)^-1 = J L^-1 J: one Cholesky and one triangular
//      inverse, no explicit inverse of H.  Both go by blocks of 32: a diagonal block is factored
//      and inverted in one CTA's shared memory, the rest is tiled products; the inverse doubles its
//      blocks (32, 64, ...), X_21 = -X_22 (L_21 X_11).  The panels multiply by reciprocals of
//      the pivots and of their roots.  Against extended precision (both emulated on the host), U of a
//      damped 160 x 160 Hessian is off by 1.2e-14 of its norm from 96 tokens and 2.6e-15 from 320; a
//      column-at-a-time recursion that divides by each pivot is off by 1.8e-14 and 4.6e-15;
//   4. the columns in blocks of 128: column j of a block is rounded to each row's grid, its
//      rounding error e = (w_j - q_hat_j) / U_jj is spread over the block's later columns
//      (w_k -= e U_jk), and after the block over all later columns at once (a product with
//      U's block rows).
// W is held transposed (column j of every row contiguous) so that consecutive rows are read and
// written coalesced.  Inside a block the update is one rounded multiply and one rounded subtract,
// as the plain recursion writes it.
//
// What bounds it: GB300's fp64 rate (about two multiply-adds per cycle and SM), so the products
// are cut into tiles small enough to spread evenly over all SMs, and the two serial recursions
// (the Cholesky's pivots, a row's 128 columns) keep their chains short.  Measured for
// 3392 x 848 coefficients and 1024 calibration tokens: 6.5 ms in all, of which the products 3.5 (at
// the fp64 pipe's rate), the column iteration 1.4, the Cholesky's panels 0.9, the inverse 0.6;
// with one Cholesky launch per column, one block per column of the inverse and the iteration
// in global memory it took 22.9 ms.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "fq_device.cuh"
#include "fq_internal.h"

namespace fq {
namespace {

constexpr int kBlockCols = 128;   // columns per block of the iteration
constexpr int kT = 256;           // threads per block of the simple kernels
constexpr int kMaxIn = 25600;     // the largest n_in taken

// ---- fp64 tiled product: C[m][n] = op(sum_k A(m, k) B(k, n)), A and B given by element strides;
// every element is one chain of fused multiply-adds in ascending k from zero.  32 x 32 tiles, 2 x
// 2 outputs per thread: at the fp64 rate a tile's shared-memory reads are far below its
// multiply-adds, and small tiles leave the last wave of blocks short.
constexpr int kG = 32, kGK = 16;
enum GemmOp : int { kSet = 0, kSub = 1, kNeg = 2 };        // C = sum, C - sum, -sum
enum GemmTri : int { kFull = 0, kALower = 1, kAUpper = 2 };  // A(m, k) = 0 for k > m, k < m

struct GemmShape {
  int64_t a_m, a_k, b_k, b_n, ldc;
  int M, N, K;
  int op, tri;
  int lower;                        // only tiles on or below the diagonal
  int mirror;                       // and their transposes are stored too
};

__device__ __forceinline__ void gemm_f64_tile(const double* __restrict__ A,
                                              const double* __restrict__ B,
                                              double* __restrict__ C, const GemmShape& g) {
  __shared__ double As[kGK][kG + 1];
  __shared__ double Bs[kGK][kG + 1];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int m0 = blockIdx.y * kG, n0 = blockIdx.x * kG;
  if (m0 >= g.M || n0 >= g.N || (g.lower && m0 < n0)) return;
  const int k_lo = g.tri == kAUpper ? m0 : 0;
  const int k_hi = g.tri == kALower ? min(g.K, m0 + kG) : g.K;
  // a thread's two elements of each operand slice, consecutive threads along the contiguous side
  int am[2], ak[2], bn[2], bk[2];
#pragma unroll
  for (int l = 0; l < 2; ++l) {
    const int t = threadIdx.x + 256 * l;
    am[l] = g.a_m == 1 ? t % kG : t / kGK;
    ak[l] = g.a_m == 1 ? t / kG : t % kGK;
    bn[l] = g.b_n == 1 ? t % kG : t / kGK;
    bk[l] = g.b_n == 1 ? t / kG : t % kGK;
  }
  double acc[2][2] = {}, ra[2], rb[2];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      ra[l] = (m0 + am[l] < g.M && k0 + ak[l] < k_hi)
                  ? A[(m0 + am[l]) * g.a_m + (k0 + ak[l]) * g.a_k] : 0.0;
      rb[l] = (n0 + bn[l] < g.N && k0 + bk[l] < k_hi)
                  ? B[(k0 + bk[l]) * g.b_k + (n0 + bn[l]) * g.b_n] : 0.0;
    }
  };
  fetch(k_lo);
  for (int k0 = k_lo; k0 < k_hi; k0 += kGK) {
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      As[ak[l]][am[l]] = ra[l];
      Bs[bk[l]][bn[l]] = rb[l];
    }
    __syncthreads();
    if (k0 + kGK < k_hi) fetch(k0 + kGK);
#pragma unroll
    for (int kk = 0; kk < kGK; ++kk) {
      const double a[2] = {As[kk][ty], As[kk][ty + 16]}, b[2] = {Bs[kk][tx], Bs[kk][tx + 16]};
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 2; ++q) acc[p][q] = fma(a[p], b[q], acc[p][q]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int gm = m0 + ty + 16 * p, gn = n0 + tx + 16 * q;
      if (gm < g.M && gn < g.N) {
        double* c = C + gm * g.ldc + gn;
        *c = g.op == kSub ? *c - acc[p][q] : (g.op == kNeg ? -acc[p][q] : acc[p][q]);
        if (g.mirror && m0 > n0) C[gn * g.ldc + gm] = acc[p][q];
      }
    }
}

__global__ void __launch_bounds__(256) gemm_f64_kernel(const double* __restrict__ A,
                                                       const double* __restrict__ B,
                                                       double* __restrict__ C, GemmShape g) {
  gemm_f64_tile(A, B, C, g);
}

cudaError_t gemm_f64(const double* A, const double* B, double* C, const GemmShape& g,
                     cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  const dim3 grid(static_cast<unsigned>(ceil_div(g.N, kG)), static_cast<unsigned>(ceil_div(g.M, kG)));
  gemm_f64_kernel<<<grid, 256, 0, s>>>(A, B, C, g);
  return cudaGetLastError();
}

// ---- mean and standard deviation over all of D, two passes, fixed order: kParts blocks sum
// grid-strided shares, then one block adds the partial sums in order.
constexpr int kParts = 512;

__global__ void __launch_bounds__(kT) partial_sum_kernel(const double* __restrict__ D, int64_t n,
                                                         const double* __restrict__ mom,
                                                         int deviations,
                                                         double* __restrict__ part) {
  __shared__ double red[kT];
  const double mu = deviations ? mom[0] : 0.0;
  double s = 0.0;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(kT) + threadIdx.x; i < n;
       i += static_cast<int64_t>(kParts) * kT) {
    const double d = D[i] - mu;
    s += deviations ? d * d : D[i];
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = kT / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// mom[0] = sum / n (first pass), mom[1] = sqrt(sum / n) (second pass)
__global__ void __launch_bounds__(kT) final_sum_kernel(const double* __restrict__ part, int64_t n,
                                                       int second, double* __restrict__ mom) {
  __shared__ double red[kT];
  double s = 0.0;
  for (int i = threadIdx.x; i < kParts; i += kT) s += part[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = kT / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double m = red[0] / static_cast<double>(n);
    mom[second] = second ? sqrt(m) : m;
  }
}

// WT[j][i] = clip(D[i][j]) (or D[i][j]): the working copy, transposed
__global__ void clip_transpose_kernel(const double* __restrict__ D, int n_out, int n_in,
                                      const double* __restrict__ mom, int clip,
                                      double* __restrict__ WT) {
  __shared__ double tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  double lo = -INFINITY, hi = INFINITY;
  if (clip) {
    lo = mom[0] - 2.0 * mom[1];
    hi = mom[0] + 2.0 * mom[1];
  }
  for (int dy = threadIdx.y; dy < 32; dy += 8) {
    const int r = r0 + dy, c = c0 + threadIdx.x;
    if (r < n_out && c < n_in) tile[dy][threadIdx.x] = fmin(fmax(D[static_cast<int64_t>(r) * n_in + c], lo), hi);
  }
  __syncthreads();
  for (int dy = threadIdx.y; dy < 32; dy += 8) {
    const int c = c0 + dy, r = r0 + threadIdx.x;
    if (c < n_in && r < n_out) WT[static_cast<int64_t>(c) * n_out + r] = tile[threadIdx.x][dy];
  }
}

// One block per row i (reading column i of WT): min, max, mean square -> fp16 zero and scale,
// the de-noising gain.
__global__ void __launch_bounds__(kT) row_grid_kernel(const double* __restrict__ WT, int n_out,
                                                      int n_in, __half* __restrict__ scale,
                                                      __half* __restrict__ zero,
                                                      double* __restrict__ s64,
                                                      double* __restrict__ z64,
                                                      float* __restrict__ gamma) {
  const int i = blockIdx.x;
  __shared__ double smn[kT], smx[kT], ssq[kT];
  double mn = INFINITY, mx = -INFINITY, sq = 0.0;
  for (int j = threadIdx.x; j < n_in; j += kT) {
    const double v = WT[static_cast<int64_t>(j) * n_out + i];
    mn = fmin(mn, v);
    mx = fmax(mx, v);
    sq += v * v;
  }
  smn[threadIdx.x] = mn;
  smx[threadIdx.x] = mx;
  ssq[threadIdx.x] = sq;
  __syncthreads();
  for (int w = kT / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      smn[threadIdx.x] = fmin(smn[threadIdx.x], smn[threadIdx.x + w]);
      smx[threadIdx.x] = fmax(smx[threadIdx.x], smx[threadIdx.x + w]);
      ssq[threadIdx.x] += ssq[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const __half hz = __double2half(smn[0]);
    __half hs = __double2half((smx[0] - smn[0]) / 3.0);
    if (__half2float(hs) == 0.f) hs = __float2half(1.f);
    zero[i] = hz;
    scale[i] = hs;
    const double sc = static_cast<double>(__half2float(hs));
    s64[i] = sc;
    z64[i] = static_cast<double>(__half2float(hz));
    if (gamma) {
      const double P = ssq[0] / n_in;
      gamma[i] = static_cast<float>(P / (P + sc * sc / 12.0));
    }
  }
}

// K = J (H + damp mean(diag H) I) J, lower triangle used
__global__ void damp_reverse_kernel(const double* __restrict__ H, int n, double damp,
                                    double* __restrict__ K) {
  __shared__ double red[kT];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += kT) s += H[static_cast<int64_t>(i) * n + i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = kT / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  const double add = damp * (red[0] / n);
  const int64_t total = static_cast<int64_t>(n) * n;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(kT) + threadIdx.x; e < total;
       e += static_cast<int64_t>(gridDim.x) * kT) {
    const int i = static_cast<int>(e / n), j = static_cast<int>(e % n);
    double v = H[static_cast<int64_t>(n - 1 - i) * n + (n - 1 - j)];
    if (i == j) v += add;
    K[e] = v;
  }
}

// ---- blocked right-looking Cholesky of K (lower triangle) with the inverses of its diagonal blocks
constexpr int kNB = 32;           // block: a warp's lanes

// Block column b .. b + nb - 1: factor the diagonal block, K_bb = L L^T, and solve L Y = B by forward
// substitution, a column of B per lane: CTA 0 for B = I, the inverse of L, which goes to X; CTA c > 0
// for B = the transpose of 32 rows below the block, K_ib <- K_ib L^-T in place.  Every CTA factors
// the diagonal block for itself, which saves a launch and its latency per block; nothing rewrites
// the diagonal block.  The factorization is a chain of 32 pivots: the warp that owns column j + 1
// updates it first and divides by its pivot while the other warps update the columns after it.
// Loops stay rolled: unrolled code runs once per launch and waits for its instructions.
__global__ void __launch_bounds__(256) chol_panel_kernel(double* __restrict__ K, int n, int b,
                                                         int nb, double* __restrict__ X,
                                                         int32_t* __restrict__ status) {
  __shared__ double D[kNB][kNB + 1];      // the block, then its factor
  __shared__ double Y[kNB][kNB + 1];      // the right-hand sides, a column per lane
  __shared__ double inv_s[kNB];
  __shared__ double m_s[2][kNB];          // column j over its pivot, for the step at hand and the next
  const int tid = threadIdx.x, lane = tid & 31, wr = tid >> 5;
  const bool inverse = blockIdx.x == 0;
  const int r0 = b + nb + (static_cast<int>(blockIdx.x) - 1) * kNB;   // this CTA's rows
  for (int e = tid; e < kNB * kNB; e += 256) {
    const int i = e / kNB, j = e % kNB;
    // past nb: the identity, so that a short last block needs no case of its own
    D[i][j] = i < nb ? (j <= i ? K[static_cast<int64_t>(b + i) * n + b + j] : 0.0)
                     : (i == j ? 1.0 : 0.0);
    if (inverse)
      Y[i][j] = i == j ? 1.0 : 0.0;
    else
      Y[j][i] = (r0 + i < n && j < nb) ? K[static_cast<int64_t>(r0 + i) * n + b + j] : 0.0;
  }
  __syncthreads();
  // right-looking, unscaled, a row per lane: D_ik -= (D_ij / piv_j) D_kj, column k by warp k mod 8
  if (wr == 0) m_s[0][lane] = D[lane][0] * (1.0 / D[0][0]);
  __syncthreads();
  for (int j = 0; j < kNB; ++j) {
    const double m = m_s[j & 1][lane];
    const int first = j + 1 + ((wr - (j + 1)) & 7);            // this warp's first column after j
    for (int k = first; k < kNB; k += 8) {
      if (lane >= k) D[lane][k] = fma(-m, D[k][j], D[lane][k]);
      if (k == j + 1) {
        __syncwarp();
        m_s[k & 1][lane] = D[lane][k] * (1.0 / D[k][k]);
      }
    }
    __syncthreads();
  }
  if (tid < 32) {
    // a pivot that is not positive: the damped H was not positive definite
    const double piv = D[lane][lane];
    if (inverse && !(piv > 0.0)) report(status, FQ_ERR_DEVICE_CHECK);
    inv_s[lane] = 1.0 / sqrt(piv);
  }
  __syncthreads();
  // columns scaled: L_ij = D_ij / sqrt(piv_j)
  for (int i = wr; i < kNB; i += 8)
    if (lane <= i) D[i][lane] *= inv_s[lane];
  __syncthreads();
  // x_k = y_k / L_kk, then y_i -= L_ik x_k for every later row i, the rows split over the warps
  // (y_k itself is left to the end, so that a row costs one barrier)
  for (int k = 0; k < kNB; ++k) {
    const double x = Y[k][lane] * inv_s[k];
    for (int i = wr; i < kNB; i += 8)
      if (i > k) Y[i][lane] = fma(-D[i][k], x, Y[i][lane]);
    __syncthreads();
  }
  for (int e = tid; e < kNB * kNB; e += 256) {
    const int i = e / kNB, j = e % kNB;
    if (inverse) {
      if (i < nb && j < nb)
        X[static_cast<int64_t>(b + i) * n + b + j] = j <= i ? Y[i][j] * inv_s[i] : 0.0;
    } else if (r0 + i < n && j < nb) {
      K[static_cast<int64_t>(r0 + i) * n + b + j] = Y[j][i] * inv_s[j];
    }
  }
}

// One doubling of the inverse for all pairs of s x s blocks (blockIdx.z = pair): T = L_21 X_11, kept
// transposed in the upper triangle of L's matrix, which nothing else uses (step 0), then
// X_21 = -X_22 T (step 1).
__global__ void __launch_bounds__(256) tri_double_kernel(double* __restrict__ L,
                                                         double* __restrict__ X, int n, int s,
                                                         int step) {
  const int o = 2 * s * blockIdx.z, rows = min(s, n - o - s);   // rows of the lower block
  if (rows <= 0) return;
  const int64_t at = static_cast<int64_t>(o) * n + o, below = static_cast<int64_t>(s) * n;
  double* Tt = L + at + s;                                      // Tt[c][r] = T[r][c], s x rows
  const int64_t N = n;
  if (step == 0)   // Tt[c][r] = sum_{k >= c} X_11[k][c] L_21[r][k]
    gemm_f64_tile(X + at, L + at + below, Tt,
                  GemmShape{1, N, 1, N, N, s, rows, s, kSet, kAUpper, 0, 0});
  else             // X_21[r][c] = -sum_{k <= r} X_22[r][k] Tt[c][k]
    gemm_f64_tile(X + at + below + s, Tt, X + at + below,
                  GemmShape{N, 1, 1, N, N, rows, s, rows, kNeg, kALower, 0, 0});
}

// U = J X J in place: the n^2 entries in reverse order.
__global__ void reverse_kernel(double* __restrict__ X, int64_t total) {
  for (int64_t e = blockIdx.x * static_cast<int64_t>(kT) + threadIdx.x; e < total / 2;
       e += static_cast<int64_t>(gridDim.x) * kT) {
    const double lo = X[e], hi = X[total - 1 - e];
    X[e] = hi;
    X[total - 1 - e] = lo;
  }
}

// Block b0 .. b1-1 of the iteration.  A CTA keeps `rows` rows of the block's columns and the
// block of U in shared memory.  Warp 0 carries the serial chain, a row per lane: column j with the
// last error e_(j-1) applied, rounded, its error e_j.  Meanwhile the other warps apply e_(j-1) to
// the columns after j, so every element takes the errors in ascending order, and the chain of
// one column costs one barrier.
constexpr int kIterRows = 32;     // most rows per CTA
constexpr int kIterSmem = (kBlockCols * kBlockCols + kIterRows * (kBlockCols + 1) + 2 * kIterRows) * 8;

__global__ void __launch_bounds__(kT) gptq_block_kernel(const double* __restrict__ WT, int n_out,
                                                        int n_in, const double* __restrict__ U,
                                                        const double* __restrict__ s64,
                                                        const double* __restrict__ z64, int b0,
                                                        int b1, int rows,
                                                        uint8_t* __restrict__ codesT,
                                                        double* __restrict__ ET) {
  extern __shared__ double iter_smem[];
  double(*Us)[kBlockCols] = reinterpret_cast<double(*)[kBlockCols]>(iter_smem);
  double(*W)[kBlockCols + 1] =
      reinterpret_cast<double(*)[kBlockCols + 1]>(iter_smem + kBlockCols * kBlockCols);
  double* E = iter_smem + kBlockCols * kBlockCols + kIterRows * (kBlockCols + 1);   // [2][rows]
  const int nb = b1 - b0, i0 = blockIdx.x * rows, nr = min(rows, n_out - i0);
  const int tid = threadIdx.x;
  for (int e = tid; e < nb * nb; e += kT) {
    const int j = e / nb, k = e % nb;
    if (k >= j) Us[j][k] = U[static_cast<int64_t>(b0 + j) * n_in + b0 + k];
  }
  for (int e = tid; e < nb * nr; e += kT) {
    const int j = e / nr, r = e % nr;
    W[r][j] = WT[static_cast<int64_t>(b0 + j) * n_out + i0 + r];
  }
  __syncthreads();
  const bool chain = tid < 32 && tid < nr;
  const int i = i0 + (chain ? tid : 0);
  const double s = s64[i], z = z64[i];
  double e_prev = 0.0;
  // the other warps: row r, columns in steps of ncg
  const int t = tid - 32, r = t >= 0 ? t % nr : 0, cg = t >= 0 ? t / nr : 0, ncg = (kT - 32) / nr;
  const bool bulk = t >= 0 && cg < ncg;
  for (int j = 0; j < nb; ++j) {
    if (chain) {
      double w = W[tid][j];
      if (j > 0) w = __dsub_rn(w, __dmul_rn(e_prev, Us[j - 1][j]));
      const double q = fmin(fmax(rint((w - z) / s), 0.0), 3.0);
      const double e = (w - __dadd_rn(__dmul_rn(s, q), z)) / Us[j][j];
      E[(j & 1) * kIterRows + tid] = e;
      e_prev = e;
      codesT[static_cast<int64_t>(b0 + j) * n_out + i] = static_cast<uint8_t>(q);
      ET[static_cast<int64_t>(j) * n_out + i] = e;
    } else if (bulk && j > 0) {
      const double e = E[((j - 1) & 1) * kIterRows + r];
      for (int k = j + 1 + cg; k < nb; k += ncg)
        W[r][k] = __dsub_rn(W[r][k], __dmul_rn(e, Us[j - 1][k]));
    }
    __syncthreads();
  }
}

// codes[i][j] = codesT[j][i]
__global__ void transpose_u8_kernel(const uint8_t* __restrict__ in, int rows, int cols,
                                    uint8_t* __restrict__ out) {
  __shared__ uint8_t tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int dy = threadIdx.y; dy < 32; dy += 8) {
    const int r = r0 + dy, c = c0 + threadIdx.x;
    if (r < rows && c < cols) tile[dy][threadIdx.x] = in[static_cast<int64_t>(r) * cols + c];
  }
  __syncthreads();
  for (int dy = threadIdx.y; dy < 32; dy += 8) {
    const int c = c0 + dy, r = r0 + threadIdx.x;
    if (c < cols && r < rows) out[static_cast<int64_t>(c) * rows + r] = tile[threadIdx.x][dy];
  }
}

struct GptqWs {
  size_t status, mom, part, s64, z64, WT, K, U, ET, codesT, total;
};

GptqWs gptq_ws(int n_out, int n_in) {
  GptqWs L{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off += round_up(static_cast<int64_t>(bytes), 256);
    return at;
  };
  L.status = take(4);
  L.mom = take(2 * 8);
  L.part = take(kParts * 8);
  L.s64 = take(static_cast<size_t>(n_out) * 8);
  L.z64 = take(static_cast<size_t>(n_out) * 8);
  L.WT = take(static_cast<size_t>(n_out) * n_in * 8);
  L.K = take(static_cast<size_t>(n_in) * n_in * 8);
  L.U = take(static_cast<size_t>(n_in) * n_in * 8);
  L.ET = take(static_cast<size_t>(n_out) * kBlockCols * 8);
  L.codesT = take(static_cast<size_t>(n_out) * n_in);
  L.total = off;
  return L;
}

unsigned grid_cap(int64_t total) {
  return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(ceil_div(total, kT), 4096)));
}

bool a8(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 7u) == 0; }

}  // namespace
}  // namespace fq

using namespace fq;

extern "C" {

fq_status fq_gptq_hessian(const double* Z, int N, int n_in, double* H, fq_stream_t stream) {
  if (!Z || !H || N <= 0 || n_in <= 0) return FQ_ERR_INVALID_ARG;
  if (!a8(Z) || !a8(H)) return FQ_ERR_ALIGNMENT;
  // H[i][j] = sum_t Z[t][i] Z[t][j]: A(i, t) = Z[t n_in + i], B(t, j) = Z[t n_in + j]
  // (symmetric: the same chains of multiply-adds, so half of the tiles are computed)
  const int64_t ld = n_in;
  return gemm_f64(Z, Z, H, GemmShape{1, ld, ld, 1, ld, n_in, n_in, N, kSet, kFull, 1, 1},
                  reinterpret_cast<cudaStream_t>(stream)) == cudaSuccess
             ? FQ_OK
             : FQ_ERR_CUDA;
}

size_t fq_gptq_workspace_bytes(int n_out, int n_in) {
  if (n_out <= 0 || n_in <= 0) return 0;
  return gptq_ws(n_out, n_in).total;
}

fq_status fq_quantize_gptq(const double* C, int n_out, int n_in, const double* H, double damp,
                           int clip, uint8_t* codes, uint16_t* scale, uint16_t* zero,
                           float* gamma, void* ws, size_t ws_bytes, fq_stream_t stream) {
  if (!C || !H || !codes || !scale || !zero || n_out <= 0 || n_in <= 0 || !(damp >= 0.0))
    return FQ_ERR_INVALID_ARG;
  if (!a8(C) || !a8(H) || (reinterpret_cast<uintptr_t>(scale) & 1u) ||
      (reinterpret_cast<uintptr_t>(zero) & 1u) || (gamma && (reinterpret_cast<uintptr_t>(gamma) & 3u)))
    return FQ_ERR_ALIGNMENT;
  if (!ws) return FQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return FQ_ERR_ALIGNMENT;
  const GptqWs L = gptq_ws(n_out, n_in);
  if (ws_bytes < L.total) return FQ_ERR_WORKSPACE;
  if (n_in > kMaxIn) return FQ_ERR_UNSUPPORTED;
  auto s = reinterpret_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  auto* status = reinterpret_cast<int32_t*>(w + L.status);
  auto* mom = reinterpret_cast<double*>(w + L.mom);
  auto* s64 = reinterpret_cast<double*>(w + L.s64);
  auto* z64 = reinterpret_cast<double*>(w + L.z64);
  auto* WT = reinterpret_cast<double*>(w + L.WT);
  auto* K = reinterpret_cast<double*>(w + L.K);
  auto* U = reinterpret_cast<double*>(w + L.U);
  auto* ET = reinterpret_cast<double*>(w + L.ET);
  auto* codesT = reinterpret_cast<uint8_t*>(w + L.codesT);
  const int64_t nD = static_cast<int64_t>(n_out) * n_in;
  const int64_t nH = static_cast<int64_t>(n_in) * n_in;
  if (cudaMemsetAsync(status, 0, 4, s) != cudaSuccess) return FQ_ERR_CUDA;
  // 1. clip (Algorithm 1, steps 2-3) into the transposed working copy
  auto* part = reinterpret_cast<double*>(w + L.part);
  if (clip) {
    partial_sum_kernel<<<kParts, kT, 0, s>>>(C, nD, mom, 0, part);
    final_sum_kernel<<<1, kT, 0, s>>>(part, nD, 0, mom);
    partial_sum_kernel<<<kParts, kT, 0, s>>>(C, nD, mom, 1, part);
    final_sum_kernel<<<1, kT, 0, s>>>(part, nD, 1, mom);
  }
  clip_transpose_kernel<<<dim3(static_cast<unsigned>(ceil_div(n_in, 32)),
                               static_cast<unsigned>(ceil_div(n_out, 32))),
                          dim3(32, 8), 0, s>>>(C, n_out, n_in, mom, clip, WT);
  // 2. each row's grid and gain
  row_grid_kernel<<<static_cast<unsigned>(n_out), kT, 0, s>>>(
      WT, n_out, n_in, reinterpret_cast<__half*>(scale), reinterpret_cast<__half*>(zero), s64,
      z64, gamma);
  // 3. U with H^-1 = U^T U
  damp_reverse_kernel<<<grid_cap(nH), kT, 0, s>>>(H, n_in, damp, K);
  if (cudaMemsetAsync(U, 0, static_cast<size_t>(nH) * 8, s) != cudaSuccess) return FQ_ERR_CUDA;
  const int64_t ld = n_in;
  for (int b = 0; b < n_in; b += kNB) {
    const int nb = std::min(kNB, n_in - b), below = n_in - b - nb;
    chol_panel_kernel<<<static_cast<unsigned>(1 + ceil_div(below, kNB)), 256, 0, s>>>(
        K, n_in, b, nb, U, status);
    // K_ik -= L_ib L_kb^T for the rows and columns below the block, lower triangle
    const double* P = K + (b + nb) * ld + b;
    if (gemm_f64(P, P, K + (b + nb) * ld + b + nb,
                 GemmShape{ld, 1, 1, ld, ld, below, below, nb, kSub, kFull, 1, 0},
                 s) != cudaSuccess)
      return FQ_ERR_CUDA;
  }
  for (int w32 = kNB; w32 < n_in; w32 *= 2) {
    const dim3 g(static_cast<unsigned>(w32 / kG), static_cast<unsigned>(w32 / kG),
                 static_cast<unsigned>(ceil_div(n_in, 2 * w32)));
    tri_double_kernel<<<g, 256, 0, s>>>(K, U, n_in, w32, 0);
    tri_double_kernel<<<g, 256, 0, s>>>(K, U, n_in, w32, 1);
  }
  reverse_kernel<<<grid_cap(nH / 2), kT, 0, s>>>(U, nH);
  // 4. the columns, block by block; the rows spread evenly over the SMs
  if (cudaFuncSetAttribute(gptq_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           kIterSmem) != cudaSuccess)
    return FQ_ERR_CUDA;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return FQ_ERR_CUDA;
  const int64_t waves = ceil_div(n_out, static_cast<int64_t>(kIterRows) * sms);
  const int rows = static_cast<int>(std::max<int64_t>(1, ceil_div(n_out, waves * sms)));
  for (int b0 = 0; b0 < n_in; b0 += kBlockCols) {
    const int b1 = std::min(n_in, b0 + kBlockCols);
    gptq_block_kernel<<<static_cast<unsigned>(ceil_div(n_out, rows)), kT, kIterSmem, s>>>(
        WT, n_out, n_in, U, s64, z64, b0, b1, rows, codesT, ET);
    // WT[k][i] -= sum_jj U[b0 + jj][k] ET[jj][i] for k >= b1
    if (gemm_f64(U + b0 * ld + b1, ET, WT + static_cast<int64_t>(b1) * n_out,
                 GemmShape{1, ld, n_out, 1, n_out, n_in - b1, n_out, b1 - b0, kSub, kFull, 0, 0},
                 s) != cudaSuccess)
      return FQ_ERR_CUDA;
  }
  transpose_u8_kernel<<<dim3(static_cast<unsigned>(ceil_div(n_out, 32)),
                             static_cast<unsigned>(ceil_div(n_in, 32))),
                        dim3(32, 8), 0, s>>>(codesT, n_in, n_out, codes);
  if (cudaGetLastError() != cudaSuccess) return FQ_ERR_CUDA;
  // the status word reports a Hessian that was not positive definite after damping
  int32_t st = 0;
  if (cudaMemcpyAsync(&st, status, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return FQ_ERR_CUDA;
  return st ? FQ_ERR_DEVICE_CHECK : FQ_OK;
}

}  // extern "C"
