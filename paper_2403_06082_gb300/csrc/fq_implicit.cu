// Forward pass with frames in structured form (the decode path, M <= 64 tokens).
//
// With d a multiple of rho, the un-rotated analysis operator T_u of the (k, rho, d) frame is
// block-diagonal (Appendix J): run j = 0 .. rho/2 - 1 covers the complex coordinates
// c = j w .. (j+1) w - 1 (w = d / rho; complex coordinate c is real coordinates 2c, 2c + 1), and
// its k frame vectors are the realified rows of exp(2 pi i k_i c / k) / sqrt(k).  The rotated
// frame is T = T_u R^T, R = Pi (Q_a kron Q_b) D (Appendix K), so
//     z = T_u (R^T x),        y = R (T_u^T u).
//
// One forward is three kernels chained with programmatic dependent launch:
//   rotate<analysis>   v = R_in^T x   (bf16)
//   the fused decode kernel with block-sparse frame operands: z = T_u,in v, the 2-bit code
//                      product, s = T_u,out^T u, all on the tensor cores (its analysis and
//                      synthesis read only the K blocks of each row tile's runs, stored as
//                      contiguous pre-swizzled 16 KiB tiles: about 1/8 of the dense operator
//                      for rho = 16)
//   rotate<synthesis>  y = R_out s   (bf16)
// Without a rotation the fused kernel reads x and writes y itself.  The rotations are two small
// products per token on CUDA cores (a x a and b x b with a b = d).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <set>
#include <vector>

#include "fq_device.cuh"
#include "fq_internal.h"

namespace fq {
namespace {


// ------------------------------------------------------------------------------ rotations
// C CTAs take one token's a x b block, each a range of the rows of Y; bf16 in and out, fp32 between.
//   analysis:  V = Pi^T x (V[perm[i]] = x_i), Y = Q_a^T V Q_b, out = D vec(Y)    A = Q_a^T, B = Q_b
//   synthesis: V = D s, Y = Q_a V Q_b^T, out = Pi vec(Y) (out[iperm[e]] = vec(Y)_e) A = Q_a, B = Q_b^T
// A CTA reads the whole token, in order, and permutes it on its way into shared memory: a gather of
// 2-byte entries from global memory costs a sector each, ten times the conflicts of the scatter into
// shared memory.  T1 = A V for its rows and Y = T1 B follow without the other CTAs, 4 rows x 2 columns
// per thread, the row values of a reduction index as one 16-byte read (A is read transposed).
// What bounds it is latency: a token is two products of a few million multiply-adds, and code that
// runs once per launch waits for its instructions, so the loops are unrolled little.  The CTA's rows of
// A and all of B do not depend on the previous kernel and are staged in shared memory before the
// wait for the input; a factor that does not fit is read from L2.
// Measured, us per call (a CTA per eight rows that staged B in chunks; a cluster per token that split
// the gather and exchanged T1; this form): 2048 x 2048 at 4 tokens 23.1, 27.3, 22.9, at 32 tokens
// 31.1, 32.7, 27.6; two 4096 to 11008 layers at 16 tokens 88, 82, 70; three 11008 to 4096 layers at 64
// tokens 266, 158, 140; 28672 to 4096 at one token (B, 200 KB, read from L2) 99, 167, 103.
constexpr int kRotThreads = 256;
constexpr size_t kMaxSmem = 227 * 1024;

// One launch rotates the tokens of up to FQ_MAX_GROUP layers (blockIdx.z = layer).
struct RotLayer {
  const __nv_bfloat16* in;
  __nv_bfloat16* out;
  int a, b;
  int bp;                 // row stride of V and of the staged B: b rounded up to 2
  int rc;                 // rows of Y per CTA, a multiple of 4, and T1t's row stride
  int stage_a, stage_b;   // (where not both factors of every layer are staged whole)
  int wide;               // At, B, perm and signs are 16-byte aligned (as fq_frame_implicit lays them)
  const float* At;        // A^T, a x a row-major: At[i][r] = A[r][i]
  const float* B;         // b x b row-major
  const int32_t* perm;
  const int32_t* iperm;
  const float* signs;
};
struct RotBatch {
  RotLayer L[FQ_MAX_GROUP];
};

template <int kBytes>
__device__ __forceinline__ void cp_async(float* smem_dst, const float* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(smem_dst)), "l"(gsrc),
               "n"(kBytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// `cols` columns of an n x n factor (row-major) into shared memory with row stride np, asynchronously:
// one copy when they are whole rows without padding, else a warp per row, in the widest pieces that
// the alignment allows (n, cols and the first column are multiples of them; `wide`: src's base is 16-byte
// aligned).  Nothing is written past the last column (such entries only reach results that are dropped).
__device__ __forceinline__ void stage_factor(float* dst, const float* __restrict__ src, int n,
                                             int cols, int np, bool wide, int tid) {
  if (wide && n % 4 == 0 && cols == n) {       // np == n
    for (int i = tid; i < n * n / 4; i += kRotThreads) cp_async<16>(dst + 4 * i, src + 4 * i);
    return;
  }
  const int lane = tid & 31;
  for (int r = tid >> 5; r < n; r += kRotThreads / 32) {
    const float* from = src + static_cast<int64_t>(r) * n;
    float* to = dst + r * np;
    if (wide && n % 2 == 0)
      for (int i = 2 * lane; i < cols; i += 64) cp_async<8>(to + i, from + i);
    else
      for (int i = lane; i < cols; i += 32) cp_async<4>(to + i, from + i);
  }
}

// acc[row][col] += sum_k rows4(k)[row] * cols2(k)[col]
template <int kUnroll, typename Rows, typename Cols>
__device__ __forceinline__ void rot_product(float (&acc)[4][2], int n, Rows rows4, Cols cols2) {
#pragma unroll kUnroll
  for (int k = 0; k < n; ++k) {
    const float4 u = rows4(k);
    const float2 v = cols2(k);
    acc[0][0] = fmaf(u.x, v.x, acc[0][0]);
    acc[0][1] = fmaf(u.x, v.y, acc[0][1]);
    acc[1][0] = fmaf(u.y, v.x, acc[1][0]);
    acc[1][1] = fmaf(u.y, v.y, acc[1][1]);
    acc[2][0] = fmaf(u.z, v.x, acc[2][0]);
    acc[2][1] = fmaf(u.z, v.y, acc[2][1]);
    acc[3][0] = fmaf(u.w, v.x, acc[3][0]);
    acc[3][1] = fmaf(u.w, v.y, acc[3][1]);
  }
}

// kStaged: both factors of every layer of the launch are in shared memory, all of A, and their arrays
// are wide.  Otherwise each may or may not be, and of A only the CTA's columns of A^T.
template <bool kSynth, bool kStaged>
__global__ void __launch_bounds__(kRotThreads) rotate_kernel(const __grid_constant__ RotBatch rb) {
  const RotLayer& ly = rb.L[blockIdx.z];
  const int a = ly.a, b = ly.b, bp = ly.bp, rc = ly.rc;
  const int tid = threadIdx.x;
  const int r0 = min(a, static_cast<int>(blockIdx.x) * rc), nr = min(rc, a - r0);   // its rows
  const bool wide = kStaged || ly.wide;
  const int al = kStaged ? (a + 3) & ~3 : rc, a0 = kStaged ? r0 : 0;   // As's row stride, and r0 in it
  extern __shared__ float4 rot_smem4[];
  float* T1t = reinterpret_cast<float*>(rot_smem4);   // [b][rc]: T1t[k][r] = T1[r0 + r][k]
  float* As = T1t + b * rc;                           // [a][al]: As[k][a0 + r] = A[r0 + r][k]
  float* V = As + (kStaged || ly.stage_a ? a * al : 0);   // [a][bp]
  float* Bs = V + a * bp + ((a * bp) & 2);            // [b][bp], 16-byte aligned
  pdl_launch_dependents();
  if (kStaged)
    stage_factor(As, ly.At, a, a, al, wide, tid);
  else if (ly.stage_a)
    stage_factor(As, ly.At + r0, a, nr, al, wide, tid);
  if (kStaged || ly.stage_b) stage_factor(Bs, ly.B, b, b, bp, wide, tid);
  cp_async_commit();
  pdl_wait();
  const int64_t tok = static_cast<int64_t>(blockIdx.y) * a * b;
  // four entries of the token at a time (a b is a multiple of 8)
  const uint2* in = reinterpret_cast<const uint2*>(ly.in + tok);
  const float* side = kSynth ? ly.signs : reinterpret_cast<const float*>(ly.perm);
#pragma unroll 4
  for (int i = tid; i < a * b / 4; i += kRotThreads) {
    const uint2 w = in[i];
    const float4 h = wide ? reinterpret_cast<const float4*>(side)[i]
                          : make_float4(side[4 * i], side[4 * i + 1], side[4 * i + 2], side[4 * i + 3]);
    const float x[4] = {__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                        __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u)};
    const float sv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int e = kSynth ? 4 * i + j : __float_as_int(sv[j]);
      V[bp == b ? e : e + e / b] = kSynth ? sv[j] * x[j] : x[j];
    }
  }
  cp_async_wait_all();
  __syncthreads();
  // T1 = A V, then Y = T1 B, rows r0 .. r0 + nr - 1; task: 4 rows x 2 columns
  const int pairs = (b + 1) / 2, tasks = (nr + 3) / 4 * pairs;
  for (int t = tid; t < tasks; t += kRotThreads) {
    const int r = t / pairs * 4, c = t % pairs * 2;
    float acc[4][2] = {};
    const auto cols = [&](int k) { return *reinterpret_cast<const float2*>(V + k * bp + c); };
    if (kStaged || ly.stage_a) {
      rot_product<4>(acc, a, [&](int k) {
        return *reinterpret_cast<const float4*>(As + k * al + a0 + r);
      }, cols);
    } else {
      rot_product<8>(acc, a, [&](int k) {
        const float* p = ly.At + static_cast<int64_t>(k) * a + r0 + r;
        return make_float4(p[0], r + 1 < nr ? p[1] : 0.f, r + 2 < nr ? p[2] : 0.f,
                           r + 3 < nr ? p[3] : 0.f);
      }, cols);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)                  // (rows past nr fall into the padding)
      if (c + q < b)
        *reinterpret_cast<float4*>(T1t + (c + q) * rc + r) =
            make_float4(acc[0][q], acc[1][q], acc[2][q], acc[3][q]);
  }
  __syncthreads();
  __nv_bfloat16* out = ly.out + tok;
  for (int t = tid; t < tasks; t += kRotThreads) {
    const int r = t / pairs * 4, c = t % pairs * 2;
    float acc[4][2] = {};
    // where the results go (or their signs), requested before the product
    int dest[4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int o = (r0 + min(r + j, nr - 1)) * b + min(c + q, b - 1);
        dest[j][q] = kSynth ? ly.iperm[o] : __float_as_int(ly.signs[o]);
      }
    const auto rows = [&](int k) { return *reinterpret_cast<const float4*>(T1t + k * rc + r); };
    if (kStaged || ly.stage_b) {
      rot_product<4>(acc, b, rows,
                     [&](int k) { return *reinterpret_cast<const float2*>(Bs + k * bp + c); });
    } else if (wide && bp == b) {                // (many loads in flight for their latency)
      rot_product<32>(acc, b, rows, [&](int k) {
        return __ldg(reinterpret_cast<const float2*>(ly.B + static_cast<int64_t>(k) * b + c));
      });
    } else {
      rot_product<8>(acc, b, rows, [&](int k) {
        const float* p = ly.B + static_cast<int64_t>(k) * b + c;
        return make_float2(p[0], c + 1 < b ? p[1] : 0.f);
      });
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (r + j >= nr || c + q >= b) continue;
        if (kSynth)
          out[dest[j][q]] = __float2bfloat16_rn(acc[j][q]);
        else
          out[(r0 + r + j) * b + c + q] =
              __float2bfloat16_rn(__int_as_float(dest[j][q]) * acc[j][q]);
      }
  }
}

// ------------------------------------------------------------------------------ host side
constexpr int kTR = 128, kTK = 64;            // operand tile: 128 rows x 64 bf16 (16 KiB)
constexpr int kTileBytes = kTR * kTK * 2;

// The row tiles of a block-sparse frame operand and the K blocks each one touches.
//   analysis  (T_u, n x d):   row tile t covers frame rows [128 t, +128); run j owns frame rows
//             [2 k j, 2 k (j+1)) and real coordinates [2 w j, 2 w (j+1)) (the K range)
//   synthesis (T_u^T, d x n): row tile t covers coordinates [128 t, +128); run j owns them in
//             [2 w j, 2 w (j+1)) and frame rows [2 k j, 2 k (j+1)) (the K range)
struct SparseShape {
  int rows, cols, RT, KB;
  int run_rows, run_cols;        // rows and columns of one run in this orientation
  std::vector<int32_t> idx;      // [RT][3]: kb_lo, kb_hi, first stored tile
  int count = 0;
};

SparseShape sparse_shape(int k, int rho, int d, bool synthesis) {
  const int n = k * rho, w = d / rho;
  SparseShape S;
  S.rows = synthesis ? d : n;
  S.cols = synthesis ? n : d;
  S.run_rows = synthesis ? 2 * w : 2 * k;
  S.run_cols = synthesis ? 2 * k : 2 * w;
  S.RT = static_cast<int>(ceil_div(S.rows, kTR));
  S.KB = static_cast<int>(ceil_div(S.cols, kTK));
  S.idx.resize(3 * static_cast<size_t>(S.RT));
  for (int t = 0; t < S.RT; ++t) {
    const int r0 = t * kTR, r1 = std::min(S.rows, r0 + kTR);
    const int j0 = r0 / S.run_rows, j1 = (r1 - 1) / S.run_rows;
    const int lo = static_cast<int>((static_cast<int64_t>(j0) * S.run_cols) / kTK);
    const int hi = static_cast<int>(std::min<int64_t>(
        S.KB, ceil_div(static_cast<int64_t>(j1 + 1) * S.run_cols, kTK)));
    S.idx[3 * t] = lo;
    S.idx[3 * t + 1] = hi;
    S.idx[3 * t + 2] = S.count;
    S.count += hi - lo;
  }
  return S;
}

// bf16 bit pattern of a float, rounding to nearest even (the operands are finite)
uint16_t bf16_bits(float f) {
  uint32_t u;
  std::memcpy(&u, &f, 4);
  u += 0x7FFFu + ((u >> 16) & 1u);
  return static_cast<uint16_t>(u >> 16);
}

// The stored tiles of one orientation: entry (r, c) of the un-rotated analysis operator is,
// for frame row r = 2 (j k + k_i) + e and real coordinate c = 2 q + f with q in run j,
// v = exp(2 pi i k_i q / k) / sqrt(k) realified as (e, f) = (0,0) Re v, (0,1) Im v,
// (1,0) -Im v, (1,1) Re v (Appendix J; 0 outside the run), computed in double, rounded to fp32
// and then to bf16 like the dense operator.  Each tile is written in the 128-byte-swizzled
// shared-memory image of a K-major 128 x 64 tile: row r's 16-byte chunk h at chunk h ^ (r mod 8).
void fill_tiles(int k, int rho, int d, const SparseShape& S, bool synthesis,
                const std::vector<double>& cs, const std::vector<double>& sn,
                std::vector<uint16_t>& out) {
  const int w = d / rho;
  const double rk = 1.0 / std::sqrt(static_cast<double>(k));
  out.assign(static_cast<size_t>(S.count) * kTR * kTK, 0);
  for (int t = 0; t < S.RT; ++t) {
    const int lo = S.idx[3 * t], hi = S.idx[3 * t + 1], first = S.idx[3 * t + 2];
    for (int kb = lo; kb < hi; ++kb) {
      uint16_t* tile = out.data() + static_cast<size_t>(first + kb - lo) * kTR * kTK;
      for (int r = 0; r < kTR; ++r) {
        const int gr = t * kTR + r;
        if (gr >= S.rows) continue;
        for (int cc = 0; cc < kTK; ++cc) {
          const int gc = kb * kTK + cc;
          if (gc >= S.cols) continue;
          const int frow = synthesis ? gc : gr, coord = synthesis ? gr : gc;
          const int b2 = frow >> 1, e = frow & 1, f = coord & 1, q = coord >> 1;
          const int j = b2 / k, ki = b2 % k;
          if (q < j * w || q >= (j + 1) * w) continue;
          const int m = static_cast<int>((static_cast<int64_t>(ki) * q) % k);
          const double re = cs[m] * rk, im = sn[m] * rk;
          const double v = e == 0 ? (f == 0 ? re : im) : (f == 0 ? -im : re);
          const int pos = r * kTK + ((((cc >> 3) ^ (r & 7)) << 3) | (cc & 7));
          tile[pos] = bf16_bits(static_cast<float>(v));
        }
      }
    }
  }
}

struct FrameBuf {
  size_t Qa, QaT, Qb, QbT, perm, iperm, signs, ana_tiles, ana_idx, syn_tiles, syn_idx, total;
};

FrameBuf frame_buf(int k, int rho, int d, int a, int b) {
  FrameBuf L{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += static_cast<size_t>(round_up(static_cast<int64_t>(bytes), 256));
    return o;
  };
  const size_t qa = static_cast<size_t>(a) * a * 4, qb = static_cast<size_t>(b) * b * 4;
  L.Qa = take(qa);
  L.QaT = take(qa);
  L.Qb = take(qb);
  L.QbT = take(qb);
  L.perm = take(static_cast<size_t>(d) * 4);
  L.iperm = take(static_cast<size_t>(d) * 4);
  L.signs = take(static_cast<size_t>(d) * 4);
  const SparseShape A = sparse_shape(k, rho, d, false), S = sparse_shape(k, rho, d, true);
  L.ana_tiles = take(static_cast<size_t>(A.count) * kTileBytes);
  L.ana_idx = take(A.idx.size() * 4);
  L.syn_tiles = take(static_cast<size_t>(S.count) * kTileBytes);
  L.syn_idx = take(S.idx.size() * 4);
  L.total = off;
  return L;
}

bool valid_triple(int k, int rho, int d) {
  return k > 0 && rho >= 2 && rho % 2 == 0 && d > 0 && d % rho == 0 && k >= d / rho;
}

bool valid_frame(const fq_frame* f) {
  if (!f || !valid_triple(f->k, f->rho, f->d)) return false;
  if (!f->ana_tiles || !f->ana_idx || !f->syn_tiles || !f->syn_idx || f->ana_count <= 0 ||
      f->syn_count <= 0)
    return false;
  if (f->a == 0 && f->b == 0) return true;
  return f->a > 0 && f->b > 0 && static_cast<int64_t>(f->a) * f->b == f->d && f->Qa && f->QaT &&
         f->Qb && f->QbT && f->perm && f->iperm && f->signs;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

struct ImplWs {
  size_t v, s, total, group;
};

// the fused kernel's workspace (header, z, u), then the rotated tokens and the un-rotated output
ImplWs impl_ws(int M, int d_in, int n_in, int n_out, int d_out) {
  ImplWs L{};
  size_t off = decode_workspace_bytes(M, d_in, n_in, n_out, d_out);
  L.group = off;
  L.v = off;
  off += static_cast<size_t>(round_up(static_cast<int64_t>(M) * d_in * 2, 256));
  L.s = off;
  off += static_cast<size_t>(round_up(static_cast<int64_t>(M) * d_out * 2, 256));
  L.total = off;
  return L;
}

// Frames taken: the sizes that this library's entry points document (a rotation with b <= 1024
// whose (d + 8 (a + b) + 8 g r + B) fp32 values fit 227 KiB, r = b rounded up to 32, g = min(4,
// 1024 / r), B = b^2 for b <= 128 where the total stays within 110 KiB and 64 b otherwise).  The
// rotation kernel itself needs less.
bool frame_fits(const fq_frame& f) {
  if (ceil_div(static_cast<int64_t>(f.k) * f.rho, kTR) > kWsMaxTiles ||
      ceil_div(f.d, kTR) > kWsMaxTiles)
    return false;
  if (f.a == 0) return true;
  if (f.b > 1024) return false;
  const int64_t r = round_up(f.b, 32), g = std::max<int64_t>(1, std::min<int64_t>(4, 1024 / r));
  const int64_t base = round_up(f.d, 4) + 8 * (static_cast<int64_t>(f.a) + f.b) + 8 * g * r;
  const int64_t whole = (base + static_cast<int64_t>(f.b) * f.b) * 4;
  return (f.b <= 128 && whole <= 110 * 1024) || (base + 64 * static_cast<int64_t>(f.b)) * 4 <=
                                                    static_cast<int64_t>(kMaxSmem);
}

// A layer's split over C CTAs per token, and its shared memory with both factors staged whole, or
// (`whole` false) with what of them fits; above kMaxSmem when it does not fit.
size_t rot_layout(RotLayer& L, int C, bool whole) {
  const int64_t a = L.a, b = L.b;
  L.bp = static_cast<int>(round_up(b, 2));
  L.rc = static_cast<int>(round_up(ceil_div(a, C), 4));
  const int64_t base = 4 * (b * L.rc + round_up(a * L.bp, 4)), bs = 4 * round_up(b * L.bp, 4);
  if (whole) return static_cast<size_t>(base + 4 * a * round_up(a, 4) + bs);
  const int64_t max = static_cast<int64_t>(kMaxSmem), as = 4 * a * L.rc;
  L.stage_a = base + as <= max;
  L.stage_b = base + (L.stage_a ? as : 0) + bs <= max;
  return static_cast<size_t>(base + (L.stage_a ? as : 0) + (L.stage_b ? bs : 0));
}

// The CTAs per token of a launch over `tokens` tokens (of all layers), the layers' layouts, and their
// shared memory.  More CTAs shorten a token's products but read it as often, so a token with little
// work takes fewer, and C is halved while the launch is more than the CTAs that fit at once (4/3 of
// them at C = 4), unless a factor would lose its place in shared memory.  Measured with C = 1, 2, 4, 8
// (us per call): 512 x 512 at 16 tokens 18.4, 18.3, 18.1, 18.9; 1024 x 1024 at 8 tokens 20.2, 20.1, 19.8,
// 19.9; 2048 x 2048 at one token 23.2, 21.9, 21.1, 21.4, at 16 tokens 28.8, 30.0, 25.6, 24.0; three
// 4096 x 4096 at 64 tokens 102, 91, 81, 86; 4096 to 11008 at 32 tokens 91, 71, 61, 63, three at 64 tokens
// 208, 196, 202, 227.  With C = 4, 8, 16: 4096 x 4096 at one token 26.9, 27.5, 27.4, at 16 tokens 37.2,
// 31.1, 29.5; 11008 x 11008 at 4 tokens 81.4, 71.9, 70.6, at 16 tokens 82.1, 74.0, 86.0.  With C = 8, 16,
// 32: 28672 to 4096 at one token 124.6, 104.0, 102.7.
constexpr int kRotPerSm = 4;      // CTAs that an SM's registers hold

struct RotPlan {
  int C;
  bool staged;              // both factors of every layer, whole, of wide arrays
  int kept, kept_a;         // factors in shared memory, and first factors (their CTAs' columns)
  size_t smem;
};

RotPlan rot_plan(RotLayer* L, int n, int64_t tokens, int sms) {
  int64_t work = 0;         // multiply-adds per token: 43 k for 24 x 32, 66 k for 32 x 32, 524 k for 64 x 64
  int a = 0;
  bool wide = true;
  for (int l = 0; l < n; ++l) {
    wide = wide && L[l].wide;
    const int64_t w = static_cast<int64_t>(L[l].a) * L[l].b * (L[l].a + L[l].b);
    if (w > work) work = w, a = L[l].a;
  }
  auto with = [&](int C) {
    RotPlan p{C, true, 2 * n, n, 0};
    for (int l = 0; l < n; ++l) p.smem = std::max(p.smem, rot_layout(L[l], C, true));
    if (wide && p.smem <= kMaxSmem) return p;
    p = RotPlan{C, false, 0, 0, 0};
    for (int l = 0; l < n; ++l) {
      p.smem = std::max(p.smem, rot_layout(L[l], C, false));
      p.kept += L[l].stage_a + L[l].stage_b;
      p.kept_a += L[l].stage_a;
    }
    return p;
  };
  int C = work <= 50000 ? 1 : (work <= 70000 ? 4 : (work <= 250000 ? (tokens <= 2 ? 4 : 8) : 16));
  while (C > 1 && work / C > 600000 && 8 * C <= a) C *= 2;
  RotPlan p = with(C);
  // (a first factor many times as long as the second: until a CTA's columns of it fit)
  while (p.kept_a < n && 8 * C <= a && tokens * 2 * C <= 4 * sms) p = with(C *= 2);
  while (p.C > 2) {
    const int64_t resident = sms * std::min<int64_t>(kRotPerSm, 228 * 1024 / (p.smem + 1024));
    const RotPlan half = with(p.C / 2);
    const int64_t most = p.C == 4 ? resident * 4 / 3 : resident;
    if (tokens * p.C <= most || half.smem > kMaxSmem || half.kept < p.kept) break;
    p = half;
  }
  return with(p.C);
}

cudaError_t set_smem_attributes() {
  static std::mutex mu;
  static std::set<int> done;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> g(mu);
  if (done.count(dev)) return cudaSuccess;
  const int bytes = static_cast<int>(kMaxSmem);
  void (*const kernels[])(RotBatch) = {rotate_kernel<false, false>, rotate_kernel<false, true>,
                                       rotate_kernel<true, false>, rotate_kernel<true, true>};
  cudaError_t e = cudaSuccess;
  for (auto* k : kernels)
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.insert(dev);
  return e;
}

// R^T x (analysis) or R s (synthesis) for M tokens of n layers in one launch, bf16 in and out;
// layers without a rotation, and those whose `in` is null, are skipped.  Launched with
// programmatic stream serialization (the kernel may start while its predecessor in the stream
// finishes; it waits with griddepcontrol.wait before reading its inputs).
template <bool kSynth>
cudaError_t rotate_batch(int n, const fq_frame* const* f, const void* const* in,
                         void* const* out, int M, cudaStream_t s) {
  RotBatch rb{};
  int nb = 0;
  for (int l = 0; l < n; ++l) {
    if (f[l]->a == 0 || !in[l]) continue;
    const fq_frame& F = *f[l];
    RotLayer& L = rb.L[nb++];
    L.in = static_cast<const __nv_bfloat16*>(in[l]);
    L.out = static_cast<__nv_bfloat16*>(out[l]);
    L.a = F.a;
    L.b = F.b;
    L.At = kSynth ? F.QaT : F.Qa;
    L.B = kSynth ? F.QbT : F.Qb;
    L.perm = F.perm;
    L.iperm = F.iperm;
    L.signs = F.signs;
    L.wide = aligned16(L.At) && aligned16(L.B) && aligned16(L.perm) && aligned16(L.signs);
  }
  if (nb == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const RotPlan p = rot_plan(rb.L, nb, static_cast<int64_t>(M) * nb, sms);
  if (p.smem > kMaxSmem) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(p.C), static_cast<unsigned>(M), static_cast<unsigned>(nb));
  cfg.blockDim = dim3(kRotThreads);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, p.staged ? rotate_kernel<kSynth, true> : rotate_kernel<kSynth, false>,
                            rb);
}

template <bool kSynth>
cudaError_t rotate(const fq_frame& f, int M, const void* in, void* out, cudaStream_t s) {
  const fq_frame* fp = &f;
  return rotate_batch<kSynth>(1, &fp, &in, &out, M, s);
}

}  // namespace
}  // namespace fq

using namespace fq;

extern "C" {

size_t fq_frame_implicit_bytes(int k, int rho, int d, int a, int b) {
  if (!valid_triple(k, rho, d) || a < 0 || b < 0) return 0;
  if ((a == 0) != (b == 0) || (a > 0 && static_cast<int64_t>(a) * b != d)) return 0;
  return frame_buf(k, rho, d, a, b).total;
}

fq_status fq_frame_implicit(int k, int rho, int d, const fq_rotation* rot, void* buf,
                            size_t bytes, fq_frame* out, fq_stream_t stream) {
  if (!out || !valid_triple(k, rho, d)) return FQ_ERR_INVALID_ARG;
  const int a = rot ? rot->a : 0, b = rot ? rot->b : 0;
  if (rot) {
    if (!rot->gauss_a || !rot->gauss_b || !rot->perm || !rot->signs || a <= 0 || b <= 0 ||
        static_cast<int64_t>(a) * b != d)
      return FQ_ERR_INVALID_ARG;
    std::vector<char> seen(d, 0);
    for (int i = 0; i < d; ++i) {
      const int64_t p = rot->perm[i];
      if (p < 0 || p >= d || seen[p] || (rot->signs[i] != 1.0 && rot->signs[i] != -1.0))
        return FQ_ERR_INVALID_ARG;
      seen[p] = 1;
    }
  }
  const FrameBuf L = frame_buf(k, rho, d, a, b);
  if (!buf || bytes < L.total) return FQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(buf) & 255u) != 0) return FQ_ERR_ALIGNMENT;
  auto s = reinterpret_cast<cudaStream_t>(stream);
  char* base = static_cast<char*>(buf);
  // the two orientations of the un-rotated operator, tile by tile (host, double precision)
  std::vector<double> cs(k), sn(k);
  const double two_pi = 6.283185307179586476925286766559;
  for (int m = 0; m < k; ++m) {
    cs[m] = std::cos(two_pi * m / k);
    sn[m] = std::sin(two_pi * m / k);
  }
  const SparseShape SA = sparse_shape(k, rho, d, false), SS = sparse_shape(k, rho, d, true);
  std::vector<uint16_t> ta, ts;
  fill_tiles(k, rho, d, SA, false, cs, sn, ta);
  fill_tiles(k, rho, d, SS, true, cs, sn, ts);
  std::vector<float> qa, qat, qb, qbt, sg;
  std::vector<int32_t> pm, ipm;
  if (rot) {
    std::vector<double> Qa, Qb;
    haar_q(rot->gauss_a, a, Qa);
    haar_q(rot->gauss_b, b, Qb);
    qa.resize(static_cast<size_t>(a) * a);
    qat.resize(qa.size());
    for (int i = 0; i < a; ++i)
      for (int j = 0; j < a; ++j) {
        qa[static_cast<size_t>(i) * a + j] = static_cast<float>(Qa[static_cast<size_t>(i) * a + j]);
        qat[static_cast<size_t>(j) * a + i] = static_cast<float>(Qa[static_cast<size_t>(i) * a + j]);
      }
    qb.resize(static_cast<size_t>(b) * b);
    qbt.resize(qb.size());
    for (int i = 0; i < b; ++i)
      for (int j = 0; j < b; ++j) {
        qb[static_cast<size_t>(i) * b + j] = static_cast<float>(Qb[static_cast<size_t>(i) * b + j]);
        qbt[static_cast<size_t>(j) * b + i] = static_cast<float>(Qb[static_cast<size_t>(i) * b + j]);
      }
    sg.resize(d);
    pm.resize(d);
    ipm.resize(d);
    for (int i = 0; i < d; ++i) {
      sg[i] = static_cast<float>(rot->signs[i]);
      pm[i] = static_cast<int32_t>(rot->perm[i]);
      ipm[pm[i]] = i;
    }
  }
  auto up = [&](size_t off, const void* src, size_t n) {
    return n == 0 || cudaMemcpyAsync(base + off, src, n, cudaMemcpyHostToDevice, s) == cudaSuccess;
  };
  if (!up(L.ana_tiles, ta.data(), ta.size() * 2) || !up(L.ana_idx, SA.idx.data(), SA.idx.size() * 4) ||
      !up(L.syn_tiles, ts.data(), ts.size() * 2) || !up(L.syn_idx, SS.idx.data(), SS.idx.size() * 4) ||
      !up(L.Qa, qa.data(), qa.size() * 4) || !up(L.QaT, qat.data(), qat.size() * 4) ||
      !up(L.Qb, qb.data(), qb.size() * 4) || !up(L.QbT, qbt.data(), qbt.size() * 4) ||
      !up(L.signs, sg.data(), sg.size() * 4) || !up(L.perm, pm.data(), pm.size() * 4) ||
      !up(L.iperm, ipm.data(), ipm.size() * 4))
    return FQ_ERR_CUDA;
  // the host vectors are released on return: the copies from them must be complete
  if (cudaStreamSynchronize(s) != cudaSuccess) return FQ_ERR_CUDA;
  fq_frame f{};
  f.k = k;
  f.rho = rho;
  f.d = d;
  f.a = a;
  f.b = b;
  f.ana_tiles = reinterpret_cast<const uint8_t*>(base + L.ana_tiles);
  f.ana_idx = reinterpret_cast<const int32_t*>(base + L.ana_idx);
  f.ana_count = SA.count;
  f.syn_tiles = reinterpret_cast<const uint8_t*>(base + L.syn_tiles);
  f.syn_idx = reinterpret_cast<const int32_t*>(base + L.syn_idx);
  f.syn_count = SS.count;
  if (rot) {
    f.Qa = reinterpret_cast<const float*>(base + L.Qa);
    f.QaT = reinterpret_cast<const float*>(base + L.QaT);
    f.Qb = reinterpret_cast<const float*>(base + L.Qb);
    f.QbT = reinterpret_cast<const float*>(base + L.QbT);
    f.perm = reinterpret_cast<const int32_t*>(base + L.perm);
    f.iperm = reinterpret_cast<const int32_t*>(base + L.iperm);
    f.signs = reinterpret_cast<const float*>(base + L.signs);
  }
  *out = f;
  return FQ_OK;
}

size_t fq_implicit_workspace_bytes(int M, int d_in, int n_in, int n_out, int d_out) {
  if (M <= 0 || M > kDecodeMaxM || d_in <= 0 || n_in <= 0 || n_out <= 0 || d_out <= 0) return 0;
  return impl_ws(M, d_in, n_in, n_out, d_out).total;
}

fq_status fq_linear_forward_implicit(const void* x, int M, const fq_frame* F_in,
                                     const fq_packed* C, const fq_frame* F_out,
                                     const float* gamma, void* y, void* ws, size_t ws_bytes,
                                     int max_sms, fq_stream_t stream) {
  if (!x || !y || !C || max_sms < 0 || M <= 0) return FQ_ERR_INVALID_ARG;
  if (const fq_status cs = check_packed(C)) return cs;
  if (!valid_frame(F_in) || !valid_frame(F_out)) return FQ_ERR_INVALID_ARG;
  const fq_frame fi = *F_in, fo = *F_out;
  const int n_in = fi.k * fi.rho, n_out = fo.k * fo.rho;
  if (C->n_in != n_in || C->n_out != n_out) return FQ_ERR_INVALID_ARG;
  if (n_in % 16 || n_out % 16 || fi.d % 8 || fo.d % 8) return FQ_ERR_ALIGNMENT;
  if (!aligned16(x) || !aligned16(y) || (gamma && !aligned16(gamma)) ||
      !aligned16(fi.ana_tiles) || !aligned16(fo.syn_tiles))
    return FQ_ERR_ALIGNMENT;
  if (!ws) return FQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return FQ_ERR_ALIGNMENT;
  if (M > kDecodeMaxM || !frame_fits(fi) || !frame_fits(fo)) return FQ_ERR_UNSUPPORTED;
  const ImplWs L = impl_ws(M, fi.d, n_in, n_out, fo.d);
  if (ws_bytes < L.total) return FQ_ERR_WORKSPACE;
  {
    int dev = 0, major = 0, minor = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess)
      return FQ_ERR_CUDA;
    if (major * 10 + minor != 103) return FQ_ERR_UNSUPPORTED;
  }
  if (set_smem_attributes() != cudaSuccess) return FQ_ERR_CUDA;
  auto s = reinterpret_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  void* v = fi.a > 0 ? static_cast<void*>(w + L.v) : const_cast<void*>(x);
  void* sy = fo.a > 0 ? static_cast<void*>(w + L.s) : y;
  if (fi.a > 0 && rotate<false>(fi, M, x, v, s) != cudaSuccess) return FQ_ERR_CUDA;
  DecGroupLayer g{v, fi.d, nullptr, *C, nullptr, fo.d, gamma, sy};
  g.tin = SparseOperand{fi.ana_tiles, fi.ana_idx, fi.ana_count};
  g.tout = SparseOperand{fo.syn_tiles, fo.syn_idx, fo.syn_count};
  const fq_status st = launch_decode_group(M, 1, &g, w, L.group, max_sms, false, nullptr, 0, 0, s);
  if (st != FQ_OK) return st;
  if (fo.a > 0 && rotate<true>(fo, M, sy, y, s) != cudaSuccess) return FQ_ERR_CUDA;
  return FQ_OK;
}


size_t fq_implicit_group_workspace_bytes(int M, int n_layers, const fq_implicit_layer* layers) {
  if (M <= 0 || M > kDecodeMaxM || n_layers < 1 || n_layers > FQ_MAX_GROUP || !layers) return 0;
  DecGroupLayer g[FQ_MAX_GROUP];
  size_t extra = 0;
  for (int l = 0; l < n_layers; ++l) {
    const fq_implicit_layer& L = layers[l];
    if (!L.C || !L.F_in || !L.F_out) return 0;
    g[l] = DecGroupLayer{nullptr, L.F_in->d, nullptr, *L.C, nullptr, L.F_out->d, nullptr, nullptr};
    extra += static_cast<size_t>(round_up(static_cast<int64_t>(M) * L.F_in->d * 2, 256)) +
             static_cast<size_t>(round_up(static_cast<int64_t>(M) * L.F_out->d * 2, 256));
  }
  const size_t base = decode_group_workspace_bytes(M, n_layers, g);
  return base == 0 ? 0 : base + extra;
}

fq_status fq_linear_forward_implicit_group(int M, int n_layers, const fq_implicit_layer* layers,
                                           void* ws, size_t ws_bytes, int max_sms,
                                           fq_stream_t stream) {
  if (!layers || n_layers < 1 || n_layers > FQ_MAX_GROUP || max_sms < 0 || M <= 0)
    return FQ_ERR_INVALID_ARG;
  for (int l = 0; l < n_layers; ++l) {
    const fq_implicit_layer& L = layers[l];
    if (!L.x || !L.y || !L.C) return FQ_ERR_INVALID_ARG;
    if (const fq_status cs = check_packed(L.C)) return cs;
    if (!valid_frame(L.F_in) || !valid_frame(L.F_out)) return FQ_ERR_INVALID_ARG;
    const fq_frame &fi = *L.F_in, &fo = *L.F_out;
    if (L.C->n_in != fi.k * fi.rho || L.C->n_out != fo.k * fo.rho) return FQ_ERR_INVALID_ARG;
    if (fi.d % 8 || fo.d % 8) return FQ_ERR_ALIGNMENT;
    if (!aligned16(L.x) || !aligned16(L.y) || (L.gamma && !aligned16(L.gamma)) ||
        !aligned16(fi.ana_tiles) || !aligned16(fo.syn_tiles))
      return FQ_ERR_ALIGNMENT;
    if (!frame_fits(fi) || !frame_fits(fo)) return FQ_ERR_UNSUPPORTED;
    for (int j = 0; j < n_layers; ++j)
      if (j != l && (layers[j].y == L.y || layers[j].x == L.y)) return FQ_ERR_INVALID_ARG;
    if (L.x == L.y) return FQ_ERR_INVALID_ARG;
  }
  if (M > kDecodeMaxM) return FQ_ERR_UNSUPPORTED;
  if (!ws) return FQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return FQ_ERR_ALIGNMENT;
  const size_t need = fq_implicit_group_workspace_bytes(M, n_layers, layers);
  if (need == 0) return FQ_ERR_INVALID_ARG;
  if (ws_bytes < need) return FQ_ERR_WORKSPACE;
  {
    int dev = 0, major = 0, minor = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess)
      return FQ_ERR_CUDA;
    if (major * 10 + minor != 103) return FQ_ERR_UNSUPPORTED;
  }
  if (set_smem_attributes() != cudaSuccess) return FQ_ERR_CUDA;
  auto s = reinterpret_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  // the fused kernel's workspace first, then every layer's rotated tokens and output
  DecGroupLayer g[FQ_MAX_GROUP];
  for (int l = 0; l < n_layers; ++l) {
    const fq_implicit_layer& L = layers[l];
    g[l] = DecGroupLayer{nullptr, L.F_in->d, nullptr, *L.C, nullptr, L.F_out->d, L.gamma, nullptr};
  }
  const fq_frame* fin[FQ_MAX_GROUP];
  const fq_frame* fout[FQ_MAX_GROUP];
  const void* xin[FQ_MAX_GROUP];
  void* vout[FQ_MAX_GROUP];
  const void* sin_[FQ_MAX_GROUP];
  void* yout[FQ_MAX_GROUP];
  size_t off = decode_group_workspace_bytes(M, n_layers, g);
  const size_t group_bytes = off;
  for (int l = 0; l < n_layers; ++l) {
    const fq_implicit_layer& L = layers[l];
    const fq_frame &fi = *L.F_in, &fo = *L.F_out;
    // layers that rotate the same tokens by the same rotation share the result
    int same = l;
    for (int j = 0; j < l && same == l; ++j) {
      const fq_frame& fj = *layers[j].F_in;
      if (layers[j].x == L.x && fj.a == fi.a && fj.b == fi.b && fj.Qa == fi.Qa && fj.Qb == fi.Qb &&
          fj.iperm == fi.iperm && fj.signs == fi.signs)
        same = j;
    }
    void* v = fi.a > 0 ? static_cast<void*>(w + off) : const_cast<void*>(L.x);
    if (same < l) v = const_cast<void*>(g[same].x);
    xin[l] = same < l ? nullptr : L.x;
    off += static_cast<size_t>(round_up(static_cast<int64_t>(M) * fi.d * 2, 256));
    void* sy = fo.a > 0 ? static_cast<void*>(w + off) : L.y;
    off += static_cast<size_t>(round_up(static_cast<int64_t>(M) * fo.d * 2, 256));
    g[l].x = v;
    g[l].y = sy;
    g[l].tin = SparseOperand{fi.ana_tiles, fi.ana_idx, fi.ana_count};
    g[l].tout = SparseOperand{fo.syn_tiles, fo.syn_idx, fo.syn_count};
  }
  for (int l = 0; l < n_layers; ++l) {
    fin[l] = layers[l].F_in;
    fout[l] = layers[l].F_out;
    vout[l] = const_cast<void*>(g[l].x);
    sin_[l] = g[l].y;
    yout[l] = layers[l].y;
  }
  if (rotate_batch<false>(n_layers, fin, xin, vout, M, s) != cudaSuccess) return FQ_ERR_CUDA;
  const fq_status st =
      launch_decode_group(M, n_layers, g, w, group_bytes, max_sms, false, nullptr, 0, 0, s);
  if (st != FQ_OK) return st;
  if (rotate_batch<true>(n_layers, fout, sin_, yout, M, s) != cudaSuccess) return FQ_ERR_CUDA;
  return FQ_OK;
}

}  // extern "C"
