// FQ_BF16 path: the three products of the frame-quantized layer on the sm_103a tensor cores.
//
// Every phase is one persistent, warp-specialised kernel computing
//     out[t][i] = epilogue( sum_k A[i][k] * B[t][k] )      (i < R rows, t < M tokens)
// with the weight-side operand A as the rows of the MMA and the tokens as its N operand.  It
// serves batches of more than 64 tokens (prefill) and every batch with rounded activations; the
// others take the fused decode kernel.  Phases (Sec. 3.2):
//   analysis   A = T_in (n_in x d_in),  B = x,  out = z (bf16)
//   core       A = 2-bit codes of C_hat (n_out x n_in) decoded to bf16 in shared memory,
//              B = z, out = u = gamma * (s * acc + zero * sum(z))   (bf16)
//   synthesis  A = T_out^T (d_out x n_out), B = u, out = y (bf16)
//
// tc_pair_kernel runs them on CTA pairs, with tiles of 256 rows x 128 or 256 tokens.  A call with a
// budget of one SM, which has no pair, takes tc_phase_kernel: tiles of 128 rows x 128 or 256 tokens
// on one SM.  So does an odd budget where that is estimated to be faster (three SMs, mostly).
//
// Operand tiles are 64 bf16 wide in K (one 128-byte swizzle atom) and staged through a ring
// of shared-memory stages guarded by mbarriers; accumulators are double-buffered in TMEM so
// the epilogue of one tile overlaps the MMAs of the next.
//
// Tiles are numbered token tile fastest (tile = row tile * TT + token tile) and taken in turn by the
// CTAs (pairs): those of a wave share each weight tile across all token tiles, so a weight
// matrix larger than L2 (T_out^T of the up and gate layers, 267 MB) streams from HBM once per wave
// instead of once per token tile (measured 8.7% faster on the 2048-token block).
//
// sum(z), needed by the core's zero term, comes from the analysis epilogue as one sum per
// 128-row tile of z and token, taken over the bf16 values stored.
//
// The three phases are chained with programmatic dependent launch (the analysis kernel too,
// so consecutive layers chain as well): a kernel's CTAs start on SMs as they free up, load
// weight tiles that do not depend on the previous kernel, and wait (griddepcontrol.wait)
// before reading activations or writing anything the previous kernel may still read.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <utility>

#include "fq_device.cuh"
#include "fq_internal.h"
#include "framequant_dense.h"

namespace fq {
namespace {

enum Phase : int { kAnalysis = 0, kCore = 1, kSynthesis = 2 };

constexpr int kBM = 128;                    // MMA M (rows of A per tile)
constexpr int kBK = 64;                     // K per stage (one 128-byte swizzle atom of bf16)
constexpr int kATileBytes = kBM * kBK * 2;  // 16 KiB
constexpr int kCodeBytes = kBM * kBK / 4;   // 2 KiB of packed codes per stage
constexpr int kSmemBudget = 200 * 1024;
constexpr int kEpi = 128;                   // epilogue threads
constexpr int kChunk = 16;                  // accumulator columns per TMEM load

struct PhaseArgs {
  int R, K, M;
  int RT, TT, KB, tiles;     // row tiles (128 rows, or 256 on a CTA pair), token tiles, K blocks
  int RT1;                   // 128-row tiles
  // On CTA pairs:
  int KS, kbs, units;        // K splits per tile, K blocks per split, tiles * KS work units
  float* part;               // KS > 1: fp32 partial tiles [tile][split][BN][128]
  int64_t part_floats;       // what `part` holds (host)
  uint32_t* cnt;             // KS > 1: arrivals per tile, 16 bits for each CTA's half (the last
                             // resets them to 0), kWsCntSlots of them in the workspace header
  const uint32_t* words;     // core: packed codes
  __nv_bfloat16* out;        // [M][R]
  float* zsum_part;          // analysis writes [RT][M] sums of z; the core reads them
  int zsum_tiles;
  const __half* scale;
  const __half* zero;
  const float* gamma;
  int32_t* status;
  int clear_status;          // this launch starts a call: clear the status word
  int transposed;            // synthesis on CTA pairs: out is [R][M] (M a multiple of 8)
  // Rounding of the frame representation of the activations (Appendix F), else all null:
  float* out32;              // analysis: z in fp32 (the bf16 z is then the rounded one)
  uint32_t* amax;            // analysis: running max |z| as float bits; the core resets it
  const float* delta;        // core: the rounding step Delta, which scales the product
};

template <int PHASE, int BN>
struct Layout {
  static constexpr bool kCodes = PHASE == kCore;
  static constexpr int kBTileBytes = BN * kBK * 2;
  static constexpr int kCodesStage = kCodes ? kCodeBytes : 0;
  static constexpr int kStageBytes = kATileBytes + kBTileBytes + kCodesStage;
  // Code rounds are decoded by warp (round mod 4), which waits for a stage's codes only in the
  // rounds it owns; that is exact only when every phase of a stage's barrier belongs to the
  // same warp, i.e. when the ring depth is a multiple of 4.
  static constexpr int kStagesRaw = std::min(12, kSmemBudget / kStageBytes);
  static constexpr int kStages = kCodes ? (kStagesRaw & ~3) : kStagesRaw;
  // double-buffered accumulators [0, 2 BN)
  static constexpr int kAccCols = 2 * BN;
  static constexpr uint32_t kTmemCols = kAccCols <= 256 ? 256 : 512;
  // byte offsets from the 1024-aligned base
  static constexpr int oA = 0;
  static constexpr int oB = oA + kStages * kATileBytes;
  static constexpr int oCodes = oB + kStages * kBTileBytes;
  static constexpr int oBar = oCodes + kStages * kCodesStage;
  static constexpr int kNumBars = 4 * kStages + 2 + 2 + 1;
  static constexpr int oMisc = oBar + kNumBars * 8;
  static constexpr int oRedSmall = oMisc + 16;                      // [4][kChunk] floats
  static constexpr int oZsum = oRedSmall + 4 * kChunk * 4;          // [2][BN] floats
  static constexpr int kBytes = oZsum + 2 * BN * 4 + 1024;          // + alignment slack
  static_assert(BN == 128 || BN == 256, "tile widths of the one-SM kernel");
  static_assert(kBTileBytes % 1024 == 0, "B tiles must keep 1024-byte alignment");
  static_assert(kBytes <= 227 * 1024, "shared memory");
  static_assert(kStages >= 2 && (!kCodes || kStages % 4 == 0), "ring depth");
};

template <int PHASE>
constexpr int threads_for() { return PHASE == kCore ? 320 : 192; }

// Decode 64 2-bit codes (4 words, layout of framequant.h) into 64 exact bf16 values and store
// them as one 128-byte row of a K-major tile with the 128-byte swizzle (16-byte chunk c of row
// r lands at chunk c ^ (r mod 8)).  q in {0..3} becomes bf16(128 + q) by placing q in the low
// mantissa bits of 128.0 (0x4300) and then 128 is subtracted exactly.
__device__ __forceinline__ void decode_row(const uint4 w4, uint8_t* tile, int r) {
  const uint32_t wv[4] = {w4.x, w4.y, w4.z, w4.w};
  const __nv_bfloat162 bias = __floats2bfloat162_rn(128.f, 128.f);
  uint8_t* row = tile + r * 128;
#pragma unroll
  for (int wi = 0; wi < 4; ++wi) {
    uint32_t h[8];
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      const uint32_t bits = ((wv[wi] >> (2 * p)) & 0x00030003u) | 0x43004300u;
      __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&bits);
      v = __hsub2(v, bias);
      h[p] = *reinterpret_cast<const uint32_t*>(&v);
    }
    // word wi holds columns 16 wi .. 16 wi + 15 = chunks 2 wi and 2 wi + 1
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int c = 2 * wi + half;
      uint4 q = make_uint4(h[4 * half], h[4 * half + 1], h[4 * half + 2], h[4 * half + 3]);
      *reinterpret_cast<uint4*>(row + ((c ^ (r & 7)) << 4)) = q;
    }
  }
}

__device__ __forceinline__ bool bar_red_or(uint32_t id, uint32_t n, bool v) {
  uint32_t out;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(out)
      : "r"(static_cast<uint32_t>(v)), "r"(id), "r"(n)
      : "memory");
  return out != 0;
}

// Without pairs (a call whose budget is one SM, or an odd number of them that pairs use badly): tiles
// of 128 rows x BN tokens, one CTA each, with one warp of TMA copies, one issuing MMAs, four of
// epilogue and, in the core, four decoders.  BN is 256 above 128 tokens: the operands of a K block
// then take 740 cycles for twice the tokens of 128 (600), see plan_one_sm.
template <int PHASE, int BN>
__global__ void __launch_bounds__(threads_for<PHASE>(), 1)
    tc_phase_kernel(const __grid_constant__ CUtensorMap tmA,
                    const __grid_constant__ CUtensorMap tmB, const PhaseArgs p) {
  using Lo = Layout<PHASE, BN>;
  constexpr int S_ = Lo::kStages;
  constexpr bool kCodes = Lo::kCodes;
  constexpr int kBTile = Lo::kBTileBytes;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* sA = smem + Lo::oA;
  uint8_t* sB = smem + Lo::oB;
  uint8_t* sCodes = smem + Lo::oCodes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + Lo::oBar);   // A (+B) landed / B landed
  uint64_t* empty = full + S_;      // stage consumed by the MMAs
  uint64_t* aready = empty + S_;    // decoded A tile written (core)
  uint64_t* cfull = aready + S_;    // codes landed (core)
  uint64_t* tfull = cfull + S_;     // accumulator ready
  uint64_t* tempty = tfull + 2;     // accumulator drained
  uint64_t* mma_done = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + Lo::oMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* red = reinterpret_cast<float*>(smem + Lo::oRedSmall);     // [4][kChunk]
  float* zsum_s = reinterpret_cast<float*>(smem + Lo::oZsum);      // [2][BN]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t cid = blockIdx.x, ncl = gridDim.x;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S_; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&aready[s], 32);     // one decoder warp per stage
      mbar_init(&cfull[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], kEpi);
    }
    mbar_init(mma_done, 1);
    *abort_flag = 0;
    fence_barrier_init();
    if (!kCodes) prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
  }
  if (warp == 1) tmem_alloc(tmem_slot, Lo::kTmemCols);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  // Let the next kernel's CTAs launch as soon as SMs free up; they wait for this grid's
  // completion (griddepcontrol.wait) before reading what it writes.
  pdl_launch_dependents();

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      const uint64_t pol_w = policy_evict_first();   // weights: streamed once
      const uint64_t pol_x = policy_evict_last();    // activations: re-read by other tiles
      // Weight tiles of the first tile do not depend on the previous kernel: issue up to a
      // full ring of them before waiting for it, and warm L2 with the rest.
      int pre = 0;
      if (static_cast<int>(cid) < p.tiles) {
        const int rt = static_cast<int>(cid) / p.TT;
        pre = min(S_, p.KB);
        for (int kb = 0; kb < pre; ++kb) {
          const int i = kb;
          if (kCodes) {
            mbar_arrive_expect_tx(&cfull[i], kCodeBytes);
            bulk_load(sCodes + i * kCodeBytes,
                      p.words + (static_cast<int64_t>(rt) * p.KB + kb) * 512, kCodeBytes,
                      &cfull[i], pol_w);
          } else {
            mbar_arrive_expect_tx(&full[i], kATileBytes + kBTile);
            tma_load_2d(sA + i * kATileBytes, &tmA, &full[i], kb * kBK, rt * kBM, pol_w);
          }
        }
        for (int kb = pre; kb < p.KB; ++kb) {
          if (kCodes) {
            const uint32_t* src = p.words + (static_cast<int64_t>(rt) * p.KB + kb) * 512;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src),
                         "r"(kCodeBytes)
                         : "memory");
          } else {
            asm volatile(
                "cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(
                    reinterpret_cast<uint64_t>(&tmA)),
                "r"(kb * kBK), "r"(rt * kBM)
                : "memory");
          }
        }
      }
      pdl_wait();   // the previous kernel is complete and its writes are visible
      if (p.clear_status && blockIdx.x == 0) *p.status = 0;       // a new call
      // the rounding kernel before this one has read the maximum: ready for the next call
      if (PHASE == kCore && p.amax && blockIdx.x == 0) *p.amax = 0u;
      int stage = 0;
      uint32_t phase = 0;
      int it = 0;
      uint32_t issued_parity[S_];
      bool issued[S_];
#pragma unroll
      for (int s = 0; s < S_; ++s) issued[s] = false, issued_parity[s] = 0;
      for (int tile = static_cast<int>(cid); tile < p.tiles && !*abort_flag;
           tile += static_cast<int>(ncl)) {
        const int rt = tile / p.TT, tt = tile % p.TT;
        for (int kb = 0; kb < p.KB; ++kb, ++it) {
          if (it >= pre) {
            if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag)) {
              report(p.status, FQ_ERR_TIMEOUT);
              *abort_flag = 1;
              break;
            }
            if (kCodes) {
              mbar_arrive_expect_tx(&cfull[stage], kCodeBytes);
              bulk_load(sCodes + stage * kCodeBytes,
                        p.words + (static_cast<int64_t>(rt) * p.KB + kb) * 512, kCodeBytes,
                        &cfull[stage], pol_w);
            } else {
              mbar_arrive_expect_tx(&full[stage], kATileBytes + kBTile);
              tma_load_2d(sA + stage * kATileBytes, &tmA, &full[stage], kb * kBK, rt * kBM,
                          pol_w);
            }
          }
          if (kCodes) mbar_arrive_expect_tx(&full[stage], kBTile);
          tma_load_2d(sB + stage * kBTile, &tmB, &full[stage], kb * kBK, tt * BN, pol_x);
          issued[stage] = true;
          issued_parity[stage] = phase;
          if (++stage == S_) stage = 0, phase ^= 1;
        }
      }
      // Never leave with copies in flight: wait (bounded) for the last round of each stage.
      for (int s = 0; s < S_; ++s) {
        if (!issued[s]) continue;
        if (!mbar_wait(&full[s], issued_parity[s], nullptr) ||
            (kCodes && !mbar_wait(&cfull[s], issued_parity[s], nullptr)))
          report(p.status, FQ_ERR_TIMEOUT);
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = umma_idesc_bf16(kBM, BN);
      int stage = 0;
      uint32_t phase = 0;
      int buf = 0;
      uint32_t acc_phase = 0;
      bool issued_any = false;
      for (int tile = static_cast<int>(cid); tile < p.tiles && !*abort_flag;
           tile += static_cast<int>(ncl)) {
        if (!mbar_wait(&tempty[buf], acc_phase ^ 1, abort_flag)) {
          report(p.status, FQ_ERR_TIMEOUT);
          *abort_flag = 1;
          break;
        }
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * BN);
        bool ok = true;
        for (int kb = 0; kb < p.KB; ++kb) {
          ok = mbar_wait(&full[stage], phase, abort_flag) &&
               (!kCodes || mbar_wait(&aready[stage], phase, abort_flag));
          if (!ok) break;
          tc_fence_after_sync();
          const uint64_t adesc = umma_desc_sw128(smem_u32(sA + stage * kATileBytes));
          const uint64_t bdesc = umma_desc_sw128(smem_u32(sB + stage * kBTile));
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)   // 16 bf16 = 32 bytes along K per step
            umma_bf16(d_tmem, adesc + 2 * k, bdesc + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          issued_any = true;
          umma_commit(&empty[stage]);
          if (++stage == S_) stage = 0, phase ^= 1;
        }
        if (!ok) {
          report(p.status, FQ_ERR_TIMEOUT);
          *abort_flag = 1;
          break;
        }
        umma_commit(&tfull[buf]);
        if (++buf == 2) buf = 0, acc_phase ^= 1;
      }
      // Drain: every MMA issued has completed before the TMEM is released.
      if (issued_any) {
        umma_commit(mma_done);
        if (!mbar_wait(mma_done, 0, nullptr)) report(p.status, FQ_ERR_TIMEOUT);
      }
    }
  } else if (warp < 6) {
    // ---------------------------------------------------------------- epilogue (rows)
    const int quarter = warp & 3;                 // TMEM lanes 32*quarter .. +31
    const int r_in_tile = quarter * 32 + lane;
    const int et = threadIdx.x - 64;              // 0..127 within the epilogue group
    const int ew = warp - 2;
    pdl_wait();
    int buf = 0;
    uint32_t acc_phase = 0;
    for (int tile = static_cast<int>(cid); tile < p.tiles; tile += static_cast<int>(ncl)) {
      const int rt = tile / p.TT, tt = tile % p.TT;
      const int row = rt * kBM + r_in_tile;
      const int t0 = tt * BN;
      const bool row_ok = row < p.R;
      float s_i = 0.f, z_i = 0.f;
      if (PHASE == kCore && row_ok) {
        s_i = __half2float(p.scale[row]);
        z_i = __half2float(p.zero[row]);
      }
      if (PHASE == kCore) {
        // sum_j z[t][j] for the tile's tokens, from the analysis phase's per-tile sums
        named_barrier_sync(1, kEpi);
        for (int q = et; q < BN; q += kEpi) {
          const int t = t0 + q;
          float s = 0.f;
          if (t < p.M)
            for (int g = 0; g < p.zsum_tiles; ++g)
              s += ldcg_f32(p.zsum_part + static_cast<int64_t>(g) * p.M + t);
          zsum_s[buf * BN + q] = s;
        }
        named_barrier_sync(1, kEpi);
      }
      const bool fail = !mbar_wait(&tfull[buf], acc_phase, abort_flag);
      if (fail) report(p.status, FQ_ERR_TIMEOUT);
      if (bar_red_or(1, kEpi, fail || *abort_flag)) {
        if (et == 0) *abort_flag = 1;
        break;
      }
      tc_fence_after_sync();
      const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) +
                             static_cast<uint32_t>(buf * BN);
      const float* zs = zsum_s + buf * BN;
      const float g_i = (PHASE == kCore && row_ok && p.gamma) ? p.gamma[row] : 1.f;
      // with rounded activations the accumulator is the exact integer sum_j q_ij zbar_j, and
      // u = Delta gamma (s acc + zero sum_j zbar_j)
      const float dl = (PHASE == kCore && p.delta) ? ldcg_f32(p.delta) : 1.f;
      float amax_t = 0.f;                         // analysis with rounding: this row's max |z|
      // the finished values of columns c .. c + 15 of this thread's row
      auto emit = [&](int c, float* v) {
        if (PHASE == kAnalysis && p.out32) {
          // fp32 z for the rounding kernel, and the running maximum of |z|
#pragma unroll
          for (int q = 0; q < kChunk; ++q) {
            const int t = t0 + c + q;
            if (row_ok && t < p.M) {
              p.out32[static_cast<int64_t>(t) * p.R + row] = v[q];
              amax_t = fmaxf(amax_t, fabsf(v[q]));
            }
          }
          return;
        }
#pragma unroll
        for (int q = 0; q < kChunk; ++q) {
          if (PHASE == kCore) v[q] = g_i * fmaf(s_i, v[q], z_i * zs[c + q]) * dl;
          const __nv_bfloat16 b = __float2bfloat16_rn(v[q]);
          v[q] = __bfloat162float(b);
          const int t = t0 + c + q;
          if (row_ok && t < p.M) p.out[static_cast<int64_t>(t) * p.R + row] = b;
        }
        if (PHASE == kAnalysis) {
          // per-token sum over the tile's 128 rows of the bf16 z actually stored
#pragma unroll
          for (int q = 0; q < kChunk; ++q) {
            float s = row_ok ? v[q] : 0.f;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            v[q] = s;
          }
          if (lane == 0) {
#pragma unroll
            for (int q = 0; q < kChunk; ++q) red[ew * kChunk + q] = v[q];
          }
          named_barrier_sync(1, kEpi);
          if (et < kChunk) {
            const int t = t0 + c + et;
            // fixed order over the TMEM quarters (rows 0.., 32.., 64.., 96..)
            const float s = (red[2 * kChunk + et] + red[3 * kChunk + et]) +
                            (red[0 * kChunk + et] + red[1 * kChunk + et]);
            if (t < p.M) p.zsum_part[static_cast<int64_t>(rt) * p.M + t] = s;
          }
          named_barrier_sync(1, kEpi);
        }
      };
#pragma unroll 1
      for (int c = 0; c < BN; c += kChunk) {
        float v[kChunk];
        tmem_ld16(t_row + c, v);
        tmem_wait_ld();
        emit(c, v);
      }
      tc_fence_before_sync();
      mbar_arrive(&tempty[buf]);
      if (PHASE == kAnalysis && p.out32) {
        // one atomic per warp and tile: the tensor's max |z| (non-negative floats order like
        // their bit patterns)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
          amax_t = fmaxf(amax_t, __shfl_xor_sync(0xffffffffu, amax_t, off));
        if (lane == 0 && amax_t > 0.f) atomicMax(p.amax, __float_as_uint(amax_t));
      }
      if (++buf == 2) buf = 0, acc_phase ^= 1;
    }
  } else {
    // ---------------------------------------------------------------- code decoders (core)
    if (kCodes) {
      // stage i of this CTA is decoded by decoder warp i mod 4, four rows per lane
      const int dw = warp - 6;
      int stage = 0;
      uint32_t phase = 0;
      int it = 0;
      bool ok = true;
      for (int tile = static_cast<int>(cid); tile < p.tiles && ok && !*abort_flag;
           tile += static_cast<int>(ncl)) {
        for (int kb = 0; kb < p.KB; ++kb, ++it) {
          if ((it & 3) == dw) {
            if (!mbar_wait(&cfull[stage], phase, abort_flag)) {
              ok = false;
              break;
            }
            const uint4* codes = reinterpret_cast<const uint4*>(sCodes + stage * kCodeBytes);
            uint8_t* tile_a = sA + stage * kATileBytes;
#pragma unroll
            for (int rr = 0; rr < 4; ++rr) decode_row(codes[lane + 32 * rr], tile_a, lane + 32 * rr);
            fence_proxy_async_smem();
            mbar_arrive(&aready[stage]);
          }
          if (++stage == S_) stage = 0, phase ^= 1;
        }
      }
      if (!ok) {
        report(p.status, FQ_ERR_TIMEOUT);
        *abort_flag = 1;
      }
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, Lo::kTmemCols);
  }
}

// ---------------------------------------------------------------------------------------------
// Tiles of 256 rows x 128 or 256 tokens on CTA pairs
// ---------------------------------------------------------------------------------------------
// A 128 x 256 tile on one SM is bound by its shared memory: each 128-cycle MMA step reads 12 KiB
// of operands and the ring refills 12 KiB, 192 B per cycle against the 128 B an SM moves.  A pair of
// SMs computing a 256 x 256 tile (tcgen05 cta_group::2) reads 4 KiB of A and its own half of B,
// 4 KiB, per SM and step, and refills as much: 128 B per cycle, and for the code product less
// (2-bit codes).  Measured with the whole path of this file: 11008 x 4096 at 2048 tokens 701 -> 573 us
// (1475 TFLOP/s under the power cap), 8192 x 8192 at 4096 tokens 1452 -> 1254 us; a 64-wide K round
// takes 515 to 570 cycles of which the MMAs need 512 (980 on one SM).
//
// Each CTA of the pair loads and decodes its own 128 rows of A and half of the tokens of B;
// rank 0 issues the MMAs for both, so the barriers the MMAs wait on live in rank 0:
//   full[s]    rank 0: one arrival of its producer with both CTAs' bytes, the copies of both,
//              and in the code product one arrival per decoder warp of both CTAs
//   tempty[b]  rank 0: one arrival per epilogue warp of both CTAs
// and the MMAs' completions are committed to both CTAs (empty[s], tfull[b]).  The producer waits
// for the last use of each of its stages before it leaves, so no copy is in flight then.
//
// The code product's round is a chain: stage free, codes expanded, MMAs, stage free.  So the
// codes do not pass through shared memory: round i is expanded by decoder i mod D, which holds the
// round's codes in registers, loaded from global memory right after it handed over round i - D
// (not earlier: the release of a hand-over to the other CTA, about 1500 cycles, waits for loads
// in flight).  For 256 tokens six decoders of two warps keep up with the MMAs' 512 cycles per
// round; for 128 tokens nine of one warp are faster (2.4% on 8192 x 8192 at 128 tokens, 9% on 4096 x
// 4096 at 100), since two warps wait for the same release, and slower for 256 (0.7 to 3%).  A
// decoder meets a stage only in some of its rounds, but it never waits for a phase more than one
// past the last one complete: at round i it has seen round i - D - S's MMAs (S stages) complete,
// the commits are in order, and D <= S.
template <int PHASE, int BN_>
struct PairLayout {
  static constexpr bool kCodes = PHASE == kCore;
  static constexpr int kBN = BN_;                       // tokens per tile
  static constexpr int kBTile = kBN / 2 * kBK * 2;      // this CTA's half of them
  // analysis: [4][kBN] sums of z; code product: [kBN] sums of z
  static constexpr int kSums = PHASE == kAnalysis ? 4 * kBN * 4 : (kCodes ? kBN * 4 : 0);
  static constexpr int kStages = (225 * 1024 - kSums) / (kATileBytes + kBTile);
  static constexpr int kEpiWarps = 8;                   // two per TMEM quarter
  static constexpr int kEpiThreads = 32 * kEpiWarps;
  static constexpr int kHalf = kBN / 2;                 // columns per epilogue warp
  static constexpr int kGroups = kCodes ? 1 : 2;        // of 16 columns at a time (registers)
  static constexpr int kDecoders = kBN == 256 ? 6 : kStages;
  static constexpr int kWarpsPer = kBN == 256 ? 2 : 1;  // warps per decoder
  static constexpr int kDecWarps = kCodes ? kDecoders * kWarpsPer : 0;
  static constexpr int kThreads = 64 + kEpiThreads + 32 * kDecWarps;
  static constexpr uint32_t kTmemCols = 512;            // all, so that both CTAs' base is 0
  static constexpr int oA = 0;
  static constexpr int oB = oA + kStages * kATileBytes;
  static constexpr int oBar = oB + kStages * kBTile;
  static constexpr int kNumBars = 2 * kStages + 4;
  static constexpr int oMisc = oBar + kNumBars * 8;     // TMEM address, abort and last-split flags
  static constexpr int oSums = (oMisc + 16 + 15) & ~15;
  static constexpr int kBytes = oSums + kSums + 1024;   // + alignment slack
  static_assert(kBN == 128 || kBN == 256, "tokens per tile");
  static_assert(2 * kBN <= 512, "two accumulators");
  static_assert(!kCodes || kDecoders <= kStages, "a decoder waits for a stage's latest phase only");
  static_assert(kBTile % 1024 == 0, "B tiles keep 1024-byte alignment");
  static_assert(kBytes <= 227 * 1024, "shared memory");
};

// Decode 64 2-bit codes (4 words) into one 128-byte row of a swizzled K-major tile, like
// decode_row, with fewer operations: a pair of codes at bits 2p (p = 0, 1, 2) of the half-words
// is ORed into the mantissa of 128.0 where it stands, giving 128 + 4^p q, and one fused
// multiply-add makes it q (every step exact); two shifts per word bring the other pairs there.
__device__ __forceinline__ void decode_row_fma(const uint4 w4, uint8_t* tile, int r) {
  const uint32_t wv[4] = {w4.x, w4.y, w4.z, w4.w};
  const __nv_bfloat162 one[3] = {__floats2bfloat162_rn(1.f, 1.f),
                                 __floats2bfloat162_rn(0.25f, 0.25f),
                                 __floats2bfloat162_rn(0.0625f, 0.0625f)};
  const __nv_bfloat162 bias[3] = {__floats2bfloat162_rn(-128.f, -128.f),
                                  __floats2bfloat162_rn(-32.f, -32.f),
                                  __floats2bfloat162_rn(-8.f, -8.f)};
  uint8_t* row = tile + r * 128;
#pragma unroll
  for (int wi = 0; wi < 4; ++wi) {
    uint32_t h[8];
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      const uint32_t w = wv[wi] >> (6 * (p / 3));
      const uint32_t bits = (w & (0x00030003u << (2 * (p % 3)))) | 0x43004300u;
      const __nv_bfloat162 v =
          __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&bits), one[p % 3], bias[p % 3]);
      h[p] = *reinterpret_cast<const uint32_t*>(&v);
    }
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int c = 2 * wi + half;
      *reinterpret_cast<uint4*>(row + ((c ^ (r & 7)) << 4)) =
          make_uint4(h[4 * half], h[4 * half + 1], h[4 * half + 2], h[4 * half + 3]);
    }
  }
}

// Sums over a warp's 32 lanes of 16 values per lane: returned to lane l for value l >> 1 (both
// lanes of a pair hold it).  Each step adds the lane 16, 8, 4, 2, 1 away and halves the values
// a lane carries, so the additions are those of a full butterfly in 16 instead of 80 shuffles.
__device__ __forceinline__ float warp_sums16(const float (&v)[kChunk], int lane) {
  float a[8], b[4], c[2];
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4, h2 = lane & 2;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float send = h16 ? v[i] : v[i + 8], keep = h16 ? v[i + 8] : v[i];
    a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float send = h8 ? a[i] : a[i + 4], keep = h8 ? a[i + 4] : a[i];
    b[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float send = h4 ? b[i] : b[i + 2], keep = h4 ? b[i + 2] : b[i];
    c[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  const float send = h2 ? c[0] : c[1], keep = h2 ? c[1] : c[0];
  const float d = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  return d + __shfl_xor_sync(0xffffffffu, d, 1);
}

// Transposes between the lanes of a warp, so that results leave in 16-byte stores: on entry lane l
// holds row l of 16 columns, on return rows of a group of consecutive rows.
//   bf16:  eight rows 8 (l / 8) .. + 7 of columns column16(l) and column16(l) + 1, in w[0..3] and w[4..7]
//   fp32:  four rows 4 (l / 4) .. + 3 of columns 8 b0 + 4 b1 + 0 .. 3 (b0, b1 the low bits of l)
// Each step exchanges half of a lane's registers with the lane 1, 2 (, 4) away.
__device__ __forceinline__ int column16(int lane) {
  return 8 * (lane & 1) + 4 * ((lane >> 1) & 1) + 2 * ((lane >> 2) & 1);
}

// The registers a lane keeps (of a) and what its partner sends, in the order of the partners'
// rows: lower rows in lo, upper rows in hi.
template <int N>
__device__ __forceinline__ void exchange(const uint32_t* a, int lane, int bit, uint32_t* lo,
                                         uint32_t* hi) {
  const bool up = lane & bit;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t send = up ? a[i] : a[i + N], keep = up ? a[i + N] : a[i];
    const uint32_t got = __shfl_xor_sync(0xffffffffu, send, bit);
    lo[i] = up ? got : keep;
    hi[i] = up ? keep : got;
  }
}

__device__ __forceinline__ void transpose_bf16(const uint32_t (&h)[8], int lane,
                                               uint32_t (&w)[8]) {
  uint32_t lo[4], hi[4], g[8];
  exchange<4>(h, lane, 1, lo, hi);               // pairs of columns, rows 2m and 2m + 1
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    g[2 * i] = __byte_perm(lo[i], hi[i], 0x5410);       // the even column of the pair
    g[2 * i + 1] = __byte_perm(lo[i], hi[i], 0x7632);   // the odd one
  }
  exchange<4>(g, lane, 2, lo, hi);               // four columns, rows 4m .. 4m + 3
#pragma unroll
  for (int i = 0; i < 4; ++i) g[2 * i] = lo[i], g[2 * i + 1] = hi[i];
  exchange<4>(g, lane, 4, lo, hi);               // two columns, rows 8m .. 8m + 7
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    w[4 * i] = lo[2 * i];
    w[4 * i + 1] = lo[2 * i + 1];
    w[4 * i + 2] = hi[2 * i];
    w[4 * i + 3] = hi[2 * i + 1];
  }
}

__device__ __forceinline__ void transpose_fp32(const float (&v)[16], int lane,
                                               uint32_t (&w)[16]) {
  uint32_t a[16], lo[8], hi[8];
#pragma unroll
  for (int i = 0; i < 16; ++i) a[i] = __float_as_uint(v[i]);
  exchange<8>(a, lane, 1, lo, hi);               // eight columns, rows 2m and 2m + 1
#pragma unroll
  for (int i = 0; i < 8; ++i) a[2 * i] = lo[i], a[2 * i + 1] = hi[i];
  exchange<8>(a, lane, 2, lo, hi);               // four columns, rows 4m .. 4m + 3
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    w[4 * i] = lo[2 * i];
    w[4 * i + 1] = lo[2 * i + 1];
    w[4 * i + 2] = hi[2 * i];
    w[4 * i + 3] = hi[2 * i + 1];
  }
}

template <int PHASE, int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PairLayout<PHASE, BN>::kThreads, 1)
    tc_pair_kernel(const __grid_constant__ CUtensorMap tmA,
                   const __grid_constant__ CUtensorMap tmB, const PhaseArgs p) {
  using Lo = PairLayout<PHASE, BN>;
  constexpr int S_ = Lo::kStages;
  constexpr bool kCodes = Lo::kCodes;
  constexpr uint32_t kFullBytes = 2 * ((kCodes ? 0 : kATileBytes) + Lo::kBTile);

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* sA = smem + Lo::oA;
  uint8_t* sB = smem + Lo::oB;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + Lo::oBar);
  uint64_t* empty = full + S_;
  uint64_t* tfull = empty + S_;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + Lo::oMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* last_flag = reinterpret_cast<volatile int*>(tmem_slot + 2);
  float* red = reinterpret_cast<float*>(smem + Lo::oSums);
  float* zsum_s = red;

  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);   // uniform
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = static_cast<int>(blockIdx.x >> 1), npairs = static_cast<int>(gridDim.x >> 1);
  // work unit u = split * tiles + tile: K blocks [split * kbs, min(KB, (split + 1) * kbs))
  auto unit_tile = [&](int u) { return u % p.tiles; };
  auto unit_k0 = [&](int u) { return (u / p.tiles) * p.kbs; };
  auto unit_k1 = [&](int u) { return min(p.KB, (u / p.tiles + 1) * p.kbs); };
  // this CTA's 128-row tile of pair row tile rt; past the last one its operand rows are zeros
  // (tensor map) or the last tile's codes, and its results are dropped
  auto row_tile = [&](int rt) { return 2 * rt + static_cast<int>(rank); };

  if (threadIdx.x == 0) {
    for (int s = 0; s < S_; ++s) {
      mbar_init(&full[s], kCodes ? 1 + 2 * Lo::kWarpsPer : 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 2 * Lo::kEpiWarps);
    }
    *abort_flag = 0;
    fence_barrier_init();
    if (!kCodes) prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, Lo::kTmemCols);
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync();       // both CTAs' barriers and TMEM exist before either signals the other
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  // (Not from the kernel that writes a rebuilt weight: the next kernel may be one of this library
  // that reads the weight as its A operand before its own wait.)
  if (!p.transposed) pdl_launch_dependents();

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      const uint64_t pol_w = policy_evict_first();
      const uint64_t pol_x = policy_evict_last();
      const bool leader = rank == 0;
      auto load_a = [&](int stage, int rt, int kb) {
        if (leader) mbar_arrive_expect_tx(&full[stage], kFullBytes);
        if (!kCodes)
          tma_load_2d_pair(sA + stage * kATileBytes, &tmA, mapa(smem_u32(&full[stage]), 0),
                           kb * kBK, row_tile(rt) * kBM, pol_w);
      };
      // weight tiles of the first unit do not depend on the previous kernel: a ring of them is
      // requested, and the rest warmed in L2, before waiting for it
      int pre = 0;
      if (pair < p.units) {
        const int rt = unit_tile(pair) / p.TT, rt1 = min(row_tile(rt), p.RT1 - 1);
        const int k0 = unit_k0(pair), k1 = unit_k1(pair);
        pre = min(S_, k1 - k0);
        for (int i = 0; i < pre; ++i) load_a(i, rt, k0 + i);
        for (int kb = k0 + pre; kb < k1; ++kb) {
          if (kCodes)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(
                             p.words + (static_cast<int64_t>(rt1) * p.KB + kb) * 512),
                         "r"(kCodeBytes)
                         : "memory");
          else
            asm volatile(
                "cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(
                    reinterpret_cast<uint64_t>(&tmA)),
                "r"(kb * kBK), "r"(rt1 * kBM)
                : "memory");
        }
      }
      pdl_wait();   // the previous kernel is complete and its writes are visible
      if (p.clear_status && blockIdx.x == 0) *p.status = 0;       // a new call
      // the rounding kernel before this one has read the maximum: ready for the next call
      if (PHASE == kCore && p.amax && blockIdx.x == 0) *p.amax = 0u;
      int stage = 0, it = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int unit = pair; unit < p.units && ok && !*abort_flag; unit += npairs) {
        const int tile = unit_tile(unit), k0 = unit_k0(unit), k1 = unit_k1(unit);
        const int rt = tile / p.TT, tt = tile % p.TT;
        for (int kb = k0; kb < k1; ++kb, ++it) {
          if (it >= pre) {
            if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag)) {
              ok = false;
              break;
            }
            load_a(stage, rt, kb);
          }
          tma_load_2d_pair(sB + stage * Lo::kBTile, &tmB, mapa(smem_u32(&full[stage]), 0),
                           kb * kBK, tt * BN + static_cast<int>(rank) * (BN / 2), pol_x);
          if (++stage == S_) stage = 0, phase ^= 1;
        }
      }
      if (!ok) {
        report(p.status, FQ_ERR_TIMEOUT);
        *abort_flag = 1;
      }
      // The MMAs of each stage's last round are complete (so its copies have landed, and every
      // commit that signals it was made): the waits of one more round of the ring.
      const int rounds = min(it, S_);
      if (it < S_) stage = 0, phase = 1;     // the first ring: stages 0 .. it - 1, phase 0
      for (int r = 0; r < rounds; ++r) {
        if (!mbar_wait(&empty[stage], phase ^ 1, nullptr)) {
          report(p.status, FQ_ERR_TIMEOUT);
          break;
        }
        if (++stage == S_) stage = 0, phase ^= 1;
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (rank 0)
    // The whole warp walks the rounds and one elected lane issues: the operands then are
    // warp-uniform where they are computed, and a round's waits, MMAs and commit take fewer
    // cycles than its MMAs (with one lane walking alone a round took 656 cycles, more than the
    // 256 of four 256 x 128 x 16 MMAs and the 512 of 256 x 256 x 16).
    if (rank == 0) {
      constexpr uint32_t idesc = umma_idesc_bf16(2 * kBM, BN);
      const uint64_t a0 = umma_desc_sw128(smem_u32(sA)), b0 = umma_desc_sw128(smem_u32(sB));
      const bool elected = elect_one();
      int stage = 0, buf = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      for (int unit = pair; unit < p.units; unit += npairs) {
        const int k0 = unit_k0(unit), k1 = unit_k1(unit);
        ok = __all_sync(0xffffffffu, mbar_wait_cluster(&tempty[buf], acc_phase ^ 1, abort_flag));
        if (!ok) break;
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * BN);
        for (int kb = k0; kb < k1; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait_cluster(&full[stage], phase, abort_flag));
          if (!ok) break;
          tc_fence_after_sync();
          if (elected) {
            const uint64_t adesc = a0 + static_cast<uint64_t>(stage * (kATileBytes >> 4));
            const uint64_t bdesc = b0 + static_cast<uint64_t>(stage * (Lo::kBTile >> 4));
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k)
              umma_bf16_pair(d_tmem, adesc + 2 * k, bdesc + 2 * k, idesc,
                             (kb > k0 || k > 0) ? 1u : 0u);
            umma_commit_pair(&empty[stage]);
          }
          __syncwarp();
          if (++stage == S_) stage = 0, phase ^= 1;
        }
        if (!ok) break;
        if (elected) umma_commit_pair(&tfull[buf]);
        __syncwarp();
        if (++buf == 2) buf = 0, acc_phase ^= 1;
      }
      if (!ok && lane == 0) {
        report(p.status, FQ_ERR_TIMEOUT);
        *abort_flag = 1;
      }
    }
  } else if (warp < 2 + Lo::kEpiWarps) {
    // ---------------------------------------------------------------- epilogue (rows)
    constexpr int kN = Lo::kEpiThreads;
    const int quarter = warp & 3;                 // TMEM lanes 32 * quarter .. + 31
    const int c_lo = (warp - 2) / 4 * Lo::kHalf;  // columns c_lo .. c_hi - 1
    const int c_hi = c_lo + Lo::kHalf;
    const int r_in_tile = quarter * 32 + lane;
    const int et = threadIdx.x - 64;
    pdl_wait();
    int buf = 0;
    uint32_t acc_phase = 0;
    for (int unit = pair; unit < p.units; unit += npairs) {
      const int tile = unit_tile(unit), split = unit / p.tiles;
      const int rt = tile / p.TT, tt = tile % p.TT;
      const int rt1 = row_tile(rt);
      const int row = rt1 * kBM + r_in_tile;
      const int t0 = tt * BN;
      const bool row_ok = row < p.R;
      float s_i = 0.f, z_i = 0.f;
      if (PHASE == kCore && row_ok) {
        s_i = __half2float(p.scale[row]);
        z_i = __half2float(p.zero[row]);
      }
      if (PHASE == kCore) {
        // sum_j z[t][j] of the tile's tokens (one per thread), from the analysis' per-tile sums
        const int t = t0 + et;
        float s = 0.f;
        if (et < BN && t < p.M)
#pragma unroll 8
          for (int g = 0; g < p.zsum_tiles; ++g)
            s += ldcg_f32(p.zsum_part + static_cast<int64_t>(g) * p.M + t);
        named_barrier_sync(1, kN);                // the previous unit's sums have been read
        if (et < BN) zsum_s[et] = s;
      }
      const bool fail = !mbar_wait(&tfull[buf], acc_phase, abort_flag);
      if (fail) report(p.status, FQ_ERR_TIMEOUT);
      if (bar_red_or(1, kN, fail || *abort_flag)) {
        if (et == 0) *abort_flag = 1;
        break;
      }
      tc_fence_after_sync();
      const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) +
                             static_cast<uint32_t>(buf * BN);
      const float g_i = (PHASE == kCore && row_ok && p.gamma) ? p.gamma[row] : 1.f;
      // with rounded activations the accumulator is the exact integer sum_j q_ij zbar_j, and
      // u = Delta gamma (s acc + zero sum_j zbar_j)
      const float dl = (PHASE == kCore && p.delta) ? ldcg_f32(p.delta) : 1.f;
      float amax_t = 0.f;
      // the finished values of columns c .. c + 15 of this thread's row, to memory (rows of R
      // are a multiple of 8: a group of 8 or 4 rows is stored whole or not at all)
      const int row_w = rt1 * kBM + quarter * 32;   // the warp's first row
      auto emit = [&](int c, float (&v)[kChunk]) {
        if (PHASE == kAnalysis && p.out32) {
          // fp32 z for the rounding kernel, and the running maximum of |z| (zero past R and M)
#pragma unroll
          for (int q = 0; q < kChunk; ++q) amax_t = fmaxf(amax_t, fabsf(v[q]));
          uint32_t w[16];
          transpose_fp32(v, lane, w);
          const int r = row_w + 4 * (lane >> 2);
          const int t = t0 + c + 8 * (lane & 1) + 4 * ((lane >> 1) & 1);
          float* dst = p.out32 + static_cast<int64_t>(t) * p.R + r;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (r < p.R && t + q < p.M)
              *reinterpret_cast<uint4*>(dst) =
                  make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
            dst += p.R;
          }
          return;
        }
        uint32_t h[8], w[8];
        if (PHASE == kCore) {
#pragma unroll
          for (int q = 0; q < kChunk; q += 4) {
            const float4 zs = *reinterpret_cast<const float4*>(zsum_s + c + q);
            v[q] = g_i * fmaf(s_i, v[q], z_i * zs.x) * dl;
            v[q + 1] = g_i * fmaf(s_i, v[q + 1], z_i * zs.y) * dl;
            v[q + 2] = g_i * fmaf(s_i, v[q + 2], z_i * zs.z) * dl;
            v[q + 3] = g_i * fmaf(s_i, v[q + 3], z_i * zs.w) * dl;
          }
        }
#pragma unroll
        for (int q = 0; q < kChunk; q += 2) {
          const __nv_bfloat162 b = __floats2bfloat162_rn(v[q], v[q + 1]);
          h[q / 2] = *reinterpret_cast<const uint32_t*>(&b);
          if (PHASE == kAnalysis) {
            v[q] = row_ok ? __low2float(b) : 0.f;
            v[q + 1] = row_ok ? __high2float(b) : 0.f;
          }
        }
        if (PHASE == kSynthesis && p.transposed) {
          // this thread's row: 16 consecutive tokens, inside M eight at a time
          __nv_bfloat16* dst = p.out + static_cast<int64_t>(row) * p.M + t0 + c;
          if (row_ok && t0 + c < p.M)
            *reinterpret_cast<uint4*>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
          if (row_ok && t0 + c + 8 < p.M)
            *reinterpret_cast<uint4*>(dst + 8) = make_uint4(h[4], h[5], h[6], h[7]);
          return;
        }
        transpose_bf16(h, lane, w);
        const int r = row_w + 8 * (lane >> 3), t = t0 + c + column16(lane);
        __nv_bfloat16* dst = p.out + static_cast<int64_t>(t) * p.R + r;
        if (r < p.R) {
          if (t < p.M) *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
          if (t + 1 < p.M)
            *reinterpret_cast<uint4*>(dst + p.R) = make_uint4(w[4], w[5], w[6], w[7]);
        }
        if (PHASE == kAnalysis) {
          // per-token sum over the warp's 32 rows of the bf16 z actually stored
          const float s = warp_sums16(v, lane);
          if ((lane & 1) == 0) red[quarter * BN + c + (lane >> 1)] = s;
        }
      };
      // the accumulator of columns c .. c + kW - 1
      constexpr int kG = Lo::kGroups, kW = kG * kChunk;
      auto load = [&](int c, float (&v)[kG][kChunk]) {
#pragma unroll
        for (int g = 0; g < kG; ++g) tmem_ld16(t_row + c + g * kChunk, v[g]);
        tmem_wait_ld();
      };
      auto release = [&]() {
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(mapa(smem_u32(&tempty[buf]), 0));
      };
      bool finish = true;
      if (p.KS == 1) {
#pragma unroll 1
        for (int c = c_lo; c < c_hi; c += kW) {
          float v[kG][kChunk];
          load(c, v);
#pragma unroll
          for (int g = 0; g < kG; ++g) emit(c + g * kChunk, v[g]);
        }
        release();
      } else {
        // Split K.  The CTAs of the 128-row tile's splits take tickets as they get here.  All
        // but the last store their partial tile in the workspace (column-major, so a warp's 32
        // rows are one 128-byte line) and count it in; the last waits for those counts, adds the
        // partials in split order with its own still in TMEM, and finishes the tile.  (The
        // CTAs it waits for are past their MMAs; the wait is bounded like every other.)
        const int64_t t1 = static_cast<int64_t>(rt1) * p.TT + tt;
        const bool mine_ok = rt1 < p.RT1;
        uint32_t* cnt = p.cnt + tile;            // this half's bits: 0-7 tickets, 8-15 stored partials
        const uint32_t shift = 16 * rank;
        if (et == 0)
          *last_flag = mine_ok ? (((atomicAdd(cnt, 1u << shift) >> shift) & 0xffu) ==
                                  static_cast<uint32_t>(p.KS - 1))
                               : 0;
        named_barrier_sync(1, kN);
        finish = *last_flag != 0;
        float* part = p.part + t1 * p.KS * BN * kBM + r_in_tile;
        if (!finish) {
          float* mine = part + static_cast<int64_t>(split) * BN * kBM;
#pragma unroll 1
          for (int c = c_lo; mine_ok && c < c_hi; c += kW) {
            float v[kG][kChunk];
            load(c, v);
#pragma unroll
            for (int q = 0; q < kW; ++q)
              mine[(c + q) * kBM] = v[q / kChunk][q % kChunk];
          }
          release();
          __threadfence();
          named_barrier_sync(1, kN);
          if (et == 0 && mine_ok) {
            __threadfence();
            atomicAdd(cnt, 0x100u << shift);
          }
        } else {
          if (et == 0) {
            const uint32_t want = (static_cast<uint32_t>(p.KS - 1) << 8) | static_cast<uint32_t>(p.KS);
            const long long w0 = clock64();
            while (((ld_acquire_gpu(cnt) >> shift) & 0xffffu) != want) {
              if (clock64() - w0 > kWaitLimitCycles || *abort_flag) {
                report(p.status, FQ_ERR_TIMEOUT);
                *abort_flag = 1;
                break;
              }
            }
            atomicAnd(cnt, ~(0xffffu << shift));   // ready for the next call
          }
          named_barrier_sync(1, kN);
#pragma unroll 1
          for (int c = c_lo; c < c_hi; c += kW) {
            float v[kG][kChunk], own[kG][kChunk];
            load(c, own);
#pragma unroll
            for (int q = 0; q < kW; ++q) v[q / kChunk][q % kChunk] = 0.f;
            for (int sp = 0; sp < p.KS; ++sp) {
              const float* other = part + (static_cast<int64_t>(sp) * BN + c) * kBM;
#pragma unroll
              for (int q = 0; q < kW; ++q)
                v[q / kChunk][q % kChunk] +=
                    sp == split ? own[q / kChunk][q % kChunk] : ldcg_f32(other + q * kBM);
            }
#pragma unroll
            for (int g = 0; g < kG; ++g) emit(c + g * kChunk, v[g]);
          }
          release();
        }
        named_barrier_sync(1, kN);               // the flag is read before it is reused
      }
      if (PHASE == kAnalysis && !p.out32 && finish) {
        // the tile's sum of z per token, quarters added in a fixed order
        named_barrier_sync(1, kN);
        if (et < BN && rt1 < p.RT1 && t0 + et < p.M)
          p.zsum_part[static_cast<int64_t>(rt1) * p.M + t0 + et] =
              (red[et] + red[BN + et]) + (red[2 * BN + et] + red[3 * BN + et]);
        named_barrier_sync(1, kN);                   // read before the next unit's sums
      }
      if (PHASE == kAnalysis && p.out32) {
        // one atomic per warp and tile: the tensor's max |z| (non-negative floats order like
        // their bit patterns)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
          amax_t = fmaxf(amax_t, __shfl_xor_sync(0xffffffffu, amax_t, off));
        if (lane == 0 && amax_t > 0.f) atomicMax(p.amax, __float_as_uint(amax_t));
      }
      if (++buf == 2) buf = 0, acc_phase ^= 1;
    }
  } else {
    // ---------------------------------------------------------------- code decoders (core)
    if (kCodes) {
      // decoder d expands the code blocks of rounds d, d + D, ..., its warps 128 / W rows each
      constexpr int D = Lo::kDecoders, W = Lo::kWarpsPer, kRows = 4 / W;   // rows per lane
      const int dw = warp - 2 - Lo::kEpiWarps;
      const int d = dw / W, row0 = dw % W * (128 / W) + lane;
      // the codes to load next: K block kb of `unit` (past k1: of a later unit), at src
      int unit = pair, kb = 0, k1 = 0;
      const uint4* src = nullptr;
      auto enter = [&](int over) {               // K block k0 + over of the unit
        while (unit < p.units) {
          const int k0 = unit_k0(unit);
          k1 = unit_k1(unit);
          if (k0 + over < k1) {
            kb = k0 + over;
            const int rt1 = min(row_tile(unit_tile(unit) / p.TT), p.RT1 - 1);
            src = reinterpret_cast<const uint4*>(
                      p.words + (static_cast<int64_t>(rt1) * p.KB + kb) * 512) + row0;
            return;
          }
          over -= k1 - k0;
          unit += npairs;
        }
      };
      enter(d);
      uint4 codes[kRows] = {};
      auto fetch = [&]() -> bool {               // the next round's codes; false past the last
        if (unit >= p.units) return false;
#pragma unroll
        for (int rr = 0; rr < kRows; ++rr) codes[rr] = ldg_stream_u4(src + 32 * rr);
        kb += D;
        src += D * (kCodeBytes / 16);
        if (kb >= k1) {
          const int over = kb - k1;
          unit += npairs;
          enter(over);
        }
        return true;
      };
      bool have = fetch();
      int stage = d;                             // round mod S_
      uint32_t phase = 0;                        // (round / S_) & 1
      while (have) {
        const bool got = mbar_wait(&empty[stage], phase ^ 1, abort_flag);
        if (!__all_sync(0xffffffffu, got)) {
          if (lane == 0) {
            report(p.status, FQ_ERR_TIMEOUT);
            *abort_flag = 1;
          }
          break;
        }
        uint8_t* tile_a = sA + stage * kATileBytes;
#pragma unroll
        for (int rr = 0; rr < kRows; ++rr) decode_row_fma(codes[rr], tile_a, row0 + 32 * rr);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(mapa(smem_u32(&full[stage]), 0));
        have = fetch();
        stage += D;
        if (stage >= S_) stage -= S_, phase ^= 1;
      }
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  cluster_sync();          // no CTA leaves while the other may still signal it or use its TMEM
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc_pair(tmem_base, Lo::kTmemCols);
  }
}

// Rounding of the frame representation of the activations (Appendix F): with the tensor's
// step Delta = max |z| / L, L = 2^(N-1) - 1, zq = nearest integer to z / Delta (ties to even,
// clamped to [-L, L]) as bf16 (exact: |zq| <= 127 needs 7 significant bits), and the per-token
// sum of zq for the zero term (exact in fp32 in any order: at most 127 * 81920 < 2^24).
//
// Memory-bound: 6 bytes per coefficient.  A token is rounded by one warp (kPer = 32) or one block
// (kPer = 256), eight coefficients per thread and step (32-byte loads, one 16-byte store; n is
// a multiple of 16).  With one block per token, 4-byte loads and 2-byte stores it took 69 us for 12608
// tokens of 848 coefficients (0.9 TB/s); the ViT fc1 layer went from 327 to 299 us with this.
constexpr int kQuantThreads = 256;

template <int kPer>
__global__ void __launch_bounds__(kQuantThreads) ff_round_kernel(
    const float* __restrict__ z32, int M, int n, float L, const uint32_t* __restrict__ amax,
    float* __restrict__ delta, __nv_bfloat16* __restrict__ zq, float* __restrict__ zsum) {
  constexpr int kTokens = kQuantThreads / kPer;      // tokens per block and round
  __shared__ float red[kQuantThreads / 32];
  pdl_launch_dependents();
  pdl_wait();                                   // the analysis is complete
  const float d = __uint_as_float(*reinterpret_cast<const volatile uint32_t*>(amax)) / L;
  if (blockIdx.x == 0 && threadIdx.x == 0) *delta = d;
  const int sub = threadIdx.x % kPer;
  for (int t0 = blockIdx.x * kTokens; t0 < M; t0 += gridDim.x * kTokens) {
    const int t = t0 + threadIdx.x / kPer;
    float s = 0.f;
    if (t < M) {
      const float* zr = z32 + static_cast<int64_t>(t) * n;
      __nv_bfloat16* qr = zq + static_cast<int64_t>(t) * n;
#pragma unroll 2
      for (int j = 8 * sub; j < n; j += 8 * kPer) {
        const float4 lo = __ldcg(reinterpret_cast<const float4*>(zr + j));
        const float4 hi = __ldcg(reinterpret_cast<const float4*>(zr + j + 4));
        const float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float q[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            q[h] = d > 0.f ? rintf(__fdiv_rn(v[2 * e + h], d)) : 0.f;
            q[h] = fminf(fmaxf(q[h], -L), L);
            s += q[h];
          }
          const __nv_bfloat162 b = __floats2bfloat162_rn(q[0], q[1]);
          w[e] = *reinterpret_cast<const uint32_t*>(&b);
        }
        *reinterpret_cast<uint4*>(qr + j) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (kPer == 32) {
      if (sub == 0 && t < M) zsum[t] = s;
    } else {
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
      __syncthreads();
      if (threadIdx.x == 0) {
        float tot = 0.f;
        for (int w = 0; w < kQuantThreads / 32; ++w) tot += red[w];
        zsum[t] = tot;
      }
      __syncthreads();
    }
  }
}

// The analysis of the d_in unit vectors, for the weight reconstruction: unit vector e_t has
// z = T_in e_t = column t of T_in, exact in bf16, so the analysis product is a transpose,
// z[t][j] = T_in[j][t], with the sums of z over each 128-row tile of T_in, as the analysis of
// tokens leaves them.  Memory-bound (4 bytes per element): a block moves 128 rows x 64 columns through
// shared memory, 16 bytes per access at both ends (a row of 68 elements puts the 16 columns x 2
// row groups that a warp gathers into 32 different banks).  For 4512 x 4096 a 2-byte transpose, a
// separate column-sum kernel and the transpose of the result took 41, 17 and 38 us; rebuilding
// that weight and multiplying 2048 tokens by it went from 336 to 271 us without them.
constexpr int kUnitRows = 128, kUnitCols = 64;

__global__ void __launch_bounds__(256) unit_analysis_kernel(const __nv_bfloat16* __restrict__ T_in,
                                                            int n_in, int d_in,
                                                            __nv_bfloat16* __restrict__ z,
                                                            float* __restrict__ zsum,
                                                            int32_t* __restrict__ status) {
  __shared__ __align__(16) uint16_t tile[kUnitRows][kUnitCols + 4];
  __shared__ float part[4][kUnitCols];
  const int t0 = blockIdx.x * kUnitCols, j0 = blockIdx.y * kUnitRows;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *status = 0;     // a new call
  // d_in is a multiple of 8: eight columns are inside or outside together
#pragma unroll
  for (int it = 0; it < 4; ++it) {
    const int r = 32 * it + tid / 8, c = 8 * (tid % 8);
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (j0 + r < n_in && t0 + c < d_in)
      v = __ldg(reinterpret_cast<const uint4*>(T_in + static_cast<int64_t>(j0 + r) * d_in + t0 + c));
    *reinterpret_cast<uint2*>(&tile[r][c]) = make_uint2(v.x, v.y);
    *reinterpret_cast<uint2*>(&tile[r][c + 4]) = make_uint2(v.z, v.w);
  }
  __syncthreads();
  // a warp and step: 16 columns of T_in, 16 of its rows (n_in is a multiple of 16)
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int q = warp + 8 * k;
    const int c = 16 * (q & 3) + (lane & 15), r = 16 * (q >> 2) + 8 * (lane >> 4);
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      w[e] = tile[r + 2 * e][c] | (static_cast<uint32_t>(tile[r + 2 * e + 1][c]) << 16);
    if (t0 + c < d_in && j0 + r < n_in)
      *reinterpret_cast<uint4*>(z + static_cast<int64_t>(t0 + c) * n_in + j0 + r) =
          make_uint4(w[0], w[1], w[2], w[3]);
  }
  const int c = tid & 63, g = tid >> 6;          // 32 rows of one column per thread
  float s = 0.f;
#pragma unroll 8
  for (int r = 32 * g; r < 32 * g + 32; ++r) s += __uint_as_float(static_cast<uint32_t>(tile[r][c]) << 16);
  part[g][c] = s;
  __syncthreads();
  if (g == 0 && t0 + c < d_in)
    zsum[static_cast<int64_t>(blockIdx.y) * d_in + t0 + c] =
        (part[0][c] + part[1][c]) + (part[2][c] + part[3][c]);
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000,
                                         cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  });
  return fn;
}

// bf16 matrix rows x cols (row-major), boxes of 64 columns x box_rows rows, 128-byte swizzle.
bool make_tmap(CUtensorMap* m, const void* base, int64_t rows, int64_t cols, int box_rows) {
  auto enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(cols) * 2};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(kBK), static_cast<cuuint32_t>(box_rows)};
  cuuint32_t estr[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The token tile that the workspace's partial tiles are sized by.
int pick_bn(int M) { return M <= 128 ? 128 : 256; }

struct DeviceInfo {
  int dev = -1;
  int sms = 0;
};

DeviceInfo device_info() {
  DeviceInfo d;
  cudaGetDevice(&d.dev);
  cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, d.dev);
  if (d.sms <= 0) d.sms = 148;
  return d;
}

template <int PHASE, int BN>
cudaError_t prepare_kernel(int dev) {
  static std::mutex mu;
  static std::map<int, bool> done;
  std::lock_guard<std::mutex> g(mu);
  if (done[dev]) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(tc_phase_kernel<PHASE, BN>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       Layout<PHASE, BN>::kBytes);
  if (e == cudaSuccess) done[dev] = true;
  return e;
}

// K splits of a phase with few tiles (on CTA pairs): up to kMaxSplits, of at least kMinSplitBlocks K
// blocks each.  At 128 tokens a 8192-row phase has only 32 tiles.
constexpr int kMaxSplits = 4;
constexpr int kMinSplitBlocks = 4;
constexpr int kMaxSplitSms = 256;      // bound on the SM count used for split-K planning

// Without pairs: whole tiles, a CTA per SM.  Returns the estimated time in cycles, waves of tiles a K
// block at a time.  On one SM, 128 and 256 tokens per tile (us per call): 4096 x 4096 at 200 tokens
// 4545, 2752, at 512 tokens 8932, 5335; 768 to 3072 at 200 tokens 1147, 772.
constexpr int kOneSmRoundCycles[2] = {600, 740};   // per K block, BN = 128, 256
constexpr int kOneSmEpilogueCycles[2] = {6000, 11000};

int one_sm_bn(int M) { return M <= 128 ? 128 : 256; }

int64_t plan_one_sm(PhaseArgs& a, int sms) {
  const int bn = one_sm_bn(a.M), w = bn / 256;
  a.RT1 = a.RT = static_cast<int>(ceil_div(a.R, kBM));
  a.TT = static_cast<int>(ceil_div(a.M, bn));
  a.KB = static_cast<int>(ceil_div(a.K, kBK));
  a.tiles = a.RT * a.TT;
  return ceil_div(a.tiles, sms) * a.KB * kOneSmRoundCycles[w] + kOneSmEpilogueCycles[w];
}

// CTA pairs: units of 256 x BN tiles (or K splits of them), one pair per unit and
// round.  BN and the K split are those with the least estimated time, in cycles: waves of units,
// each a K block at a time (256 tokens: the MMAs' 512 cycles and a little; 128: 24 KiB of operands
// per CTA from L2), the last tile's epilogue, and for a split the partial tiles' way through L2.
// Measured (us per call; 256-token tiles and every split that fits, then this rule): 768 x 768 at
// 700 tokens 61, 22; 4096 x 4096 at 200 tokens 88, 52, at 300 tokens 77, 68, at 1000 tokens 93, 94;
// 2048 x 2048 at 200 tokens 75, 35; 8192 x 8192 at 256 tokens 116, 114 (128-token tiles: 133).
constexpr int kRoundCycles[2] = {440, 540};       // per K block, BN = 128, 256
constexpr int kEpilogueCycles[2] = {6000, 11000};
constexpr int kSplitFixed[2] = {5000, 10000};     // a split tile, and each of its splits
constexpr int kSplitEach[2] = {1500, 3000};

// Returns the tokens per tile and the estimate.
std::pair<int, int64_t> plan_pairs(PhaseArgs& a, int pairs) {
  a.RT1 = static_cast<int>(ceil_div(a.R, kBM));
  a.RT = static_cast<int>(ceil_div(a.R, 2 * kBM));
  a.KB = static_cast<int>(ceil_div(a.K, kBK));
  int64_t best = INT64_MAX;
  int best_bn = 128;
  for (int w = 0; w < 2; ++w) {
    const int bn = 128 << w, tt = static_cast<int>(ceil_div(a.M, bn)), tiles = a.RT * tt;
    for (int ks = 1; ks <= std::min(kMaxSplits, a.KB / kMinSplitBlocks) || ks == 1; ++ks) {
      const int kbs = static_cast<int>(ceil_div(a.KB, ks));
      if (ks > 1 && (ceil_div(a.KB, kbs) != ks || tiles * ks > pairs || tiles > kWsCntSlots ||
                     static_cast<int64_t>(a.RT1) * tt * ks * bn * kBM > a.part_floats))
        continue;
      const int64_t cost = ceil_div(static_cast<int64_t>(tiles) * ks, pairs) * kbs * kRoundCycles[w] +
                           kEpilogueCycles[w] + (ks > 1 ? kSplitFixed[w] + ks * kSplitEach[w] : 0);
      if (cost < best) {
        best = cost;
        best_bn = bn;
        a.TT = tt;
        a.tiles = tiles;
        a.KS = ks;
        a.kbs = kbs;
      }
    }
  }
  a.units = a.tiles * a.KS;
  return {best_bn, best};
}

struct WsLayout {
  size_t z, u, zsum, part, z32, total;
  int64_t part_floats;       // size of part
};

// Partial tiles for split K, sized for any device with at most kMaxSplitSms SMs: a phase with
// t < kMaxSplitSms tiles keeps at most min(kMaxSplitSms, t * kMaxSplits) partial tiles.
WsLayout ws_layout(int M, int d_in, int n_in, int n_out, int d_out, int act_bits) {
  WsLayout L{};
  size_t off = kWsHeader;
  L.z = off;
  off += round_up(static_cast<int64_t>(M) * n_in * 2, 256);
  L.u = off;
  off += round_up(static_cast<int64_t>(M) * n_out * 2, 256);
  L.zsum = off;
  off += round_up(ceil_div(n_in, kBM) * M * 4, 256);
  const int BN = pick_bn(M);
  const int64_t TT = ceil_div(M, BN);
  const int64_t rows[3] = {n_in, n_out, d_out};
  int64_t slots = 0;
  for (int64_t r : rows) {
    const int64_t tiles = ceil_div(r, kBM) * TT;
    if (tiles < kMaxSplitSms)
      slots = std::max(slots, std::min<int64_t>(kMaxSplitSms, tiles * kMaxSplits));
  }
  (void)d_in;
  L.part = off;
  L.part_floats = slots * BN * kBM;
  off += static_cast<size_t>(slots) * BN * kBM * 4;
  L.z32 = off;
  if (act_bits > 0) off += round_up(static_cast<int64_t>(M) * n_in * 4, 256);
  L.total = off;
  return L;
}

// CTA pairs of this kernel that fit the device at once (0 on an error); sets the kernel's shared
// memory attribute on the device's first call.
template <int PHASE, int BN>
int resident_pairs(int dev) {
  static std::mutex mu;
  static std::map<int, int> cache;
  std::lock_guard<std::mutex> g(mu);
  const auto it = cache.find(dev);
  if (it != cache.end()) return it->second;
  using Lo = PairLayout<PHASE, BN>;
  if (cudaFuncSetAttribute(tc_pair_kernel<PHASE, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           Lo::kBytes) != cudaSuccess)
    return 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(Lo::kThreads);
  cfg.dynamicSmemBytes = Lo::kBytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, tc_pair_kernel<PHASE, BN>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  cache[dev] = n;
  return n;
}

// Launch configuration chained to the previous kernel with programmatic dependent launch.
struct ChainedLaunch {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  ChainedLaunch(int grid, int threads, int smem, cudaStream_t s) {
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = static_cast<size_t>(smem);
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  ChainedLaunch(const ChainedLaunch&) = delete;
};

// One phase of a call, planned with its tensor maps before anything is launched.
struct PhasePlan {
  CUtensorMap A, B;
  bool pairs;                // on CTA pairs, else the one-SM kernel
  int bn;                    // tokens per tile
  int grid;
};

// A: the weight operand (R x K; not used by the code product), B: the tokens (M x K).  CTA pairs for
// budgets of two SMs and more; an odd budget leaves an SM without a partner, so there the one-SM
// kernel on all of them is taken where its estimate is lower.  At three SMs (us per call, one pair and
// three CTAs): 4096 x 4096 at 129 tokens 1013, 949, at 512 tokens 2015, 1834; 768 to 3072 at 128
// tokens 232, 207, at 512 tokens 595, 546.  At five, two pairs beat five CTAs: 4096 x 4096 at 512
// tokens 1018, 1147.
template <int PHASE>
bool plan_call_phase(PhasePlan& pl, PhaseArgs& a, const void* A, const void* B,
                     const DeviceInfo& d) {
  int64_t cost = INT64_MAX;
  pl.pairs = d.sms >= 2;
  if (pl.pairs) {
    const int pairs = std::min({resident_pairs<PHASE, 128>(d.dev), resident_pairs<PHASE, 256>(d.dev),
                                d.sms / 2});
    if (pairs < 1) return false;
    std::tie(pl.bn, cost) = plan_pairs(a, pairs);
    pl.grid = 2 * std::min(a.units, pairs);
  }
  if (d.sms % 2 && !a.transposed) {            // (the one-SM kernel has no transposed store)
    PhaseArgs one = a;
    const int64_t one_cost = plan_one_sm(one, d.sms);
    if (one_cost < cost) {
      cost = one_cost;
      a = one;
      pl.pairs = false;
      pl.bn = one_sm_bn(a.M);
      pl.grid = std::min(a.tiles, d.sms);
      if ((pl.bn == 128 ? prepare_kernel<PHASE, 128>(d.dev) : prepare_kernel<PHASE, 256>(d.dev)) !=
          cudaSuccess)
        return false;
    }
  }
  if (cost == INT64_MAX) return false;
  // a pair's CTAs load half of a tile's tokens each
  if (!make_tmap(&pl.B, B, a.M, a.K, pl.pairs ? pl.bn / 2 : pl.bn)) return false;
  if (PHASE == kCore) {
    pl.A = pl.B;
    return true;
  }
  return make_tmap(&pl.A, A, a.R, a.K, kBM);
}

template <int PHASE, int BN>
cudaError_t launch_pairs(const PhasePlan& pl, const PhaseArgs& a, cudaStream_t s) {
  using Lo = PairLayout<PHASE, BN>;
  const ChainedLaunch l(pl.grid, Lo::kThreads, Lo::kBytes, s);
  return cudaLaunchKernelEx(&l.cfg, tc_pair_kernel<PHASE, BN>, pl.A, pl.B, a);
}

template <int PHASE, int BN>
cudaError_t launch_one_sm(const PhasePlan& pl, const PhaseArgs& a, cudaStream_t s) {
  const ChainedLaunch l(pl.grid, threads_for<PHASE>(), Layout<PHASE, BN>::kBytes, s);
  return cudaLaunchKernelEx(&l.cfg, tc_phase_kernel<PHASE, BN>, pl.A, pl.B, a);
}

template <int PHASE>
cudaError_t launch_phase(const PhasePlan& pl, const PhaseArgs& a, cudaStream_t s) {
  if (pl.pairs)
    return pl.bn == 128 ? launch_pairs<PHASE, 128>(pl, a, s) : launch_pairs<PHASE, 256>(pl, a, s);
  return pl.bn == 128 ? launch_one_sm<PHASE, 128>(pl, a, s) : launch_one_sm<PHASE, 256>(pl, a, s);
}

cudaError_t launch_round(const PhaseArgs& an, int n_in, int act_bits, const DeviceInfo& d,
                         float* delta, __nv_bfloat16* zq, float* zsum, cudaStream_t s) {
  // A warp per token once there are tokens for most of the SMs' warps, sooner where a token has work
  // for few of a block's threads; a block per token otherwise.  Whole layers, us with a block and
  // with a warp per token: n_in = 288 at 608 tokens 19.5, 20.3, at 1216 22.5, 20.5; 848 at 2432 33.0, 34.9,
  // at 4864 47.6, 46.7, at 12608 85.7, 79.4; 2256 at 2432 90.2, 92.2, at 4864 130.6, 125.3; 3392 at 4864
  // 128.6, 134.7, at 12608 348, 335; 4512 at 4864 357, 361, at 12608 1071, 1054.
  const bool warps = an.M >= (n_in <= 512 ? 8 : (n_in <= 2304 ? 32 : 64)) * d.sms;
  const int blocks = static_cast<int>(ceil_div(an.M, warps ? kQuantThreads / 32 : 1));
  const ChainedLaunch l(std::min(blocks, 8 * d.sms), kQuantThreads, 0, s);
  const float L = static_cast<float>((1 << (act_bits - 1)) - 1);
  return cudaLaunchKernelEx(&l.cfg, warps ? ff_round_kernel<32> : ff_round_kernel<kQuantThreads>,
                            static_cast<const float*>(an.out32), an.M, n_in, L,
                            static_cast<const uint32_t*>(an.amax), delta, zq, zsum);
}

// The dense product of the weight-reconstruction path: one synthesis-phase kernel with the
// reconstructed weight as its A operand.
WsLayout dense_ws_layout(int M, int d_out) {
  WsLayout L{};
  const int BN = pick_bn(M);
  const int64_t tiles = ceil_div(d_out, kBM) * ceil_div(M, BN);
  int64_t slots = 0;
  if (tiles < kMaxSplitSms) slots = std::min<int64_t>(kMaxSplitSms, tiles * kMaxSplits);
  L.part = kWsHeader;
  L.part_floats = slots * BN * kBM;
  L.total = L.part + static_cast<size_t>(slots) * BN * kBM * 4;
  return L;
}

fq_status launch_tc_dense(const void* x, int M, int d_in, const void* W, int d_out, void* y,
                          char* ws, size_t ws_bytes, cudaStream_t s) {
  const WsLayout L = dense_ws_layout(M, d_out);
  if (ws_bytes < L.total) return FQ_ERR_WORKSPACE;
  PhaseArgs a{};
  a.R = d_out;
  a.K = d_in;
  a.M = M;
  a.out = reinterpret_cast<__nv_bfloat16*>(y);
  a.clear_status = 1;
  a.status = reinterpret_cast<int32_t*>(ws);
  a.cnt = reinterpret_cast<uint32_t*>(ws + kWsCnt);
  a.part = reinterpret_cast<float*>(ws + L.part);
  a.part_floats = L.part_floats;
  PhasePlan pl;
  if (!plan_call_phase<kSynthesis>(pl, a, W, x, device_info())) return FQ_ERR_CUDA;
  return launch_phase<kSynthesis>(pl, a, s) == cudaSuccess ? FQ_OK : FQ_ERR_CUDA;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

size_t tc_workspace_bytes(int M, int d_in, int n_in, int n_out, int d_out, int act_bits) {
  return ws_layout(M, d_in, n_in, n_out, d_out, act_bits).total;
}

fq_status launch_tc_forward(const void* x, int M, int d_in, const void* T_in,
                            const fq_packed& Cq, const void* T_out_t, int d_out,
                            const float* gamma, void* y, char* ws, size_t ws_bytes,
                            int max_sms, int act_bits, cudaStream_t s) {
  const int n_in = Cq.n_in, n_out = Cq.n_out;
  const WsLayout L = ws_layout(M, d_in, n_in, n_out, d_out, act_bits);
  if (ws_bytes < L.total) return FQ_ERR_WORKSPACE;
  auto* status = reinterpret_cast<int32_t*>(ws);
  auto* z = reinterpret_cast<__nv_bfloat16*>(ws + L.z);
  auto* u = reinterpret_cast<__nv_bfloat16*>(ws + L.u);
  auto* zsum = reinterpret_cast<float*>(ws + L.zsum);

  PhaseArgs a[3];
  const int R[3] = {n_in, n_out, d_out};
  const int K[3] = {d_in, n_in, n_out};
  __nv_bfloat16* outs[3] = {z, u, reinterpret_cast<__nv_bfloat16*>(y)};
  for (int ph = 0; ph < 3; ++ph) {
    a[ph] = PhaseArgs{};
    a[ph].R = R[ph];
    a[ph].K = K[ph];
    a[ph].M = M;
    a[ph].out = outs[ph];
    a[ph].zsum_part = zsum;
    a[ph].status = status;
    a[ph].cnt = reinterpret_cast<uint32_t*>(ws + kWsCnt);
    a[ph].part = reinterpret_cast<float*>(ws + L.part);
    a[ph].part_floats = L.part_floats;
  }
  a[0].clear_status = 1;
  a[1].words = Cq.words;
  a[1].scale = reinterpret_cast<const __half*>(Cq.scale_f16);
  a[1].zero = reinterpret_cast<const __half*>(Cq.zero_f16);
  a[1].gamma = gamma;
  float* delta = nullptr;
  if (act_bits > 0) {
    a[0].out32 = reinterpret_cast<float*>(ws + L.z32);
    a[0].amax = reinterpret_cast<uint32_t*>(ws + kWsAmax);
    delta = reinterpret_cast<float*>(ws + kWsDelta);
    a[1].amax = a[0].amax;
    a[1].delta = delta;
  }

  DeviceInfo d = device_info();
  if (max_sms > 0) d.sms = std::min(d.sms, max_sms);
  a[1].zsum_tiles =
      act_bits > 0 ? 1 : static_cast<int>(ceil_div(n_in, kBM));   // rounded: one exact sum
  PhasePlan pl[3];
  if (!plan_call_phase<kAnalysis>(pl[0], a[0], T_in, x, d) ||
      !plan_call_phase<kCore>(pl[1], a[1], nullptr, z, d) ||
      !plan_call_phase<kSynthesis>(pl[2], a[2], T_out_t, u, d))
    return FQ_ERR_CUDA;
  if (launch_phase<kAnalysis>(pl[0], a[0], s) != cudaSuccess) return FQ_ERR_CUDA;
  if (act_bits > 0 &&
      launch_round(a[0], n_in, act_bits, d, delta, a[0].out, a[0].zsum_part, s) != cudaSuccess)
    return FQ_ERR_CUDA;
  if (launch_phase<kCore>(pl[1], a[1], s) != cudaSuccess ||
      launch_phase<kSynthesis>(pl[2], a[2], s) != cudaSuccess)
    return FQ_ERR_CUDA;
  return FQ_OK;
}

fq_status launch_tc_unit_forward(const void* T_in, int d_in, const fq_packed& Cq,
                                 const void* T_out_t, int d_out, const float* gamma, void* W_hat,
                                 char* ws, size_t ws_bytes, cudaStream_t s) {
  const int M = d_in, n_in = Cq.n_in, n_out = Cq.n_out;
  const WsLayout L = ws_layout(M, d_in, n_in, n_out, d_out, 0);
  if (ws_bytes < L.total) return FQ_ERR_WORKSPACE;
  auto* status = reinterpret_cast<int32_t*>(ws);
  auto* z = reinterpret_cast<__nv_bfloat16*>(ws + L.z);
  auto* u = reinterpret_cast<__nv_bfloat16*>(ws + L.u);
  auto* zsum = reinterpret_cast<float*>(ws + L.zsum);
  const auto* Tin = static_cast<const __nv_bfloat16*>(T_in);

  PhaseArgs a[3];
  const int R[3] = {n_in, n_out, d_out};
  const int K[3] = {d_in, n_in, n_out};
  __nv_bfloat16* outs[3] = {z, u, reinterpret_cast<__nv_bfloat16*>(W_hat)};
  for (int ph = 1; ph < 3; ++ph) {
    a[ph] = PhaseArgs{};
    a[ph].R = R[ph];
    a[ph].K = K[ph];
    a[ph].M = M;
    a[ph].out = outs[ph];
    a[ph].zsum_part = zsum;
    a[ph].status = status;
    a[ph].cnt = reinterpret_cast<uint32_t*>(ws + kWsCnt);
    a[ph].part = reinterpret_cast<float*>(ws + L.part);
    a[ph].part_floats = L.part_floats;
  }
  a[1].words = Cq.words;
  a[1].scale = reinterpret_cast<const __half*>(Cq.scale_f16);
  a[1].zero = reinterpret_cast<const __half*>(Cq.zero_f16);
  a[1].gamma = gamma;
  a[2].transposed = 1;                           // the output's rows are those of W_hat

  a[1].zsum_tiles = static_cast<int>(ceil_div(n_in, kUnitRows));
  const DeviceInfo d = device_info();
  PhasePlan pl[2];
  if (!plan_call_phase<kCore>(pl[0], a[1], nullptr, z, d) ||
      !plan_call_phase<kSynthesis>(pl[1], a[2], T_out_t, u, d))
    return FQ_ERR_CUDA;

  unit_analysis_kernel<<<dim3(static_cast<unsigned>(ceil_div(d_in, kUnitCols)),
                              static_cast<unsigned>(ceil_div(n_in, kUnitRows))),
                         256, 0, s>>>(Tin, n_in, d_in, z, zsum, status);
  if (cudaGetLastError() != cudaSuccess) return FQ_ERR_CUDA;
  return launch_phase<kCore>(pl[0], a[1], s) == cudaSuccess &&
                 launch_phase<kSynthesis>(pl[1], a[2], s) == cudaSuccess
             ? FQ_OK
             : FQ_ERR_CUDA;
}

}  // namespace fq

extern "C" {

size_t fq_dense_workspace_bytes(int M, int d_in, int d_out) {
  if (M <= 0 || d_in <= 0 || d_out <= 0) return 0;
  return fq::dense_ws_layout(M, d_out).total;
}

fq_status fq_dense_forward(const void* x, int M, int d_in, const void* W_hat, int d_out, void* y,
                           void* ws, size_t ws_bytes, fq_stream_t stream) {
  if (!x || !W_hat || !y || M <= 0 || d_in <= 0 || d_out <= 0) return FQ_ERR_INVALID_ARG;
  if (d_in % 8 || d_out % 8 || !fq::aligned16(x) || !fq::aligned16(W_hat) || !fq::aligned16(y))
    return FQ_ERR_ALIGNMENT;
  if (!ws) return FQ_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0) return FQ_ERR_ALIGNMENT;
  if (ws_bytes < fq_dense_workspace_bytes(M, d_in, d_out)) return FQ_ERR_WORKSPACE;
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess)
    return FQ_ERR_CUDA;
  if (major * 10 + minor != 103) return FQ_ERR_UNSUPPORTED;
  return fq::launch_tc_dense(x, M, d_in, W_hat, d_out, y, static_cast<char*>(ws), ws_bytes,
                             reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"
