// us_ffn_hidden: the two GEMMs that end in the hidden layer of the FFN block as ONE launch.
//
//   H  = alpha  * X W1                                   (first forward GEMM,          K = d_model)
//   A  = round(act_out * gelu(act_in * H))               (to FP8, or to the 16-bit operand format)
//   dA = beta_x * G W2^T                                 (second layer's input gradient, K = d_model)
//   dH = round(grad_out * act_in * gelu'(act_in * round16(H)) * dA)
//
// Both GEMMs produce a [tokens x d_ff] matrix and the GELU gradient needs, element for element, the
// pre-activation H the forward GEMM has just produced.  Launched separately, H travels to memory in
// 16 bits and back (2 x 2 bytes per element of the largest tensor of the block), and both kernels'
// stores compete with their operand loads for the SM's memory path.  Here a CTA pair computes, for
// one 256 x 256 output tile, first X W1 into accumulator 0 and then G W2^T into accumulator 1 of
// tensor memory.  The sixteen epilogue warps turn accumulator 0 into A while the MMAs
// of accumulator 1 run (stored as FP8 or in the 16-bit operand format), keep H -- rounded to the 16-bit format the unfused path stores it in -- in
// registers, and turn accumulator 1 into dH while the next tile's X W1 runs: the two
// accumulators alternate exactly as two consecutive tiles of gemm_kernel do, and H never leaves the SM
// (unless the caller asks for a copy).  Results are bit-identical to us_linear_fwd + GELU epilogue
// followed by us_linear_bwd_x + GELU-gradient epilogue.
//
// Bound: tensor pipe, in a long run the power cap.  Measured, separate launches -> this one, us:
// FP8 8192 x 1024 x 4096: 86 -> 67;  BF16 8192 x 1024 x 4096 (H copy kept): 171 -> 138;  FP8 16384 x 2048 x 8192:
// 550 -> 507;  FP8 256 x 128 x 512 on 128 x 128 tiles: 12.3 + a launch gap -> 7.2, with the columns of a tile split over four CTAs
// (and the grouped launch over two) the whole three-launch step 16.4 -> 12.3.
#include <cuda.h>

#include <algorithm>

#include <type_traits>

#include "gemm_kernel.cuh"
#include "host.h"

namespace us {
namespace {

constexpr int kHidEW = 16;
// Shared-memory plan: 32 KB operand stages (this CTA's 128 rows of A and 128 rows of B, 128 bytes of K each) and one
// output box of 32 rows per epilogue warp, BN / 4 columns of OES bytes.  The kept pre-activation lives in registers,
// which leaves room for six stages (five with 16-bit outputs and 256-column tiles).
// NB: columns of the products a CTA computes, 64 where several share a tile; then 24 KB stages, or smaller ones with fewer
// rows of A than 128, in as many as fit.
template <int BN, int OES, int NB>
struct HidSmem {
  static constexpr int kABytes = kBM * kStageKBytes;
  static constexpr int kBBytes = (NB == 64 ? 64 : 128) * kStageKBytes;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kRowBytes = BN / 4 * OES;                     // of an output box: 32, 64 or 128
  static constexpr int kEpiWarpBytes = 32 * kRowBytes;
  static constexpr int kEpiBytes = kHidEW * kEpiWarpBytes;
  static constexpr int kStages = (229376 - kEpiBytes) / kStageBytes;
  static constexpr int kMaxStages = NB == 64 ? 16 : kStages;
  static constexpr int kBarrierBytes = 512;
  static constexpr int kTotal = kStages * kStageBytes + kEpiBytes + kBarrierBytes + 1024;   // + alignment slack
};

struct HiddenParams {
  int M, N, K1, K2;                 // outputs are [M x N]; contraction lengths of X W1 and of G W2^T
  int tiles_m, tiles_n;
  FastDiv d_tiles_m;
  uint32_t idesc1, idesc2;
  float scale1, scale2;             // alpha, beta_x
  float act_in, act_out, grad_out;  // s_in, alpha_g, beta_g
  uint8_t* h_ptr; long long h_ld;   // optional copy of the rounded pre-activation (NULL: none); ld in elements
  int h_sectors;                    // its rows start on 32-byte boundaries
  uint8_t *a_ptr, *d_ptr; long long a_ld, d_ld;   // A and dH, for SPLIT > 1 (otherwise reached by TMA)
  unsigned int* status;
  uint32_t wait_limit;
  uint32_t x_bytes; int stages;     // SPLIT > 1: bytes of X or G in a stage (the rows that exist), and the stages that fit
  int starved, served;              // test hook (starved_cta)
};

// ES: operand bytes per element (1 = FP8, 2 = BF16 / F16).  BN, CG: tiles of 256 x 256 per CTA pair (256, 2), or of
// 128 x 128 per CTA (128, 1) where the large ones would leave more than half of the pairs idle (hidden_impl).
// SPLIT (128 x 128 tiles): CTAs that share a tile, each computing 64 of its columns (of four, two the same ones) and turning 128 / SPLIT
// into outputs.  In a small problem the arithmetic of the epilogue (3700 + 2800 cycles of one SM's issue slots for a tile) is the
// longest part of the launch while most SMs are idle.  With all 128 columns computed by each they fetched a third more bytes (32 KB a K block
// instead of 24, with few rows twice as many): captured steps, us, 48 x 1024 x 4096 30.7 -> 28.7, 16 x 1024 x 4096 32.4 -> 29.1, 512 x 512 x 1456 15.0 -> 14.8.
// OUT_A, OUT_D: output formats of A and dH (us_dtype).  H_BF16: pre-activation rounded to BF16 (else F16).
template <int ES, int BN, int CG, int SPLIT, int OUT_A, int OUT_D, bool H_BF16>
__global__ void __launch_bounds__(gemm_threads(kHidEW), 1)
ffn_hidden_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w1,
                  const __grid_constant__ CUtensorMap tm_g, const __grid_constant__ CUtensorMap tm_w2,
                  const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_dh,
                  const HiddenParams p) {
  constexpr int kOes = OUT_A == US_E4M3 || OUT_A == US_E5M2 ? 1 : 2;
  constexpr int kNB = SPLIT > 1 ? 64 : BN;          // columns of an accumulator
  using S = HidSmem<BN, kOes, kNB>;
  static_assert(BN / CG == 128, "128 rows of B per CTA");
  constexpr int kBK = 128 / ES;                     // K elements per stage
  constexpr int kTileM = kBM * CG;
  static_assert(SPLIT == 1 || (CG == 1 && BN == 128 && (SPLIT == 2 || SPLIT == 4)), "split tiles are 128 x 128");
  constexpr int kWarpCols = SPLIT > 1 ? 16 : BN / 4;            // columns of a tile one epilogue warp handles,
  constexpr int kSliceCols = SPLIT > 1 ? 16 : 32, kSlices = kWarpCols / kSliceCols;   // worked in slices
  constexpr int kWarpsUsed = SPLIT > 1 ? 4 * (BN / SPLIT / kWarpCols) : kHidEW;
  constexpr uint32_t kChunkBytes = kBK * 128;       // a box of an MN-major operand tile: kBK rows of K x 128 bytes
  constexpr uint32_t kTmemCols = 2 * kNB;
  constexpr bool kHalfRowB = SPLIT > 1 && ES == 1;  // W1 in rows of 64 bytes
  const uint32_t x_bytes = SPLIT > 1 ? p.x_bytes : (uint32_t)S::kABytes, stage_bytes = x_bytes + S::kBBytes;
  const int stages = SPLIT > 1 ? p.stages : S::kStages;

  ptx::grid_release_next();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (ptx::smem_addr(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - ptx::smem_addr(smem_raw));
  const uint32_t epi_base = smem_base + S::kStages * S::kStageBytes;
  const uint32_t bars = epi_base + S::kEpiBytes;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (S::kMaxStages + s); };
  auto acc_full_bar = [&](int a) { return bars + 8u * (2 * S::kMaxStages + a); };
  auto acc_empty_bar = [&](int a) { return bars + 8u * (2 * S::kMaxStages + 2 + a); };
  const uint32_t drained_bar = bars + 8u * (2 * S::kMaxStages + 4);
  static_assert(8 * (2 * S::kMaxStages + 5) + 8 <= S::kBarrierBytes, "barrier area too small");
  uint8_t* tail = smem_gen + S::kStages * S::kStageBytes + S::kEpiBytes + 8 * (2 * S::kMaxStages + 5);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(tail);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = CG == 2 ? (int)ptx::cluster_ctarank() : 0;
  const int pair = blockIdx.x / (CG * SPLIT), num_pairs = gridDim.x / (CG * SPLIT);      // tile-walking unit: CTA pair or CTA(s)
  const int split_col = SPLIT > 1 ? (int)(blockIdx.x % SPLIT) * (BN / SPLIT) : 0;        // this CTA's first output column of the tile
  const int split_acc = SPLIT > 1 ? split_col % 64 : 0;                                  // and where it is in the accumulators
  const int num_tiles = p.tiles_m * p.tiles_n;
  const int kb1 = (p.K1 + kBK - 1) / kBK, kb2 = (p.K2 + kBK - 1) / kBK;
  // column-major over the tiles: pairs that run side by side share a panel of W1 and of W2
  auto tile_mn2 = [&](int tile, int& tm, int& tn) { tn = p.d_tiles_m.div(tile); tm = tile - tn * p.tiles_m; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { ptx::mbar_init(full_bar(s), 1); ptx::mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < 2; ++a) { ptx::mbar_init(acc_full_bar(a), 1); ptx::mbar_init(acc_empty_bar(a), CG * kWarpsUsed); }
    ptx::mbar_init(drained_bar, 1);
    *abort_flag = 0;
    ptx::mbar_init_fence();
    ptx::prefetch_tensormap(&tm_x);
    ptx::prefetch_tensormap(&tm_w1);
    ptx::prefetch_tensormap(&tm_g);
    ptx::prefetch_tensormap(&tm_w2);
  }
  if (warp == 1) {
    if (CG == 2) { ptx::tmem_alloc_pair(ptx::smem_addr(const_cast<uint32_t*>(tmem_slot)), kTmemCols); ptx::tmem_relinquish_pair(); }
    else { ptx::tmem_alloc(ptx::smem_addr(const_cast<uint32_t*>(tmem_slot)), kTmemCols); ptx::tmem_relinquish(); }
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (CG == 2) ptx::cluster_meet();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (every CTA)
    if (ptx::elect_one()) {
      uint32_t issued = 0;
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      const int end = starved_cta(p.starved, rank) ? min(num_tiles, pair + p.served * num_pairs) : num_tiles;
      for (int tile = pair; ok && tile < end; tile += num_pairs) {
        int tm, tn;
        tile_mn2(tile, tm, tn);
        const int m0 = tm * kTileM + rank * 128, n0 = tn * BN + rank * 128 + (split_col - split_acc);
        for (int sub = 0; ok && sub < 2; ++sub) {
          const int num_kb = sub ? kb2 : kb1;
          for (int kb = 0; kb < num_kb; ++kb) {
            ok = wait_bounded(empty_bar(stage), phase ^ 1u, abort_flag, p.status, p.wait_limit);
            if (!ok) break;
            const uint32_t a_dst = smem_base + stage * stage_bytes, b_dst = a_dst + x_bytes;
            const int k0 = kb * kBK;
            if (issued == 0) ptx::grid_wait_previous();       // coordinates and barriers are ready: only the loads wait
            const uint32_t fb = CG == 2 ? ptx::in_even_cta(full_bar(stage)) : full_bar(stage);
            if (rank == 0) ptx::mbar_expect_tx(full_bar(stage), CG * stage_bytes);
            auto load = [&](uint32_t dst, const void* tmap, int x, int y) {
              if (CG == 2) ptx::tma_load_2d_pair(dst, tmap, fb, x, y); else ptx::tma_load_2d(dst, tmap, fb, x, y);
            };
            if (sub == 0) {
              load(a_dst, &tm_x, k0, m0);                           // X  [M x K1], K-major
#pragma unroll
              for (int c = 0; c < (SPLIT > 1 ? 1 : ES); ++c) load(b_dst + c * kChunkBytes, &tm_w1, n0 + c * kBK, k0);   // W1 [K1 x N], N-major, 128 / ES columns per box
            } else {
              load(a_dst, &tm_g, k0, m0);                           // G  [M x K2], K-major
              load(b_dst, &tm_w2, k0, n0);                          // W2 [N x K2], K-major
            }
            ++issued;
            if (++stage == stages) { stage = 0; phase ^= 1u; }
          }
        }
      }
      if (*abort_flag && rank == 0) {
        // Let copies that are still in flight land before the CTA gives up its shared memory.
        const uint32_t n = issued < (uint32_t)stages ? issued : (uint32_t)stages;
        for (uint32_t i = 0; i < n; ++i) {
          if (stage == 0) { stage = stages; phase ^= 1u; }
          --stage;
          for (uint32_t it = 0; it < p.wait_limit && !ptx::mbar_try_wait(full_bar(stage), phase); ++it) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (even CTA of a pair only)
    if (ptx::elect_one() && rank == 0) {
      ptx::grid_wait_previous();                       // no operand comes earlier: the bounded waits begin when the loads do
      int stage = 0; uint32_t phase = 0, local = 0;
      bool ok = true;
      const uint32_t stage_step = stage_bytes >> 4;
      const uint64_t a_desc = ptx::smem_desc_sw128(smem_base, 16, 1024);                              // K-major
      const uint64_t b_desc_mn = kHalfRowB ? ptx::smem_desc_sw64(smem_base + x_bytes, 16, 512)
                                           : ptx::smem_desc_sw128(smem_base + x_bytes, kChunkBytes, 1024);    // W1: N-major
      const uint64_t b_desc_k = ptx::smem_desc_sw128(smem_base + x_bytes, 16, 1024);                  // W2: K-major
      const uint32_t a_hi = (uint32_t)(a_desc >> 32), a_lo0 = (uint32_t)a_desc;
      for (int tile = pair; ok && tile < num_tiles; tile += num_pairs, ++local) {
        const uint32_t acc_phase = local & 1u;
        for (int sub = 0; ok && sub < 2; ++sub) {
          const uint64_t b_desc = sub ? b_desc_k : b_desc_mn;
          const uint32_t b_hi = (uint32_t)(b_desc >> 32), b_lo0 = (uint32_t)b_desc;
          const uint32_t b_step = (sub ? 32u : (kHalfRowB ? kChunkBytes / 2 : kChunkBytes) / kKSteps) >> 4;
          const uint32_t idesc = sub ? p.idesc2 : p.idesc1;
          const int num_kb = sub ? kb2 : kb1;
          ok = wait_bounded(acc_empty_bar(sub), acc_phase ^ 1u, abort_flag, p.status, p.wait_limit);
          if (!ok) break;
          ptx::tc_fence_after_sync();
          const uint32_t d_tmem = tmem_base + sub * kNB;
          uint32_t accumulate = 0;
          for (int kb = 0; kb < num_kb; ++kb) {
            if (!ptx::mbar_try_wait(full_bar(stage), phase)) {
              ok = wait_bounded(full_bar(stage), phase, abort_flag, p.status, p.wait_limit);
              if (!ok) break;
            }
            ptx::tc_fence_after_sync();
            const uint32_t a_lo = a_lo0 + stage * stage_step, b_lo = b_lo0 + stage * stage_step;
#pragma unroll
            for (int k = 0; k < kKSteps; ++k) {
              const uint64_t adesc = ((uint64_t)a_hi << 32) | (a_lo + k * 2u);
              const uint64_t bdesc = ((uint64_t)b_hi << 32) | (b_lo + k * b_step);
              if (CG == 2) ptx::mma_ss_pair<ES == 1>(d_tmem, adesc, bdesc, idesc, accumulate);
              else ptx::mma_ss<ES == 1>(d_tmem, adesc, bdesc, idesc, accumulate);
              accumulate = 1;
            }
            if (CG == 2) ptx::mma_commit_pair(empty_bar(stage), 3); else ptx::mma_commit(empty_bar(stage));
            if (++stage == stages) { stage = 0; phase ^= 1u; }
          }
          if (ok) { if (CG == 2) ptx::mma_commit_pair(acc_full_bar(sub), 3); else ptx::mma_commit(acc_full_bar(sub)); }
        }
      }
      if (*abort_flag) {
        if (CG == 2) ptx::mma_commit_pair(drained_bar, 1); else ptx::mma_commit(drained_bar);
        for (uint32_t it = 0; it < p.wait_limit && !ptx::mbar_try_wait(drained_bar, 0); ++it) {}
      }
    }
  } else if (warp - 2 < kWarpsUsed) {
    // ------------------------------------------------------------ epilogue warps
    ptx::grid_wait_previous();
    // Warp (lane quarter q, part) owns 32 rows x kWarpCols columns of the tile; a lane holds one row of them.  The
    // rounded pre-activation of a tile stays in registers as packed 16-bit pairs (hst) between the two phases; staging
    // is one output box of 32 rows per warp, swizzled with the pattern of its row width (32-byte rows: none).
    const int q = warp & 3, part = (warp - 2) >> 2;
    const uint32_t buf_out = epi_base + (warp - 2) * S::kEpiWarpBytes;
    const uint32_t box_row = (uint32_t)lane * S::kRowBytes;
    const uint32_t box_sw = S::kRowBytes == 128 ? (uint32_t)(lane & 7) : S::kRowBytes == 64 ? (uint32_t)((lane >> 1) & 3) : 0u;
    const f32x2 s1 = splat2(p.scale1), s2 = splat2(p.scale2), in2 = splat2(p.act_in), os2 = splat2(p.grad_out * p.act_in);
    const float tail_k = fabsf(p.act_in) * (1.0f / kTailRange), act_oi = p.act_out * p.act_in;

    auto release_acc = [&](int a, int tile) {                   // (where no later tile takes it nobody waits)
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0 && tile + num_pairs < num_tiles) {
        if (CG == 2) ptx::mbar_arrive_cluster(ptx::in_even_cta(acc_empty_bar(a)));
        else ptx::mbar_arrive(acc_empty_bar(a));
      }
    };
    // Eight outputs of this lane's row, group g of slice s, into the box: 16-byte chunk c at c ^ box_sw.
    // (SPLIT > 1: straight to memory, the 16-byte pieces of this lane's row.)
    uint8_t* direct = nullptr;
    int direct_cols = 0;                                        // columns of the lane's part that exist
    auto put = [&](uint32_t c, uint4 v, int es) {               // 16 / es values from column c * 16 / es of the warp's part
      if constexpr (SPLIT == 1) {
        ptx::sts128(buf_out + box_row + ((c ^ box_sw) << 4), v);
      } else {
        const int per = 16 / es, col = (int)c * per;
        if (col + per <= direct_cols) {
          *reinterpret_cast<uint4*>(direct + c * 16u) = v;
        } else {
          const uint32_t w[4] = {v.x, v.y, v.z, v.w};
          for (int i = 0; i < per && col + i < direct_cols; ++i) {
            if (es == 1) direct[c * 16u + i] = (uint8_t)(w[i >> 2] >> (8 * (i & 3)));
            else reinterpret_cast<uint16_t*>(direct + c * 16u)[i] = (uint16_t)(w[i >> 1] >> (16 * (i & 1)));
          }
        }
      }
    };
    auto stage_out = [&](auto fmt, const float (&y)[8], uint32_t (&held)[2], int s, int g) {
      constexpr int F = decltype(fmt)::value;
      if constexpr (F == US_E4M3 || F == US_E5M2) {
        const uint32_t lo = cvt_fp8x4<F == US_E5M2>(y[0], y[1], y[2], y[3]);
        const uint32_t hi = cvt_fp8x4<F == US_E5M2>(y[4], y[5], y[6], y[7]);
        if ((g & 1) == 0) { held[0] = lo; held[1] = hi; }
        else put((uint32_t)(2 * s + (g >> 1)), make_uint4(held[0], held[1], lo, hi), 1);
      } else {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = F == US_BF16 ? pack_bf16x2(y[2 * k], y[2 * k + 1]) : pack_f16x2(y[2 * k], y[2 * k + 1]);
        put((uint32_t)(4 * s + g), make_uint4(w[0], w[1], w[2], w[3]), 2);
      }
    };
    uint32_t hst[kSliceCols / 2 * kSlices];
    // One 32-column slice s of accumulator 0: scale, keep round16(H), GELU, round, stage.
    auto slice_fwd = [&](const uint32_t (&r)[kSliceCols], int s) {
      uint32_t held[2];
#pragma unroll
      for (int g = 0; g < kSliceCols / 8; ++g) {
        f32x2 x[4];
        float y[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          x[k] = mul2(pack2(__uint_as_float(r[8 * g + 2 * k]), __uint_as_float(r[8 * g + 2 * k + 1])), s1);
          float a, b;
          unpack2(x[k], a, b);
          hst[kSliceCols / 2 * s + 4 * g + k] = H_BF16 ? pack_bf16x2(a, b) : pack_f16x2(a, b);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) gelu_scaled2<kOes == 1>(x[k], tail_k, act_oi, y[2 * k], y[2 * k + 1]);   // the form the separate launch takes for this output
        stage_out(std::integral_constant<int, OUT_A>(), y, held, s, g);
      }
    };
    // The same slice of accumulator 1: scale, GELU gradient from the kept pre-activation, round, stage.
    auto slice_bwd = [&](const uint32_t (&r)[kSliceCols], int s) {
      uint32_t held[2];
#pragma unroll
      for (int g = 0; g < kSliceCols / 8; ++g) {
        float y[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const f32x2 x = mul2(pack2(__uint_as_float(r[8 * g + 2 * k]), __uint_as_float(r[8 * g + 2 * k + 1])), s2);
          const float2 h = H_BF16 ? unpack_bf16x2(hst[kSliceCols / 2 * s + 4 * g + k]) : unpack_f16x2(hst[kSliceCols / 2 * s + 4 * g + k]);
          unpack2(gelu_grad_scaled2(pack2(h.x, h.y), x, in2, os2), y[2 * k], y[2 * k + 1]);
        }
        stage_out(std::integral_constant<int, OUT_D>(), y, held, s, g);
      }
    };

    uint32_t local = 0;
    bool ok = true;
    for (int tile = pair; ok && tile < num_tiles; tile += num_pairs, ++local) {
      int tm, tn;
      tile_mn2(tile, tm, tn);
      const int row0 = tm * kTileM + rank * 128 + q * 32, n_w = tn * BN + split_col + part * kWarpCols;
      const bool active = n_w < p.N;                            // warp-uniform
      const uint32_t acc_phase = local & 1u;
#pragma unroll
      for (int sub = 0; sub < 2; ++sub) {
        ok = wait_bounded(acc_full_bar(sub), acc_phase, abort_flag, p.status, p.wait_limit);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        ptx::tc_fence_after_sync();
        const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + sub * kNB + split_acc + part * kWarpCols;
        uint32_t r0[kSliceCols], r1[kSliceCols];
        if (SPLIT > 1) {
          const long long at = sub == 0 ? (long long)(row0 + lane) * p.a_ld : (long long)(row0 + lane) * p.d_ld;
          direct = (sub == 0 ? p.a_ptr : p.d_ptr) + (at + n_w) * kOes;
          direct_cols = row0 + lane < p.M ? p.N - n_w : 0;
        }
        if (active) {
          ptx::tmem_ld_32x32_issue(t_row, r0);
          if (SPLIT == 1) {
            if (ptx::elect_one()) ptx::bulk_wait_group_read<0>();      // earlier stores have read the staging boxes
            __syncwarp();
          }
          ptx::tmem_ld_fence(r0);
          if (kSlices == 2) {
            ptx::tmem_ld_32x32_issue(t_row + 32, r1);
            if (sub == 0) slice_fwd(r0, 0); else slice_bwd(r0, 0);
            ptx::tmem_ld_fence(r1);
          }
        }
        release_acc(sub, tile);                                       // the values are in registers
        if (active) {
          if (kSlices == 2) { if (sub == 0) slice_fwd(r1, 1); else slice_bwd(r1, 1); }
          else { if (sub == 0) slice_fwd(r0, 0); else slice_bwd(r0, 0); }
          if (sub == 0 && p.h_ptr != nullptr && row0 + lane < p.M) {
            // the copy of the rounded pre-activation: this lane's columns, 16 at a time (a whole 32-byte sector per lane and
            // store: with 16 bytes each sector crosses to L2 twice; BF16 8192 x 1024 x 4096 132 -> 123 us, 117 without a copy), or
            // 8 at a time where the rows allow no more
            uint8_t* dst = p.h_ptr + ((long long)(row0 + lane) * p.h_ld + n_w) * 2;
            const bool sectors = kOes == 2 && p.h_sectors && n_w + kWarpCols <= p.N;      // (FP8 blocks rarely keep the copy; there the registers matter more)
            if (sectors) {
#pragma unroll
              for (int c = 0; c < kWarpCols / 16; ++c) ptx::stg256(dst + 32 * c, &hst[8 * c]);
            }
#pragma unroll
            for (int c = 0; c < kWarpCols / 8; ++c) {
              if (sectors) break;
              const int col = n_w + 8 * c;
              if (col + 8 <= p.N) {
                *reinterpret_cast<uint4*>(dst + 16 * c) = make_uint4(hst[4 * c], hst[4 * c + 1], hst[4 * c + 2], hst[4 * c + 3]);
              } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                  if (col + j < p.N)
                    *reinterpret_cast<uint16_t*>(dst + 16 * c + 2 * j) = (uint16_t)(hst[4 * c + (j >> 1)] >> (16 * (j & 1)));
              }
            }
          }
          if (SPLIT == 1) {
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (ptx::elect_one()) {
              if (sub == 0) {
                ptx::tma_store_2d(&tm_a, buf_out, n_w, row0);
              } else {
                ptx::tma_store_2d(&tm_dh, buf_out, n_w, row0);
              }
              ptx::bulk_commit_group();
            }
          }
        }
      }
    }
    // Leaving (early too, when a wait ran out somewhere in the CTA): tensor-memory loads have landed and
    // the stores have read shared memory before the CTA may give up its resources.
    ptx::tmem_ld_wait_all();
    if (ptx::elect_one()) ptx::bulk_wait_group_read<0>();
    __syncwarp();
  }

  ptx::tc_fence_before_sync();
  __syncthreads();
  if (CG == 2) ptx::cluster_part(*abort_flag != 0);
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    if (CG == 2) ptx::tmem_dealloc_pair(tmem_base, kTmemCols); else ptx::tmem_dealloc(tmem_base, kTmemCols);
  }
}

using host::make_tmap;

bool aligned16(const us_mat* m) {
  return reinterpret_cast<uintptr_t>(m->ptr) % 16 == 0 && (m->ld * dtype_size(m->dtype)) % 16 == 0;
}
bool valid_mat(const us_mat* m) {
  return m && m->ptr && m->rows >= 1 && m->cols >= 1 && m->ld >= m->cols && m->rows < (1ll << 31) && m->cols < (1ll << 31) &&
         m->dtype >= US_F32 && m->dtype <= US_E5M2;
}
bool is_fp8(int dt) { return dt == US_E4M3 || dt == US_E5M2; }

template <int ES, int BN, int CG, int SPLIT, int OUT_A, int OUT_D, bool H_BF16>
us_status launch_hidden(const CUtensorMap* t, const HiddenParams& p, int units, cudaStream_t stream) {
  auto kern = ffn_hidden_kernel<ES, BN, CG, SPLIT, OUT_A, OUT_D, H_BF16>;
  constexpr int smem = HidSmem<BN, OUT_A == US_E4M3 || OUT_A == US_E5M2 ? 1 : 2, (SPLIT > 1 ? 64 : BN)>::kTotal;
  static std::atomic<uint64_t> smem_set{0};
  return host::launch(kern, &smem_set, CG * SPLIT * units, gemm_threads(kHidEW), smem, CG, stream, t[0], t[1], t[2], t[3], t[4], t[5], p);
}
template <int ES, int OUT_A, int OUT_D, bool H_BF16>
us_status pick_tile(bool pair, int split, const CUtensorMap* t, const HiddenParams& p, int units, cudaStream_t st) {
  if (pair) return launch_hidden<ES, 256, 2, 1, OUT_A, OUT_D, H_BF16>(t, p, units, st);
  if (split == 4) return launch_hidden<ES, 128, 1, 4, OUT_A, OUT_D, H_BF16>(t, p, units, st);
  if (split == 2) return launch_hidden<ES, 128, 1, 2, OUT_A, OUT_D, H_BF16>(t, p, units, st);
  return launch_hidden<ES, 128, 1, 1, OUT_A, OUT_D, H_BF16>(t, p, units, st);
}
template <int ES, int OUT_A, int OUT_D>
us_status pick_hidden(bool pair, int split, bool h_bf16, const CUtensorMap* t, const HiddenParams& p, int units, cudaStream_t st) {
  return h_bf16 ? pick_tile<ES, OUT_A, OUT_D, true>(pair, split, t, p, units, st) : pick_tile<ES, OUT_A, OUT_D, false>(pair, split, t, p, units, st);
}

// any: 16-bit operands (outputs in the same format) and any size are covered too.
us_status hidden_impl(const us_mat* X, const us_mat* W1, float alpha, const us_mat* G, const us_mat* W2, float beta_x,
                      float act_in_scale, float act_out_scale, float grad_out_scale, int h_dtype, const us_mat* H,
                      const us_mat* A, const us_mat* dH, void* ws, size_t ws_bytes, void* stream, uint32_t wait_limit,
                      int starved, int served, bool any) {
  if (!valid_mat(X) || !valid_mat(W1) || !valid_mat(G) || !valid_mat(W2) || !valid_mat(A) || !valid_mat(dH)) return US_ERR_INVALID_ARG;
  const bool keep_h = H && H->ptr;
  if (keep_h && !valid_mat(H)) return US_ERR_INVALID_ARG;
  if (h_dtype != US_BF16 && h_dtype != US_F16) return US_ERR_INVALID_ARG;
  const int64_t M = X->rows, K1 = X->cols, N = W1->cols, K2 = G->cols;
  if (W1->rows != K1 || G->rows != M || W2->rows != N || W2->cols != K2) return US_ERR_INVALID_ARG;
  if (A->rows != M || A->cols != N || dH->rows != M || dH->cols != N) return US_ERR_INVALID_ARG;
  if (keep_h && (H->rows != M || H->cols != N || H->dtype != h_dtype)) return US_ERR_INVALID_ARG;
  if (!ws || ws_bytes < us_workspace_bytes()) return US_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(ws) % 16) return US_ERR_ALIGNMENT;
  if (!aligned16(X) || !aligned16(W1) || !aligned16(G) || !aligned16(W2) || !aligned16(A) || !aligned16(dH) ||
      (keep_h && !aligned16(H)))
    return US_ERR_ALIGNMENT;
  const us_mat* ms[6] = {X, W1, G, W2, A, dH};
  bool f8 = true, h16 = X->dtype == US_BF16 || X->dtype == US_F16;
  for (const us_mat* m : ms) { f8 = f8 && is_fp8(m->dtype); h16 = h16 && m->dtype == X->dtype; }
  if (!f8 && !(any && h16)) return US_ERR_UNSUPPORTED;
  if (!any && (M <= 128 || N <= 128)) return US_ERR_UNSUPPORTED;
  const int sms = host::sm_count();
  if (sms <= 0) return US_ERR_CUDA;

  // The rule of the single launches: 256 x 256 tiles per CTA pair unless they would leave more than half of the pairs idle
  // (1000 x 528 x 2096, 36 such tiles: 13.0 us with them, 9.5 us with 128 x 128).
  const bool pair = 4 * ((M + 255) / 256) * ((N + 255) / 256) >= sms;
  const int tile = pair ? 256 : 128, es = f8 ? 1 : 2, one = f8 ? US_E5M2 : US_BF16;
  HiddenParams p{};
  p.M = (int)M; p.N = (int)N; p.K1 = (int)K1; p.K2 = (int)K2;
  p.tiles_m = (int)((M + tile - 1) / tile); p.tiles_n = (int)((N + tile - 1) / tile);
  if ((int64_t)p.tiles_m * p.tiles_n >= (1ll << 30)) return US_ERR_UNSUPPORTED;
  p.d_tiles_m = make_fast_div(p.tiles_m);
  const int tiles = p.tiles_m * p.tiles_n, most = pair ? sms / 2 : sms;
  const int units = tiles < most ? tiles : most;
  const int split = pair ? 1 : 4 * tiles <= sms ? 4 : 2 * tiles <= sms ? 2 : 1;
  const int cols = split > 1 ? 64 : tile;                        // of an accumulator
  p.idesc1 = make_idesc(X->dtype == one, W1->dtype == one, false, true, tile, cols);
  p.idesc2 = make_idesc(G->dtype == one, W2->dtype == one, false, false, tile, cols);
  // a short X or G: its rows in groups of eight.  The MMA still reads 128; what lies behind them ends up in rows that do not exist.
  const int x_rows = split > 1 && M < 128 ? (int)((M + 7) / 8 * 8) : 128;
  p.x_bytes = (uint32_t)x_rows * kStageKBytes;
  using Half1 = HidSmem<128, 1, 64>;
  using Half2 = HidSmem<128, 2, 64>;
  const int room = f8 ? Half1::kStages * Half1::kStageBytes : Half2::kStages * Half2::kStageBytes;
  p.stages = std::min(Half1::kMaxStages, room / ((int)p.x_bytes + Half1::kBBytes));
  p.scale1 = alpha; p.scale2 = beta_x;
  p.act_in = act_in_scale; p.act_out = act_out_scale; p.grad_out = grad_out_scale;
  p.h_ptr = keep_h ? static_cast<uint8_t*>(H->ptr) : nullptr;
  p.h_ld = keep_h ? H->ld : 0;
  p.h_sectors = keep_h && reinterpret_cast<uintptr_t>(H->ptr) % 32 == 0 && H->ld % 16 == 0;
  p.a_ptr = static_cast<uint8_t*>(A->ptr); p.a_ld = A->ld;
  p.d_ptr = static_cast<uint8_t*>(dH->ptr); p.d_ld = dH->ld;
  p.status = static_cast<unsigned int*>(ws);
  p.wait_limit = wait_limit;
  p.starved = starved; p.served = served;

  CUtensorMap t[6];
  const int out_box = tile / 4 * es;                             // bytes per row of an epilogue warp's output box
  if (!make_tmap(&t[0], X, es, x_rows, 128) || !make_tmap(&t[1], W1, es, 128 / es, split > 1 && es == 1 ? 64 : 128) ||
      !make_tmap(&t[2], G, es, x_rows, 128) || !make_tmap(&t[3], W2, es, split > 1 ? 64 : 128, 128))
    return US_ERR_CUDA;
  t[4] = t[5] = t[0];                                            // (CTAs that share a tile store without them)
  if (split == 1 && (!make_tmap(&t[4], A, es, 32, out_box) || !make_tmap(&t[5], dH, es, 32, out_box)))
    return US_ERR_CUDA;

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const bool bf = h_dtype == US_BF16;
  if (!f8) return X->dtype == US_BF16 ? pick_hidden<2, US_BF16, US_BF16>(pair, split, bf, t, p, units, st) : pick_hidden<2, US_F16, US_F16>(pair, split, bf, t, p, units, st);
  const bool a5 = A->dtype == US_E5M2, d5 = dH->dtype == US_E5M2;
  if (!a5 && d5) return pick_hidden<1, US_E4M3, US_E5M2>(pair, split, bf, t, p, units, st);
  if (!a5 && !d5) return pick_hidden<1, US_E4M3, US_E4M3>(pair, split, bf, t, p, units, st);
  if (a5 && d5) return pick_hidden<1, US_E5M2, US_E5M2>(pair, split, bf, t, p, units, st);
  return pick_hidden<1, US_E5M2, US_E4M3>(pair, split, bf, t, p, units, st);
}

}  // namespace
}  // namespace us

extern "C" us_status us_ffn_hidden(const us_mat* X, const us_mat* W1, float alpha, const us_mat* G, const us_mat* W2,
                                   float beta_x, float act_in_scale, float act_out_scale, float grad_out_scale,
                                   int32_t h_dtype, const us_mat* H, const us_mat* A, const us_mat* dH, void* ws,
                                   size_t ws_bytes, void* stream) {
  return us::hidden_impl(X, W1, alpha, G, W2, beta_x, act_in_scale, act_out_scale, grad_out_scale, h_dtype, H, A, dH, ws,
                         ws_bytes, stream, us::kWaitLimit, 0, 0, false);
}

extern "C" us_status us_ffn_hidden_any(const us_mat* X, const us_mat* W1, float alpha, const us_mat* G, const us_mat* W2,
                                       float beta_x, float act_in_scale, float act_out_scale, float grad_out_scale,
                                       int32_t h_dtype, const us_mat* H, const us_mat* A, const us_mat* dH, void* ws,
                                       size_t ws_bytes, void* stream) {
  return us::hidden_impl(X, W1, alpha, G, W2, beta_x, act_in_scale, act_out_scale, grad_out_scale, h_dtype, H, A, dH, ws,
                         ws_bytes, stream, us::kWaitLimit, 0, 0, true);
}

extern "C" us_status us_test_ffn_hidden_starved(const us_mat* X, const us_mat* W1, const us_mat* G, const us_mat* W2,
                                                const us_mat* A, const us_mat* dH, void* ws, size_t ws_bytes,
                                                uint32_t wait_limit, void* stream) {
  if (wait_limit == 0 || wait_limit > (1u << 16)) return US_ERR_INVALID_ARG;
  return us::hidden_impl(X, W1, 1.f, G, W2, 1.f, 1.f, 1.f, 1.f, US_BF16, nullptr, A, dH, ws, ws_bytes, stream, wait_limit, 1, 0, false);
}
extern "C" us_status us_test_ffn_hidden_starved_cta(const us_mat* X, const us_mat* W1, const us_mat* G, const us_mat* W2, const us_mat* A, const us_mat* dH,
                                                    void* ws, size_t ws_bytes, uint32_t wait_limit, int cta, int tiles, void* stream) {
  if (wait_limit == 0 || wait_limit > (1u << 16) || cta < -1 || cta > 1 || tiles < 0 || tiles > 1024) return US_ERR_INVALID_ARG;
  return us::hidden_impl(X, W1, 1.f, G, W2, 1.f, 1.f, 1.f, 1.f, US_BF16, nullptr, A, dH, ws, ws_bytes, stream, wait_limit, cta + 2, tiles, false);
}
