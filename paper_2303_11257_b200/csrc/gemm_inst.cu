// Kernel instantiations of the unit-scaled GEMM for one (operand width, A layout, B layout)
// combination, selected by the macros US_INST_ES, US_INST_AMN, US_INST_BMN.  The build compiles
// this file once per combination, in parallel.
#include <cuda.h>

#include <algorithm>

#include "gemm_kernel.cuh"
#include "gemm_launch.h"
#include "host.h"

#ifndef US_INST_ES
#error "compile with -DUS_INST_ES=<1|2> -DUS_INST_AMN=<0|1> -DUS_INST_BMN=<0|1>"
#endif

namespace us {
namespace {

// host::make_tmap, or with a batch (bstride: elements between problems) a map of rank 4: column, row, inner batch index, outer batch
// index; a box never spans problems.
static bool make_tmap(CUtensorMap* tm, const us_mat* m, int es, int box_rows, int box_bytes = 128,
                      const BatchDesc* bd = nullptr, const int64_t* bstride = nullptr) {
  if (!bd) return host::make_tmap(tm, m, es, box_rows, box_bytes);
  host::EncodeTiledFn fn = host::encode_tiled_fn();
  if (!fn) return false;
  const CUtensorMapDataType type = es == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                                 : es == 2 ? CU_TENSOR_MAP_DATA_TYPE_UINT16 : CU_TENSOR_MAP_DATA_TYPE_UINT32;
  cuuint64_t dims[4] = {(cuuint64_t)m->cols, (cuuint64_t)m->rows, (cuuint64_t)bd->nb1, (cuuint64_t)bd->nb0};
  cuuint64_t strides[3] = {(cuuint64_t)m->ld * es, (cuuint64_t)bstride[1] * es, (cuuint64_t)bstride[0] * es};
  cuuint32_t box[4] = {(cuuint32_t)(box_bytes / es), (cuuint32_t)box_rows, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(tm, type, 4, m->ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            box_bytes == 32 ? CU_TENSOR_MAP_SWIZZLE_NONE : box_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int ES, bool A_MN, bool B_MN, int BN, int CG, int EPI, int EW, bool BATCHED = false>
static us_status launch(const us_mat* A, const us_mat* B, const GemmParams& p, const EpiMats& em, cudaStream_t stream,
                        const BatchDesc* bd = nullptr) {
  constexpr int kBK = kStageKBytes / ES;
  CUtensorMap ta, tb, t_out, t_aux, t_skip;
  const BatchDesc* b4 = BATCHED ? bd : nullptr;
  if (!make_tmap(&ta, A, ES, A_MN ? kBK : BN == 64 ? (int)p.a_bytes / kStageKBytes : kBM, 128, b4, b4 ? bd->a : nullptr)) return US_ERR_CUDA;
  if (!make_tmap(&tb, B, ES, B_MN ? kBK : BN / CG, B_MN && BN / CG * ES < 128 ? 64 : 128, b4, b4 ? bd->b : nullptr)) return US_ERR_CUDA;
  // epilogue boxes: 32 rows x the bytes of a warp's columns, 128 at most (the 16-warp epilogue: 64 FP8 codes); unused maps alias the
  // output's so that every parameter is valid
  const int out_es = dtype_size(em.out->dtype);
  if (!make_tmap(&t_out, em.out, out_es, 32, EW == 16 ? 64 : out_row_bytes(BN, out_es), b4, b4 ? bd->out : nullptr)) return US_ERR_CUDA;
  t_aux = t_out; t_skip = t_out;
  // the 16-warp GELU-gradient epilogue reads the stored pre-activation as 32-row x 64-byte boxes (one per 32-column slice)
  const int aux_row = EPI == kEpiGeluGrad ? (EW == 16 ? 64 : 128) : out_row_bytes(BN, 2);
  if (EPI != kEpiLegacy && em.aux && !make_tmap(&t_aux, em.aux, dtype_size(em.aux->dtype), 32, aux_row)) return US_ERR_CUDA;
  if (EPI != kEpiLegacy && em.skip && !make_tmap(&t_skip, em.skip, dtype_size(em.skip->dtype), 32)) return US_ERR_CUDA;
  auto kern = gemm_kernel<ES, A_MN, B_MN, BN, CG, EPI, EW, BATCHED>;
  constexpr int smem = GemmSmem<BN, CG, EW, EPI == kEpiPlain16>::kTotal;
  const int sms = host::sm_count();
  if (sms <= 0) return US_ERR_CUDA;
  const int tiles = p.tiles_m * p.tiles_n * p.nb0 * p.nb1;
  const int groups = sms / CG;                        // one CTA per SM; pairs share a TPC
  const int grid = CG * (tiles < groups ? tiles : groups);
  static std::atomic<uint64_t> smem_set{0};
  return host::launch(kern, &smem_set, grid, gemm_threads(EW), smem, CG, stream, ta, tb, t_out, t_aux, t_skip, p);
}

template <int ES, bool A_MN, bool B_MN, int BN, int CG>
static us_status pick_epilogue(const us_mat* A, const us_mat* B, const GemmParams& p, const EpiMats& em, int epi,
                               const BatchDesc& bd, cudaStream_t stream) {
  if (bd.batched()) {                                  // batched problems: plain epilogue only (checked by the caller)
    return launch<ES, A_MN, B_MN, BN, CG, kEpiPlain, 8, true>(A, B, p, em, stream, &bd);
  }
  // The GELU epilogues with an FP8 output (the FFN's forward and backward hidden layer) are ALU
  // bound with eight epilogue warps; they run with sixteen.
  const bool fp8_out = (em.out->dtype == US_E4M3 || em.out->dtype == US_E5M2) && p.fn == US_FN_GELU;   // the 16-warp epilogue is the GELU pair's
  if constexpr (BN != 64) {                            // (a warp has 32 columns of a narrow tile: eight are enough there)
    if (fp8_out && epi == kEpiGelu) return launch<ES, A_MN, B_MN, BN, CG, kEpiGelu, 16>(A, B, p, em, stream);
    if (fp8_out && epi == kEpiGeluGrad) return launch<ES, A_MN, B_MN, BN, CG, kEpiGeluGrad, 16>(A, B, p, em, stream);
  }
  if constexpr (!A_MN && B_MN) {
    if (epi == kEpiSkipCopy) return launch<ES, A_MN, B_MN, BN, CG, kEpiSkipCopy, 8>(A, B, p, em, stream);
  }
  switch (epi) {
    case kEpiPlain:
      if constexpr (CG == 2) {
        // FP8 outputs of contractions of up to 32 K blocks: sixteen epilogue warps (beyond, equal or, at 64, 2 % slower).  Not 16-bit ones,
        // whose tiles are bound by the bytes they write (FP8 operands into BF16, eight / sixteen warps, us: 8192 x 128 x 3072 12.1 / 11.3,
        // x 1024 x 3072 22.6 / 23.8, 2048 x 1024 x 30528 57.6 / 60.2).
        if ((em.out->dtype == US_E4M3 || em.out->dtype == US_E5M2) && (long long)p.K * ES <= 4096)
          return launch<ES, A_MN, B_MN, BN, CG, kEpiPlain16, 16>(A, B, p, em, stream);
      }
      return em.out->dtype == US_F32 ? launch<ES, A_MN, B_MN, BN, CG, kEpiPlainF32, 8>(A, B, p, em, stream)
                                     : launch<ES, A_MN, B_MN, BN, CG, kEpiPlain, 8>(A, B, p, em, stream);
    case kEpiGelu:     return launch<ES, A_MN, B_MN, BN, CG, kEpiGelu, 8>(A, B, p, em, stream);
    case kEpiGeluGrad: return launch<ES, A_MN, B_MN, BN, CG, kEpiGeluGrad, 8>(A, B, p, em, stream);
    case kEpiSkip:
      return em.out->dtype == US_F32 ? launch<ES, A_MN, B_MN, BN, CG, kEpiSkipF32, 8>(A, B, p, em, stream)
                                     : launch<ES, A_MN, B_MN, BN, CG, kEpiSkip, 8>(A, B, p, em, stream);
    default:           return launch<ES, A_MN, B_MN, BN, CG, kEpiLegacy, 8>(A, B, p, em, stream);
  }
}

// Whether the contraction is shared by several CTAs, and in which tiles.  now: the tiles taken otherwise; sectors: the operands' rows
// start on 32-byte boundaries (a box of other rows takes TMA about twice as long).
//
// Both ways are estimated by tiling_time.  Measured, us, FP8 into BF16, one CTA a tile / two / four / eight CTAs on tiles of 128 x 64 / the same on 128 x 128 /
// two and four pairs on 256 x 256 (-: more CTAs than SMs, or more clusters than run at once), rows x K x columns:
//     48 x 1920 x 1024    4.7 / 4.8 4.7 - / 6.0 6.2 7.1 / -           48 x 2560 x 1024   5.4 / 5.2 4.8 - / 6.4 6.2 7.4 / -
//     48 x 4096 x 1024    7.3 / 6.0 5.2 - / 7.2 6.7 7.2 / -           48 x 8192 x 1024  12.2 / 8.2 6.4 - / 9.7 7.9 7.9 / -
//    300 x 4096 x 704     7.4 / 6.2 6.4 - / 7.9 7.1 - / 11.3 11.1    512 x 8192 x 1024  12.7 / 9.6 - - / 10.4 10.2 - / 15.9 14.2
//    128 x 512 weight gradient, K 16384  21.8 / 13.0 8.7 7.2 / 14.6 10.5 8.7 / -
//    2048 x 30528 x 1024 67.6 / - - - / - - - / 52.8 -
// 110 drawn ops (16 to 16384 rows, FP8 and BF16) against one CTA a tile: 0.99 to 5.5 times as fast.  From 20 K blocks on; weight gradients from
// 48 on, so that with fewer the grouped launch (one accumulator per tile) gives the same bits; up to the 8192 blocks that were measured.
template <int ES, bool A_MN, bool B_MN>
static Tiling split_tiling(const GemmParams& p, Tiling now, bool sectors) {
  const int kb = (p.K + kStageKBytes / ES - 1) / (kStageKBytes / ES), sms = host::sm_count();
  if (kb < (A_MN ? 48 : 20) || kb > kSplitMostBlocks || sms <= 0) return now;
  const auto tiles = [&](const Tiling& t) { return (long long)((p.M + kBM * t.cg - 1) / (kBM * t.cg)) * ((p.N + t.bn - 1) / t.bn); };
  const auto cost = [&](const Tiling& t) { return tiling_time(t, tiles(t), kb, split_a_bytes(t.bn, A_MN, p.M), sectors, sms); };
  Tiling pick = now;
  double best = 0.92 * cost(now);
  for (int form = 0; form < 3; ++form) {
    Tiling t{form == 0 ? 64 : form == 1 ? 128 : 256, form == 2 ? 2 : 1, 2};
    if (!split_form_fits(t, p.M, p.N)) continue;
    for (; t.splits * t.cg <= 8; t.splits *= 2) {
      if (kb < 4 * t.splits || tiles(t) * t.splits * t.cg > sms || cost(t) >= best) continue;
      if (tiles(t) > split_capacity(ES, t)) continue;
      best = cost(t);
      pick = t;
    }
  }
  return pick;
}

}  // namespace

template <int ES, bool A_MN, bool B_MN>
us_status launch_gemm(const us_mat* A, const us_mat* B, GemmParams& p, const EpiMats& em, int epi, const BatchDesc& bd,
                      cudaStream_t stream, Tiling* only) {
  // CTA pairs with 256 x 256 tiles whenever such a tile is not mostly empty and there are enough of them to occupy at
  // least half of the machine's CTA pairs; 128 x 128 tiles otherwise (a 1024 x 1024 output is 16 pair tiles on 74
  // pairs, but 64 single-CTA tiles).
  const int sms = host::sm_count();
  const long long pair_tiles = (long long)((p.M + 2 * kBM - 1) / (2 * kBM)) * ((p.N + 255) / 256) * bd.nb0 * bd.nb1;
  const bool pair = p.N > 128 && p.M > kBM && (sms <= 0 || 4 * pair_tiles >= sms);
  // 128 x 64 tiles where the machine has an SM for each of them (or, batched, where the outputs are no wider): half the operand
  // bytes and epilogue of a 128 x 128 tile per CTA.  us, 128 x 128 -> 128 x 64 tiles, outputs x contraction, FP8 unless said: 48 x 4096 x 512
  // 4.1 -> 3.4, 200 x 4700 x 512 weight gradient 5.5 -> 5.1, 1000 x 528 x 512 4.2 -> 3.4, 9000 x 128 x 512 4.3 -> 4.0, 128 x 9472 x 2048
  // 6.2 -> 6.2; batched 256 x (512 x 64) 13.4 -> 12.0.  Two exceptions:
  //  - An MN-major A with rows shorter than a 128-byte box is fetched by every tile in pieces of its short rows, so fewer tiles are better
  //    sooner.  Weight gradients, contraction of 2048, 32 / 48 / 64 / 96 tiles of 128 x 64 against the 128 x 128 ones: 16-byte rows
  //    7.6 / 8.0 / 9.6 / 14.4 against 7.6 / 7.8 / 8.1 / 8.6, 48 bytes 8.6 / 8.8 / 9.6 / 13.5 against 8.8 / 8.9 / 9.1 / 9.2, 96 bytes (BF16)
  //    7.8 / 7.8 / 8.0 / 9.9 against 9.4 / 9.4 / 9.4 / 9.5; 200 bytes 10.9 / 10.9 / 11.0 / 11.8 against 12.5 / 12.5 / 12.7 / 12.8.
  //  - 65 to 95 columns are two tiles instead of one, the second mostly empty (9400 x 80 x 1024: 4.7 -> 5.3, 5000 x 100 4.9 -> 4.3).
  const long long narrow_tiles = (long long)((p.M + kBM - 1) / kBM) * ((p.N + 63) / 64);
  const int short_a = A_MN ? p.M * ES : kStageKBytes;
  const int most = short_a < 32 ? 32 : short_a < 96 ? 48 : short_a < kStageKBytes ? 64 : p.N > 64 && p.N < 96 ? sms * 3 / 4 : sms;
  const bool narrow = !pair && (bd.batched() ? p.N <= 64 : narrow_tiles <= most);
  using Narrow = GemmSmem<64, 1, 8>;
  p.a_bytes = (A_MN || p.M >= kBM ? kBM : (p.M + 7) / 8 * 8) * kStageKBytes;
  p.stages = std::min((uint32_t)Narrow::kMaxStages, (uint32_t)(Narrow::kStages * Narrow::kStageBytes) / (p.a_bytes + Narrow::kBBytes));
  Tiling t{pair ? 256 : narrow ? 64 : 128, pair ? 2 : 1, 1};
  if (!bd.batched() && (epi == kEpiPlain || epi == kEpiSkip || epi == kEpiSkipCopy)) {
    const bool sectors = A->ld * ES % 32 == 0 && B->ld * ES % 32 == 0;
    t = split_tiling<ES, A_MN, B_MN>(p, t, sectors);
  }
  if (only) {
    *only = t;
    return US_OK;
  }
  const int bn = t.bn, cg = t.cg;
  if (t.splits > 1) {
    const SplitCall call{A, B, em.out, em.skip, em.copy, A_MN, B_MN, p.scale, p.skip_coef, p.out_coef};
    return launch_split(1, &call, t, p.status, p.wait_limit, p.served ? 0 : p.starved, stream);
  }
  p.tiles_m = (p.M + kBM * cg - 1) / (kBM * cg);
  p.tiles_n = (p.N + bn - 1) / bn;
  p.nb0 = (int)bd.nb0; p.nb1 = (int)bd.nb1;
  // A (M x K operand) is re-read by every column of tiles: keep the plain order while it fits well
  // inside the 126 MB L2, switch to bands of 8 tile rows beyond that.
  p.band_m = ((long long)p.M * p.K * ES <= (80ll << 20)) ? p.tiles_m : 8;
  // A short contraction mostly writes: tiles that run together then cover whole rows of a few bands (us, FP8 operands, outputs x K: 8192 x
  // 8192 float32 x 512 55.7 -> 49.7, repeated runs of either up to 8 apart; 16384 x 8192 BF16 x 1024 115 -> 108, 16384 x 1024 x 256 13.9 ->
  // 11.7; 8192 x 4096 x 1024, 1024 x 30528 float32 x 512, 65536 x 512 x 128 and batched scores equal; 1024 x 30528 with K = 2048 loses that
  // way from two bands down).
  if ((long long)p.K * ES <= 1024 && p.tiles_m > 4) p.band_m = 4;
  p.full_bands = p.tiles_m / p.band_m;
  p.d_problem = make_fast_div(p.tiles_m * p.tiles_n);
  p.d_band = make_fast_div(p.band_m * p.tiles_n);
  p.d_rows = make_fast_div(p.band_m);
  p.d_rows_last = make_fast_div(p.tiles_m % p.band_m ? p.tiles_m % p.band_m : 1);
  p.d_nb1 = make_fast_div(p.nb1);
  p.idesc = (p.idesc & ~((0x3fu << 17) | (0x1fu << 24))) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)((kBM * cg) >> 4) << 24);
  return pair ? pick_epilogue<ES, A_MN, B_MN, 256, 2>(A, B, p, em, epi, bd, stream)
       : narrow ? pick_epilogue<ES, A_MN, B_MN, 64, 1>(A, B, p, em, epi, bd, stream)
                : pick_epilogue<ES, A_MN, B_MN, 128, 1>(A, B, p, em, epi, bd, stream);
}

template us_status launch_gemm<US_INST_ES, (US_INST_AMN != 0), (US_INST_BMN != 0)>(const us_mat*, const us_mat*, GemmParams&,
                                                                                 const EpiMats&, int, const BatchDesc&, cudaStream_t, Tiling*);

}  // namespace us
