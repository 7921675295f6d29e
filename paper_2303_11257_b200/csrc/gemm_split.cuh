// GEMMs whose contractions are shared by the CTAs of a cluster (one, or up to four in a launch).
//
// An output of few tiles with a long contraction leaves most SMs idle, and the ones at work are bound by what an SM can take in (a K
// block of 128 x 128 operands, 32 KB, every 150 ns; every 380 ns, 86 bytes per ns, where rows start inside a 32-byte sector).  Here p.splits CTAs (or CTA pairs, CG = 2) of a
// cluster compute the same tile over consecutive parts of K.  When all have finished, every block of 32 rows x 32 columns belongs to
// one of them: the others store their partial sums into its operand ring through distributed shared memory, and it adds them to its
// own in float32, in a fixed order, and finishes the block.  One tile per cluster, no workspace, no atomics: results do not depend on scheduling.
//
// Two hardware cluster barriers carry the exchange: after the first nobody reads operands any more, after the second the partial sums
// are there.  Every thread reaches both whatever its waits returned, so a wait that ran out in one CTA leaves no other one waiting.
#pragma once

#include "gemm_group.cuh"

namespace us {

struct SplitProblem {
  GroupProblem g;                           // out boxes: 32 rows x 32 columns
  int tiles_m, tile_end;                    // tile rows; tiles of the problems up to and including this one
  uint32_t a_bytes; int stages;             // bytes of A in a stage (narrow tiles of few rows: those that exist), and the stages that fit
};
template <int PROBLEMS>
struct SplitParams {
  SplitProblem prob[PROBLEMS];
  int splits;                               // CTAs (pairs) per tile: 2, 4 or 8
  unsigned int* status;
  uint32_t wait_limit;
  int starved;                              // test hook (starved_cta)
};

// MULTI: several problems; the parameters of one alone are at fixed addresses and need not be fetched ahead.
template <int ES, int BN, int CG, bool MULTI>
__global__ void __launch_bounds__(gemm_threads(8), 1)
gemm_split_kernel(const __grid_constant__ SplitParams<MULTI ? kGroupMaxProblems : 1> p) {
  using S = GemmSmem<BN, CG, 8>;
  constexpr int kBK = kStageKBytes / ES;
  constexpr uint32_t kChunkBytes = kBK * 128;
  constexpr int kBRows = BN / CG;
  constexpr int kSlices = BN / 64;                              // blocks of 32 columns per epilogue warp
  constexpr uint32_t kBlockBytes = 4096u;                       // partial sums of a block: [16-byte chunk][row]
  static_assert(8 * kSlices * kBlockBytes <= (uint32_t)(S::kStages * S::kStageBytes), "partial sums fit the operand ring");

  ptx::grid_release_next();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (ptx::smem_addr(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - ptx::smem_addr(smem_raw));
  const uint32_t epi_base = smem_base + S::kStages * S::kStageBytes;
  const uint32_t bars = epi_base + S::kEpiBytes;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (S::kMaxStages + s); };
  const uint32_t acc_full_bar = bars + 8u * (2 * S::kMaxStages), drained_bar = acc_full_bar + 8u;
  auto epi_in_bar = [&](int w) { return bars + 8u * (2 * S::kMaxStages + 2 + w); };
  uint8_t* tail = smem_gen + S::kStages * S::kStageBytes + S::kEpiBytes + 8 * (2 * S::kMaxStages + 2 + kEpilogueWarps);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(tail);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int splits = p.splits, cluster_rank = (int)ptx::cluster_ctarank();
  const int part = cluster_rank / CG, rank = cluster_rank % CG;     // part of K; position in the pair
  const uint32_t even = (uint32_t)(cluster_rank - rank);            // the pair's even CTA
  int tile = blockIdx.x / (CG * splits), pi = 0;
  if (MULTI) {
    while (tile >= p.prob[pi].tile_end) ++pi;
    if (pi > 0) tile -= p.prob[pi - 1].tile_end;
  }
  const SplitProblem& sp = p.prob[pi];
  const GroupProblem& P = sp.g;
  // the problem's fields, fetched once where they are reached through an index (see gemm_group.cuh)
  auto once = [](int x) { return MULTI ? ptx::once(x) : x; };
  const int tiles_m = once(sp.tiles_m), stages = once(sp.stages), rows = once(P.M), cols = once(P.N), all_k = once(P.K);
  const uint32_t a_bytes = (uint32_t)once((int)sp.a_bytes), stage_bytes = a_bytes + S::kBBytes;
  const bool a_mn = once(P.a_mn) != 0, b_mn = once(P.b_mn) != 0, skip = once(P.has_skip) != 0;
  const int tn = tile / tiles_m, tm = tile - tn * tiles_m;
  const int all_kb = (all_k + kBK - 1) / kBK;
  const int kb0 = (int)((int64_t)all_kb * part / splits), num_kb = (int)((int64_t)all_kb * (part + 1) / splits) - kb0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { ptx::mbar_init(full_bar(s), 1); ptx::mbar_init(empty_bar(s), 1); }
    ptx::mbar_init(acc_full_bar, 1);
    ptx::mbar_init(drained_bar, 1);
    for (int w = 0; w < kEpilogueWarps; ++w) ptx::mbar_init(epi_in_bar(w), 1);
    *abort_flag = 0;
    ptx::mbar_init_fence();
    ptx::prefetch_tensormap(&P.ta);
    ptx::prefetch_tensormap(&P.tb);
  }
  if (warp == 1) {
    if (CG == 2) { ptx::tmem_alloc_pair(ptx::smem_addr(const_cast<uint32_t*>(tmem_slot)), BN); ptx::tmem_relinquish_pair(); }
    else { ptx::tmem_alloc(ptx::smem_addr(const_cast<uint32_t*>(tmem_slot)), BN); ptx::tmem_relinquish(); }
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (CG == 2) ptx::cluster_meet();                  // the partner's barriers and TMEM are ready too
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  // Epilogue warp (quarter q, half) has 32 rows x BN / 2 columns, as kSlices blocks.  The tile's 8 * kSlices blocks, slice by slice, are
  // dealt to the parts in runs of `run`.
  const int q = warp & 3, half = ((warp - 2) >> 2) & 1, spot = 2 * q + half;
  const int run = 8 * kSlices / splits;
  const int row0 = tm * (kBM * CG) + rank * kBM + q * 32, n_w = tn * BN + half * (BN / 2);
  auto block = [&](int sl) { return 8 * sl + spot; };
  auto mine = [&](int sl) { return block(sl) / run == part && n_w + 32 * sl < cols; };
  const uint32_t buf_in = epi_base + (uint32_t)(warp - 2) * epi_warp_bytes(8), buf_out = buf_in + 4096u;
  const uint32_t in_bar = epi_in_bar(warp - 2);
  bool ok = true, in_pending = false;
  uint32_t in_phase = 0;
  auto issue_in = [&](int sl) {                      // this warp's block sl of the skip tensor (16-bit types: and 32 columns more)
    if (ptx::elect_one()) {
      ptx::mbar_expect_tx(in_bar, 4096);
      ptx::tma_load_2d(buf_in, &P.tskip, in_bar, n_w + 32 * sl, row0);
    }
    in_pending = true;
  };
  int first = 0;                                     // this warp's first block of its own
  while (first < kSlices && !mine(first)) ++first;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (every CTA)
    if (ptx::elect_one()) {
      const int m0 = tm * (kBM * CG) + rank * kBM, n0 = tn * BN + rank * kBRows;
      uint32_t issued = 0;
      int stage = 0; uint32_t phase = 0;
      ptx::grid_wait_previous();
      with_layout(a_mn, b_mn, [&](auto amn, auto bmn) {
        constexpr bool A_MN = decltype(amn)::value, B_MN = decltype(bmn)::value;
        const int end = starved_cta(p.starved, cluster_rank) ? 0 : num_kb;
        for (int kb = 0; ok && kb < end; ++kb) {
          ok = wait_bounded(empty_bar(stage), phase ^ 1u, abort_flag, p.status, p.wait_limit);
          if (!ok) break;
          const uint32_t a_dst = smem_base + stage * stage_bytes, b_dst = a_dst + a_bytes;
          const int k0 = (kb0 + kb) * kBK;
          const uint32_t fb = CG == 2 ? ptx::in_cta(full_bar(stage), even) : full_bar(stage);
          if (rank == 0) ptx::mbar_expect_tx(full_bar(stage), CG * stage_bytes);
          auto load = [&](uint32_t dst, const void* map, int x, int y) {
            if (CG == 2) ptx::tma_load_2d_pair(dst, map, fb, x, y); else ptx::tma_load_2d(dst, map, fb, x, y);
          };
          if (A_MN) {
#pragma unroll
            for (int c = 0; c < ES; ++c) load(a_dst + c * kChunkBytes, &P.ta, m0 + c * kBK, k0);      // 128 / ES elements per box
          } else {
            load(a_dst, &P.ta, k0, m0);
          }
          if (B_MN) {
#pragma unroll
            for (int c = 0; c < (kBRows * ES + 127) / 128; ++c) load(b_dst + c * kChunkBytes, &P.tb, n0 + c * kBK, k0);
          } else {
            load(b_dst, &P.tb, k0, n0);
          }
          ++issued;
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
      });
      if (*abort_flag && rank == 0) {
        // Let copies that are still in flight land before the CTA's shared memory is used for anything else.
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
      const uint16_t pair_mask = (uint16_t)(3u << even);
      const uint32_t idesc = P.idesc;
      ptx::grid_wait_previous();                       // no operand comes earlier: the bounded waits begin when the loads do
      // The loop is compiled per operand layout: steps and descriptors that are known then leave the four MMAs of a block to uniform
      // registers (with run-time layouts a K block of a narrow tile took 0.21 us instead of 0.15).
      with_layout(a_mn, b_mn, [&](auto amn, auto bmn) {
        constexpr bool A_MN = decltype(amn)::value, B_MN = decltype(bmn)::value, kHalfRowB = ES == 1 && BN == 64 && B_MN;
        const uint64_t a_desc0 = A_MN ? ptx::smem_desc_sw128(smem_base, kChunkBytes, 1024) : ptx::smem_desc_sw128(smem_base, 16, 1024);
        const uint64_t b_desc0 = kHalfRowB ? ptx::smem_desc_sw64(smem_base + a_bytes, 16, 512)
                                 : B_MN    ? ptx::smem_desc_sw128(smem_base + a_bytes, kChunkBytes, 1024)
                                           : ptx::smem_desc_sw128(smem_base + a_bytes, 16, 1024);
        const uint32_t a_hi = (uint32_t)(a_desc0 >> 32), b_hi = (uint32_t)(b_desc0 >> 32);
        const uint32_t a_lo0 = (uint32_t)a_desc0, b_lo0 = (uint32_t)b_desc0, stage_step = stage_bytes >> 4;
        constexpr uint32_t kAStep = (A_MN ? kChunkBytes / kKSteps : 32u) >> 4;
        constexpr uint32_t kBStep = (kHalfRowB ? kChunkBytes / 2 / kKSteps : B_MN ? kChunkBytes / kKSteps : 32u) >> 4;
        int stage = 0; uint32_t phase = 0, accumulate = 0;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!ptx::mbar_try_wait(full_bar(stage), phase)) {
            ok = wait_bounded(full_bar(stage), phase, abort_flag, p.status, p.wait_limit);
            if (!ok) break;
          }
          ptx::tc_fence_after_sync();
          const uint32_t a_lo = a_lo0 + stage * stage_step, b_lo = b_lo0 + stage * stage_step;
#pragma unroll
          for (int k = 0; k < kKSteps; ++k) {
            const uint64_t adesc = ((uint64_t)a_hi << 32) | (a_lo + k * kAStep);
            const uint64_t bdesc = ((uint64_t)b_hi << 32) | (b_lo + k * kBStep);
            if (CG == 2) ptx::mma_ss_pair<ES == 1>(tmem_base, adesc, bdesc, idesc, accumulate);
            else ptx::mma_ss<ES == 1>(tmem_base, adesc, bdesc, idesc, accumulate);
            accumulate = 1;
          }
          if (CG == 2) ptx::mma_commit_pair(empty_bar(stage), pair_mask); else ptx::mma_commit(empty_bar(stage));
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
      });
      if (ok) { if (CG == 2) ptx::mma_commit_pair(acc_full_bar, pair_mask); else ptx::mma_commit(acc_full_bar); }
      if (*abort_flag) {
        if (CG == 2) ptx::mma_commit_pair(drained_bar, (uint16_t)(1u << even)); else ptx::mma_commit(drained_bar);
        for (uint32_t it = 0; it < p.wait_limit && !ptx::mbar_try_wait(drained_bar, 0); ++it) {}
      }
    }
  } else {
    ptx::grid_wait_previous();
    if (first < kSlices && skip) issue_in(first);
    ok = wait_bounded(acc_full_bar, 0, abort_flag, p.status, p.wait_limit);
    ok = __all_sync(0xffffffffu, ok);
  }
  __syncwarp();

  ptx::cluster_sync();                               // all operands of the cluster have been read: its rings take partial sums now
  const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + half * (BN / 2);
  if (warp >= 2 && ok) {
    ptx::tc_fence_after_sync();
#pragma unroll 1
    for (int sl = 0; sl < kSlices; ++sl) {
      const int owner = block(sl) / run;
      if (owner == part || n_w + 32 * sl >= cols) continue;
      const int from = part - (part > owner ? 1 : 0);
      const uint32_t to = ptx::in_cta(smem_base + (uint32_t)(from * run + block(sl) % run) * kBlockBytes, (uint32_t)(owner * CG + rank)) + (uint32_t)lane * 16u;
      float v[32];
      ptx::tmem_ld_32x32(t_row + 32 * sl, v);
#pragma unroll
      for (int c = 0; c < 8; ++c) ptx::st_cluster_v4(to + (uint32_t)c * 512u, &v[4 * c]);
    }
    ptx::tc_fence_before_sync();
  }
  __syncwarp();
  ptx::cluster_sync();                               // the partial sums have arrived

  if (warp >= 2 && first < kSlices && ok) {
    ptx::tc_fence_after_sync();
    const int out_dt = once(P.out_dt), skip_dt = once(P.skip_dt), out_es = dtype_size(out_dt), out_row = 32 * out_es;      // an output box: one block
    const uint32_t sw = (uint32_t)(lane & 7);
    const uint32_t out_sw = out_row == 128 ? sw : out_row == 64 ? (uint32_t)((lane >> 1) & 3) : 0u;
    const f32x2 scale2 = splat2(P.scale), skip2 = splat2(P.skip_coef), oc2 = splat2(P.out_coef);
#pragma unroll 1
    for (int sl = first; sl < kSlices && mine(sl); ++sl) {
      const int col = n_w + 32 * sl;
      uint4 raw[8];
      if (skip) {
        ok = wait_bounded(in_bar, in_phase, abort_flag, p.status, p.wait_limit);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        in_phase ^= 1u;
        in_pending = false;
        const int nchunk = 2 * dtype_size(skip_dt);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (j < nchunk) raw[j] = ptx::lds128(buf_in + (uint32_t)lane * 128u + ((j ^ sw) << 4));
        if (sl + 1 < kSlices && mine(sl + 1)) {
          __syncwarp();                              // every lane has read the box
          issue_in(sl + 1);
        }
      }
      float y[32];
      ptx::tmem_ld_32x32(t_row + 32 * sl, y);
      uint32_t at = smem_base + (uint32_t)(block(sl) % run) * kBlockBytes + (uint32_t)lane * 16u;
#pragma unroll 1
      for (int s = 1; s < splits; ++s, at += (uint32_t)run * kBlockBytes) {
        uint4 w[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) w[c] = ptx::lds128(at + (uint32_t)c * 512u);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          y[4 * c] += __uint_as_float(w[c].x); y[4 * c + 1] += __uint_as_float(w[c].y);
          y[4 * c + 2] += __uint_as_float(w[c].z); y[4 * c + 3] += __uint_as_float(w[c].w);
        }
      }
#pragma unroll
      for (int k = 0; k < 16; ++k) unpack2(mul2(pack2(y[2 * k], y[2 * k + 1]), scale2), y[2 * k], y[2 * k + 1]);
      if (skip) residual_row32(skip_dt, raw, skip2, oc2, y);
      if (P.copy && row0 + lane < rows) {             // an FP8 copy of the result
        uint32_t copy[8];
        copy_codes32(out_dt, P.copy_dt, y, copy);
        copy_store(P.copy + (int64_t)(row0 + lane) * P.copy_ld + col, copy, cols - col, P.copy_sectors != 0);
      }
      if (sl > first) {                              // the output box is about to be refilled
        if (ptx::elect_one()) ptx::bulk_wait_group_read<0>();
        __syncwarp();
      }
      stage_row32(out_dt, y, buf_out + (uint32_t)(lane * out_row), 0u, out_sw);
      ptx::fence_proxy_async_smem();
      __syncwarp();
      if (ptx::elect_one()) { ptx::tma_store_2d(&P.tout, buf_out, col, row0); ptx::bulk_commit_group(); }
    }
    ptx::tc_fence_before_sync();
    if (ptx::elect_one()) ptx::bulk_wait_group_read<0>();
  }
  if (in_pending && lane == 0)                       // (a wait ran out: the box may still be on its way)
    for (uint32_t it = 0; it < p.wait_limit && !ptx::mbar_try_wait(in_bar, in_phase); ++it) {}
  __syncwarp();

  ptx::tc_fence_before_sync();
  __syncthreads();
  if (CG == 2) ptx::cluster_meet();                  // (nothing has been signalled since the barriers above)
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    if (CG == 2) ptx::tmem_dealloc_pair(tmem_base, BN); else ptx::tmem_dealloc(tmem_base, BN);
  }
}

}  // namespace us
