// Several independent unit-scaled GEMMs in ONE launch (us_linear_group).
//
// The last four GEMMs of an FFN step (the second forward GEMM, the two weight-gradient GEMMs
// and the input-gradient GEMM of the first layer) depend on nothing but tensors that exist already.
// Launched one after the other, each pays its own set-up and tail and leaves a partly filled last
// wave (64 or 128 tiles of 256 x 256 on 74 CTA pairs).  Here the tiles of all problems form one
// list that the host deals out to the CTA pairs longest-first, so that every pair gets about the
// same number of K blocks; a pair walks its share with the usual roles (TMA producer, MMA issuer,
// eight epilogue warps), and the main loop of a pair's next tile runs while its previous tile's
// epilogue drains, across problem boundaries too.
//
// Scope: FP8 or 16-bit operands (all problems of a launch the same width; either layout each), plain
// or residual (skip) epilogue, any output dtype, up to kGroupMaxProblems problems.  CTA-pair tiles of
// 256 x 256 (cta_group::2), or, when those would leave too many pairs idle, single-CTA tiles of 128 x 128.
// Everything that differs between problems is run-time data here: tensor maps, operand layouts (a K-major
// tile is one box of 128 rows x 128 bytes; an MN-major one has 128 / ES rows of K per box, one box of 128 bytes
// for FP8 and two for 16-bit elements), instruction descriptor, scale, epilogue kind.
// Measured, four separate launches -> this one, us: FP8 8192 x 1024 x 4096 122 -> 101; BF16 216 -> 199;
// FP8 16384 x 2048 x 8192 (21 tiles per pair) 912 of kernel time, partly side by side, -> 809; FP8 256 x 128 x 512 26 -> 7.
//
// The run-time data are kernel parameters reached through an index: loads of 100 cycles and more, which a store or a wait
// between two uses makes the compiler repeat.  So every role fetches a tile's fields once, the first tile's before it waits for the
// previous kernel, and the epilogue takes its choices (skip type, output type) once per 32-column slice.  With the choices inside the
// groups of eight columns a slice with a skip tensor took 1550 cycles after its data were there, and its reading another 800.
// Captured steps, us: 256 x 128 x 512 9.5 -> 8.8, 512 x 512 x 1456 18.0 -> 16.8, 1000 x 528 x 2096 27.4 -> 25.2, 4096 x 256 x 704
// 24.6 -> 23.4, 2048 x 1024 x 3008 55.1 -> 54.3; BF16 8192 x 1024 x 4096 412 -> 402.
#pragma once

#include "gemm_kernel.cuh"

namespace us {

constexpr int kGroupMaxProblems = 4;
constexpr int kGroupMaxItems = 2048;    // entries of the work list (a kernel parameter: 8 KB)
constexpr int kGroupMaxUnits = 160;     // CTA pairs or CTAs that share the list

struct GroupProblem {
  CUtensorMap ta, tb, tout, tskip;      // A and B: operand boxes (above); out / skip: 32-row x 128-byte boxes
  int M, N, K;
  int a_mn, b_mn;                       // operand stored MN-major ([K x M] resp. [K x N] row-major)
  uint32_t idesc;
  float scale;
  int out_dt;
  int has_skip, skip_dt;
  float skip_coef, out_coef;
  uint8_t* copy; int64_t copy_ld;       // an FP8 copy of the output (null: none)
  int copy_dt, copy_sectors;            // its rows start on 32-byte boundaries
};

struct GroupParams {
  GroupProblem prob[kGroupMaxProblems];
  int count, rounds, units;             // units: CTA pairs, or CTAs with single-CTA tiles
  unsigned int* status;
  uint32_t wait_limit;
  int starved, served;                  // test hook (starved_cta)
  // work list: entry [round * units + unit] = problem << 28 | tile row << 14 | tile column, or -1
  int32_t table[kGroupMaxItems];
};

__device__ __forceinline__ void group_decode(int32_t e, int& prob, int& tm, int& tn) {
  prob = e >> 28; tm = (e >> 14) & 0x3fff; tn = e & 0x3fff;
}

constexpr int kGroupEW = 8;

// SPLIT = 2 (128 x 128 tiles): two CTAs compute the same tile and each writes half of its columns, where the problems are so
// small that half of the SMs would be idle: the epilogue of a tile takes longer than a short main loop.
//
// COPY: some problem's output is also written as FP8 codes.  A variant of its own, because the code of the copy, never taken,
// cost the launches without one 3 to 4 % (1000 x 528 x 2096: 15.3 to 16.0 us).
template <int ES, int BN, int CG, int SPLIT, bool COPY>
__global__ void __launch_bounds__(gemm_threads(kGroupEW), 1)
gemm_group_kernel(const __grid_constant__ GroupParams g) {
  using S = GemmSmem<BN, CG, kGroupEW>;
  static_assert(BN / CG == 128, "128 rows of B per CTA");
  constexpr int kBK = 128 / ES;                     // K elements per stage
  constexpr int kTileM = kBM * CG;
  static_assert(SPLIT == 1 || (BN == 128 && CG == 1), "split tiles are 128 x 128");
  constexpr int kWarpCols = BN / 2 / SPLIT;         // columns of a tile one epilogue warp handles
  // first column a warp handles, and its offset in the tile: a tile column of the work list is tn * SPLIT + part
  auto warp_col = [](int tn, int half) { return tn * (BN / SPLIT) + half * kWarpCols; };
  constexpr uint32_t kChunkBytes = kBK * 128;       // a box of an MN-major operand tile: kBK rows of K x 128 bytes
  constexpr uint32_t kTmemCols = 2 * BN;

  ptx::grid_release_next();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (ptx::smem_addr(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - ptx::smem_addr(smem_raw));
  const uint32_t epi_base = smem_base + S::kStages * S::kStageBytes;
  const uint32_t bars = epi_base + S::kEpiBytes;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (S::kStages + s); };
  auto acc_full_bar = [&](int a) { return bars + 8u * (2 * S::kStages + a); };
  auto acc_empty_bar = [&](int a) { return bars + 8u * (2 * S::kStages + 2 + a); };
  const uint32_t drained_bar = bars + 8u * (2 * S::kStages + 4);
  auto epi_in_bar = [&](int w) { return bars + 8u * (2 * S::kStages + 5 + w); };
  uint8_t* tail = smem_gen + S::kStages * S::kStageBytes + S::kEpiBytes + 8 * (2 * S::kStages + 5 + kGroupEW);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(tail);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = CG == 2 ? (int)ptx::cluster_ctarank() : 0;
  const int unit = blockIdx.x / CG;
  auto entry = [&](int r) { return g.table[r * g.units + unit]; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < S::kStages; ++s) { ptx::mbar_init(full_bar(s), 1); ptx::mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < 2; ++a) { ptx::mbar_init(acc_full_bar(a), 1); ptx::mbar_init(acc_empty_bar(a), CG * kGroupEW); }
    ptx::mbar_init(drained_bar, 1);
    for (int w = 0; w < kGroupEW; ++w) ptx::mbar_init(epi_in_bar(w), 1);
    *abort_flag = 0;
    ptx::mbar_init_fence();
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
      const int end = starved_cta(g.starved, rank) ? min(g.rounds, g.served) : g.rounds;
      for (int r = 0; ok && r < end; ++r) {
        const int32_t e = entry(r);
        if (e < 0) continue;
        int pi, tm, tn;
        group_decode(e, pi, tm, tn);
        const GroupProblem& P = g.prob[pi];
        const int m0 = tm * kTileM + rank * 128, n0 = tn / SPLIT * BN + rank * 128;
        const int num_kb = (P.K + kBK - 1) / kBK, a_mn = P.a_mn, b_mn = P.b_mn;
        if (r == 0) { ptx::prefetch_tensormap(&P.ta); ptx::prefetch_tensormap(&P.tb); }
        for (int kb = 0; kb < num_kb; ++kb) {
          ok = wait_bounded(empty_bar(stage), phase ^ 1u, abort_flag, g.status, g.wait_limit);
          if (!ok) break;
          const uint32_t a_dst = smem_base + stage * S::kStageBytes, b_dst = a_dst + S::kABytes;
          const int k0 = kb * kBK;
          if (issued == 0) ptx::grid_wait_previous();
          const uint32_t fb = CG == 2 ? ptx::in_even_cta(full_bar(stage)) : full_bar(stage);
          if (rank == 0) ptx::mbar_expect_tx(full_bar(stage), CG * S::kStageBytes);
          auto load = [&](uint32_t dst, const void* tmap, int x, int y) {
            if (CG == 2) ptx::tma_load_2d_pair(dst, tmap, fb, x, y); else ptx::tma_load_2d(dst, tmap, fb, x, y);
          };
          auto operand = [&](uint32_t dst, const void* tmap, int mn, int mn0) {
            if (mn) {
#pragma unroll
              for (int c = 0; c < ES; ++c) load(dst + c * kChunkBytes, tmap, mn0 + c * kBK, k0);   // 128 / ES elements per box
            } else {
              load(dst, tmap, k0, mn0);
            }
          };
          operand(a_dst, &P.ta, a_mn, m0);
          operand(b_dst, &P.tb, b_mn, n0);
          ++issued;
          if (++stage == S::kStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (*abort_flag && rank == 0) {
        const uint32_t n = issued < (uint32_t)S::kStages ? issued : (uint32_t)S::kStages;
        for (uint32_t i = 0; i < n; ++i) {
          if (stage == 0) { stage = S::kStages; phase ^= 1u; }
          --stage;
          for (uint32_t it = 0; it < g.wait_limit && !ptx::mbar_try_wait(full_bar(stage), phase); ++it) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (even CTA of a pair only)
    if (ptx::elect_one() && rank == 0) {
      int stage = 0; uint32_t phase = 0, local = 0;
      bool ok = true;
      constexpr uint32_t kStageStep = S::kStageBytes >> 4;
      for (int r = 0; ok && r < g.rounds; ++r) {
        const int32_t e = entry(r);
        if (e < 0) continue;
        int pi, tm, tn;
        group_decode(e, pi, tm, tn);
        const GroupProblem& P = g.prob[pi];
        const int num_kb = (P.K + kBK - 1) / kBK;
        const uint64_t a_desc0 = P.a_mn ? ptx::smem_desc_sw128(smem_base, kChunkBytes, 1024) : ptx::smem_desc_sw128(smem_base, 16, 1024);
        const uint64_t b_desc0 = P.b_mn ? ptx::smem_desc_sw128(smem_base + S::kABytes, kChunkBytes, 1024)
                                        : ptx::smem_desc_sw128(smem_base + S::kABytes, 16, 1024);
        const uint32_t a_hi = (uint32_t)(a_desc0 >> 32), b_hi = (uint32_t)(b_desc0 >> 32);
        const uint32_t a_lo0 = (uint32_t)a_desc0, b_lo0 = (uint32_t)b_desc0;
        const uint32_t a_step = (P.a_mn ? kChunkBytes / kKSteps : 32u) >> 4, b_step = (P.b_mn ? kChunkBytes / kKSteps : 32u) >> 4;
        const uint32_t idesc = P.idesc;
        const uint32_t acc = local & 1u, acc_phase = (local >> 1) & 1u;
        if (local == 0) ptx::grid_wait_previous();       // no operand comes earlier: the bounded waits begin when the loads do
        ++local;
        ok = wait_bounded(acc_empty_bar(acc), acc_phase ^ 1u, abort_flag, g.status, g.wait_limit);
        if (!ok) break;
        ptx::tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + acc * BN;
        uint32_t accumulate = 0;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!ptx::mbar_try_wait(full_bar(stage), phase)) {
            ok = wait_bounded(full_bar(stage), phase, abort_flag, g.status, g.wait_limit);
            if (!ok) break;
          }
          ptx::tc_fence_after_sync();
          const uint32_t a_lo = a_lo0 + stage * kStageStep, b_lo = b_lo0 + stage * kStageStep;
#pragma unroll
          for (int k = 0; k < kKSteps; ++k) {
            const uint64_t adesc = ((uint64_t)a_hi << 32) | (a_lo + k * a_step);
            const uint64_t bdesc = ((uint64_t)b_hi << 32) | (b_lo + k * b_step);
            if (CG == 2) ptx::mma_ss_pair<ES == 1>(d_tmem, adesc, bdesc, idesc, accumulate);
            else ptx::mma_ss<ES == 1>(d_tmem, adesc, bdesc, idesc, accumulate);
            accumulate = 1;
          }
          if (CG == 2) ptx::mma_commit_pair(empty_bar(stage), 3); else ptx::mma_commit(empty_bar(stage));
          if (++stage == S::kStages) { stage = 0; phase ^= 1u; }
        }
        if (ok) { if (CG == 2) ptx::mma_commit_pair(acc_full_bar(acc), 3); else ptx::mma_commit(acc_full_bar(acc)); }
      }
      if (*abort_flag) {
        if (CG == 2) ptx::mma_commit_pair(drained_bar, 1); else ptx::mma_commit(drained_bar);
        for (uint32_t it = 0; it < g.wait_limit && !ptx::mbar_try_wait(drained_bar, 0); ++it) {}
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps
    // Warp (quarter q, half) owns 32 rows x half of the columns of a tile, worked in 32-column slices.  Staging: box 0
    // (4 KB) receives the skip tensor's boxes by TMA, box 1 (4 KB) collects output and leaves by TMA store.
    const int q = warp & 3, half = (warp - 2) >> 2;
    const uint32_t buf_in = epi_base + (warp - 2) * epi_warp_bytes(kGroupEW), buf_out = buf_in + 4096u;
    const uint32_t in_bar = epi_in_bar(warp - 2);
    const uint32_t row_off = (uint32_t)lane * 128u, sw = (uint32_t)(lane & 7);
    uint32_t in_phase = 0, local = 0;
    bool in_pending = false, ok = true;

    auto issue_in = [&](const CUtensorMap* map, int col, int row0) {
      if (ptx::elect_one()) {
        ptx::mbar_expect_tx(in_bar, 4096);
        ptx::tma_load_2d(buf_in, map, in_bar, col, row0);
      }
      in_pending = true;
    };
    // The entry of a round, and the first box of the skip tensor that its tile has for this warp (map null: none).  A round is looked at
    // while the one before waits for its accumulator, the first one before the previous kernel is waited for.
    int mine = g.rounds;                                       // entries of this unit
    while (mine > 0 && entry(mine - 1) < 0) --mine;
    struct Next { int32_t e; const CUtensorMap* map; int col, row; };
    auto look = [&](int r) {
      Next n{r < mine ? entry(r) : -1, nullptr, 0, 0};
      if (n.e < 0) return n;
      int pi, tm, tn;
      group_decode(n.e, pi, tm, tn);
      const GroupProblem& P = g.prob[pi];
      n.col = warp_col(tn, half); n.row = tm * kTileM + rank * 128 + q * 32;
      if (P.has_skip && n.col < P.N) n.map = &P.tskip;
      return n;
    };
    Next next = look(0);
    ptx::grid_wait_previous();
    if (next.map) issue_in(next.map, next.col, next.row);

    for (int r = 0; ok && next.e >= 0; ++r) {
      int pi, tm, tn;
      group_decode(next.e, pi, tm, tn);
      const GroupProblem& P = g.prob[pi];
      const uint32_t acc = local & 1u, acc_phase = (local >> 1) & 1u;
      ++local;
      const int row0 = tm * kTileM + rank * 128 + q * 32, n_w = warp_col(tn, half);
      // The problem's fields are fetched once per tile: a parameter reached through an index is a long load, and would be loaded again after
      // every instruction that may write memory.
      const bool skip = ptx::once(P.has_skip) != 0;
      const int skip_dt = ptx::once(P.skip_dt), out_dt = ptx::once(P.out_dt), cols = ptx::once(P.N);
      const float scale = __int_as_float(ptx::once(__float_as_int(P.scale))), skip_coef = __int_as_float(ptx::once(__float_as_int(P.skip_coef))),
                  out_coef = __int_as_float(ptx::once(__float_as_int(P.out_coef)));
      const int in_es = dtype_size(skip_dt), out_es = dtype_size(out_dt);
      // an output box holds 128-byte rows, or the fewer bytes that a warp's columns are (swizzled accordingly; 32-byte rows: not)
      const int out_row = min(128, kWarpCols * out_es);
      const int in_box_cols = 128 / in_es, out_box_cols = out_row / out_es;
      const uint32_t out_sw = out_row == 128 ? sw : out_row == 64 ? (uint32_t)((lane >> 1) & 3) : 0u;
      next = look(r + 1);
      ok = wait_bounded(acc_full_bar(acc), acc_phase, abort_flag, g.status, g.wait_limit);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      ptx::tc_fence_after_sync();
      const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + acc * BN + (tn % SPLIT) * (BN / SPLIT) + half * kWarpCols;
      auto release_acc = [&]() {
        ptx::tc_fence_before_sync();
        __syncwarp();
        if (lane == 0 && r + 2 < mine) {                     // (where no later tile takes it nobody waits)
          if (CG == 2) ptx::mbar_arrive_cluster(ptx::in_even_cta(acc_empty_bar(acc)));
          else ptx::mbar_arrive(acc_empty_bar(acc));
        }
      };
      bool released = false, looked_ahead = false;
      if (n_w < cols) {
        const f32x2 scale2 = splat2(scale), skip2 = splat2(skip_coef), oc2 = splat2(out_coef);
#pragma unroll 1
        for (int sl = 0; sl < kWarpCols / 32; ++sl) {
          const int col = n_w + 32 * sl;
          if (col >= cols) break;
          const bool last_slice = sl == kWarpCols / 32 - 1 || col + 32 >= cols;
          uint4 raw[8];
          if (skip) {
            const int off = (32 * sl) & (in_box_cols - 1);
            if (off == 0) {
              ok = wait_bounded(in_bar, in_phase, abort_flag, g.status, g.wait_limit);
              ok = __all_sync(0xffffffffu, ok);
              if (!ok) break;
              in_phase ^= 1u;
              in_pending = false;
            }
            const uint32_t cb = (uint32_t)(off * in_es) >> 4;
            const int nchunk = 2 * in_es;
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (j < nchunk) raw[j] = ptx::lds128(buf_in + row_off + (((cb + j) ^ sw) << 4));
            if (off + 32 == in_box_cols || last_slice) {
              __syncwarp();                                    // every lane has read the box
              if (!last_slice) issue_in(&P.tskip, col + 32, row0);
              else { if (next.map) issue_in(next.map, next.col, next.row); looked_ahead = true; }
            }
          }
          const int out_off = (32 * sl) & (out_box_cols - 1);
          if (out_off == 0) {                                  // the output box is about to be refilled
            if (ptx::elect_one()) ptx::bulk_wait_group_read<0>();
            __syncwarp();
          }
          float v[32];
          ptx::tmem_ld_32x32(t_row + 32 * sl, v);
          if (last_slice) { release_acc(); released = true; }
          const uint32_t out_cb = (uint32_t)(out_off * out_es) >> 4;
          const uint32_t dst = buf_out + (uint32_t)(lane * out_row);
          uint32_t copy[8];
          float y[32];
          // The choices of a tile are taken once per slice, not once per eight columns.
#pragma unroll
          for (int k = 0; k < 16; ++k) unpack2(mul2(pack2(v[2 * k], v[2 * k + 1]), scale2), y[2 * k], y[2 * k + 1]);
          if (skip) {
            residual_row32(skip_dt, raw, skip2, oc2, y);
            if (COPY && P.copy) copy_codes32(out_dt, P.copy_dt, y, copy);
          }
          stage_row32(out_dt, y, dst, out_cb, out_sw);
          if (COPY && skip && P.copy && row0 + lane < P.M)
            copy_store(P.copy + (int64_t)(row0 + lane) * P.copy_ld + col, copy, cols - col, P.copy_sectors != 0);
          if (out_off + 32 == out_box_cols || last_slice) {
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (ptx::elect_one()) { ptx::tma_store_2d(&P.tout, buf_out, col - out_off, row0); ptx::bulk_commit_group(); }
          }
        }
      }
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      if (!released) release_acc();
      if (!looked_ahead && next.map) issue_in(next.map, next.col, next.row);   // plain tile, or no columns here: the input box is free, fetch for the next tile
    }
    if (in_pending && lane == 0)
      for (uint32_t it = 0; it < g.wait_limit && !ptx::mbar_try_wait(in_bar, in_phase); ++it) {}
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

}  // namespace us
