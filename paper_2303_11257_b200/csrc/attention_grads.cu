// Fused scaled dot-product attention, whole backward pass (us_attention_bwd_all): per (sequence, head) problem
//     dP = beta_p dC V^T,   dS = softmax_beta * p (dP - sum_j p_j dP_j),  p = P / softmax_alpha
//     dQ = beta_q dS K,     dK = beta_k dS^T Q,     dV = beta_v P^T dC
// in ONE persistent kernel.  us_attention_bwd followed by two batched GEMMs for dK and dV computes the same and reads the two
// score-sized tensors P and dS three times from memory and writes one; here P is read once and dS written once.
//
// A CTA has 128 keys of a problem, a cluster of two or four CTAs (up to 128 keys: one CTA) all of them; the cluster walks the problem in tiles of 128
// query rows.  Two groups of eight softmax warps take the tiles in turn, so that one group's waits (for the tensor cores, the
// cluster, memory) run under the other's arithmetic.  Tensor memory of a CTA: per group dP of its tile (128 x 128 float32; dQ
// of the tile takes the first 64 of these columns once dP is dead), and for two problems in turn the sums dV and dK over the
// tiles (128 keys x 64 columns each).  Per tile:
//   * dC V^T fills dP; P^T dC is added to dV (A operand: the tile of P as it lies in shared memory, read MN-major);
//   * the group (two warps per TMEM lane quarter, a query row per lane) forms the row sums of P dP over the CTA's keys, the
//     CTAs of the cluster exchange them through distributed shared memory, and the group turns P into dS in place;
//   * dS K gives dQ over the CTA's keys, and dS^T Q is added to dK; the tile of dS leaves by TMA store;
//   * dQ: lane quarter q belongs to CTA q mod (cluster size), to which every CTA sends its part (4 KB a warp), and where two warps
//     of their own add them up, so that no softmax warp starts its next tile late.
// FP8: dC and dS are E5M2, P, Q, K, V E4M3.  A head row is then 64 bytes, and Q, K, V and dC tiles take the 64-byte swizzle.
//
// Bound: the serial chain of a tile (dP, row sums, the cluster's exchange, dS, dQ), of which two are under way in an SM, and beside it the
// 16-bit conversions of the softmax warps; at 128 keys HBM (64 x 16 x 128: 159 MB in 28.8 us, 0.84 of a copy's rate); at shorter lengths the
// same chain again, on tiles that are mostly empty rows (32: three quarters).  128 keys a CTA, because dP of two tiles and the sums of two
// problems fill tensor memory.  16-bit / FP8 operands, E5M2 results of contiguous heads, us against us_attention_bwd and the two GEMMs
// (sequences x heads x length): 16 x 16 x 512 104 / 93 against 130 / 91; 20 x 12 x 400 104 / 92 against 99 / 81; 24 x 16 x 320 123 / 117 against
// 96 / 76; 32 x 16 x 256 57 / 50 against 80 / 58; 64 x 16 x 128 28.8 / 21.4 against 54 / 42; 256 x 16 x 32 64 / 71 against 128 / 129.  The
// store of dS (dS = NULL leaves it out) is 7 / 2 us of 16 x 16 x 512, 4.5 / 3.3 of 32 x 16 x 256.
//
// Every wait is on an mbarrier and bounded, remote arrivals included, and no role waits at a hardware barrier between the
// start and the end, so a wait that runs out (in any CTA of a cluster) only makes the others' waits run out too; the
// cluster then meets at its last barrier, its own copies landed, and a CTA that gave up waits for what its partners had sent it.
#include <cuda.h>
#include <cuda_runtime.h>

#include "attention_host.h"
#include "common.cuh"
#include "gemm_kernel.cuh"
#include "host.h"
#include "sm100.cuh"

namespace us {
namespace {

constexpr int kGrWarps = 8, kGrParts = 2;                 // softmax warps of a group; per TMEM lane quarter
// warp 0: MMA issue; warp 1: TMA and TMEM owner; two groups of softmax warps; in a cluster, two warps that finish dQ
constexpr int gr_threads(bool cluster) { return 64 + 2 * 32 * kGrWarps + (cluster ? 64 : 0); }
constexpr int kGrPieces = 4 * kGrParts;                      // parts of dQ that a CTA gets per tile: 4 / (cluster size) quarters from each CTA, by column half
constexpr int kGrKeys = 128, kGrMaxCluster = kAttnMaxKeys / kGrKeys;
constexpr uint32_t kGrBlock = 128 * 128;                  // 128 query rows x 128 bytes of P / dS
constexpr unsigned int kStatusNotLanded = 2;              // beside kStatusTimeout: stores of a partner did not come in
constexpr uint32_t kColAcc = 256, kColDk = 64;            // sums of problem i: columns 256 + 128 (i mod 2): dV, then dK

// Shared memory.  A tile of P is one block of FP8 or two of 16 bits; a slot holds a tile.
template <bool F8>
struct GradSmem {
  static constexpr uint32_t kRow = F8 ? 64 : 128;                       // bytes of a head row
  static constexpr uint32_t kHead = 128 * kRow;                         // 128 rows of dC, Q, K or V
  static constexpr uint32_t kSlot = (F8 ? 1 : 2) * kGrBlock;
  static constexpr int kSlots = F8 ? 6 : 3;
  static constexpr uint32_t kExchange = 32 * 1024;                      // parts of dQ: eight warp-sized pieces of 4 KB
  static constexpr uint32_t kSums = 4 * kGrMaxCluster * kGrParts * 128 * 4;   // row sums by tile mod 4, rank and part
  static constexpr uint32_t kV = 0, kK = kHead, kDc = 2 * kHead, kQ = 4 * kHead, kP = 5 * kHead, kX = kP + kSlots * kSlot,
                            kS = kX + kExchange, kBars = kS + kSums, kSent = kBars + 512,
                            kTotal = kSent + kGrMaxCluster * 2 * kGrWarps * 8 + 16 + 1024 /* alignment */;
  static_assert(kTotal <= 232448, "shared memory of an SM");
};

struct AttnGradParams {
  int s_q, s_k;
  int q_tiles, nb1, problems;
  float inv_alpha;          // 1 / softmax_alpha
  float ds_scale;           // softmax_beta * beta_p / softmax_alpha
  float beta_q, beta_k, beta_v;
  void *dq, *dk, *dv;
  int dq_dt, dk_dt, dv_dt;
  int64_t dq_ld, dk_ld, dv_ld, dq_st[2], dk_st[2], dv_st[2];
  int store_ds;
  uint32_t idesc_dp, idesc_dv, idesc_dk, idesc_dq;
  unsigned int* status;
  uint32_t wait_limit;
  int stall_rank, stall_tile;   // test hook: this CTA of every cluster loads dC up to this tile only (-1: none), so that the waits run out
  uint32_t zero;            // 0; not a constant to the compiler (see the hand-over of the exchange area)
};

// BF16: 16-bit operands are BF16 (else F16).  CLUSTER: launched in clusters of two or four CTAs (more than 128 keys); without one the
// kernel contains none of the cluster's instructions, some of which a CTA outside a cluster must not even come across.
template <bool F8, bool BF16, bool CLUSTER>
__global__ void __launch_bounds__(gr_threads(CLUSTER), 1)
attention_grads_kernel(const __grid_constant__ CUtensorMap tdc, const __grid_constant__ CUtensorMap tq,
                       const __grid_constant__ CUtensorMap tk, const __grid_constant__ CUtensorMap tv,
                       const __grid_constant__ CUtensorMap tp, const __grid_constant__ CUtensorMap tds, const AttnGradParams a) {
  using S = GradSmem<F8>;
  ptx::grid_release_next();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (ptx::smem_addr(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - ptx::smem_addr(smem_raw));
  const uint32_t q_s = base + S::kQ, xch_s = base + S::kX, bars = base + S::kBars;
  // Tiles of the CTA's whole run are numbered n = 0, 1, ...; group n mod 2 works on tile n.  Barriers of tile n: per group
  // (phase n / 2), row sums by n mod 4 (phase n / 4), slots by n mod kSlots; bar_q once per tile; bar_v, bar_k and bar_acc by
  // problem mod 2.
  auto bar_at = [&](int i) { return bars + 8u * (uint32_t)i; };
  const uint32_t bar_q = bar_at(0), bar_drained = bar_at(35);
  auto bar_xfree = [&](int n) { return bar_at(1 + (n & 1)); };
  auto bar_v = [&](int i) { return bar_at(3 + (i & 1)); };
  auto bar_k = [&](int i) { return bar_at(5 + (i & 1)); };
  auto bar_acc = [&](int i) { return bar_at(7 + (i & 1)); };
  auto bar_dc = [&](int n) { return bar_at(9 + (n & 1)); };
  auto bar_dp = [&](int n) { return bar_at(11 + (n & 1)); };
  auto bar_dv = [&](int n) { return bar_at(13 + (n & 1)); };
  auto bar_ds = [&](int n) { return bar_at(15 + (n & 1)); };
  auto bar_dq = [&](int n) { return bar_at(17 + (n & 1)); };
  auto bar_dk = [&](int n) { return bar_at(19 + (n & 1)); };
  auto bar_free = [&](int n) { return bar_at(21 + (n & 1)); };
  auto bar_xch = [&](int n) { return bar_at(23 + (n & 1)); };
  auto bar_sum = [&](int n) { return bar_at(25 + (n & 3)); };
  auto bar_p = [&](int n) { return bar_at(29 + n % S::kSlots); };
  auto slot = [&](int n) { return base + S::kP + (uint32_t)(n % S::kSlots) * S::kSlot; };
  auto slot_phase = [&](int n) { return (uint32_t)(n / S::kSlots) & 1u; };
  auto dc_s = [&](int n) { return base + S::kDc + (uint32_t)(n & 1) * S::kHead; };
  auto half_phase = [&](int n) { return (uint32_t)(n >> 1) & 1u; };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gen + S::kBars + 288);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gen + S::kBars + 292);
  // What the cluster's softmax warps have sent this CTA, in tiles of their group: row sums and parts of dQ, [rank][warp][2]; behind it the
  // tiles whose parts were expected.  Written at the end, for a CTA that gave up.
  constexpr int kSenders = 2 * kGrWarps;
  auto sent_at = [&](int from, int w) { return (uint32_t)((from * kSenders + w) * 8); };
  constexpr uint32_t kExpected = kGrMaxCluster * kSenders * 8;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cl = CLUSTER ? (int)ptx::cluster_nctarank() : 1, rank = CLUSTER ? (int)ptx::cluster_ctarank() : 0;
  const int first = blockIdx.x / cl, stride = gridDim.x / cl;
  constexpr int kBlockKeys = F8 ? 128 : 64;                 // keys in a 128-byte row of P / dS
  const int key0 = rank * kGrKeys, keys = min(kGrKeys, a.s_k - key0);
  // key blocks of this CTA with at least one key; the last CTA of four has none at 384 keys or fewer: its P, dS, dK and dV are empty
  const int blocks = max(0, (keys + kBlockKeys - 1) / kBlockKeys);
  const int my_problems = first < a.problems ? (a.problems - first + stride - 1) / stride : 0;
  const int steps = my_problems * a.q_tiles;
  // Without a cluster the exchange area is a second buffer for K and V: with one or two tiles in a problem their loads would
  // otherwise be waited for.
  constexpr int ahead = CLUSTER ? 1 : 2;
  auto v_s = [&](int prob) { return base + (ahead == 2 && (prob & 1) ? S::kX : S::kV); };
  auto k_s = [&](int prob) { return base + (ahead == 2 && (prob & 1) ? S::kX + S::kHead : S::kK); };
  auto prob_phase = [&](int prob) { return (uint32_t)(prob >> 1) & 1u; };
  auto coords = [&](int n, int& q0, int& b1, int& b0) {
    const int i = n / a.q_tiles, pr = first + i * stride;
    q0 = (n - i * a.q_tiles) * 128; b0 = pr / a.nb1; b1 = pr - b0 * a.nb1;
  };
  if (threadIdx.x == 0) {
    for (uint32_t b : {bar_q, bar_drained}) ptx::mbar_init(b, 1);
    for (int i = 0; i < 2; ++i) {
      for (uint32_t b : {bar_v(i), bar_k(i), bar_dc(i), bar_dp(i), bar_dv(i), bar_dq(i), bar_dk(i), bar_xch(i)}) ptx::mbar_init(b, 1);
      for (uint32_t b : {bar_acc(i), bar_ds(i), bar_free(i)}) ptx::mbar_init(b, kGrWarps);
    }
    for (int i = 0; i < 4; ++i) ptx::mbar_init(bar_sum(i), kGrWarps);
    for (int i = 0; i < S::kSlots; ++i) ptx::mbar_init(bar_p(i), 1);
    for (int i = 0; i < 2; ++i) ptx::mbar_init(bar_xfree(i), (uint32_t)(cl * kGrParts));   // the cluster's warps that finish dQ have added up a tile
    *abort_flag = 0;
    ptx::mbar_init_fence();
  }
  if (warp == 1) { ptx::tmem_alloc(ptx::smem_addr(const_cast<uint32_t*>(tmem_slot)), 512); ptx::tmem_relinquish(); }
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (CLUSTER) ptx::cluster_sync();                         // the partners' barriers are ready too
  ptx::tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  ptx::grid_wait_previous();

  // Head tiles (dC, Q, K, V): rows of 64 elements; 128-byte rows, FP8 64-byte rows.  As a K-major operand 32 bytes along the
  // row are one MMA's K; as an MN-major one (64 columns, rows are K) an MMA takes 16 rows, FP8 32: 2048 bytes either way.
  auto head_desc = [&](uint32_t addr) { return F8 ? ptx::smem_desc_sw64(addr, 16, 512) : ptx::smem_desc_sw128(addr, 16, 1024); };
  constexpr uint32_t kHeadStep = 2048u >> 4;
  auto wait1 = [&](uint32_t bar, uint32_t parity) { return wait_bounded(bar, parity, abort_flag, a.status, a.wait_limit); };
  // for what other CTAs of the cluster have written or handed back
  auto wait1_cluster = [&](uint32_t bar, uint32_t parity) { return wait_bounded<CLUSTER>(bar, parity, abort_flag, a.status, a.wait_limit); };

  if (warp == 0) {
    if (ptx::elect_one()) {
      // ---------------------------------------------------------------- MMA issue
      // dP and dV of tile n, before dQ and dK of tile n - 1
      auto opening = [&](int n) -> bool {
        const int prob = n / a.q_tiles;
        const bool opens = n == prob * a.q_tiles;
        if (!wait1(bar_dc(n), half_phase(n)) || (opens && !wait1(bar_v(prob), prob_phase(prob))) ||
            (n > 1 && !wait1(bar_free(n), half_phase(n) ^ 1u)))
          return false;
        ptx::tc_fence_after_sync();
        const uint64_t cd = head_desc(dc_s(n)), vd = head_desc(v_s(prob));
#pragma unroll
        for (int k = 0; k < (F8 ? 2 : 4); ++k) ptx::mma_ss<F8>(tmem + 128u * (n & 1), cd + 2u * k, vd + 2u * k, a.idesc_dp, k > 0);
        ptx::mma_commit(bar_dp(n));
        if (!wait1(bar_p(n), slot_phase(n)) || (opens && prob > 1 && !wait1(bar_acc(prob), prob_phase(prob) ^ 1u))) return false;
        ptx::tc_fence_after_sync();
        // P (or dS) as an MN-major A operand: 4096 (2048) bytes of query rows per MMA
        const uint64_t pd = ptx::smem_desc_sw128(slot(n), kGrBlock, 1024);
#pragma unroll
        for (int k = 0; k < (F8 ? 4 : 8); ++k)
          ptx::mma_ss<F8>(tmem + kColAcc + 128u * (prob & 1), pd + ((F8 ? 4096u : 2048u) >> 4) * k, cd + kHeadStep * k, a.idesc_dv, !opens || k > 0);
        ptx::mma_commit(bar_dv(n));
        return true;
      };
      auto closing = [&](int n) -> bool {
        const int prob = n / a.q_tiles;
        const bool opens = n == prob * a.q_tiles;
        if ((opens && !wait1(bar_k(prob), prob_phase(prob))) || !wait1(bar_ds(n), half_phase(n))) return false;
        ptx::tc_fence_after_sync();
        const uint64_t kd = head_desc(k_s(prob)), qd = head_desc(q_s);
        for (int b = 0; b < blocks; ++b) {
          const uint64_t sd = ptx::smem_desc_sw128(slot(n) + (uint32_t)b * kGrBlock, 16, 1024);
#pragma unroll
          for (int k = 0; k < 4; ++k)                        // 32 bytes along a row of dS
            ptx::mma_ss<F8>(tmem + 128u * (n & 1), sd + 2u * k, kd + kHeadStep * (4 * b + k), a.idesc_dq, (b | k) != 0);
        }
        ptx::mma_commit(bar_dq(n));
        if (!wait1(bar_q, (uint32_t)n & 1u)) return false;
        ptx::tc_fence_after_sync();
        const uint64_t sd = ptx::smem_desc_sw128(slot(n), kGrBlock, 1024);
#pragma unroll
        for (int k = 0; k < (F8 ? 4 : 8); ++k)
          ptx::mma_ss<F8>(tmem + kColAcc + 128u * (prob & 1) + kColDk, sd + ((F8 ? 4096u : 2048u) >> 4) * k, qd + kHeadStep * k, a.idesc_dk, !opens || k > 0);
        ptx::mma_commit(bar_dk(n));
        return true;
      };
      bool ok = true;
      for (int n = 0; ok && n <= steps; ++n) {
        if (n < steps) ok = opening(n);
        if (ok && n > 0) ok = closing(n - 1);
      }
      if (*abort_flag) {                                     // MMAs that were issued finish before the CTA gives up its memory
        ptx::mma_commit(bar_drained);
        for (uint32_t it = 0; it < a.wait_limit && !ptx::mbar_try_wait(bar_drained, 0); ++it) {}
      }
    }
  } else if (warp == 1) {
    if (ptx::elect_one()) {
      // ---------------------------------------------------------------- loads, and dS out
      auto load = [&](uint32_t dst, const CUtensorMap* tm, uint32_t bar, int row, int n) {      // row < 0: the tile's query rows
        int q0, b1, b0;
        coords(n, q0, b1, b0);
        ptx::mbar_expect_tx(bar, S::kHead);
        ptx::tma_load_4d(dst, tm, bar, 0, row < 0 ? q0 : row, b1, b0);
      };
      auto load_p = [&](int n) {
        int q0, b1, b0;
        coords(n, q0, b1, b0);
        ptx::mbar_expect_tx(bar_p(n), S::kSlot);
        ptx::tma_load_4d(slot(n), &tp, bar_p(n), key0, q0, b1, b0);
        if (!F8) ptx::tma_load_4d(slot(n) + kGrBlock, &tp, bar_p(n), key0 + kBlockKeys, q0, b1, b0);
      };
      int n_p = 0, n_dc = 0, n_q = 0, n_v = 0, n_k = 0;      // loads asked for
      const int stall = rank == a.stall_rank ? a.stall_tile : 0x7fffffff;
      auto load_dc = [&](int n) {
        if (n >= stall) return;
        load(dc_s(n), &tdc, bar_dc(n), -1, n);
        ++n_dc;
      };
      auto load_v = [&]() { load(v_s(n_v), &tv, bar_v(n_v), key0, n_v * a.q_tiles); ++n_v; };      // of the next problem
      auto load_k = [&]() { load(k_s(n_k), &tk, bar_k(n_k), key0, n_k * a.q_tiles); ++n_k; };
      if (steps > 0) {
        load_dc(0);
        load_v();
        load_p(n_p++);
        if (steps > 1) { load_dc(1); load_p(n_p++); }
        load_k();
        load(q_s, &tq, bar_q, -1, 0); ++n_q;
        if (ahead == 2 && my_problems > 1) { load_v(); load_k(); }
        while (n_p < steps && n_p < S::kSlots) load_p(n_p++);
      }
      for (int n = 0; n < steps; ++n) {
        const bool closes = (n + 1) % a.q_tiles == 0;        // last tile of its problem
        if (closes && n_v < my_problems) {                   // V has been read for the last time in this problem
          if (!wait1(bar_dp(n), half_phase(n))) break;
          load_v();
        }
        if (!wait1(bar_dv(n), half_phase(n))) break;         // ... and dC of this tile
        if (n + 2 < steps) load_dc(n + 2);
        if (!wait1(bar_ds(n), half_phase(n))) break;
        if (a.store_ds) {
          int q0, b1, b0;
          coords(n, q0, b1, b0);
          for (int b = 0; b < blocks; ++b) ptx::tma_store_4d(&tds, slot(n) + (uint32_t)b * kGrBlock, key0 + b * kBlockKeys, q0, b1, b0);
          ptx::bulk_commit_group();
        }
        if (!wait1(bar_dk(n), half_phase(n))) break;         // the MMAs have read dS, Q and (dQ's, before them) K
        if (n + 1 < steps) { load(q_s, &tq, bar_q, -1, n + 1); ++n_q; }
        if (closes && n_k < my_problems) load_k();
        ptx::bulk_wait_group_read<0>();                      // ... and the store dS: this tile's slot is free
        if (n_p < steps) load_p(n_p++);
      }
      ptx::bulk_wait_group_read<0>();
      if (*abort_flag) {
        // every copy that was asked for lands before the CTA gives up its shared memory: each barrier's latest phases
        auto landed = [&](uint32_t bar, int count) {
          if (count > 0) for (uint32_t it = 0; it < a.wait_limit && !ptx::mbar_try_wait(bar, (uint32_t)(count - 1) & 1u); ++it) {}
        };
        landed(bar_q, n_q);
        for (int i = 0; i < 2; ++i) { landed(bar_v(i), (n_v + 1 - i) / 2); landed(bar_k(i), (n_k + 1 - i) / 2); landed(bar_dc(i), (n_dc + 1 - i) / 2); }
        for (int i = max(0, n_p - S::kSlots); i < n_p; ++i)
          for (uint32_t it = 0; it < a.wait_limit && !ptx::mbar_try_wait(bar_p(i), slot_phase(i)); ++it) {}
      }
    }
  } else if (CLUSTER && warp >= 2 + 2 * kGrWarps) {
    // ------------------------------------------------------------------ dQ of this CTA's lane quarters (in a cluster)
    // The exchange area: by quarter, part and sender, pieces of 32 rows x 32 columns, a lane's 16-byte piece i at 512 i.
    const int part = warp - (2 + 2 * kGrWarps);
    int expected = 0;
    for (int n = 0; n < steps; ++n) {
      int q0, b1, b0;
      coords(n, q0, b1, b0);
      if (part == 0 && lane == 0) ptx::mbar_expect_tx(bar_xch(n), kGrPieces * 4096u);
      ++expected;
      if (!__all_sync(0xffffffffu, wait1_cluster(bar_xch(n), half_phase(n)))) break;
      uint32_t seen = 0;
      for (int i = 0; i < 4 / cl; ++i) {
        const uint32_t buf = xch_s + (uint32_t)((i * kGrParts + part) * cl) * 4096u + (uint32_t)lane * 16u;
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = 0.f;
#pragma unroll 1
        for (int k = 0; k < cl; ++k) {                         // in rank order
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint4 o = ptx::lds128(buf + (uint32_t)k * 4096u + 512u * j);
            v[4 * j] += __uint_as_float(o.x); v[4 * j + 1] += __uint_as_float(o.y);
            v[4 * j + 2] += __uint_as_float(o.z); v[4 * j + 3] += __uint_as_float(o.w);
          }
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) seen |= __float_as_uint(v[j]);
        if (i == 4 / cl - 1) {
          // The pieces may be overwritten.  The arrivals are ordered behind the reads of all lanes by a dependency: their address
          // contains every value that was read (and a zero that only the host knows to be one), so they cannot be made before the
          // last of these has come, and the partners' stores follow from the arrivals.  A release at cluster scope orders the same and
          // waits for the stores to global memory too: 104 -> 123 us at 16 x 16 x 512, 57 -> 63 at 32 x 16 x 256, 16 bits.
          const uint32_t none = __reduce_or_sync(0xffffffffu, seen) & a.zero;
          if (lane < cl) ptx::mbar_arrive_relaxed_cluster(ptx::in_cta(bar_xfree(n), (uint32_t)lane) + none);
        }
        const int row = q0 + (rank + i * cl) * 32 + lane;
        if (row < a.s_q) {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] *= a.beta_q;
          char* dst = static_cast<char*>(a.dq) + ((int64_t)b0 * a.dq_st[0] + (int64_t)b1 * a.dq_st[1] + (int64_t)row * a.dq_ld + 32 * part) * dtype_size(a.dq_dt);
          store_vec<32>(dst, a.dq_dt, v);
        }
      }
    }
    if (part == 0 && lane == 0) *reinterpret_cast<volatile int*>(gen + S::kSent + kExpected) = expected;
  } else {
    // ------------------------------------------------------------------ softmax gradient, dQ, dK, dV
    // Warp (group, q, part): query rows 32 q .. + 31 of a tile, one per lane; the 32-key chunks part and part + 2 of the CTA's
    // keys, 32 of dQ's columns, and at the end of a problem 32 keys of dV (part 0) or dK.
    const int group = (warp - 2) >> 3, q = warp & 3, part = ((warp - 2) >> 2) & 1, r = q * 32 + lane;
    const uint32_t t_row = tmem + ((uint32_t)(q * 32) << 16), t_dp = t_row + 128u * group;
    constexpr int kPerBlock = kBlockKeys / 32;                // chunks in a key block
    constexpr int kPieces = F8 ? 2 : 4;                       // 16-byte pieces of a chunk: 16 FP8 or 8 16-bit values each
    constexpr int kVals = F8 ? 16 : 8;
    const int c_end = blocks * kPerBlock;
    const uint32_t row_off = (uint32_t)r * 128u, sw = (uint32_t)(r & 7);
    uint32_t sent_sums = 0, sent_dq = 0;
    auto values = [&](const uint4& raw, float (&pv)[16]) {
      const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (F8) {
          const float2 lo = unpack_fp8x2((uint16_t)(w[i] & 0xffffu), false), hi = unpack_fp8x2((uint16_t)(w[i] >> 16), false);
          pv[4 * i] = lo.x; pv[4 * i + 1] = lo.y; pv[4 * i + 2] = hi.x; pv[4 * i + 3] = hi.y;
        } else {
          const float2 f = BF16 ? unpack_bf16x2(w[i]) : unpack_f16x2(w[i]);
          pv[2 * i] = f.x; pv[2 * i + 1] = f.y;
        }
      }
    };
    auto wait = [&](uint32_t bar, uint32_t parity) { return (bool)__all_sync(0xffffffffu, wait1(bar, parity)); };
    auto wait_cluster = [&](uint32_t bar, uint32_t parity) { return (bool)__all_sync(0xffffffffu, wait1_cluster(bar, parity)); };
#pragma unroll 1
    for (int n = group; n < steps; n += 2) {
      const uint32_t ph = half_phase(n);
      int q0, b1, b0;
      coords(n, q0, b1, b0);
      if (!wait(bar_dp(n), ph) || !wait(bar_p(n), slot_phase(n))) break;
      ptx::tc_fence_after_sync();
      auto p_addr = [&](int c, int g) {                       // 16-byte piece g of chunk c of this row
        return slot(n) + (uint32_t)(c / kPerBlock) * kGrBlock + row_off + ((((uint32_t)((c % kPerBlock) * kPieces + g)) ^ sw) << 4);
      };
      // sum_j P_j dP_j over this warp's keys (keys beyond s_k are zeros in both factors)
      float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
      for (int c = part; c < c_end; c += kGrParts) {
        uint32_t x[32];
        ptx::tmem_ld_32x32_issue(t_dp + 32u * c, x);
        uint4 raw[kPieces];
#pragma unroll
        for (int g = 0; g < kPieces; ++g) raw[g] = ptx::lds128(p_addr(c, g));
        ptx::tmem_ld_fence(x);
#pragma unroll
        for (int g = 0; g < kPieces; ++g) {
          float pv[16];
          values(raw[g], pv);
#pragma unroll
          for (int i = 0; i < kVals; ++i) s4[i & 3] = fmaf(pv[i], __uint_as_float(x[kVals * g + i]), s4[i & 3]);
        }
      }
      const float mine = (s4[0] + s4[1]) + (s4[2] + s4[3]);
      // Every CTA of the cluster gets every part, 16 bytes at a time (4-byte stores, each counted on the barrier, took 6000 cycles).
      // Four sets of sums and barriers in turn: a partner sends those of tile n + 4 only after it has this CTA's of tile n + 2, which
      // a warp here sends when it has read the sums of tile n.  One warp's arrival brings the bytes to expect.
      const uint32_t set = (uint32_t)((n & 3) * kGrMaxCluster * kGrParts * 128);
      const uint32_t at = base + S::kS + 4u * (set + (uint32_t)((rank * kGrParts + part) * 128 + q * 32));
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(at + 4u * (uint32_t)lane), "f"(mine) : "memory");
      if constexpr (CLUSTER) {
        float four[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) four[i] = __shfl_sync(0xffffffffu, mine, 4 * (lane & 7) + i);
        if (lane < 8) {
          for (int k = 0; k < cl; ++k)
            if (k != rank) ptx::st_async128(ptx::in_cta(at + 16u * (uint32_t)lane, (uint32_t)k), four, ptx::in_cta(bar_sum(n), (uint32_t)k));
        }
      }
      __syncwarp();
      if (lane == 0) {
        if (CLUSTER && q == rank && part == 0) {
          ptx::mbar_expect_tx(bar_sum(n), (uint32_t)((cl - 1) * kGrWarps) * 128u);
        } else {
          ptx::mbar_arrive(bar_sum(n));
        }
      }
      ++sent_sums;
      if (!wait_cluster(bar_sum(n), (uint32_t)(n >> 2) & 1u)) break;
      const volatile float* sums = reinterpret_cast<const volatile float*>(gen + S::kS) + set + r;      // [rank][part][row]
      float total = 0.f;
      for (int k = 0; k < cl; ++k) total += sums[k * kGrParts * 128] + sums[k * kGrParts * 128 + 128];
      const float mean = total * a.inv_alpha;                  // sum_j p_j dP_j in units of the raw accumulator
      if (!wait(bar_dv(n), ph)) break;                         // P^T dC has read the tile
      // dS = ds_scale * P * (dP - mean), rounded, over P in place
#pragma unroll 1
      for (int c = part; c < c_end; c += kGrParts) {
        float x[32];
        ptx::tmem_ld_32x32(t_dp + 32u * c, x);
#pragma unroll
        for (int g = 0; g < kPieces; ++g) {
          const uint32_t addr = p_addr(c, g);
          float pv[16], d[16];
          values(ptx::lds128(addr), pv);
#pragma unroll
          for (int i = 0; i < kVals; ++i) d[i] = a.ds_scale * pv[i] * (x[kVals * g + i] - mean);
          uint32_t o[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (F8) o[i] = cvt_fp8x4<true>(d[4 * i], d[4 * i + 1], d[4 * i + 2], d[4 * i + 3]);     // gradients: E5M2
            else o[i] = BF16 ? pack_bf16x2(d[2 * i], d[2 * i + 1]) : pack_f16x2(d[2 * i], d[2 * i + 1]);
          }
          ptx::sts128(addr, make_uint4(o[0], o[1], o[2], o[3]));
        }
      }
      ptx::fence_proxy_async_smem();                           // the MMAs and the TMA store read these bytes
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(bar_ds(n));
      // ---------------------------------------------------------------- dQ: this warp's 32 of the 64 columns
      if (!wait(bar_dq(n), ph)) break;
      ptx::tc_fence_after_sync();
      float v[32];
      ptx::tmem_ld_32x32(t_dp + 32u * part, v);
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(bar_free(n));            // the group's next dP may overwrite dQ
      if constexpr (CLUSTER) {
        // to the CTA that finishes this quarter, once the cluster has added up the tile before
        if (blocks == 0) {
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = 0.f;
        }
        // (a wait by parity is sound only for a waiter that has seen every earlier phase: hence a barrier for the tiles of each group)
        if (n > 0 && !wait_cluster(bar_xfree(n - 1), half_phase(n - 1))) break;
        const uint32_t owner = (uint32_t)(q % cl), bar = ptx::in_cta(bar_xch(n), owner);
        const uint32_t dst = ptx::in_cta(xch_s + (uint32_t)(((q / cl) * kGrParts + part) * cl + rank) * 4096u + (uint32_t)lane * 16u, owner);
#pragma unroll
        for (int i = 0; i < 8; ++i) ptx::st_async128(dst + 512u * i, &v[4 * i], bar);
        ++sent_dq;
      } else if (q0 + r < a.s_q) {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] *= a.beta_q;
        char* dst = static_cast<char*>(a.dq) + ((int64_t)b0 * a.dq_st[0] + (int64_t)b1 * a.dq_st[1] + (int64_t)(q0 + r) * a.dq_ld + 32 * part) * dtype_size(a.dq_dt);
        store_vec<32>(dst, a.dq_dt, v);
      }
      // ---------------------------------------------------------------- end of a problem: dV or dK of this lane's key
      if (q0 + 128 >= a.s_q) {
        if (!wait(bar_dk(n), ph)) break;
        ptx::tc_fence_after_sync();
        const int prob = n / a.q_tiles, key = key0 + r;
        const bool of_k = part == 1;
        const int dt = of_k ? a.dk_dt : a.dv_dt;
        const float scale = of_k ? a.beta_k : a.beta_v;
        char* dst = static_cast<char*>(of_k ? a.dk : a.dv) +
                    ((int64_t)b0 * (of_k ? a.dk_st[0] : a.dv_st[0]) + (int64_t)b1 * (of_k ? a.dk_st[1] : a.dv_st[1]) +
                     (int64_t)key * (of_k ? a.dk_ld : a.dv_ld)) * dtype_size(dt);
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
          float y[32];
          ptx::tmem_ld_32x32(t_row + kColAcc + 128u * (prob & 1) + kColDk * part + 32u * i, y);
          if (i == 1) {
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar_acc(prob));    // the problem after next may overwrite these
          }
          if (key < a.s_k) {
#pragma unroll
            for (int e = 0; e < 32; ++e) y[e] *= scale;
            store_vec<32>(dst + (int64_t)32 * i * dtype_size(dt), dt, y);
          }
        }
      }
    }
    if constexpr (CLUSTER) {
      if (lane < cl) ptx::st_cluster_v2(ptx::in_cta(base + S::kSent + sent_at(rank, warp - 2), (uint32_t)lane), sent_sums, sent_dq);
    }
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (CLUSTER) ptx::cluster_sync();                          // no CTA leaves while a partner may still signal it
  if constexpr (CLUSTER) {
    if (*abort_flag && threadIdx.x == 0) {
      // Stores that the partners had under way when this CTA gave up land before it leaves.  The senders of a group are at most one
      // tile apart (each tile of one needs something of the tile before from all): of the first tile that not all have sent, what is
      // missing is made up for here, so that its phase completes with the last of the stores that were issued.
      const volatile uint32_t* sent = reinterpret_cast<const volatile uint32_t*>(gen + S::kSent);
      const int begun = *reinterpret_cast<volatile int*>(gen + S::kSent + kExpected);
      auto land = [&](uint32_t bar, int phase) {
        uint32_t it = 0;
        while (it < a.wait_limit && !ptx::mbar_try_wait_cluster(bar, (uint32_t)phase & 1u)) ++it;
        if (it == a.wait_limit) atomicOr(a.status, kStatusNotLanded);
      };
      for (int g = 0; g < 2; ++g) {
        for (int what = 0; what < 2; ++what) {                 // row sums, parts of dQ
          auto for_senders = [&](auto&& f) {                   // from, tiles sent; of dQ those that send it to this CTA
            for (int from = 0; from < cl; ++from)
              for (int w = g * kGrWarps; w < (g + 1) * kGrWarps; ++w)
                if (what == 0 || ((w + 2) & 3) % cl == rank) f(from, sent[sent_at(from, w) / 4 + what]);
          };
          uint32_t least = 0xffffffffu;
          for_senders([&](int, uint32_t tiles) { least = min(least, tiles); });
          int own = 0, others = 0;                             // that have sent tile number `least` of the group
          for_senders([&](int from, uint32_t tiles) { if (tiles > least) ++(what == 0 && from == rank ? own : others); });
          const int n = g + 2 * (int)least;                    // that tile
          if (what == 0) {
            if (least > 0) land(bar_sum(n - 2), (n - 2) >> 2);
            if (others == 0) continue;
            // the own warp that brings the bytes to expect is the one of quarter `rank`, part 0
            if (sent[sent_at(rank, g * kGrWarps + ((rank + 2) & 3)) / 4] > least) ptx::mbar_complete_tx(bar_sum(n), (uint32_t)((cl - 1) * kGrWarps - others) * 128u);
            else ptx::mbar_expect_only(bar_sum(n), (uint32_t)others * 128u);
            for (; own < kGrWarps; ++own) ptx::mbar_arrive(bar_sum(n));
            land(bar_sum(n), n >> 2);
          } else {
            const int last = others > 0 ? n : n - 2, parts = others > 0 ? others : kGrPieces;       // the last tile with parts under way
            if (last < 0) continue;
            if (last < begun) ptx::mbar_complete_tx(bar_xch(last), (uint32_t)(kGrPieces - parts) * 4096u);
            else ptx::mbar_expect_tx(bar_xch(last), (uint32_t)parts * 4096u);
            land(bar_xch(last), last >> 1);
          }
        }
      }
    }
  }
  if (warp == 1) { ptx::tc_fence_after_sync(); ptx::tmem_dealloc(tmem, 512); }
}

template <bool F8, bool BF16, bool CLUSTER>
us_status launch_grads(const CUtensorMap* t, const AttnGradParams& a, cudaStream_t stream) {
  auto kern = attention_grads_kernel<F8, BF16, CLUSTER>;
  constexpr int smem = GradSmem<F8>::kTotal;
  static std::atomic<uint64_t> smem_set{0};
  const int cl = !CLUSTER ? 1 : a.s_k > 2 * kGrKeys ? 4 : 2;
  static host::ClusterCount count;
  const int fit = host::resident_clusters(reinterpret_cast<const void*>(kern), gr_threads(CLUSTER), smem, cl, count);
  if (fit <= 0) return US_ERR_CUDA;
  return host::launch(kern, &smem_set, cl * (a.problems < fit ? a.problems : fit), gr_threads(CLUSTER), smem, cl, stream, t[0], t[1], t[2], t[3], t[4], t[5], a);
}
template <bool F8, bool BF16>
us_status pick_grads(const CUtensorMap* t, const AttnGradParams& a, cudaStream_t stream) {
  return a.s_k > kGrKeys ? launch_grads<F8, BF16, true>(t, a, stream) : launch_grads<F8, BF16, false>(t, a, stream);
}

// Failure-path test settings of one call.
struct Stall {
  uint32_t wait_limit;
  int rank, tile;
};

us_status bwd_all(const us_mat* dC, const us_mat* P, const us_mat* Q, const us_mat* K, const us_mat* V, float beta_p, float softmax_alpha,
                  float softmax_beta, float beta_q, float beta_k, float beta_v, const us_mat* dS, const us_mat* dQ, const us_mat* dK,
                  const us_mat* dV, const us_attention_bwd_all_batch* batch, void* ws, size_t ws_bytes, void* stream, const Stall& test) {
  if (!dC || !P || !Q || !K || !V || !dQ || !dK || !dV || !batch) return US_ERR_INVALID_ARG;
  if (dS && !dS->ptr) dS = nullptr;
  const int64_t* cnt = batch->count;
  if (cnt[0] < 1 || cnt[1] < 1 || cnt[0] > 65535 || cnt[1] > 65535) return US_ERR_INVALID_ARG;
  const us_mat* all[9] = {dC, P, Q, K, V, dQ, dK, dV, dS};
  const int64_t* strides[9] = {batch->dc_stride, batch->p_stride, batch->q_stride, batch->k_stride, batch->v_stride,
                               batch->dq_stride, batch->dk_stride, batch->dv_stride, batch->ds_stride};
  for (int i = 0; i < 9; ++i) {
    const us_mat* m = all[i];
    if (!m) continue;
    if (m->rows < 0 || m->cols < 0 || m->ld < m->cols) return US_ERR_INVALID_ARG;
    if (m->rows * m->cols > 0 && !m->ptr) return US_ERR_INVALID_ARG;
    for (int j = 0; j < 2; ++j)
      if (cnt[j] > 1 && strides[i][j] <= 0) return US_ERR_INVALID_ARG;
  }
  const int64_t s_q = dC->rows, s_k = K->rows, hd = dC->cols;
  const us_mat *qs[3] = {dC, Q, dQ}, *ks[4] = {K, V, dK, dV};
  for (const us_mat* m : qs)
    if (m->rows != s_q || m->cols != hd) return US_ERR_INVALID_ARG;
  for (const us_mat* m : ks)
    if (m->rows != s_k || m->cols != hd) return US_ERR_INVALID_ARG;
  if (P->rows != s_q || P->cols != s_k || (dS && (dS->rows != s_q || dS->cols != s_k))) return US_ERR_INVALID_ARG;
  if (!(softmax_alpha > 0.f)) return US_ERR_INVALID_ARG;
  const bool h16 = (dC->dtype == US_BF16 || dC->dtype == US_F16) && Q->dtype == dC->dtype && K->dtype == dC->dtype &&
                   V->dtype == dC->dtype && P->dtype == dC->dtype && (!dS || dS->dtype == dC->dtype);
  const bool f8 = dC->dtype == US_E5M2 && P->dtype == US_E4M3 && Q->dtype == US_E4M3 && K->dtype == US_E4M3 && V->dtype == US_E4M3 &&
                  (!dS || dS->dtype == US_E5M2);           // gradients E5M2, activations E4M3
  if (!(h16 || f8)) return US_ERR_UNSUPPORTED;
  for (int i = 5; i < 8; ++i)
    if (all[i]->dtype < US_F32 || all[i]->dtype > US_E5M2) return US_ERR_UNSUPPORTED;
  if (hd != kAttnD || s_k > kAttnMaxKeys) return US_ERR_UNSUPPORTED;
  if (!ws || ws_bytes < us_workspace_bytes()) return US_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(ws) % 16) return US_ERR_ALIGNMENT;
  if (s_q == 0 || s_k == 0) return US_ERR_UNSUPPORTED;     // empty sums: the separate calls say what becomes of each result
  const int es = f8 ? 1 : 2;
  for (int i = 0; i < 9; ++i)
    if (all[i] && !attn_aligned(all[i], strides[i], cnt, i >= 5 && i < 8 ? (int)dtype_size(all[i]->dtype) : es)) return US_ERR_ALIGNMENT;

  AttnGradParams a{};
  a.s_q = (int)s_q; a.s_k = (int)s_k;
  const int64_t q_tiles = (s_q + 127) / 128, problems = cnt[0] * cnt[1];
  if (q_tiles * problems > 0x3fffffff) return US_ERR_INVALID_ARG;
  a.q_tiles = (int)q_tiles; a.nb1 = (int)cnt[1]; a.problems = (int)problems;
  a.inv_alpha = 1.0f / softmax_alpha;
  a.ds_scale = softmax_beta * beta_p / softmax_alpha;
  a.beta_q = beta_q; a.beta_k = beta_k; a.beta_v = beta_v;
  a.dq = dQ->ptr; a.dq_dt = dQ->dtype; a.dq_ld = dQ->ld;
  a.dk = dK->ptr; a.dk_dt = dK->dtype; a.dk_ld = dK->ld;
  a.dv = dV->ptr; a.dv_dt = dV->dtype; a.dv_ld = dV->ld;
  for (int j = 0; j < 2; ++j) {
    a.dq_st[j] = cnt[j] > 1 ? batch->dq_stride[j] : 0;
    a.dk_st[j] = cnt[j] > 1 ? batch->dk_stride[j] : 0;
    a.dv_st[j] = cnt[j] > 1 ? batch->dv_stride[j] : 0;
  }
  a.store_ds = dS != nullptr;
  const bool bf16 = dC->dtype == US_BF16;
  const int grad = f8 ? 1 : bf16, act = f8 ? 0 : bf16;      // kind::f8f6f4: 0 = E4M3, 1 = E5M2; kind::f16: 0 = F16, 1 = BF16
  a.idesc_dp = make_idesc(grad, act, false, false, 128, 128);
  a.idesc_dv = make_idesc(act, grad, true, true, 128, 64);
  a.idesc_dk = make_idesc(grad, act, true, true, 128, 64);
  a.idesc_dq = make_idesc(grad, act, false, true, 128, 64);
  a.status = static_cast<unsigned int*>(ws);
  a.wait_limit = test.wait_limit; a.stall_rank = test.rank; a.stall_tile = test.tile;

  CUtensorMap t[6];                                        // dC, Q, K, V, P, dS
  const int row = f8 ? 64 : 128;
  if (!attn_tmap(&t[0], dC, batch->dc_stride, cnt, 128, es, row) || !attn_tmap(&t[1], Q, batch->q_stride, cnt, 128, es, row) ||
      !attn_tmap(&t[2], K, batch->k_stride, cnt, kGrKeys, es, row) || !attn_tmap(&t[3], V, batch->v_stride, cnt, kGrKeys, es, row) ||
      !attn_tmap(&t[4], P, batch->p_stride, cnt, 128, es))
    return US_ERR_CUDA;
  t[5] = t[4];
  if (dS && !attn_tmap(&t[5], dS, batch->ds_stride, cnt, 128, es)) return US_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return f8 ? pick_grads<true, false>(t, a, st) : bf16 ? pick_grads<false, true>(t, a, st) : pick_grads<false, false>(t, a, st);
}

}  // namespace
}  // namespace us

extern "C" us_status us_attention_bwd_all(const us_mat* dC, const us_mat* P, const us_mat* Q, const us_mat* K, const us_mat* V,
                                          float beta_p, float softmax_alpha, float softmax_beta, float beta_q, float beta_k,
                                          float beta_v, const us_mat* dS, const us_mat* dQ, const us_mat* dK, const us_mat* dV,
                                          const us_attention_bwd_all_batch* batch, void* ws, size_t ws_bytes, void* stream) {
  return us::bwd_all(dC, P, Q, K, V, beta_p, softmax_alpha, softmax_beta, beta_q, beta_k, beta_v, dS, dQ, dK, dV, batch, ws, ws_bytes, stream,
                     {us::kWaitLimit, -1, 0});
}
extern "C" us_status us_test_attention_bwd_all_starved(const us_mat* dC, const us_mat* P, const us_mat* Q, const us_mat* K, const us_mat* V,
                                                       float softmax_alpha, const us_mat* dS, const us_mat* dQ, const us_mat* dK,
                                                       const us_mat* dV, const us_attention_bwd_all_batch* batch, void* ws, size_t ws_bytes,
                                                       unsigned int wait_limit, int rank, int tile, void* stream) {
  if (wait_limit < 1 || wait_limit > (1u << 16) || rank < 0 || tile < 0) return US_ERR_INVALID_ARG;
  return us::bwd_all(dC, P, Q, K, V, 1.f, softmax_alpha, 1.f, 1.f, 1.f, 1.f, dS, dQ, dK, dV, batch, ws, ws_bytes, stream, {wait_limit, rank, tile});
}
