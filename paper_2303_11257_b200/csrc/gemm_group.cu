// us_linear_group: several independent linear ops in one launch (host side: checks, work list, launch).
#include <cuda.h>

#include <algorithm>

#include "gemm_group.cuh"
#include "gemm_launch.h"
#include "host.h"

namespace us {
namespace {

using host::make_tmap;

bool aligned16(const us_mat* m) {
  return reinterpret_cast<uintptr_t>(m->ptr) % 16 == 0 && (m->ld * dtype_size(m->dtype)) % 16 == 0;
}
bool valid_mat(const us_mat* m) {
  return m && m->ptr && m->rows >= 1 && m->cols >= 1 && m->ld >= m->cols && m->rows < (1ll << 31) && m->cols < (1ll << 31) &&
         m->dtype >= US_F32 && m->dtype <= US_E5M2;
}
bool is_fp8(int dt) { return dt == US_E4M3 || dt == US_E5M2; }

struct Shape { int64_t M, N, K; };

// Host checks of one call of the group; US_ERR_UNSUPPORTED for a valid call this launch form does not cover.
// any: 16-bit operands and outputs of any size are covered too.
us_status check_call(const us_linear_call* c, bool any, Shape* sh) {
  if (c->op < US_OP_FWD || c->op > US_OP_BWD_W) return US_ERR_INVALID_ARG;
  if (!valid_mat(&c->a) || !valid_mat(&c->b) || !valid_mat(&c->out)) return US_ERR_INVALID_ARG;
  int64_t M, N, K;
  bool ok;
  switch (c->op) {
    case US_OP_FWD:   M = c->a.rows; K = c->a.cols; N = c->b.cols; ok = c->b.rows == K; break;
    case US_OP_BWD_X: M = c->a.rows; K = c->a.cols; N = c->b.rows; ok = c->b.cols == K; break;
    default:          M = c->a.cols; K = c->a.rows; N = c->b.cols; ok = c->b.rows == K; break;
  }
  if (!ok || c->out.rows != M || c->out.cols != N) return US_ERR_INVALID_ARG;
  if (!aligned16(&c->a) || !aligned16(&c->b) || !aligned16(&c->out)) return US_ERR_ALIGNMENT;
  if (!(is_fp8(c->a.dtype) && is_fp8(c->b.dtype))) {
    const bool h16 = (c->a.dtype == US_BF16 || c->a.dtype == US_F16) && c->a.dtype == c->b.dtype;
    if (!h16 || !any) return US_ERR_UNSUPPORTED;
  }
  if (c->ep.act != US_ACT_NONE) return c->ep.act < US_ACT_NONE || c->ep.act > US_ACT_SIGMOID_GRAD ? US_ERR_INVALID_ARG : US_ERR_UNSUPPORTED;
  if (c->ep.skip.ptr) {
    const us_mat* s = &c->ep.skip;
    if (s->rows != M || s->cols != N || s->ld < N) return US_ERR_INVALID_ARG;
    if (s->dtype != US_F32 && s->dtype != US_BF16 && s->dtype != US_F16) return US_ERR_UNSUPPORTED;
    if (!aligned16(s)) return US_ERR_ALIGNMENT;
  }
  if (!any && (M <= 128 || N <= 128)) return US_ERR_UNSUPPORTED;
  if (M > 4095ll * 256 || N > 4095ll * 256) return US_ERR_UNSUPPORTED;
  sh->M = M; sh->N = N; sh->K = K;
  return US_OK;
}

// Deals the tiles of all problems to the units, longest contraction first, each tile to the unit with the least work
// so far (ties: lowest unit), in a fixed order: the same arguments always give the same work list, and a tile's result
// never depends on it anyway (one unit, one accumulator).  False if a unit would get more than max_rounds tiles.
bool deal(GroupParams& g, int es, int tile_m, int bn, int split, int units, int max_rounds) {
  int order[kGroupMaxProblems];
  for (int i = 0; i < g.count; ++i) order[i] = i;
  std::stable_sort(order, order + g.count, [&](int x, int y) { return g.prob[x].K > g.prob[y].K; });
  uint32_t heap[kGroupMaxUnits];                        // load << 8 | unit, a binary heap with the least on top
  int filled[kGroupMaxUnits] = {0};
  for (int u = 0; u < units; ++u) heap[u] = (uint32_t)u;
  const auto more = [](uint32_t x, uint32_t y) { return x > y; };
  int rounds = 0;
  const int kbk = 128 / es;
  for (int o = 0; o < g.count; ++o) {
    const GroupProblem& P = g.prob[order[o]];
    const int tiles_m = (P.M + tile_m - 1) / tile_m, tiles_n = (P.N + bn - 1) / bn * split;      // split: entries per tile, one per part of its columns
    const uint32_t cost = (uint32_t)((P.K + kbk - 1) / kbk) + 4;            // K blocks plus a change-over
    // column-major over the tiles of a problem (neighbours in the list share a B panel) while A stays in L2, bands of
    // eight tile rows beyond that, as for the single launches
    const int band = (int64_t)P.M * P.K * es <= (80ll << 20) ? tiles_m : 8;
    for (int m0 = 0; m0 < tiles_m; m0 += band)
      for (int tn = 0; tn < tiles_n; ++tn)
        for (int tm = m0; tm < m0 + band && tm < tiles_m; ++tm) {
          std::pop_heap(heap, heap + units, more);
          const uint32_t top = heap[units - 1], unit = top & 0xffu;
          const int slot = filled[unit] * units + (int)unit;
          if (filled[unit] >= max_rounds || slot >= kGroupMaxItems || (top >> 8) + cost >= (1u << 24)) return false;
          if (++filled[unit] > rounds) {                            // a new round: nobody has an entry yet
            std::fill(g.table + rounds * units, g.table + std::min((rounds + 1) * units, kGroupMaxItems), -1);
            ++rounds;
          }
          g.table[slot] = (order[o] << 28) | (tm << 14) | tn;
          heap[units - 1] = (((top >> 8) + cost) << 8) | unit;
          std::push_heap(heap, heap + units, more);
        }
  }
  if (rounds * units > kGroupMaxItems) return false;
  g.rounds = rounds; g.units = units;
  return true;
}

// 256 x 256 tiles per CTA pair unless they would leave a quarter of the pairs idle (measured over FFN steps, FP8 / BF16,
// us: 48 such tiles 14.3 / 19.2 against 10.7 / 17.1 with 128 x 128 tiles, 64 tiles 14.9 / 20.0 against 16.3 / 27.3).
bool pair_tiles_pay(int64_t pair_tiles, int sms) { return 8 * pair_tiles >= 3 * sms; }

// Estimated time, us, of the grouped launch of the calls in `which` (a bit each): the busiest unit's K blocks, an epilogue counted as eight.
// Measured / estimated, FP8, all four GEMMs of a step or the two that are not weight gradients: 2048 x 256 x 1024 7.0 / 6.8, 4.7 / 5.6; 4096 x 256 x
// 1024 10.0 / 9.4, 5.8 / 5.6; 1500 x 768 x 2304 12.9 / 11.2, 7.9 / 7.2; 8192 x 144 x 512 23.1 / 24.6, 7.2 / 6.6; 8192 x 256 x 768 23.0 / 24.6, 8.1 / 7.2;
// 16384 x 256 x 512 41.2 / 43.8, 11.1 / 9.2; low with much output, whose bytes it leaves
// out (8192 x 512 x 2048 29.2 / 24.8, 20.1 / 15.5), and for few tiles of very long contractions (16000 x 144 x 400 56.7 / 42.9, 30000 x 144 x 288 99 / 76).
double group_time(const Shape* sh, int count, unsigned which, int es, int sms) {
  int64_t pair_tiles = 0, blocks = 0, longest = 0;
  for (int i = 0; i < count; ++i)
    if (which >> i & 1) pair_tiles += ((sh[i].M + 255) / 256) * ((sh[i].N + 255) / 256);
  if (pair_tiles == 0) return 0.0;
  const bool pair = pair_tiles_pay(pair_tiles, sms);
  const int tile = pair ? 256 : 128, kbk = 128 / es;
  for (int i = 0; i < count; ++i) {
    if (!(which >> i & 1)) continue;
    const int64_t kb = (sh[i].K + kbk - 1) / kbk + 8;
    blocks += ((sh[i].M + tile - 1) / tile) * ((sh[i].N + tile - 1) / tile) * kb;
    longest = std::max(longest, kb);
  }
  const int units = pair ? sms / 2 : sms;
  return 3.0 + std::max((double)longest, (double)blocks / units) * (pair ? 0.3 : 0.16);
}

// The calls (a bit each) whose contractions several CTAs share in a launch of their own, in tiles t; 0: none.  A few tiles with a far
// longer contraction than the rest of the work per unit (the weight gradients of many tokens and a narrow block) leave the other
// units of the grouped launch idle; a second launch costs what its estimate says and has to save 2 us, about what the estimates are off, beyond
// it.  Captured FFN steps, one grouped launch -> two, us: FP8 8192 x 128 x 512 39.9 -> 31.6, 8192 x 256 x 768 44.6 -> 38.8, 16000 x 128 x 400 65.5 ->
// 44.3; BF16 4096 x 128 x 256 25.5 -> 18.5, 9000 x 256 x 768 74.6 -> 54.2; F16 16384 x 256 x 1024 141.9 -> 101.8.  Of 260 drawn groups that go out in two
// launches (2900 to 46000 tokens; of a whole step or of a backward pass alone) the geometric mean is 1.6 times as fast, the best 4.8; eleven are 2
// to 12 % slower (7520 x 336 x 656 25.9 -> 29.6, 5200 x 448 x 1360 in BF16 28.9 -> 31.4), all with two shares or pairs; a margin that spares them costs
// as many others up to 1.3 times.
unsigned shared_calls(const us_linear_call* calls, const Shape* sh, int count, int es, int sms, Tiling* t) {
  const int kbk = 128 / es;
  int64_t longest = 0;
  for (int i = 0; i < count; ++i) longest = std::max(longest, sh[i].K);
  if (longest < 48ll * kbk) return 0;
  const unsigned all = (1u << count) - 1;
  double best = group_time(sh, count, all, es, sms) - 2.0;
  unsigned pick = 0;
  for (int k = 0; k < count; ++k) {                       // every call of at least sh[k].K
    const int64_t K = sh[k].K;
    if (K < 48ll * kbk) continue;
    unsigned which = 0;
    bool sectors = true;
    int64_t most = 0;
    for (int i = 0; i < count; ++i) {
      if (sh[i].K < K) continue;
      which |= 1u << i;
      most = std::max(most, sh[i].K);
      sectors = sectors && calls[i].a.ld * es % 32 == 0 && calls[i].b.ld * es % 32 == 0;
    }
    if (most > (int64_t)kSplitMostBlocks * kbk) continue;
    const double rest = group_time(sh, count, all & ~which, es, sms);
    for (int form = 0; form < 3; ++form)
      for (int s = 2; s * (form == 2 ? 2 : 1) <= 8; s *= 2) {
        const Tiling c{form == 0 ? 64 : form == 1 ? 128 : 256, form == 2 ? 2 : 1, s};
        int64_t tiles = 0;
        int a_bytes = 0;
        bool fits = true;
        for (int i = 0; i < count; ++i)
          if (which >> i & 1) {
            fits = fits && split_form_fits(c, sh[i].M, sh[i].N);
            tiles += ((sh[i].M + 128 * c.cg - 1) / (128 * c.cg)) * ((sh[i].N + c.bn - 1) / c.bn);
            a_bytes = std::max(a_bytes, split_a_bytes(c.bn, calls[i].op == US_OP_BWD_W, sh[i].M));
          }
        if (!fits || tiles * c.cg * s > sms) continue;
        const double time = rest + tiling_time(c, tiles, (int)((most + kbk - 1) / kbk), a_bytes, sectors, sms);
        if (time < best && tiles <= split_capacity(es, c)) { best = time; pick = which; *t = c; }
      }
  }
  return pick;
}

template <int ES, int BN, int CG, int SPLIT, bool COPY>
us_status launch_variant(const GroupParams& g, cudaStream_t stream) {
  auto kern = gemm_group_kernel<ES, BN, CG, SPLIT, COPY>;
  constexpr int smem = GemmSmem<BN, CG, kGroupEW>::kTotal;
  static std::atomic<uint64_t> smem_set{0};
  return host::launch(kern, &smem_set, CG * g.units, gemm_threads(kGroupEW), smem, CG, stream, g);
}
template <int ES, int BN, int CG, int SPLIT>
us_status launch_group(const GroupParams& g, bool copy, cudaStream_t stream) {
  return copy ? launch_variant<ES, BN, CG, SPLIT, true>(g, stream) : launch_variant<ES, BN, CG, SPLIT, false>(g, stream);
}

// copies: NULL, or for each call the FP8 copy of its output (ptr NULL: none).
// test: NULL, or a short wait limit and which CTAs get no operands.  launches: NULL, or receives the number of kernels, and nothing is launched.
struct GroupTest { uint32_t wait_limit; int starved, served; };
us_status group_impl(int count, const us_linear_call* calls, const us_mat* copies, bool any, void* ws, size_t ws_bytes, void* stream,
                     const GroupTest* test = nullptr, int* launches = nullptr) {
  if (count < 1 || count > kGroupMaxProblems || !calls) return count >= 1 && calls ? US_ERR_UNSUPPORTED : US_ERR_INVALID_ARG;
  if (!launches && (!ws || ws_bytes < us_workspace_bytes())) return US_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(ws) % 16) return US_ERR_ALIGNMENT;
  static_assert(sizeof(GroupParams) < 32000, "kernel parameter limit");
  Shape sh[kGroupMaxProblems];
  for (int i = 0; i < count; ++i) {
    us_status s = check_call(&calls[i], any, &sh[i]);
    if (s != US_OK) return s;
    if (dtype_size(calls[i].a.dtype) != dtype_size(calls[0].a.dtype)) return US_ERR_UNSUPPORTED;   // one operand width per launch
    if (copies && copies[i].ptr) {
      s = check_copy(&copies[i], &calls[i].out, calls[i].ep.skip.ptr != nullptr);
      if (s != US_OK) return s;
    }
  }
  const int sms = host::sm_count();
  if (sms <= 0) return US_ERR_CUDA;
  const int es = dtype_size(calls[0].a.dtype);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const GroupTest tt = test ? *test : GroupTest{kWaitLimit, 0, 0};
  const int starved = tt.served ? 0 : tt.starved;         // of a launch in which a CTA has one tile
  Tiling t{};
  const unsigned shared = any ? shared_calls(calls, sh, count, es, sms, &t) : 0;
  SplitCall split_calls[kGroupMaxProblems];
  int splits = 0, left = 0, at[kGroupMaxProblems];
  int64_t pair_tiles = 0;
  bool copy = false;
  for (int i = 0; i < count; ++i) {
    const us_linear_call& c = calls[i];
    const us_mat* q = copies && copies[i].ptr ? &copies[i] : nullptr;
    if (shared >> i & 1) {
      const bool skip = c.ep.skip.ptr != nullptr;
      split_calls[splits++] = SplitCall{&c.a, &c.b, &c.out, skip ? &c.ep.skip : nullptr, q, c.op == US_OP_BWD_W, c.op != US_OP_BWD_X, c.scale,
                                        skip ? c.ep.skip_coef : 0.f, skip ? c.ep.out_coef : 1.f};
      continue;
    }
    at[left++] = i;
    copy = copy || q;
    pair_tiles += ((sh[i].M + 255) / 256) * ((sh[i].N + 255) / 256);
  }
  if (launches) *launches = (splits > 0) + (left > 0);
  if (left == 0) return launches ? US_OK : launch_split(splits, split_calls, t, static_cast<unsigned int*>(ws), tt.wait_limit, starved, st);
  const bool pair = pair_tiles_pay(pair_tiles, sms);
  const int tile_m = pair ? 256 : 128, bn = pair ? 256 : 128;
  int64_t tiles = 0;
  for (int j = 0; j < left; ++j) tiles += ((sh[at[j]].M + tile_m - 1) / tile_m) * ((sh[at[j]].N + bn - 1) / bn);
  const int most = std::min(pair ? sms / 2 : sms, kGroupMaxUnits);
  const int split = !pair && 2 * tiles <= most ? 2 : 1;
  const int units = (int)std::min<int64_t>(most, tiles * split);
  GroupParams g;
  g.count = left;
  for (int j = 0; j < left; ++j) {
    const int i = at[j];
    GroupProblem& P = g.prob[j];
    const us_linear_call& c = calls[i];
    P.M = (int)sh[i].M; P.N = (int)sh[i].N; P.K = (int)sh[i].K;
    P.a_mn = c.op == US_OP_BWD_W; P.b_mn = c.op != US_OP_BWD_X;
    const int one = es == 1 ? US_E5M2 : US_BF16;         // the format the descriptor numbers 1
    P.idesc = make_idesc(c.a.dtype == one, c.b.dtype == one, P.a_mn != 0, P.b_mn != 0, tile_m, bn);
    P.scale = c.scale;
    P.out_dt = c.out.dtype;
    P.has_skip = c.ep.skip.ptr != nullptr;
    P.skip_dt = P.has_skip ? c.ep.skip.dtype : US_F32;
    P.skip_coef = P.has_skip ? c.ep.skip_coef : 0.f;
    P.out_coef = P.has_skip ? c.ep.out_coef : 1.f;
    P.copy = copies ? static_cast<uint8_t*>(copies[i].ptr) : nullptr;
    P.copy_ld = P.copy ? copies[i].ld : 0;
    P.copy_dt = P.copy ? copies[i].dtype : US_E4M3;
    P.copy_sectors = reinterpret_cast<uintptr_t>(P.copy) % 32 == 0 && P.copy_ld % 32 == 0;
    if (launches) continue;
    if (!make_tmap(&P.ta, &c.a, es, P.a_mn ? 128 / es : 128) || !make_tmap(&P.tb, &c.b, es, P.b_mn ? 128 / es : 128)) return US_ERR_CUDA;
    const int oes = dtype_size(c.out.dtype);
    if (!make_tmap(&P.tout, &c.out, oes, 32, std::min(128, bn / 2 / split * oes))) return US_ERR_CUDA;
    P.tskip = P.tout;
    if (P.has_skip && !make_tmap(&P.tskip, &c.ep.skip, dtype_size(c.ep.skip.dtype), 32)) return US_ERR_CUDA;
  }
  if (!deal(g, es, tile_m, bn, split, units, any ? kGroupMaxItems : 12)) return US_ERR_UNSUPPORTED;      // too many tiles per unit for the work list
  if (launches) return US_OK;
  g.status = static_cast<unsigned int*>(ws);
  g.wait_limit = tt.wait_limit; g.starved = tt.starved; g.served = tt.served;
  if (splits) {                                            // (a grouped launch that is refused has launched nothing)
    const us_status s = launch_split(splits, split_calls, t, static_cast<unsigned int*>(ws), tt.wait_limit, starved, st);
    if (s != US_OK) return s;
  }
  if (es == 1) return pair ? launch_group<1, 256, 2, 1>(g, copy, st) : split == 2 ? launch_group<1, 128, 1, 2>(g, copy, st) : launch_group<1, 128, 1, 1>(g, copy, st);
  return pair ? launch_group<2, 256, 2, 1>(g, copy, st) : split == 2 ? launch_group<2, 128, 1, 2>(g, copy, st) : launch_group<2, 128, 1, 1>(g, copy, st);
}

}  // namespace
}  // namespace us

extern "C" us_status us_linear_group(int count, const us_linear_call* calls, void* ws, size_t ws_bytes, void* stream) {
  return us::group_impl(count, calls, nullptr, false, ws, ws_bytes, stream);
}
extern "C" us_status us_linear_group_any(int count, const us_linear_call* calls, void* ws, size_t ws_bytes, void* stream) {
  return us::group_impl(count, calls, nullptr, true, ws, ws_bytes, stream);
}
extern "C" us_status us_linear_group_cast(int count, const us_linear_call* calls, const us_mat* copies, void* ws, size_t ws_bytes, void* stream) {
  return copies ? us::group_impl(count, calls, copies, true, ws, ws_bytes, stream) : US_ERR_INVALID_ARG;
}
extern "C" us_status us_linear_group_launches(int count, const us_linear_call* calls, int* launches) {
  if (!launches) return US_ERR_INVALID_ARG;
  return us::group_impl(count, calls, nullptr, true, nullptr, 0, nullptr, nullptr, launches);
}
extern "C" us_status us_test_linear_group_starved(int count, const us_linear_call* calls, void* ws, size_t ws_bytes, unsigned int wait_limit, int cta, int tiles,
                                                  void* stream) {
  if (wait_limit < 1 || wait_limit > (1u << 16) || cta < -1 || cta > 7 || tiles < 0 || tiles > 1024) return US_ERR_INVALID_ARG;
  const us::GroupTest test = {wait_limit, cta + 2, tiles};
  return us::group_impl(count, calls, nullptr, true, ws, ws_bytes, stream, &test);
}
