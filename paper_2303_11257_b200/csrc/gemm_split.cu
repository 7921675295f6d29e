// Launches of gemm_split_kernel (gemm_split.cuh): tensor maps, work split over blocks, cluster launch.
#include <cuda.h>

#include <algorithm>

#include "gemm_launch.h"
#include "gemm_split.cuh"
#include "host.h"

namespace us {
namespace {

using host::make_tmap;

template <int ES, int BN, int CG, int PROBLEMS>
us_status launch(const SplitParams<PROBLEMS>& p, int tiles, cudaStream_t stream) {
  static std::atomic<uint64_t> smem_set{0};
  return host::launch(gemm_split_kernel<ES, BN, CG, (PROBLEMS > 1)>, &smem_set, CG * p.splits * tiles, gemm_threads(8), GemmSmem<BN, CG, 8>::kTotal,
                      CG * p.splits, stream, p);
}
template <int ES, int BN, int CG>
int capacity(int splits) {
  static host::ClusterCount count;
  return host::resident_clusters(reinterpret_cast<const void*>(gemm_split_kernel<ES, BN, CG, false>), gemm_threads(8), GemmSmem<BN, CG, 8>::kTotal, CG * splits, count);
}
template <int PROBLEMS>
us_status launch_problems(int count, const SplitCall* calls, const Tiling& t, unsigned int* status, uint32_t wait_limit, int starved, cudaStream_t stream) {
  SplitParams<PROBLEMS> p;
  p.splits = t.splits; p.status = status; p.wait_limit = wait_limit; p.starved = starved;
  const int es = dtype_size(calls[0].a->dtype), one = es == 1 ? US_E5M2 : US_BF16;      // the format the descriptor numbers 1
  int tiles = 0;
  for (int i = 0; i < count; ++i) {
    const SplitCall& c = calls[i];
    SplitProblem& s = p.prob[i];
    GroupProblem& P = s.g;
    P.M = (int)c.out->rows; P.N = (int)c.out->cols; P.K = (int)(c.a_mn ? c.a->rows : c.a->cols);
    P.a_mn = c.a_mn; P.b_mn = c.b_mn;
    P.idesc = make_idesc(c.a->dtype == one, c.b->dtype == one, c.a_mn, c.b_mn, kBM * t.cg, t.bn);
    P.scale = c.scale;
    P.out_dt = c.out->dtype;
    P.has_skip = c.skip != nullptr;
    P.skip_dt = c.skip ? c.skip->dtype : US_F32;
    P.skip_coef = c.skip_coef; P.out_coef = c.out_coef;
    P.copy = c.copy ? static_cast<uint8_t*>(c.copy->ptr) : nullptr;
    P.copy_ld = c.copy ? c.copy->ld : 0;
    P.copy_dt = c.copy ? c.copy->dtype : US_E4M3;
    P.copy_sectors = reinterpret_cast<uintptr_t>(P.copy) % 32 == 0 && P.copy_ld % 32 == 0;
    s.a_bytes = (uint32_t)us::split_a_bytes(t.bn, c.a_mn, c.out->rows);
    using Narrow = GemmSmem<64, 1, 8>;
    s.stages = t.bn == 64    ? std::min((int)Narrow::kMaxStages, Narrow::kStages * Narrow::kStageBytes / ((int)s.a_bytes + Narrow::kBBytes))
               : t.bn == 128 ? GemmSmem<128, 1, 8>::kStages : GemmSmem<256, 2, 8>::kStages;
    s.tiles_m = (P.M + kBM * t.cg - 1) / (kBM * t.cg);
    tiles += s.tiles_m * ((P.N + t.bn - 1) / t.bn);
    s.tile_end = tiles;
    const int box_a = c.a_mn ? 128 / es : (int)s.a_bytes / kStageKBytes, rows_b = t.bn / t.cg;
    const int out_es = dtype_size(c.out->dtype);
    if (!make_tmap(&P.ta, c.a, es, box_a) || !make_tmap(&P.tb, c.b, es, c.b_mn ? 128 / es : rows_b, c.b_mn && rows_b * es < 128 ? 64 : 128)) return US_ERR_CUDA;
    if (!make_tmap(&P.tout, c.out, out_es, 32, 32 * out_es)) return US_ERR_CUDA;
    P.tskip = P.tout;
    if (c.skip && !make_tmap(&P.tskip, c.skip, dtype_size(c.skip->dtype), 32)) return US_ERR_CUDA;
  }
  for (int i = count; i < PROBLEMS; ++i) p.prob[i].tile_end = tiles;
  if (es == 1) return t.bn == 64 ? launch<1, 64, 1>(p, tiles, stream) : t.bn == 128 ? launch<1, 128, 1>(p, tiles, stream) : launch<1, 256, 2>(p, tiles, stream);
  return t.bn == 64 ? launch<2, 64, 1>(p, tiles, stream) : t.bn == 128 ? launch<2, 128, 1>(p, tiles, stream) : launch<2, 256, 2>(p, tiles, stream);
}

}  // namespace

// Bytes of A in a stage of a narrow tile: an MN-major A is fetched whole, of a K-major one only the rows that exist.
int split_a_bytes(int bn, bool a_mn, int64_t rows) { return (bn != 64 || a_mn || rows >= kBM ? kBM : (int)((rows + 7) / 8 * 8)) * kStageKBytes; }

// A base and a time per K block, which is bound by the tensor core (128 x 128 and narrower tiles 0.152 us, pairs 0.28), by what the L2 cache
// hands to all CTAs together (15 bytes per ps), or, with rows that start inside a sector, by TMA (86 bytes per ns).  The bases hold
// the exchange: partial sums cross between SMs at some 25 bytes per ns.
double tiling_time(const Tiling& t, long long tiles, int kb, int a_bytes, bool sectors, int sms) {
  const double bytes = a_bytes + t.bn / t.cg * kStageKBytes;
  const long long all = tiles * t.cg * t.splits, ctas = std::min<long long>(all, sms), waves = (all + sms - 1) / sms;
  const double block = std::max(t.cg == 2 ? 0.28 : 0.152, std::max(ctas * bytes / 15e6, sectors ? 0.0 : bytes / 86e3));
  const int s = t.splits;
  const double base = s == 1 ? 2.4 : t.cg == 2 ? (s == 2 ? 7.0 : 8.2) : t.bn == 128 ? (s == 2 ? 4.8 : s == 4 ? 5.4 : 6.6) : s == 2 ? 3.4 : s == 4 ? 4.0 : 4.4;
  return base + (ctas > 100 ? 0.8 : 0.0) + waves * ((kb + s - 1) / s) * block;
}

int split_capacity(int es, const Tiling& t) {
  if (es == 1) return t.bn == 64 ? capacity<1, 64, 1>(t.splits) : t.bn == 128 ? capacity<1, 128, 1>(t.splits) : capacity<1, 256, 2>(t.splits);
  return t.bn == 64 ? capacity<2, 64, 1>(t.splits) : t.bn == 128 ? capacity<2, 128, 1>(t.splits) : capacity<2, 256, 2>(t.splits);
}

us_status launch_split(int count, const SplitCall* calls, const Tiling& t, unsigned int* status, uint32_t wait_limit, int starved, cudaStream_t stream) {
  return count == 1 ? launch_problems<1>(count, calls, t, status, wait_limit, starved, stream)
                    : launch_problems<kGroupMaxProblems>(count, calls, t, status, wait_limit, starved, stream);
}

}  // namespace us
