// Interface between the argument-checking front end (gemm.cu) and the kernel instantiations
// (gemm_inst.cu, compiled once per operand width and layout).
#pragma once
#include <cuda_runtime.h>

#include "../../include/unitscale.h"

namespace us {

struct GemmParams;

// The matrices the epilogue reaches through TMA (aux / skip NULL when unused).
struct EpiMats {
  const us_mat* out;
  const us_mat* aux;
  const us_mat* skip;
  const us_mat* copy;
};

// Whether q can take the FP8 copy of a residual epilogue's output.
us_status check_copy(const us_mat* q, const us_mat* out, bool residual);

// Batch description of one launch: nb0 x nb1 problems; element strides of each matrix between
// consecutive problems of the outer (index 0) and inner (index 1) batch dimension.
struct BatchDesc {
  int64_t nb0 = 1, nb1 = 1;
  int64_t a[2] = {0, 0}, b[2] = {0, 0}, out[2] = {0, 0};
  bool batched() const { return nb0 * nb1 > 1; }
};

// How an output is tiled: columns of a tile, CTAs that cooperate on it as a pair (1: none), CTAs (pairs) that share its contraction.
struct Tiling { int bn, cg, splits; };

// One GEMM of a launch with shared contractions (gemm_split.cu); skip and copy may be NULL.
struct SplitCall {
  const us_mat *a, *b, *out, *skip, *copy;
  bool a_mn, b_mn;
  float scale, skip_coef, out_coef;
};
// Tiles of the calls' outputs all t; t.splits is 2, 4 or 8 and t.splits * t.cg at most 8.
us_status launch_split(int count, const SplitCall* calls, const Tiling& t, unsigned int* status, uint32_t wait_limit, int starved, cudaStream_t stream);
int split_a_bytes(int bn, bool a_mn, int64_t rows);
// Contractions that may be shared have at most this many K blocks (128 bytes of an operand's K): what was measured.
constexpr int kSplitMostBlocks = 8192;
// Whether an M x N output can be tiled that way: pairs only where both halves of a tile have rows and columns.
inline bool split_form_fits(const Tiling& t, int64_t M, int64_t N) { return t.cg == 1 || (M > 128 && N > 128); }
// Estimated time, us, of a launch of `tiles` tiles of kb K blocks.  sectors: the operands' rows start on 32-byte boundaries.
double tiling_time(const Tiling& t, long long tiles, int kb, int a_bytes, bool sectors, int sms);
// Clusters of such a launch that run at once.
int split_capacity(int es, const Tiling& t);

// Builds the tensor maps, picks the tile configuration and launches the kernel for
// ES-byte operands (1 = FP8, 2 = BF16 / F16) with the given operand layouts and epilogue kind.  only: NULL, or takes the configuration, and
// nothing is launched.
template <int ES, bool A_MN, bool B_MN>
us_status launch_gemm(const us_mat* A, const us_mat* B, GemmParams& p, const EpiMats& em, int epi, const BatchDesc& bd,
                      cudaStream_t stream, Tiling* only);

}  // namespace us
