// Host-only entry points of libunitscale: scale-factor helpers, status strings, device queries.
#include <math.h>

#include "host.h"

namespace us {
namespace host {
int sm_count() {
  static int cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  if (cached[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return -1;
    cached[dev] = n;
  }
  return cached[dev];
}

int resident_clusters(const void* kern, int threads, size_t smem, int cluster, ClusterCount& count) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || cluster < 1 || cluster > 8) return -1;
  if (cluster == 1) return sm_count();
  int n = count.cached[dev][cluster].load(std::memory_order_relaxed);
  if (n > 0) return n;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) { (void)failed(); return -1; }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(cluster * (sm_count() / cluster)));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) { (void)failed(); return -1; }
  count.cached[dev][cluster].store(n, std::memory_order_relaxed);
  return n;
}

EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = nullptr;     // idempotent: concurrent first calls store the same pointer
  if (!fn) {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(sym);
  }
  return fn;
}

bool make_tmap(CUtensorMap* tm, const us_mat* m, int es, int box_rows, int box_bytes) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const CUtensorMapDataType type = es == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                                 : es == 2 ? CU_TENSOR_MAP_DATA_TYPE_UINT16 : CU_TENSOR_MAP_DATA_TYPE_UINT32;
  cuuint64_t dims[2] = {(cuuint64_t)m->cols, (cuuint64_t)m->rows};
  cuuint64_t strides[1] = {(cuuint64_t)m->ld * es};
  cuuint32_t box[2] = {(cuuint32_t)(box_bytes / es), (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(tm, type, 2, m->ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            box_bytes == 32 ? CU_TENSOR_MAP_SWIZZLE_NONE : box_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
}  // namespace host
}  // namespace us

// 1 / std(gelu(z)) and 1 / rms(gelu'(z)) for z ~ N(0,1), gelu(x) = x Phi(x): the values the
// table of unit scaling factors prints as 1.701 and 1.481, here to double precision.
static const double kGeluAlpha = 1.7009262433633;
static const double kGeluBeta = 1.4811144127083;

extern "C" us_status us_scales_linear(int64_t b, int64_t m, int64_t n, int constrained, float* alpha,
                                      float* beta_x, float* beta_w) {
  if (b < 1 || m < 1 || n < 1 || !alpha || !beta_x || !beta_w) return US_ERR_INVALID_ARG;
  double a = 1.0 / sqrt((double)m), bx = 1.0 / sqrt((double)n), bw = 1.0 / sqrt((double)b);
  if (constrained) a = bx = sqrt(a * bx);  // geometric mean of the constrained pair
  *alpha = (float)a;
  *beta_x = (float)bx;
  *beta_w = (float)bw;
  return US_OK;
}

extern "C" us_status us_scales_gelu(int constrained, float* alpha, float* beta) {
  if (!alpha || !beta) return US_ERR_INVALID_ARG;
  double a = kGeluAlpha, b = kGeluBeta;
  if (constrained) a = b = sqrt(a * b);
  *alpha = (float)a;
  *beta = (float)b;
  return US_OK;
}

extern "C" us_status us_scales_activation(us_fn fn, int constrained, float* alpha, float* beta) {
  if (!alpha || !beta) return US_ERR_INVALID_ARG;
  // 1 / std f(Z) and 1 / rms f'(Z) for Z ~ N(0, 1): relu in closed form (sqrt(2 / (1 - 1/pi)), sqrt 2),
  // the others by numerical integration to the digits kept here (the table prints three of them).
  double a, b;
  switch (fn) {
    case US_FN_GELU: a = kGeluAlpha; b = kGeluBeta; break;
    case US_FN_RELU: a = 1.7128585504496627; b = 1.4142135623730951; break;
    case US_FN_TANH: a = 1.5925374197228314; b = 1.4674135916307951; break;
    case US_FN_SIGMOID: a = 4.8013133720399622; b = 4.7226460859379743; break;
    default: return US_ERR_INVALID_ARG;
  }
  if (constrained) a = b = sqrt(a * b);
  *alpha = (float)a;
  *beta = (float)b;
  return US_OK;
}

extern "C" us_status us_scales_residual(float tau, float* skip_coef, float* branch_coef) {
  if (!skip_coef || !branch_coef || !(tau >= 0.f && tau <= 1.f)) return US_ERR_INVALID_ARG;
  *skip_coef = (float)sqrt(1.0 - (double)tau);
  *branch_coef = (float)sqrt((double)tau);
  return US_OK;
}

extern "C" us_status us_scales_attention(int64_t s, int64_t d_head, int constrained, float* alpha_scores, float* beta_scores,
                                         float* softmax_scale, float* alpha_context, float* beta_p, float* beta_v) {
  if (s < 1 || d_head < 1 || !alpha_scores || !beta_scores || !softmax_scale || !alpha_context || !beta_p || !beta_v)
    return US_ERR_INVALID_ARG;
  // scores Q K^T: 1 / sqrt(d_head) in both passes; context P V is an ordinary matmul with fan_in = batch = s, fan_out = d_head
  const double a_s = 1.0 / sqrt((double)d_head);
  double a_c = 1.0 / sqrt((double)s), b_p = 1.0 / sqrt((double)d_head);
  if (constrained) a_c = b_p = sqrt(a_c * b_p);
  *alpha_scores = (float)a_s;
  *beta_scores = (float)a_s;
  *softmax_scale = (float)s;
  *alpha_context = (float)a_c;
  *beta_p = (float)b_p;
  *beta_v = (float)(1.0 / sqrt((double)s));
  return US_OK;
}

extern "C" const char* us_status_string(us_status s) {
  switch (s) {
    case US_OK: return "ok";
    case US_ERR_INVALID_ARG: return "invalid argument";
    case US_ERR_UNSUPPORTED: return "unsupported dtype combination";
    case US_ERR_ALIGNMENT: return "pointer or row pitch not 16-byte aligned";
    case US_ERR_WORKSPACE: return "workspace missing or too small";
    case US_ERR_CUDA: return "CUDA call failed";
    case US_ERR_TIMEOUT: return "device-side wait timed out";
  }
  return "unknown status";
}

extern "C" int us_version(void) { return 100; }
