// Host-side helpers shared by the translation units of libunitscale.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <type_traits>

#include "../../include/unitscale.h"

namespace us {
namespace host {
// The status of a failed runtime call.  The runtime also remembers the error; it is taken back here, or the next launch whose
// status is read with cudaGetLastError would report it as its own.
inline us_status failed() {
  (void)cudaGetLastError();
  return US_ERR_CUDA;
}

// Launches a kernel that calls ptx::grid_wait_previous (programmatic dependent launch): its CTAs may take their
// places and set up barriers and tensor memory while the previous kernel of the stream still drains, and wait there
// for that kernel's completion before they touch memory.  In such a kernel at least one thread of every CTA waits, so that
// a grid never completes ahead of its predecessors, and so does every thread that touches global memory or makes bounded
// waits (whose limit is then not spent on the predecessor).  Worth its while where the grid is resident at once (the three launches of a
// 256 x 128 x 512 step 18.4 -> 16.4 us, of a 8192 x 1024 x 4096 one 199 -> 193 us); a grid of many waves pays for the wait
// in every CTA (cross-entropy rows, 2048 CTAs: 39 -> 44 us) and is launched plainly.  cluster: CTAs per cluster (1: none).
// smem_set: one static word per kernel, a bit per device on which its dynamic shared memory limit is set (nullptr: within 48 KB).
template <class... P, class... A>
us_status launch(void (*kern)(P...), std::atomic<uint64_t>* smem_set, int grid, int threads, size_t smem, int cluster,
                 cudaStream_t stream, const A&... args) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return failed();
  const uint64_t bit = 1ull << (dev & 63);
  const bool known = !smem_set || (smem_set->load(std::memory_order_relaxed) & bit);
  if (!known) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return failed();
    smem_set->fetch_or(bit, std::memory_order_relaxed);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  static_assert((std::is_same_v<P, A> && ...), "parameters are handed over as they are, without a copy");
  void* params[] = {const_cast<void*>(static_cast<const void*>(&args))...};
  return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(kern), params) == cudaSuccess ? US_OK : failed();
}

// Number of SMs of the current device (cached per device), or -1 on error.
int sm_count();
// Clusters of `cluster` CTAs (1 .. 8) of a kernel of one CTA per SM that run at once on the current device: a cluster stays within
// one group of SMs, whose number need not be a multiple of the cluster's.  Cached per device and size in `count`, a static of the
// kernel's own (another kernel's threads and shared memory fit another number); -1 on error.
struct ClusterCount { std::atomic<int> cached[64][9]; };
int resident_clusters(const void* kern, int threads, size_t smem, int cluster, ClusterCount& count);
// cuTensorMapEncodeTiled, looked up through the runtime (the library does not link against libcuda); nullptr if unavailable.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn();
// Tensor map of a row-major matrix of es-byte elements in boxes of box_rows rows x box_bytes, swizzled with the pattern of that width (32
// bytes: none); out-of-range parts of a box read as zero and are not written.
bool make_tmap(CUtensorMap* tm, const us_mat* m, int es, int box_rows, int box_bytes = 128);
// A launch without that overlap, of a kernel that may take up to max_smem bytes of dynamic shared memory.
template <class... P, class... A>
us_status launch_plain(void (*kern)(P...), std::atomic<uint64_t>* smem_set, int grid, int threads, int max_smem, size_t smem,
                       cudaStream_t stream, const A&... args) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return failed();
  const uint64_t bit = 1ull << (dev & 63);
  if (!(smem_set->load(std::memory_order_relaxed) & bit)) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem) != cudaSuccess) return failed();
    smem_set->fetch_or(bit, std::memory_order_relaxed);
  }
  kern<<<(unsigned)grid, (unsigned)threads, smem, stream>>>(P(args)...);
  return cudaGetLastError() == cudaSuccess ? US_OK : US_ERR_CUDA;
}
}  // namespace host
}  // namespace us
