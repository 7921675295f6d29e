// Scaled softmax over the rows of a matrix, forward and backward (table "Table of unit scaling
// factors", row softmax: alpha = beta = s for rows of s elements; appendix paragraph "Softmax
// (followed by matmul)").  One warp per row, 128-bit loads and stores, warp-shuffle reductions;
// rows of up to 2048 elements are held in registers between the reduction and the write.
#include "common.cuh"
#include "host.h"
#include "rowwise.cuh"
#include "sm100.cuh"

namespace us {

constexpr int kSmThreads = 256;            // 8 rows per CTA
constexpr float kLog2e = 1.4426950408889634f;

struct SmArgs {
  const void* in0; int in0_dt; int64_t in0_ld;      // S (forward) or P (backward)
  const void* in1; int in1_dt; int64_t in1_ld;      // dP (backward only)
  void* out; int out_dt; int64_t out_ld;
  int64_t rows; int cols;
  int vec_ok;                                       // all row starts 16-byte aligned and cols % 8 == 0
  float alpha, beta;
};

// NCH > 0: the row fits in NCH chunks of 8 elements per lane, kept in registers.
// NCH == 0: any length; the row is re-read from global memory (cache) in each pass.
template <int NCH>
__global__ void __launch_bounds__(kSmThreads) softmax_fwd_kernel(const SmArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t row = (int64_t)blockIdx.x * (kSmThreads / 32) + (threadIdx.x >> 5);
  if (row >= a.rows) return;
  const int64_t in_off = row * a.in0_ld, out_off = row * a.out_ld;
  const bool vec = a.vec_ok != 0;
  const int nch = NCH > 0 ? NCH : (a.cols + 255) / 256;
  float x[NCH > 0 ? NCH : 1][8];
  float m = -INFINITY;
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    float t[8];
    if (col < a.cols) {
      load8(a.in0, a.in0_dt, in_off, col, a.cols, vec, -INFINITY, t);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) t[i] = -INFINITY;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) { m = fmaxf(m, t[i]); if (NCH > 0) x[c][i] = t[i]; }
  }
  m = warp_max(m);
  const float mb = m * kLog2e;
  float sum = 0.f;
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    float t[8];
    if (NCH > 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) t[i] = x[c][i];
    } else if (col < a.cols) {
      load8(a.in0, a.in0_dt, in_off, col, a.cols, vec, -INFINITY, t);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) t[i] = -INFINITY;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float e = ex2_approx(fmaf(t[i], kLog2e, -mb));    // exp(x - max); exp(-inf) = 0 for the padding
      sum += e;
      if (NCH > 0) x[c][i] = e;
    }
  }
  sum = warp_sum(sum);
  const float inv = a.alpha / sum;
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    if (col >= a.cols) continue;
    float t[8];
    if (NCH > 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) t[i] = x[c][i] * inv;
    } else {
      load8(a.in0, a.in0_dt, in_off, col, a.cols, vec, -INFINITY, t);
#pragma unroll
      for (int i = 0; i < 8; ++i) t[i] = ex2_approx(fmaf(t[i], kLog2e, -mb)) * inv;
    }
    store8(a.out, a.out_dt, out_off, col, a.cols, vec, t);
  }
}

template <int NCH>
__global__ void __launch_bounds__(kSmThreads) softmax_bwd_kernel(const SmArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t row = (int64_t)blockIdx.x * (kSmThreads / 32) + (threadIdx.x >> 5);
  if (row >= a.rows) return;
  const int64_t p_off = row * a.in0_ld, g_off = row * a.in1_ld, out_off = row * a.out_ld;
  const bool vec = a.vec_ok != 0;
  const int nch = NCH > 0 ? NCH : (a.cols + 255) / 256;
  const float inv_alpha = 1.0f / a.alpha;
  float pt[NCH > 0 ? NCH : 1][8], g[NCH > 0 ? NCH : 1][8];
  float dot = 0.f;
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    float tp[8], tg[8];
    if (col < a.cols) {
      load8(a.in0, a.in0_dt, p_off, col, a.cols, vec, 0.f, tp);
      load8(a.in1, a.in1_dt, g_off, col, a.cols, vec, 0.f, tg);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) { tp[i] = 0.f; tg[i] = 0.f; }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      tp[i] *= inv_alpha;                                   // softmax(S) recovered from the scaled output
      dot = fmaf(tp[i], tg[i], dot);
      if (NCH > 0) { pt[c][i] = tp[i]; g[c][i] = tg[i]; }
    }
  }
  dot = warp_sum(dot);
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    if (col >= a.cols) continue;
    float tp[8], tg[8], t[8];
    if (NCH > 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) { tp[i] = pt[c][i]; tg[i] = g[c][i]; }
    } else {
      load8(a.in0, a.in0_dt, p_off, col, a.cols, vec, 0.f, tp);
      load8(a.in1, a.in1_dt, g_off, col, a.cols, vec, 0.f, tg);
#pragma unroll
      for (int i = 0; i < 8; ++i) tp[i] *= inv_alpha;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) t[i] = a.beta * tp[i] * (tg[i] - dot);
    store8(a.out, a.out_dt, out_off, col, a.cols, vec, t);
  }
}

// ---------------------------------------------------------------- 16-bit inputs, rows of at most 1024 elements
// Persistent warps: each walks rows grid-stride and fetches its next row, still packed, before working on
// the current one, so that a warp always has a row in flight.  Padding chunks (beyond the row) read as zero
// and are masked out of the maximum and the sums.
template <int NCH>
__global__ void __launch_bounds__(kSmThreads, 2) softmax_fwd16_kernel(const SmArgs a) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int64_t stride = (int64_t)gridDim.x * nw;
  int64_t row = (int64_t)blockIdx.x * nw + (threadIdx.x >> 5) + ptx::grid_wait_previous();
  uint4 cur[NCH], nxt[NCH];
  if (row < a.rows) load_row16<NCH>(a.in0, row * a.in0_ld, lane, a.cols, cur);
  for (; row < a.rows; row += stride) {
    if (row + stride < a.rows) load_row16<NCH>(a.in0, (row + stride) * a.in0_ld, lane, a.cols, nxt);
    float x[NCH][8];
    float m = -INFINITY;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      unpack16x8(cur[c], a.in0_dt, x[c]);
      if ((c * 32 + lane) * 8 < a.cols) {
#pragma unroll
        for (int i = 0; i < 8; ++i) m = fmaxf(m, x[c][i]);
      }
    }
    m = warp_max(m);
    const float mb = m * kLog2e;
    float sum = 0.f;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      if ((c * 32 + lane) * 8 < a.cols) {
#pragma unroll
        for (int i = 0; i < 8; ++i) { x[c][i] = ex2_approx(fmaf(x[c][i], kLog2e, -mb)); sum += x[c][i]; }
      }
    }
    sum = warp_sum(sum);
    const float inv = a.alpha / sum;
    const int64_t out_off = row * a.out_ld;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const int col = (c * 32 + lane) * 8;
      if (col < a.cols) {
        float t[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = x[c][i] * inv;
        store8(a.out, a.out_dt, out_off, col, a.cols, true, t);
      }
    }
#pragma unroll
    for (int c = 0; c < NCH; ++c) cur[c] = nxt[c];
  }
}

// dP 16-bit; P 16-bit of the same format, or (P8) FP8 codes as stored for an FP8 matmul.
template <int NCH, bool P8>
__global__ void __launch_bounds__(kSmThreads, 2) softmax_bwd16_kernel(const SmArgs a) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int64_t stride = (int64_t)gridDim.x * nw;
  const float inv_alpha = 1.0f / a.alpha;
  int64_t row = (int64_t)blockIdx.x * nw + (threadIdx.x >> 5) + ptx::grid_wait_previous();
  uint4 cp[P8 ? 1 : NCH], cg[NCH], np_[P8 ? 1 : NCH], ng[NCH];
  uint2 cp8[P8 ? NCH : 1], np8[P8 ? NCH : 1];
  if (row < a.rows) {
    if (P8) load_row8<P8 ? NCH : 1>(a.in0, row * a.in0_ld, lane, a.cols, cp8);
    else load_row16<P8 ? 1 : NCH>(a.in0, row * a.in0_ld, lane, a.cols, cp);
    load_row16<NCH>(a.in1, row * a.in1_ld, lane, a.cols, cg);
  }
  for (; row < a.rows; row += stride) {
    if (row + stride < a.rows) {
      if (P8) load_row8<P8 ? NCH : 1>(a.in0, (row + stride) * a.in0_ld, lane, a.cols, np8);
      else load_row16<P8 ? 1 : NCH>(a.in0, (row + stride) * a.in0_ld, lane, a.cols, np_);
      load_row16<NCH>(a.in1, (row + stride) * a.in1_ld, lane, a.cols, ng);
    }
    float pt[NCH][8], g[NCH][8];
    float dot = 0.f;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      if (P8) unpack8x8(cp8[P8 ? c : 0], a.in0_dt, pt[c]);
      else unpack16x8(cp[P8 ? 0 : c], a.in0_dt, pt[c]);
      unpack16x8(cg[c], a.in1_dt, g[c]);
#pragma unroll
      for (int i = 0; i < 8; ++i) { pt[c][i] *= inv_alpha; dot = fmaf(pt[c][i], g[c][i], dot); }   // padding: 0 * 0
    }
    dot = warp_sum(dot);
    const int64_t out_off = row * a.out_ld;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const int col = (c * 32 + lane) * 8;
      if (col < a.cols) {
        float t[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = a.beta * pt[c][i] * (g[c][i] - dot);
        store8(a.out, a.out_dt, out_off, col, a.cols, true, t);
      }
    }
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      if (P8) cp8[P8 ? c : 0] = np8[P8 ? c : 0];
      else cp[P8 ? 0 : c] = np_[P8 ? 0 : c];
      cg[c] = ng[c];
    }
  }
}

// ---------------------------------------------------------------- softmax cross-entropy
// softmax_xent(x, t) = log softmax(x)_t (table row "softmax_xent": alpha = 1, beta = s / sqrt(s - 1)).
// Three kernels, chosen by the class count and the number of rows (xent_launch_dt): one CTA per row for vocabulary-sized
// rows, held in registers or staged in shared memory, one warp per row for short ones.
struct XentArgs {
  const void* x; int x_dt; int64_t x_ld;
  const int32_t* t;
  const float* g;          // backward: one gradient per row, or null for ones
  void* out; int out_dt; int64_t out_ld;   // forward: float32 [rows]; backward: dX
  int64_t rows; int cols;
  int vec_ok;              // every row start of every tensor is 16-byte aligned
  float beta;
};

// One CTA per row; bound: HBM.  The row is read once, as NCH chunks of eight elements per thread that stay packed
// in registers through the maximum, the sum of exponentials and (backward) the write of beta * g * (onehot(t) -
// softmax(x)); all loads of a row are in flight together and the CTAs of an SM overlap one another's reductions.
// A row end inside a chunk costs one thread scalar accesses, not the row its vector path.  2048 rows of 30522 BF16
// logits, E5M2 gradient: forward 39 us = 3.2 TB/s, backward 66 us = 2.8 TB/s (a warp per row, re-reading it and
// scalar because 30522 is no multiple of 8: 265 and 491 us).  NCH == 0: rows beyond the register range, re-read from cache.
// DT: storage format of the row (US_F32, US_BF16 or US_F16).
template <int DT>
struct XentChunk { uint4 v[DT == US_F32 ? 2 : 1]; };
template <int DT>
__device__ __forceinline__ void xent_load(const XentArgs& a, int64_t off, int col, XentChunk<DT>& c) {
  if (a.vec_ok && col + 8 <= a.cols) {
    const uint4* q = reinterpret_cast<const uint4*>(static_cast<const char*>(a.x) + (off + col) * (DT == US_F32 ? 4 : 2));
    c.v[0] = __ldg(q);
    if (DT == US_F32) c.v[DT == US_F32 ? 1 : 0] = __ldg(q + 1);
  } else {
    // the packed words of -infinity wherever the row has ended
    uint32_t w[DT == US_F32 ? 8 : 4];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool in = col + i < a.cols;
      if (DT == US_F32) {
        w[i % (DT == US_F32 ? 8 : 4)] = in ? reinterpret_cast<const uint32_t*>(a.x)[off + col + i] : 0xff800000u;
      } else {
        const uint32_t h = in ? reinterpret_cast<const uint16_t*>(a.x)[off + col + i] : (DT == US_BF16 ? 0xff80u : 0xfc00u);
        if (i & 1) w[i >> 1] |= h << 16; else w[i >> 1] = h;
      }
    }
    c.v[0] = make_uint4(w[0], w[1], w[2], w[3]);
    if (DT == US_F32) c.v[DT == US_F32 ? 1 : 0] = make_uint4(w[DT == US_F32 ? 4 : 0], w[DT == US_F32 ? 5 : 0], w[DT == US_F32 ? 6 : 0], w[DT == US_F32 ? 7 : 0]);
  }
}
template <int DT>
__device__ __forceinline__ void xent_unpack(const XentChunk<DT>& c, float (&v)[8]) {
  if (DT == US_F32) {
    const uint4 lo = c.v[0], hi = c.v[DT == US_F32 ? 1 : 0];
    v[0] = __uint_as_float(lo.x); v[1] = __uint_as_float(lo.y); v[2] = __uint_as_float(lo.z); v[3] = __uint_as_float(lo.w);
    v[4] = __uint_as_float(hi.x); v[5] = __uint_as_float(hi.y); v[6] = __uint_as_float(hi.z); v[7] = __uint_as_float(hi.w);
  } else {
    unpack16x8(c.v[0], DT, v);
  }
}
// k (onehot - p) for eight consecutive classes, the target being number `at` of them: the comparison is made once for all eight.  (A gain of 2
// to 4 % with a warp per row; the branch keeps the chunks of the register form apart, 1000 x 10752 float32 gradients 14.1 -> 15.4 us.)
__device__ __forceinline__ void xent_grad(float (&p)[8], float k, unsigned at) {
  if (at < 8u) {
#pragma unroll
    for (unsigned i = 0; i < 8u; ++i) p[i] = k * ((i == at ? 1.0f : 0.f) - p[i]);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i] = k * (0.f - p[i]);
  }
}
// Sum or maximum over the CTA: warps by shuffles, then every thread combines the warps' values in warp order.
template <bool MAX>
__device__ __forceinline__ float cta_reduce(float v, float* slots) {
  v = MAX ? warp_max(v) : warp_sum(v);
  if ((threadIdx.x & 31) == 0) slots[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = slots[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) r = MAX ? fmaxf(r, slots[w]) : r + slots[w];
  return r;
}

// Packed maximum, and pairs of 16-bit values widened (see softmax_xent_staged_kernel).
template <int DT>
__device__ __forceinline__ uint32_t max16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  if (DT == US_BF16) asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  else asm("max.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
template <int DT>
__device__ __forceinline__ f32x2 pair16(uint32_t w) {
  const float2 f = DT == US_BF16 ? unpack_bf16x2(w) : unpack_f16x2(w);
  return pack2(f.x, f.y);
}
// Factors of a row's gradients k (onehot - e / sum), e the exponential of a class: k (1 - e / sum) at the target, e (-k / sum) elsewhere, one
// product a class.  (The target's is not the same product plus k: with an infinite k that would be NaN.  The zero that is added makes the
// gradient of a class of weight zero +0, as k (0 - 0) is.)
struct XentScale {
  float k, inv;
  f32x2 each;
  __device__ __forceinline__ XentScale(float k, float inv) : k(k), inv(inv), each(splat2(-k * inv)) {}
  __device__ __forceinline__ float target(float e) const { return k * (1.0f - e * inv); }
  __device__ __forceinline__ f32x2 others(f32x2 e) const { return fma2(e, each, splat2(0.f)); }
};
// Eight gradients into a row at a column that is a multiple of eight, all of them in the row.
__device__ __forceinline__ void xent_put_e5m2(const XentArgs& a, int64_t out_off, int col, const float (&v)[8]) {
  *reinterpret_cast<uint2*>(static_cast<char*>(a.out) + out_off + col) =
      make_uint2(cvt_fp8x4<true>(v[0], v[1], v[2], v[3]), cvt_fp8x4<true>(v[4], v[5], v[6], v[7]));
}
__device__ __forceinline__ void xent_put(const XentArgs& a, int64_t out_off, int col, const float (&v)[8]) {
  if (a.out_dt == US_E5M2) xent_put_e5m2(a, out_off, col, v);
  else store8(a.out, a.out_dt, out_off, col, a.cols, true, v);
}

template <bool BWD, int DT, int NCH>
__global__ void __launch_bounds__(1024) softmax_xent_row_kernel(const XentArgs a) {
  __shared__ float slots[2][32];
  const int64_t row = blockIdx.x;
  const int64_t x_off = row * a.x_ld;
  const int step = (int)blockDim.x * 8, col0 = (int)threadIdx.x * 8;
  const int nch = NCH > 0 ? NCH : (a.cols + step - 1) / step;
  const int t = a.t[row];
  const bool valid = t >= 0 && t < a.cols;                   // a target outside the row: NaN forward, no one-hot term backward
  float xt = __int_as_float(0x7fc00000), gr = 1.0f;
  // kPairs: float32 pairs, and one product a gradient; gradients of one or two chunks a thread, of float32 rows up to three, stay scalar (2048 x
  // 1500 BF16 logits 6.4 us, in pairs 6.8; 2048 x 3000 8.4 -> 7.9, 4000 x 12000 44.1 -> 38.6, forward 25.3 -> 21.1; float32 logits and gradients
  // 4000 x 12000 74, in pairs 76 to 79).
  constexpr bool kPairs = !BWD || NCH == 0 || NCH > (DT == US_F32 ? 3 : 2);
  if (!BWD && threadIdx.x == 0 && valid) xt = load_one(a.x, DT, x_off + t);
  if (BWD && a.g) gr = a.g[row];
  XentChunk<DT> keep[NCH > 0 ? NCH : 1];
  auto for_chunks = [&](auto&& fn) {
#pragma unroll
    for (int c = 0; c < nch; ++c) {
      const int col = col0 + c * step;
      if (col < a.cols) {
        XentChunk<DT>& k = keep[NCH > 0 ? c : 0];
        if (NCH == 0) xent_load<DT>(a, x_off, col, k);
        float v[8];
        xent_unpack<DT>(k, v);
        fn(col, v);
      }
    }
  };
  if (NCH > 0) {
#pragma unroll
    for (int c = 0; c < nch; ++c)
      if (col0 + c * step < a.cols) xent_load<DT>(a, x_off, col0 + c * step, keep[c]);
  }
  float m = -INFINITY;
  if constexpr (DT != US_F32 && NCH > 0 && (!BWD || NCH > 2)) {
    uint32_t m2 = DT == US_BF16 ? 0xff80ff80u : 0xfc00fc00u;
#pragma unroll
    for (int c = 0; c < nch; ++c)
      if (col0 + c * step < a.cols) {
        const uint4& r = keep[c].v[0];
        m2 = max16x2<DT>(max16x2<DT>(m2, max16x2<DT>(r.x, r.y)), max16x2<DT>(r.z, r.w));
      }
    float lo, hi;
    unpack2(pair16<DT>(m2), lo, hi);
    m = fmaxf(lo, hi);
  } else {
    for_chunks([&](int, float (&v)[8]) {
#pragma unroll
      for (int i = 0; i < 8; ++i) m = fmaxf(m, v[i]);
    });
  }
  m = cta_reduce<true>(m, slots[0]);
  const float mb = m * kLog2e;
  const f32x2 l2 = splat2(kLog2e), neg = splat2(-mb);
  f32x2 sum2 = pack2(0.f, 0.f);
  float sum = 0.f;
  for_chunks([&](int, float (&v)[8]) {
    if constexpr (!kPairs) {
#pragma unroll
      for (int i = 0; i < 8; ++i) sum += ex2_approx(fmaf(v[i], kLog2e, -mb));   // -infinity beyond the row's end adds 0
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float a0, a1;
        unpack2(fma2(pack2(v[2 * i], v[2 * i + 1]), l2, neg), a0, a1);
        sum2 = add2(sum2, pack2(ex2_approx(a0), ex2_approx(a1)));
      }
    }
  });
  if (kPairs) {
    float so;
    unpack2(sum2, sum, so);
    sum += so;
  }
  sum = cta_reduce<false>(sum, slots[1]);
  if (!BWD) {
    if (threadIdx.x == 0) static_cast<float*>(a.out)[row] = (xt - m) - 0.6931471805599453f * __log2f(sum);
    return;
  }
  const float k = a.beta * gr;
  const float inv = 1.0f / sum;
  const XentScale f(k, inv);
  const int64_t out_off = row * a.out_ld;
  // The target's gradient is written over what the same thread has put there: chosen among its chunk's eight in the loop it takes registers that
  // the longest rows lack (us, in the loop / behind it: 2048 x 9000 in BF16 18.7 / 17.2, 2048 x 4500 into E5M2 12.2 / 11.0).
  const bool mine = kPairs && valid && (t >> 3) % (int)blockDim.x == (int)threadIdx.x;        // the target is in a chunk of this thread
  if (mine) xt = load_one(a.x, DT, x_off + t);
  for_chunks([&](int col, float (&v)[8]) {
    if constexpr (!kPairs) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float p = ex2_approx(fmaf(v[i], kLog2e, -mb)) * inv;
        v[i] = k * ((col + i == t ? 1.0f : 0.f) - p);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float a0, a1;
        unpack2(fma2(pack2(v[2 * i], v[2 * i + 1]), l2, neg), a0, a1);
        unpack2(f.others(pack2(ex2_approx(a0), ex2_approx(a1))), v[2 * i], v[2 * i + 1]);
      }
    }
    store8(a.out, a.out_dt, out_off, col, a.cols, a.vec_ok && col + 8 <= a.cols, v);
  });
  if (mine) store_one(a.out, a.out_dt, out_off + t, f.target(ex2_approx(fmaf(xt, kLog2e, -mb))));
}

// One CTA per row of 16-bit logits staged in shared memory by one bulk copy, for vocabularies whose rows the register form
// holds with 512 threads: three CTAs per SM instead of two (40 registers a thread instead of 64), so that one row's load
// runs under two others' reductions.  2048 rows of 30522 BF16 logits: forward 39 -> 31 us (4.1 TB/s), backward with an E5M2
// gradient 66 -> 56 us (3.3 TB/s; two exponentials per class make 28 us of it).  A wait that runs out falls back to loads
// from global memory.
// The maximum of packed 16-bit values, sums and scalings of float32 pairs, one product a class instead of three operations, and the E5M2
// store chosen once a row, us: 2048 x 30522 forward 29.7 -> 27.1, backward E5M2 55.8 -> 44.2, BF16 54.4 -> 48.3; 2048 x 16400 E5M2 36.8 -> 30.4.
constexpr int kXentStagedThreads = 512;
constexpr uint32_t kXentWaitLimit = 1u << 20;               // polls of a wait for a bulk copy
template <bool BWD, int DT>
__global__ void __launch_bounds__(kXentStagedThreads, 3) softmax_xent_staged_kernel(const XentArgs a) {
  extern __shared__ __align__(16) uint8_t xent_smem[];
  __shared__ float slots[2][32];
  __shared__ __align__(8) uint64_t bar_word;
  const uint32_t data = ptx::smem_addr(xent_smem), bar = ptx::smem_addr(&bar_word);
  const int64_t row = blockIdx.x, x_off = row * a.x_ld;
  const int tid = (int)threadIdx.x;
  const int full = a.cols / 8, tail = a.cols - 8 * full;      // whole chunks of eight; elements behind them
  if (tid == 0) {
    ptx::mbar_init(bar, 1);
    ptx::mbar_init_fence();
    ptx::mbar_expect_tx(bar, (uint32_t)full * 16u);
    ptx::bulk_load_1d(data, static_cast<const char*>(a.x) + x_off * 2, (uint32_t)full * 16u, bar);
  }
  const int t = a.t[row];
  const bool valid = t >= 0 && t < a.cols;                   // a target outside the row: NaN forward, no one-hot term backward
  float xt = __int_as_float(0x7fc00000), gr = 1.0f;
  if ((BWD || tid == 0) && valid) xt = load_one(a.x, DT, x_off + t);
  if (BWD && a.g) gr = a.g[row];
  const float last = tid < tail ? load_one(a.x, DT, x_off + 8 * full + tid) : -INFINITY;
  __syncthreads();
  bool staged = false;
  for (uint32_t it = 0; it < kXentWaitLimit && !(staged = ptx::mbar_try_wait(bar, 0)); ++it) {}
  auto for_chunks = [&](auto&& fn) {
#pragma unroll 2
    for (int c = tid; c < full; c += kXentStagedThreads) {
      const uint4 raw = staged ? ptx::lds128(data + (uint32_t)c * 16u)
                               : __ldg(reinterpret_cast<const uint4*>(static_cast<const char*>(a.x) + x_off * 2) + c);
      const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
      fn(8 * c, w);
    }
  };
  uint32_t m2 = DT == US_BF16 ? 0xff80ff80u : 0xfc00fc00u;    // the maximum of 16-bit values needs no widening
  for_chunks([&](int, const uint32_t (&w)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) m2 = max16x2<DT>(m2, w[i]);
  });
  float m, mo;
  unpack2(pair16<DT>(m2), m, mo);
  m = cta_reduce<true>(fmaxf(last, fmaxf(m, mo)), slots[0]);
  const float mb = m * kLog2e;
  const f32x2 l2 = splat2(kLog2e), neg = splat2(-mb);
  f32x2 sum2 = pack2(tid < tail ? ex2_approx(fmaf(last, kLog2e, -mb)) : 0.f, 0.f);
  for_chunks([&](int, const uint32_t (&w)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float a0, a1;
      unpack2(fma2(pair16<DT>(w[i]), l2, neg), a0, a1);
      sum2 = add2(sum2, pack2(ex2_approx(a0), ex2_approx(a1)));
    }
  });
  float sum, so;
  unpack2(sum2, sum, so);
  sum = cta_reduce<false>(sum + so, slots[1]);
  if (!BWD) {
    if (tid == 0) static_cast<float*>(a.out)[row] = (xt - m) - 0.6931471805599453f * __log2f(sum);
  } else {
    const float k = a.beta * gr, inv = 1.0f / sum;
    const int64_t out_off = row * a.out_ld;
    const XentScale f(k, inv);
    const float gt = f.target(ex2_approx(fmaf(xt, kLog2e, -mb)));
    auto gradients = [&](auto&& put) {
      for_chunks([&](int col, const uint32_t (&w)[4]) {
        float v[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float a0, a1;
          unpack2(fma2(pair16<DT>(w[i]), l2, neg), a0, a1);
          unpack2(f.others(pack2(ex2_approx(a0), ex2_approx(a1))), v[2 * i], v[2 * i + 1]);
        }
        if ((unsigned)t - (unsigned)col < 8u) {                // the target's class
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (col + i == t) v[i] = gt;
        }
        put(col, v);
      });
    };
    if (a.out_dt == US_E5M2) {
      gradients([&](int col, const float (&v)[8]) { xent_put_e5m2(a, out_off, col, v); });
    } else {
      gradients([&](int col, const float (&v)[8]) { store8(a.out, a.out_dt, out_off, col, a.cols, true, v); });
    }
    if (tid < tail) {
      const int col = 8 * full + tid;
      store_one(a.out, a.out_dt, out_off + col, k * ((col == t ? 1.0f : 0.f) - ex2_approx(fmaf(last, kLog2e, -mb)) * inv));
    }
  }
  if (!staged && tid == 0)                                   // the copy lands before the CTA gives up its shared memory
    for (uint32_t it = 0; it < kXentWaitLimit && !ptx::mbar_try_wait(bar, 0); ++it) {}
}

// Persistent CTAs of T threads, 1024 / T of them per SM, walk the rows of a 16-bit vocabulary: a ring of kXentRing rows in shared
// memory is filled by bulk copies ahead of the row that is worked on, and a thread holds its (at most 32) elements of that
// row in registers, widened, from the maximum to the write.  Each exponential is computed once (twice in the other forms, which the
// ex2 unit bounds).  E5M2 gradient of 4096 rows of BF16 logits, the register form / this one: 16384 classes 59.8 / 46.1 us, 12000 45.7 / 39.0,
// 8192 32.5 / 22.6, 5000 20.0 / 17.5 (xent_launch_dt has the lines).  Rows of up to 4096 classes gain nothing, longer ones than 16384 leave room for one CTA an SM and
// lose, and so does the forward pass, which has no second exponential to save.
// A wait that runs out falls back to loads from global memory.
constexpr int kXentRing = 3;
template <bool MAX, int T>
__device__ __forceinline__ float ring_reduce(float v, float* slots) {
  v = MAX ? warp_max(v) : warp_sum(v);
  const int lane = threadIdx.x & 31;
  if (lane == 0) slots[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = slots[lane & (T / 32 - 1)];                      // the warps' values, combined in the same order by every warp
#pragma unroll
  for (int o = T / 64; o > 0; o >>= 1) { const float w = __shfl_xor_sync(0xffffffffu, r, o); r = MAX ? fmaxf(r, w) : r + w; }
  return r;
}
template <int DT, int T>
__global__ void __launch_bounds__(T, 1024 / T) softmax_xent_ring_kernel(const XentArgs a) {
  extern __shared__ __align__(16) uint8_t xent_smem[];
  __shared__ float slots[2][2][32];
  __shared__ __align__(8) uint64_t bar_words[kXentRing];
  constexpr int kCh = 4;                                     // chunks of eight elements per thread
  const int tid = (int)threadIdx.x;
  const int full = a.cols / 8, tail = a.cols - 8 * full;     // whole chunks of eight; elements behind them
  const uint32_t bytes = (uint32_t)full * 16u;
  const int rows = (int)a.rows, step = (int)gridDim.x;
  auto bar = [&](int i) { return ptx::smem_addr(&bar_words[i % kXentRing]); };
  auto data = [&](int i) { return ptx::smem_addr(xent_smem) + (uint32_t)(i % kXentRing) * bytes; };
  auto fetch = [&](int i) {                                  // the CTA's row number i (one thread)
    const int64_t row = blockIdx.x + (int64_t)i * step;
    if (row >= rows) return;
    ptx::mbar_expect_tx(bar(i), bytes);
    ptx::bulk_load_1d(data(i), static_cast<const char*>(a.x) + row * a.x_ld * 2, bytes, bar(i));
  };
  if (tid == 0) {
    for (int i = 0; i < kXentRing; ++i) ptx::mbar_init(bar(i), 1);
    ptx::mbar_init_fence();
    for (int i = 0; i < kXentRing; ++i) fetch(i);
  }
  __syncthreads();
  int i = 0;
  bool late = false;                                         // this thread gave up on a copy, of its row number late_at
  int late_at = 0;
  for (int row = blockIdx.x; row < rows; row += step, ++i) {
    const int64_t x_off = row * a.x_ld;
    const int t = a.t[row];
    const float gr = a.g ? a.g[row] : 1.0f;
    const float last = tid < tail ? load_one(a.x, DT, x_off + 8 * full + tid) : -INFINITY;
    bool staged = false;
    for (uint32_t it = 0; !late && it < kXentWaitLimit && !(staged = ptx::mbar_try_wait(bar(i), (uint32_t)(i / kXentRing) & 1u)); ++it) {}
    if (!late && !staged) { late = true; late_at = i; }
    f32x2 v[kCh][4];
    uint32_t m2 = DT == US_BF16 ? 0xff80ff80u : 0xfc00fc00u;
#pragma unroll
    for (int c = 0; c < kCh; ++c) {
      const int k = tid + c * T;
      if (k < full) {
        const uint4 raw = staged ? ptx::lds128(data(i) + (uint32_t)k * 16u)
                                 : __ldg(reinterpret_cast<const uint4*>(static_cast<const char*>(a.x) + x_off * 2) + k);
        const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) { m2 = max16x2<DT>(m2, w[e]); v[c][e] = pair16<DT>(w[e]); }
      }
    }
    float m, mo;
    unpack2(pair16<DT>(m2), m, mo);
    m = ring_reduce<true, T>(fmaxf(last, fmaxf(m, mo)), slots[i & 1][0]);
    if (tid == 0 && !late) fetch(i + kXentRing);             // every thread has taken its elements of this row
    const float mb = m * kLog2e;
    float e_last = tid < tail ? ex2_approx(fmaf(last, kLog2e, -mb)) : 0.f;
    const f32x2 l2 = splat2(kLog2e), neg = splat2(-mb);
    f32x2 sum2 = pack2(e_last, 0.f);
#pragma unroll
    for (int c = 0; c < kCh; ++c) {
      if (tid + c * T < full) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float a0, a1;
          unpack2(fma2(v[c][e], l2, neg), a0, a1);
          v[c][e] = pack2(ex2_approx(a0), ex2_approx(a1));
          sum2 = add2(sum2, v[c][e]);
        }
      }
    }
    float sum, so;
    unpack2(sum2, sum, so);
    sum = ring_reduce<false, T>(sum + so, slots[i & 1][1]);
    const float k = a.beta * gr, inv = 1.0f / sum;
    const XentScale f(k, inv);
    const int64_t out_off = row * a.out_ld;
#pragma unroll
    for (int c = 0; c < kCh; ++c) {
      const int col = 8 * (tid + c * T);
      if (tid + c * T < full) {
        float g[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) unpack2(f.others(v[c][e]), g[2 * e], g[2 * e + 1]);
        if ((unsigned)t - (unsigned)col < 8u) {                // the target's class
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            float lo, hi;
            unpack2(v[c][e / 2], lo, hi);
            if (col + e == t) g[e] = f.target(e & 1 ? hi : lo);
          }
        }
        xent_put(a, out_off, col, g);
      }
    }
    if (tid < tail) {
      const int col = 8 * full + tid;
      store_one(a.out, a.out_dt, out_off + col, k * ((col == t ? 1.0f : 0.f) - e_last * inv));
    }
  }
  // Copies that are still in flight after a wait that ran out land before the CTA gives up its shared memory.
  if (tid == 0 && late)
    for (int r = late_at; r < late_at + kXentRing && blockIdx.x + (int64_t)r * step < rows; ++r)
      for (uint32_t it = 0; it < kXentWaitLimit && !ptx::mbar_try_wait(bar(r), (uint32_t)(r / kXentRing) & 1u); ++it) {}
}

// One warp per row, for short rows: read twice (maximum, then sum of exponentials) and in the backward pass a third
// time, from cache.
// RAGGED: rows end inside a chunk of eight (the test costs 3 %).
template <bool BWD, bool RAGGED>
__global__ void __launch_bounds__(kSmThreads) softmax_xent_kernel(const XentArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t row = (int64_t)blockIdx.x * (kSmThreads / 32) + (threadIdx.x >> 5);
  if (row >= a.rows) return;
  const int64_t x_off = row * a.x_ld;
  const bool vec = a.vec_ok != 0;
  const int nch = (a.cols + 255) / 256;
  float m = -INFINITY;
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    if (col >= a.cols) continue;
    float v[8];
    load8(a.x, a.x_dt, x_off, col, a.cols, vec && (!RAGGED || col + 8 <= a.cols), -INFINITY, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) m = fmaxf(m, v[i]);
  }
  m = warp_max(m);
  const float mb = m * kLog2e;
  float sum = 0.f;
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    if (col >= a.cols) continue;
    float v[8];
    load8(a.x, a.x_dt, x_off, col, a.cols, vec && (!RAGGED || col + 8 <= a.cols), -INFINITY, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) sum += ex2_approx(fmaf(v[i], kLog2e, -mb));
  }
  sum = warp_sum(sum);
  const int t = a.t[row];
  const bool valid = t >= 0 && t < a.cols;                   // a target outside the row: NaN forward, no one-hot term backward
  if (!BWD) {
    if (lane == 0) {
      const float xt = valid ? load_one(a.x, a.x_dt, x_off + t) : __int_as_float(0x7fc00000);
      static_cast<float*>(a.out)[row] = (xt - m) - 0.6931471805599453f * __log2f(sum);
    }
    return;
  }
  const float k = a.beta * (a.g ? a.g[row] : 1.0f);
  const float inv = 1.0f / sum;
  const int64_t out_off = row * a.out_ld;
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    if (col >= a.cols) continue;
    float v[8];
    load8(a.x, a.x_dt, x_off, col, a.cols, vec && (!RAGGED || col + 8 <= a.cols), -INFINITY, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = ex2_approx(fmaf(v[i], kLog2e, -mb)) * inv;
    xent_grad(v, k, (unsigned)t - (unsigned)col);
    store8(a.out, a.out_dt, out_off, col, a.cols, vec && (!RAGGED || col + 8 <= a.cols), v);
  }
}

static bool rows_aligned(const us_mat* m) {
  return reinterpret_cast<uintptr_t>(m->ptr) % 16 == 0 && (m->ld * dtype_size(m->dtype)) % 16 == 0;
}

template <bool BWD>
static us_status launch_softmax(const SmArgs& a, cudaStream_t st) {
  if (a.rows == 0 || a.cols == 0) return US_OK;
  const int64_t grid64 = (a.rows + kSmThreads / 32 - 1) / (kSmThreads / 32);
  if (grid64 > 0x7fffffff) return US_ERR_INVALID_ARG;
  const int grid = (int)grid64;
  const int nch = (a.cols + 255) / 256;
  const bool in16 = a.in0_dt == US_BF16 || a.in0_dt == US_F16;
  const bool p8 = BWD && (a.in0_dt == US_E4M3 || a.in0_dt == US_E5M2) && (a.in1_dt == US_BF16 || a.in1_dt == US_F16);
  if (a.vec_ok && nch <= 4 && ((in16 && (!BWD || a.in1_dt == a.in0_dt)) || p8)) {
    const int sms = host::sm_count();
    if (sms <= 0) return US_ERR_CUDA;
    const int pgrid = grid < 2 * sms ? grid : 2 * sms;        // two resident CTAs per SM, warps walk the rows
#define US_SM16(N)                                                                   \
  do {                                                                               \
    if (BWD && p8) return host::launch(softmax_bwd16_kernel<N, true>, nullptr, pgrid, kSmThreads, 0, 1, st, a);  \
    if (BWD) return host::launch(softmax_bwd16_kernel<N, false>, nullptr, pgrid, kSmThreads, 0, 1, st, a);       \
    return host::launch(softmax_fwd16_kernel<N>, nullptr, pgrid, kSmThreads, 0, 1, st, a);                       \
  } while (0)
    if (nch <= 1) US_SM16(1);
    else if (nch <= 2) US_SM16(2);
    else US_SM16(4);
#undef US_SM16
  }
#define US_SM_LAUNCH(N)                                                          \
  do {                                                                           \
    if (BWD) softmax_bwd_kernel<N><<<grid, kSmThreads, 0, st>>>(a);              \
    else softmax_fwd_kernel<N><<<grid, kSmThreads, 0, st>>>(a);                  \
  } while (0)
  if (nch <= 1) US_SM_LAUNCH(1);
  else if (nch <= 2) US_SM_LAUNCH(2);
  else if (nch <= 4) US_SM_LAUNCH(4);
  else if (nch <= 8 && !BWD) US_SM_LAUNCH(8);
  else US_SM_LAUNCH(0);
#undef US_SM_LAUNCH
  return cudaGetLastError() == cudaSuccess ? US_OK : US_ERR_CUDA;
}

// input: a tensor the kernel reads (float formats; FP8 too where fp8_in says so).
static us_status check_mat(const us_mat* m, const us_mat* like, bool input, bool fp8_in = false) {
  if (!m || m->rows < 0 || m->cols < 0 || m->ld < m->cols) return US_ERR_INVALID_ARG;
  if (like && (m->rows != like->rows || m->cols != like->cols)) return US_ERR_INVALID_ARG;
  if (m->rows * m->cols > 0 && !m->ptr) return US_ERR_INVALID_ARG;
  if (m->cols > 0x7ffffff0) return US_ERR_INVALID_ARG;
  const bool is_fp8 = m->dtype == US_E4M3 || m->dtype == US_E5M2;
  if (input ? !(m->dtype == US_F32 || m->dtype == US_BF16 || m->dtype == US_F16 || (fp8_in && is_fp8)) : !(m->dtype >= US_F32 && m->dtype <= US_E5M2))
    return US_ERR_UNSUPPORTED;
  if (m->ptr && reinterpret_cast<uintptr_t>(m->ptr) % dtype_size(m->dtype)) return US_ERR_ALIGNMENT;
  return US_OK;
}

}  // namespace us

using namespace us;

extern "C" us_status us_softmax_fwd(const us_mat* S, float alpha, const us_mat* P, void* stream) {
  us_status s = check_mat(S, nullptr, true);
  if (s == US_OK) s = check_mat(P, S, false);
  if (s != US_OK) return s;
  SmArgs a{};
  a.in0 = S->ptr; a.in0_dt = S->dtype; a.in0_ld = S->ld;
  a.out = P->ptr; a.out_dt = P->dtype; a.out_ld = P->ld;
  a.rows = S->rows; a.cols = (int)S->cols; a.alpha = alpha; a.beta = 0.f;
  a.vec_ok = rows_aligned(S) && rows_aligned(P) && S->cols % 8 == 0;
  return launch_softmax<false>(a, static_cast<cudaStream_t>(stream));
}

extern "C" us_status us_softmax_bwd(const us_mat* P, const us_mat* dP, float alpha, float beta, const us_mat* dS,
                                    void* stream) {
  us_status s = check_mat(P, nullptr, true, true);           // the stored forward output may be FP8
  if (s == US_OK) s = check_mat(dP, P, true);
  if (s == US_OK) s = check_mat(dS, P, false);
  if (s != US_OK) return s;
  if (!(alpha > 0.f)) return US_ERR_INVALID_ARG;
  SmArgs a{};
  a.in0 = P->ptr; a.in0_dt = P->dtype; a.in0_ld = P->ld;
  a.in1 = dP->ptr; a.in1_dt = dP->dtype; a.in1_ld = dP->ld;
  a.out = dS->ptr; a.out_dt = dS->dtype; a.out_ld = dS->ld;
  a.rows = P->rows; a.cols = (int)P->cols; a.alpha = alpha; a.beta = beta;
  a.vec_ok = rows_aligned(P) && rows_aligned(dP) && rows_aligned(dS) && P->cols % 8 == 0;
  return launch_softmax<true>(a, static_cast<cudaStream_t>(stream));
}

template <bool BWD, int DT>
static us_status xent_launch_dt(const XentArgs& a, cudaStream_t st) {
  // A warp per row up to 512 classes (two chunks per lane), and in the forward pass up to 1280 (16-bit: 1536) where there
  // are rows enough to fill the chip that way.  BF16 logits, us, a warp per row against a CTA per row: forward 16384 x 512 /
  // 640 / 1024 / 1280 / 2048: 9.4 / 9.6 / 12.2 / 14.1 / 23.8 against 14.7 / 13.9 / 14.5 / 16.6 / 20.9, 2048 x 640 / 1024: 3.5 / 4.2
  // against 3.2 / 3.4, even at 2400 x 640, 3600 x 1024, 5000 x 1280 and 14000 x 1536, 65536 x 1536 63 against 75 (F32: 77, 72);
  // backward 16384 x 512 / 640 / 1024: 14.7 / 17.8 / 22.9 against 17.2 / 18.2 / 20.8.
  // Beyond, the smallest CTA whose threads hold the row in at most 8 chunks of 16-bit or 4 chunks of float32 elements (32
  // registers of data each): few warps with many loads in flight each and two or more CTAs per SM (30522 classes: 512 threads
  // x 8 chunks 39 / 66 us forward / backward, 1024 x 4 42 / 92 us, because one CTA then fills the SM and nothing overlaps its
  // reductions).
  constexpr int kMaxCh = DT == US_F32 ? 4 : 8;
  const int64_t grid = (a.rows + kSmThreads / 32 - 1) / (kSmThreads / 32);
  if (grid > 0x7fffffff) return US_ERR_INVALID_ARG;
  const int sms = host::sm_count();
  if (sms <= 0) return US_ERR_CUDA;
  const int limit = DT == US_F32 ? 1280 : 1536;
  const bool many_rows = !BWD && a.vec_ok && a.cols <= limit && a.rows >= 16 * sms && a.rows >= (a.cols <= 1280 ? 4ll : 10ll) * a.cols;
  if (a.cols <= 512 || many_rows || a.rows > 0x7fffffff) {
    if (a.cols % 8 == 0) softmax_xent_kernel<BWD, false><<<(int)grid, kSmThreads, 0, st>>>(a);
    else softmax_xent_kernel<BWD, true><<<(int)grid, kSmThreads, 0, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? US_OK : US_ERR_CUDA;
  }
  const int chunks = (a.cols + 7) / 8;
  int threads = 128;
  while (threads < 1024 && chunks > threads * kMaxCh) threads *= 2;
  const int nch = (chunks + threads - 1) / threads;
  const int rows = (int)a.rows;
  if constexpr (DT != US_F32) {
    // The ring: wherever every row has a CTA of its own; with more rows not for float32 gradients, whose writes bound both forms and are
    // less even from fewer CTAs, not for 8193 to 10240 classes, where the register form has five chunks a thread and 256 threads, the
    // ring 512 of which few have more than two, and not below 5000.  Registers over ring, BF16 logits, 4104 / 5000 / 6000 / 8192 / 8200 / 10000 /
    // 10752 / 12000 / 16384 classes: 148 rows, E5M2 1.34 1.33 1.50 1.71 1.33 1.33 1.40 1.38 1.58, BF16 1.21 to 1.55, float32 1.18 1.20 1.23 1.34 1.01 0.96 1.00 0.98
    // 1.01; 1000 rows, E5M2 1.03 1.06 1.12 1.32 0.95 1.04 1.07 1.07 1.19, BF16 0.94 0.97 1.05 1.18 0.88 0.95 1.00 1.00 1.08, float32 0.87 0.91 0.98 1.07 0.76 0.82
    // 0.84 0.82 0.92; 4096 rows, E5M2 1.10 1.14 1.24 1.43 1.07 1.11 1.16 1.17 1.30, BF16 0.97 1.01 1.13 1.20 0.98 1.01 1.06 1.06 1.18, float32 0.81 to 1.00.
    const int t = a.cols > 8192 ? 512 : 256, units = sms * (1024 / t);
    const bool walks = a.out_dt != US_F32 && ((a.cols >= 5000 && a.cols <= 8192) || a.cols > 10240);
    if (BWD && a.vec_ok && a.cols > 4096 && a.cols <= 16384 && (rows <= units || walks)) {
      static std::atomic<uint64_t> ring_set[2];
      const int g = rows < units ? rows : units, max_smem = kXentRing * 64 * t;
      const size_t smem = (size_t)kXentRing * (a.cols / 8) * 16;
      if (t == 512) return host::launch_plain(softmax_xent_ring_kernel<DT, 512>, &ring_set[0], g, t, max_smem, smem, st, a);
      return host::launch_plain(softmax_xent_ring_kernel<DT, 256>, &ring_set[1], g, t, max_smem, smem, st, a);
    }
    // Rows of 16385 to 36000 classes: three of them fit an SM's shared memory, and the register form needs 512 threads a row
    // (2048 x 16384 / 16400 / 24576 BF16 logits, forward and backward: staged 20.9 + 37.3 / 20.8 + 37.6 / 25.5 + 48.8 us, in
    // registers 18.7 + 35.2 / 21.0 + 43.5 / 33.1 + 56.0)
    if (a.vec_ok && (threads == 512 || (threads == 1024 && a.cols <= 36000))) {
      static std::atomic<uint64_t> smem_set{0};
      return host::launch_plain(softmax_xent_staged_kernel<BWD, DT>, &smem_set, rows, kXentStagedThreads, 72000, a.cols / 8 * 16, st, a);
    }
  }
  switch (nch > kMaxCh ? 0 : nch) {
    case 1: softmax_xent_row_kernel<BWD, DT, 1><<<rows, threads, 0, st>>>(a); break;
    case 2: softmax_xent_row_kernel<BWD, DT, 2><<<rows, threads, 0, st>>>(a); break;
    case 3: softmax_xent_row_kernel<BWD, DT, 3><<<rows, threads, 0, st>>>(a); break;
    case 4: softmax_xent_row_kernel<BWD, DT, 4><<<rows, threads, 0, st>>>(a); break;
    case 5: softmax_xent_row_kernel<BWD, DT, kMaxCh == 8 ? 5 : 0><<<rows, threads, 0, st>>>(a); break;
    case 6: softmax_xent_row_kernel<BWD, DT, kMaxCh == 8 ? 6 : 0><<<rows, threads, 0, st>>>(a); break;
    case 7: softmax_xent_row_kernel<BWD, DT, kMaxCh == 8 ? 7 : 0><<<rows, threads, 0, st>>>(a); break;
    case 8: softmax_xent_row_kernel<BWD, DT, kMaxCh == 8 ? 8 : 0><<<rows, threads, 0, st>>>(a); break;
    default: softmax_xent_row_kernel<BWD, DT, 0><<<rows, threads, 0, st>>>(a);
  }
  return cudaGetLastError() == cudaSuccess ? US_OK : US_ERR_CUDA;
}
template <bool BWD>
static us_status xent_launch(const XentArgs& a, cudaStream_t st) {
  switch (a.x_dt) {
    case US_F32: return xent_launch_dt<BWD, US_F32>(a, st);
    case US_BF16: return xent_launch_dt<BWD, US_BF16>(a, st);
    default: return xent_launch_dt<BWD, US_F16>(a, st);
  }
}

static us_status check_xent(const us_mat* X, const int32_t* targets) {
  us_status s = check_mat(X, nullptr, true);
  if (s != US_OK) return s;
  if (X->rows > 0 && !targets) return US_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(targets) % 4) return US_ERR_ALIGNMENT;
  if (X->rows > 0 && X->cols < 1) return US_ERR_INVALID_ARG;
  return US_OK;
}

extern "C" us_status us_softmax_xent_fwd(const us_mat* X, const int32_t* targets, float* out, void* stream) {
  us_status s = check_xent(X, targets);
  if (s != US_OK) return s;
  if (X->rows == 0) return US_OK;
  if (!out || reinterpret_cast<uintptr_t>(out) % 4) return US_ERR_INVALID_ARG;
  XentArgs a{};
  a.x = X->ptr; a.x_dt = X->dtype; a.x_ld = X->ld; a.t = targets; a.out = out;
  a.rows = X->rows; a.cols = (int)X->cols;
  a.vec_ok = rows_aligned(X);
  return xent_launch<false>(a, static_cast<cudaStream_t>(stream));
}

extern "C" us_status us_softmax_xent_bwd(const us_mat* X, const int32_t* targets, const float* g, float beta,
                                         const us_mat* dX, void* stream) {
  us_status s = check_xent(X, targets);
  if (s == US_OK) s = check_mat(dX, X, false);
  if (s != US_OK) return s;
  if (g && reinterpret_cast<uintptr_t>(g) % 4) return US_ERR_ALIGNMENT;
  if (X->rows == 0) return US_OK;
  XentArgs a{};
  a.x = X->ptr; a.x_dt = X->dtype; a.x_ld = X->ld; a.t = targets; a.g = g;
  a.out = dX->ptr; a.out_dt = dX->dtype; a.out_ld = dX->ld;
  a.rows = X->rows; a.cols = (int)X->cols; a.beta = beta;
  a.vec_ok = rows_aligned(X) && rows_aligned(dX);
  return xent_launch<true>(a, static_cast<cudaStream_t>(stream));
}
