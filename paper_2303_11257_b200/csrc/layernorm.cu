// Scaled layer norm over the rows of a matrix, forward and backward (table "Table of unit scaling
// factors", row layer_norm: alpha = 1, beta_x = 1, beta_w = beta_c = b^-1/2 for a b x n input).
//
// Forward and the input gradient are row-wise: one warp per row, 128-bit loads and stores, warp-shuffle
// reductions, the row held in registers when it has at most 1024 elements (re-read from cache otherwise).  The
// backward pass of 16-bit rows of up to 2048 elements shares a row among several warps (ln_bwd_rows_kernel).
// The variance is taken about the mean (sum of (x - mu)^2), which equals the table's
// mean(x^2) - mu^2 without its cancellation in float32.
//
// Weight and bias gradients are column sums over all rows.  The backward kernel keeps, per lane, the
// partial sums of the columns that lane owns (in registers, or in shared memory for long rows) over
// the rows its warp walks, combines the warps of a CTA in a fixed order and writes one partial row
// per CTA to the caller's workspace; a second kernel adds the CTAs' partials in a fixed order and
// applies beta.  No atomics: results do not depend on scheduling.
#include <algorithm>

#include "common.cuh"
#include "host.h"
#include "rowwise.cuh"
#include "sm100.cuh"

namespace us {

constexpr int kLnThreads = 256;             // 8 warps = 8 rows in flight per CTA
constexpr int kLnWarps = kLnThreads / 32;
constexpr int kLnMaxBwdCols = 4096;         // backward, long rows: column partials of 4 warps in 128 KB of shared memory

struct LnArgs {
  const void* x; int x_dt; int64_t x_ld;
  const void* g; int g_dt; int64_t g_ld;    // backward only
  const void* w; int w_dt;                  // [cols]
  const void* c; int c_dt;                  // [cols], forward only
  void* out; int out_dt; int64_t out_ld;    // Y (forward) or dX (backward)
  void* q; int q_dt; int64_t q_ld;          // an FP8 copy of it (COPY variants)
  float* partial;                           // backward: [gridDim.x][2][cols]
  int64_t rows; int cols;
  int vec_ok;                               // all row starts 16-byte aligned and cols % 8 == 0
  float eps, beta_x;
};

// Eight results: stored, and (COPY) the stored values once more in FP8 for a caller that wants them as the operand of a matmul.  The
// kernels have variants for it, because the code of the copy, never taken, cost the passes without one 2 to 4 % (backward 8192 x 1024
// BF16 19.7 -> 20.3 us, forward 1000 x 1024 3.71 -> 3.82).
template <bool COPY>
__device__ __forceinline__ void ln_store8(const LnArgs& a, int64_t row, int col, bool vec, const float (&t)[8]) {
  store8(a.out, a.out_dt, row * a.out_ld, col, a.cols, vec, t);
  if (COPY) {
    float r[8];
    as_stored8(a.out_dt, t, r);
    store8(a.q, a.q_dt, row * a.q_ld, col, a.cols, vec, r);
  }
}

// Mean and reciprocal standard deviation of a row given as nch chunks per lane.
template <int NCH>
__device__ __forceinline__ void row_stats(const LnArgs& a, int64_t x_off, int lane, int nch, float (&x)[NCH > 0 ? NCH : 1][8],
                                          float& mu, float& rstd) {
  const bool vec = a.vec_ok != 0;
  float s = 0.f;
#pragma unroll
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    float t[8];
    if (col < a.cols) {
      load8(a.x, a.x_dt, x_off, col, a.cols, vec, 0.f, t);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) t[i] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) { s += t[i]; if (NCH > 0) x[c][i] = t[i]; }
  }
  mu = warp_sum(s) / (float)a.cols;
  float q = 0.f;
#pragma unroll
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    float t[8];
    if (NCH > 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) t[i] = x[c][i];
    } else if (col < a.cols) {
      load8(a.x, a.x_dt, x_off, col, a.cols, vec, 0.f, t);
    }
    if (col < a.cols) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float d = (col + i < a.cols) ? t[i] - mu : 0.f;
        q = fmaf(d, d, q);
      }
    }
  }
  rstd = rsqrtf(warp_sum(q) / (float)a.cols + a.eps);
}

// NCH > 0: rows of up to 256 * NCH elements, held in registers.  NCH == 0: any length, re-read.
template <int NCH, bool COPY>
__global__ void __launch_bounds__(kLnThreads) ln_fwd_kernel(const LnArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t row = (int64_t)blockIdx.x * kLnWarps + (threadIdx.x >> 5);
  if (row >= a.rows) return;
  const int64_t x_off = row * a.x_ld;
  const bool vec = a.vec_ok != 0;
  const int nch = NCH > 0 ? NCH : (a.cols + 255) / 256;
  float x[NCH > 0 ? NCH : 1][8];
  float mu, rstd;
  row_stats<NCH>(a, x_off, lane, nch, x, mu, rstd);
#pragma unroll
  for (int c = 0; c < nch; ++c) {
    const int col = (c * 32 + lane) * 8;
    if (col >= a.cols) continue;
    float t[8], w[8], b[8];
    if (NCH > 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) t[i] = x[c][i];
    } else {
      load8(a.x, a.x_dt, x_off, col, a.cols, vec, 0.f, t);
    }
    load8(a.w, a.w_dt, 0, col, a.cols, vec, 0.f, w);
    load8(a.c, a.c_dt, 0, col, a.cols, vec, 0.f, b);
#pragma unroll
    for (int i = 0; i < 8; ++i) t[i] = fmaf(w[i], (t[i] - mu) * rstd, b[i]);
    ln_store8<COPY>(a, row, col, vec, t);
  }
}

// Input gradient of the rows this warp walks, and the CTA's partial column sums of G * xhat and G.
template <int NCH, bool COPY>
__global__ void __launch_bounds__(kLnThreads) ln_bwd_kernel(const LnArgs a) {
  extern __shared__ __align__(16) float ln_smem[];          // NCH > 0: [warps][cols] for the combine; NCH == 0: [warps][2][cols]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;             // 8 warps per CTA, 4 for long rows
  const bool vec = a.vec_ok != 0;
  const int nch = NCH > 0 ? NCH : (a.cols + 255) / 256;
  const float inv_n = 1.0f / (float)a.cols;
  float sw[NCH > 0 ? NCH : 1][8], sc[NCH > 0 ? NCH : 1][8];
  float* my_w = ln_smem + (size_t)warp * 2 * a.cols;      // NCH == 0 only
  float* my_c = my_w + a.cols;
  if (NCH > 0) {
#pragma unroll
    for (int c = 0; c < (NCH > 0 ? NCH : 1); ++c)
#pragma unroll
      for (int i = 0; i < 8; ++i) { sw[c][i] = 0.f; sc[c][i] = 0.f; }
  } else {
    for (int j = lane; j < a.cols; j += 32) { my_w[j] = 0.f; my_c[j] = 0.f; }
    __syncwarp();
  }
  for (int64_t row = (int64_t)blockIdx.x * nw + warp; row < a.rows; row += (int64_t)gridDim.x * nw) {
    const int64_t x_off = row * a.x_ld, g_off = row * a.g_ld;
    float x[NCH > 0 ? NCH : 1][8], u[NCH > 0 ? NCH : 1][8];
    float mu, rstd;
    row_stats<NCH>(a, x_off, lane, nch, x, mu, rstd);
    // pass 1: xhat, u = g w; row sums of u and u xhat; column partials of g xhat and g
    float su = 0.f, sux = 0.f;
#pragma unroll
    for (int c = 0; c < nch; ++c) {
      const int col = (c * 32 + lane) * 8;
      if (col >= a.cols) continue;
      float t[8], g[8], w[8];
      if (NCH > 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = x[c][i];
      } else {
        load8(a.x, a.x_dt, x_off, col, a.cols, vec, 0.f, t);
      }
      load8(a.g, a.g_dt, g_off, col, a.cols, vec, 0.f, g);
      load8(a.w, a.w_dt, 0, col, a.cols, vec, 0.f, w);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const bool in = col + i < a.cols;
        const float xh = in ? (t[i] - mu) * rstd : 0.f;
        const float uu = in ? g[i] * w[i] : 0.f;
        su += uu;
        sux = fmaf(uu, xh, sux);
        if (NCH > 0) {
          x[c][i] = xh; u[c][i] = uu;
          sw[c][i] = fmaf(g[i], xh, sw[c][i]);
          sc[c][i] += in ? g[i] : 0.f;
        } else if (in) {
          my_w[col + i] = fmaf(g[i], xh, my_w[col + i]);
          my_c[col + i] += g[i];
        }
      }
    }
    const float mean_u = warp_sum(su) * inv_n, mean_ux = warp_sum(sux) * inv_n;
    const float k = a.beta_x * rstd;
    // pass 2: dX = beta_x rstd (u - mean(u) - xhat mean(u xhat))
#pragma unroll
    for (int c = 0; c < nch; ++c) {
      const int col = (c * 32 + lane) * 8;
      if (col >= a.cols) continue;
      float d[8];
      if (NCH > 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) d[i] = k * (u[c][i] - mean_u - x[c][i] * mean_ux);
      } else {
        float t[8], g[8], w[8];
        load8(a.x, a.x_dt, x_off, col, a.cols, vec, 0.f, t);
        load8(a.g, a.g_dt, g_off, col, a.cols, vec, 0.f, g);
        load8(a.w, a.w_dt, 0, col, a.cols, vec, 0.f, w);
#pragma unroll
        for (int i = 0; i < 8; ++i) d[i] = k * (g[i] * w[i] - mean_u - (t[i] - mu) * rstd * mean_ux);
      }
      ln_store8<COPY>(a, row, col, vec, d);
    }
  }
  // ---- combine the CTA's warps in warp order; one partial row (G xhat sums, then G sums) per CTA
  float* dst = a.partial + (size_t)blockIdx.x * 2 * a.cols;
  if (NCH > 0) {
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
      __syncthreads();
#pragma unroll
      for (int c = 0; c < (NCH > 0 ? NCH : 1); ++c) {
        const int col = (c * 32 + lane) * 8;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (col + i < a.cols) ln_smem[(size_t)warp * a.cols + col + i] = pass == 0 ? sw[c][i] : sc[c][i];
      }
      __syncthreads();
      for (int j = threadIdx.x; j < a.cols; j += blockDim.x) {
        float s = 0.f;
        for (int wq = 0; wq < nw; ++wq) s += ln_smem[(size_t)wq * a.cols + j];
        dst[(size_t)pass * a.cols + j] = s;
      }
    }
  } else {
    __syncthreads();
    for (int j = threadIdx.x; j < 2 * a.cols; j += blockDim.x) {
      const int which = j >= a.cols, col = j - which * a.cols;
      float s = 0.f;
      for (int wq = 0; wq < nw; ++wq) s += ln_smem[((size_t)wq * 2 + which) * a.cols + col];
      dst[j] = s;
    }
  }
}

// ---------------------------------------------------------------- 16-bit inputs, rows in registers
// The common case (BF16 / F16 activations and gradients, rows of at most 2048 elements, aligned) of the forward pass
// gets persistent warps that fetch their next row, still packed, before working on the current one,
// and read the weight (and bias) from a float32 copy in shared memory; the backward pass has two kernels further down.

// Mean and reciprocal standard deviation of a row held as floats (zeros beyond the row's end).
template <int NCH>
__device__ __forceinline__ void stats_regs(const float (&x)[NCH][8], int lane, int cols, float eps, float& mu, float& rstd) {
  float s = 0.f;
#pragma unroll
  for (int c = 0; c < NCH; ++c)
#pragma unroll
    for (int i = 0; i < 8; ++i) s += x[c][i];
  mu = warp_sum(s) / (float)cols;
  float q = 0.f;
#pragma unroll
  for (int c = 0; c < NCH; ++c) {
    if ((c * 32 + lane) * 8 < cols) {
#pragma unroll
      for (int i = 0; i < 8; ++i) { const float d = x[c][i] - mu; q = fmaf(d, d, q); }
    }
  }
  rstd = rsqrtf(warp_sum(q) / (float)cols + eps);
}

template <int NCH, bool COPY>
__global__ void __launch_bounds__(kLnThreads, NCH <= 4 ? 3 : 2) ln_fwd16_kernel(const LnArgs a) {
  extern __shared__ __align__(16) float ln_smem[];                         // w[cols], c[cols] as float32
  float* w_s = ln_smem;
  float* c_s = ln_smem + a.cols;
  const int zero = ptx::grid_wait_previous();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t stride = (int64_t)gridDim.x * nw;
  int64_t row = (int64_t)blockIdx.x * nw + warp + zero;
  uint4 cur[NCH], nxt[NCH];
  if (row < a.rows) load_row16<NCH>(a.x, row * a.x_ld, lane, a.cols, cur);   // the first row and w, c are on their way together
  for (int j = threadIdx.x; j < a.cols; j += blockDim.x) { w_s[j] = load_one(a.w, a.w_dt, j + zero); c_s[j] = load_one(a.c, a.c_dt, j + zero); }
  __syncthreads();
  for (; row < a.rows; row += stride) {
    if (row + stride < a.rows) load_row16<NCH>(a.x, (row + stride) * a.x_ld, lane, a.cols, nxt);
    float x[NCH][8];
#pragma unroll
    for (int c = 0; c < NCH; ++c) unpack16x8(cur[c], a.x_dt, x[c]);
    float mu, rstd;
    stats_regs<NCH>(x, lane, a.cols, a.eps, mu, rstd);
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const int col = (c * 32 + lane) * 8;
      if (col < a.cols) {
        const float4 w0 = *reinterpret_cast<const float4*>(w_s + col), w1 = *reinterpret_cast<const float4*>(w_s + col + 4);
        const float4 b0 = *reinterpret_cast<const float4*>(c_s + col), b1 = *reinterpret_cast<const float4*>(c_s + col + 4);
        const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
        const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        float t[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = fmaf(w[i], (x[c][i] - mu) * rstd, b[i]);
        ln_store8<COPY>(a, row, col, true, t);
      }
    }
#pragma unroll
    for (int c = 0; c < NCH; ++c) cur[c] = nxt[c];
  }
}

// Rows beyond what L2 holds, with a gradient of X's 16-bit type: one warp per row.
//
// The rows reach the SM through a ring of kLnStages slots per warp in shared memory, filled by bulk
// copies (cp.async.bulk, completion counted on one mbarrier per slot): with one row per warp in
// registers the kernel is bound by memory latency (a few tens of KB in flight per SM), the ring keeps
// kLnStages rows per warp in flight.  A wait on a slot is bounded; if it ever runs out the warp reads
// that row and all later ones with ordinary loads (same result), and before leaving it gives the
// copies it issued time to land.
constexpr int kLnStages = 3;
constexpr uint32_t kLnWaitLimit = 1u << 20;

// XBF: X (and a 16-bit gradient) are BF16 rather than F16; fixed at compile time, because a run-time choice
// in the unpacking costs more instructions than the arithmetic it feeds.
template <int NCH, bool XBF, bool COPY>
__global__ void __launch_bounds__(128, 3) ln_bwd16_kernel(const LnArgs a) {
  extern __shared__ __align__(16) float ln_smem[];             // w[cols] as float32, [warps][cols] for the combine, the ring, its mbarriers
  float* w_s = ln_smem;                                        // NCH * 256 floats
  float* comb = ln_smem + NCH * 256;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t xb = (uint32_t)a.cols * 2u, gb = xb, slot = xb + gb;
  char* ring_gen = reinterpret_cast<char*>(comb + (size_t)nw * a.cols) + (size_t)warp * kLnStages * slot;
  const uint32_t ring = ptx::smem_addr(ring_gen);
  const uint32_t bars = ptx::smem_addr(reinterpret_cast<char*>(comb + (size_t)nw * a.cols) + (size_t)nw * kLnStages * slot) +
                        8u * (uint32_t)(warp * kLnStages);
  if (lane == 0) {
    for (int st = 0; st < kLnStages; ++st) ptx::mbar_init(bars + 8u * st, 1);
    ptx::mbar_init_fence();
  }
  // w in shared memory, laid out for conflict-free 16-byte reads: a lane's eight consecutive weights
  // (columns 8 q .. 8 q + 7) are split into a low and a high half; low halves at [4 q, 4 q + 4), high halves
  // kLnHi floats further.
  const int kLnHi = NCH * 32 * 4;
  const int zero = ptx::grid_wait_previous();
  for (int j = threadIdx.x + zero; j < a.cols; j += blockDim.x)
    w_s[(j >> 3) * 4 + (j & 3) + ((j & 4) ? kLnHi : 0)] = load_one(a.w, a.w_dt, j);
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * nw;
  const float inv_n = 1.0f / (float)a.cols;
  f32x2 sw[NCH][4], sc[NCH][4];                                // column sums of g * xhat and of g, as float32 pairs
#pragma unroll
  for (int c = 0; c < NCH; ++c)
#pragma unroll
    for (int j = 0; j < 4; ++j) { sw[c][j] = pack2(0.f, 0.f); sc[c][j] = pack2(0.f, 0.f); }
  int64_t row = (int64_t)blockIdx.x * nw + warp + zero;
  auto issue = [&](int64_t r, int st) {                        // lane 0
    const uint32_t bar = bars + 8u * st;
    ptx::mbar_expect_tx(bar, slot);
    ptx::bulk_load_1d(ring + st * slot, static_cast<const char*>(a.x) + r * a.x_ld * 2, xb, bar);
    ptx::bulk_load_1d(ring + st * slot + xb, static_cast<const char*>(a.g) + r * a.g_ld * 2, gb, bar);
  };
  int issued = 0;                                              // rows asked for so far (warp-uniform)
  for (; issued < kLnStages && row + issued * stride < a.rows; ++issued)
    if (lane == 0) issue(row + issued * stride, issued);
  bool direct = false;                                         // ordinary loads instead of the ring, after a wait ran out
  int it = 0, unconsumed = 0;                                  // unconsumed: first row whose copy was never waited for
  uint4 cx[NCH], cg[NCH];
  for (; row < a.rows; row += stride, ++it) {
    const int st = it % kLnStages;
    const uint32_t parity = (uint32_t)(it / kLnStages) & 1u;
    if (!direct) {
      bool ok = false;
      for (uint32_t k = 0; k < kLnWaitLimit && !(ok = ptx::mbar_try_wait(bars + 8u * st, parity)); ++k) {}
      direct = !__all_sync(0xffffffffu, ok);
      if (direct) unconsumed = it;
    }
    if (!direct) {
      const char* sx = ring_gen + (size_t)st * slot;
#pragma unroll
      for (int c = 0; c < NCH; ++c) {
        const int col = (c * 32 + lane) * 8;
        if (col < a.cols) {
          cx[c] = *reinterpret_cast<const uint4*>(sx + col * 2);
          cg[c] = *reinterpret_cast<const uint4*>(sx + xb + col * 2);
        } else {
          cx[c] = make_uint4(0, 0, 0, 0);
          cg[c] = make_uint4(0, 0, 0, 0);
        }
      }
      __syncwarp();                                            // every lane holds its part: the slot can be refilled
      const int64_t nxt = row + (int64_t)kLnStages * stride;
      if (nxt < a.rows) {
        if (lane == 0) issue(nxt, st);
        ++issued;
      }
    } else {
      load_row16<NCH>(a.x, row * a.x_ld, lane, a.cols, cx);
      load_row16<NCH>(a.g, row * a.g_ld, lane, a.cols, cg);
    }
    // From here on the row is worked on as pairs of float32 in 64-bit registers (add / mul / fma .f32x2):
    // the kernel is bound by instruction issue, and the packed forms halve the arithmetic instructions.
    f32x2 xp[NCH][4];
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const uint32_t wx[4] = {cx[c].x, cx[c].y, cx[c].z, cx[c].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 f = XBF ? unpack_bf16x2(wx[j]) : unpack_f16x2(wx[j]);
        xp[c][j] = pack2(f.x, f.y);
      }
    }
    auto g_pair = [&](int c, int j) -> f32x2 {                 // gradient values 2 j, 2 j + 1 of chunk c
      const uint4& r = cg[c];
      const uint32_t w = j == 0 ? r.x : j == 1 ? r.y : j == 2 ? r.z : r.w;
      const float2 f = XBF ? unpack_bf16x2(w) : unpack_f16x2(w);
      return pack2(f.x, f.y);
    };
    auto w_pairs = [&](int col, f32x2 (&w2)[4]) {
      const ulonglong2 lo = *reinterpret_cast<const ulonglong2*>(w_s + (col >> 1)), hi = *reinterpret_cast<const ulonglong2*>(w_s + (col >> 1) + kLnHi);
      w2[0] = lo.x; w2[1] = lo.y; w2[2] = hi.x; w2[3] = hi.y;
    };
    // mean, then variance about the mean (chunks beyond the row's end hold zeros and are left out of the second sum)
    f32x2 acc = pack2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < NCH; ++c)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc = add2(acc, xp[c][j]);
    float lo, hi;
    unpack2(acc, lo, hi);
    const float mu = warp_sum(lo + hi) * inv_n;
    const f32x2 neg_mu = splat2(-mu);
    acc = pack2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      if ((c * 32 + lane) * 8 < a.cols) {
#pragma unroll
        for (int j = 0; j < 4; ++j) { const f32x2 dm = add2(xp[c][j], neg_mu); acc = fma2(dm, dm, acc); }
      }
    }
    unpack2(acc, lo, hi);
    const float rstd = rsqrtf(warp_sum(lo + hi) * inv_n + a.eps);
    const f32x2 rstd2 = splat2(rstd), shift2 = splat2(-mu * rstd);
    f32x2 su2 = pack2(0.f, 0.f), sux2 = pack2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const int col = (c * 32 + lane) * 8;
      if (col < a.cols) {
        f32x2 w2[4];
        w_pairs(col, w2);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const f32x2 g2 = g_pair(c, j);
          const f32x2 xh = fma2(xp[c][j], rstd2, shift2);      // normalised input, kept for the second loop
          xp[c][j] = xh;
          const f32x2 uu = mul2(g2, w2[j]);
          su2 = add2(su2, uu);
          sux2 = fma2(uu, xh, sux2);
          sw[c][j] = fma2(g2, xh, sw[c][j]);
          sc[c][j] = add2(sc[c][j], g2);
        }
      }
    }
    unpack2(su2, lo, hi);
    const float mean_u = warp_sum(lo + hi) * inv_n;
    unpack2(sux2, lo, hi);
    const float mean_ux = warp_sum(lo + hi) * inv_n;
    const float k = a.beta_x * rstd;
    const f32x2 k2 = splat2(k), c0 = splat2(-k * mean_u), c1 = splat2(-k * mean_ux);
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const int col = (c * 32 + lane) * 8;
      if (col < a.cols) {
        f32x2 w2[4];
        w_pairs(col, w2);
        float d[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // k (g w - mean_u - xh mean_ux)
          const f32x2 t = fma2(mul2(g_pair(c, j), w2[j]), k2, c0);
          unpack2(fma2(xp[c][j], c1, t), d[2 * j], d[2 * j + 1]);
        }
        ln_store8<COPY>(a, row, col, true, d);
      }
    }
  }
  if (direct && lane == 0) {
    // copies issued but never consumed: one per slot at most
    for (int k = unconsumed; k < issued; ++k) {
      const uint32_t bar = bars + 8u * (k % kLnStages), parity = (uint32_t)(k / kLnStages) & 1u;
      for (uint32_t n = 0; n < kLnWaitLimit && !ptx::mbar_try_wait(bar, parity); ++n) {}
    }
  }
  float* dst = a.partial + (size_t)blockIdx.x * 2 * a.cols;
#pragma unroll
  for (int pass = 0; pass < 2; ++pass) {
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const int col = (c * 32 + lane) * 8;
      if (col < a.cols) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<f32x2*>(comb + (size_t)warp * a.cols + col + 2 * j) = pass == 0 ? sw[c][j] : sc[c][j];
      }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < a.cols; j += blockDim.x) {
      float s = 0.f;
      for (int wq = 0; wq < nw; ++wq) s += comb[(size_t)wq * a.cols + j];
      dst[(size_t)pass * a.cols + j] = s;
    }
  }
}

// Sums over the warp of four values per lane; lane l gets that of v[l & 3].  (Six shuffles instead of twenty.)
__device__ __forceinline__ float warp_sum4(const float (&v)[4], int lane) {
  const bool b0 = lane & 1, b1 = lane & 2;
  float x = (b0 ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, b0 ? v[0] : v[1], 1);
  const float z = (b0 ? v[3] : v[2]) + __shfl_xor_sync(0xffffffffu, b0 ? v[2] : v[3], 1);
  x = (b1 ? z : x) + __shfl_xor_sync(0xffffffffu, b1 ? x : z, 2);
#pragma unroll
  for (int o = 4; o <= 16; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// The same for the B rows of a turn, four or one.
__device__ __forceinline__ float sum_rows(const float (&v)[4], int lane) { return warp_sum4(v, lane); }
__device__ __forceinline__ float sum_rows(const float (&v)[1], int) { return warp_sum(v[0]); }

// The 16-bit cases of the backward pass (rows of at most 2048 elements): a row belongs to wpr = cols / 256 warps, eight columns a lane, so
// that a lane's share of the column sums is 16 registers and two CTAs of eight warps fit an SM; the warps of a row take four rows at
// a time, which hides the latency of their loads and shares two exchanges through shared memory among four rows: the means, then the
// sums of (x - mu)^2, g w and g w (x - mu).  B: rows of a turn, four, or one where each group has but one row (300 x 128 4.4 -> 3.9 us, 100 x 512
// 5.3 -> 4.6: less code to fetch).  G32: the gradient is float32 (the gradient of a layer's output often is) instead of the 16-bit
// type of X.  XBF: X (and a 16-bit gradient) are BF16 rather than F16.  Bound: latency of the exchanges, 16 warps an SM; beyond L2
// memory.  us, a warp per row -> this, BF16 with an FP8 copy: 8192 x 1024 22.9 -> 18.3, its float32 gradient 25.9 -> 19.0, 2048 x 768 12.2 -> 8.2, 4096 x
// 256 9.1 -> 5.8, 256 x 1024 9.1 -> 6.3; 2048 x 2048, which the general kernel took, 65 -> 13.
constexpr int kLnBatch = 4, kLnCtasPerSm = 2;
enum LnOut { kLnSame = 0, kLnSameE4 = 1, kLnSameE5 = 2, kLnAny = 3, kLnAnyCopy = 4 };   // dX of X's type (and its FP8 copy), or of any type
template <bool G32, bool XBF, int OUT, int B>
__global__ void __launch_bounds__(kLnThreads, kLnCtasPerSm) ln_bwd_rows_kernel(const LnArgs a, const int wpr) {
  extern __shared__ __align__(16) float ln_smem[];             // exchanges [warps][1 + 3][4], then the combine [groups][2][cols]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int groups = nw / wpr, group = warp / wpr, col = ((warp - group * wpr) * 32 + lane) * 8;
  const bool has = col < a.cols;
  float4* means = reinterpret_cast<float4*>(ln_smem) + group * wpr;                       // of this row group: one per warp
  float4* sums = reinterpret_cast<float4*>(ln_smem) + nw + 3 * group * wpr;               // three per warp
  float* comb = ln_smem + 16 * nw;
  const float inv_n = 1.0f / (float)a.cols, inv_rest = fmaf(-inv_n, (float)a.cols, 1.0f) * inv_n;
  // s / cols as a division rounds it, or the value next to that
  auto mean = [&](float s) { return fmaf(s, inv_n, isinf(s) ? 0.f : s * inv_rest); };
  auto meet = [&]() { ptx::named_barrier_sync(1 + group, 32 * wpr); };
  const int zero = ptx::grid_wait_previous();
  f32x2 w2[4], sw[4], sc[4];                                   // weights; column sums of g * xhat and of g
  {
    float w[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (has) load8(a.w, a.w_dt, 0, col + zero, a.cols, true, 0.f, w);
#pragma unroll
    for (int j = 0; j < 4; ++j) { w2[j] = pack2(w[2 * j], w[2 * j + 1]); sw[j] = sc[j] = pack2(0.f, 0.f); }
  }
  auto unpack = [](uint32_t w) { const float2 f = XBF ? unpack_bf16x2(w) : unpack_f16x2(w); return pack2(f.x, f.y); };
  // The rows stay packed between the exchanges: without this the compiler keeps what it has unpacked, and spills.
  auto packed = [](uint4& r) { asm volatile("" : "+r"(r.x), "+r"(r.y), "+r"(r.z), "+r"(r.w)); };
  auto word = [](const uint4& r, int j) { return j == 0 ? r.x : j == 1 ? r.y : j == 2 ? r.z : r.w; };
  const int64_t stride = (int64_t)gridDim.x * groups;
  for (int64_t row0 = (int64_t)blockIdx.x * groups + group + zero; row0 < a.rows; row0 += B * stride) {
    const int64_t rest = (a.rows - row0 + stride - 1) / stride;
    const int here = rest < B ? (int)rest : B;   // rows of this turn
    uint4 cx[B], cg[B], ch[G32 ? B : 1];  // packed rows; a float32 gradient takes two vectors
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int64_t row = row0 + b * stride;
      cx[b] = cg[b] = make_uint4(0, 0, 0, 0);
      if (G32) ch[G32 ? b : 0] = make_uint4(0, 0, 0, 0);
      if (has && b < here) {
        cx[b] = __ldg(reinterpret_cast<const uint4*>(static_cast<const char*>(a.x) + (row * a.x_ld + col) * 2));
        const uint4* g = reinterpret_cast<const uint4*>(static_cast<const char*>(a.g) + (row * a.g_ld + col) * (G32 ? 4 : 2));
        cg[b] = __ldg(g);
        if (G32) ch[G32 ? b : 0] = __ldg(g + 1);
      }
    }
    auto g_pair = [&](int b, int j) -> f32x2 {                 // gradient values 2 j, 2 j + 1 of row b
      if (!G32) return unpack(word(cg[b], j));
      const uint4& r = j < 2 ? cg[b] : ch[G32 ? b : 0];
      return j & 1 ? pack2(__uint_as_float(r.z), __uint_as_float(r.w)) : pack2(__uint_as_float(r.x), __uint_as_float(r.y));
    };
    // ---- means
    float v[B], lo, hi;
#pragma unroll
    for (int b = 0; b < B; ++b) {
      v[b] = 0.f;
      if (b >= here) continue;
      unpack2(add2(add2(unpack(cx[b].x), unpack(cx[b].y)), add2(unpack(cx[b].z), unpack(cx[b].w))), lo, hi);
      v[b] = lo + hi;
    }
    const float m = sum_rows(v, lane);
    float mu[B] = {};
    if (wpr == 1) {
#pragma unroll
      for (int b = 0; b < B; ++b) mu[b] = __shfl_sync(0xffffffffu, m, b);
    } else {
      if (lane < B) reinterpret_cast<float*>(&means[warp - group * wpr])[lane] = m;
      meet();
      for (int k = 0; k < wpr; ++k) {
        const float4 t = means[k];
        mu[0] += t.x;
        if constexpr (B == 4) { mu[1] += t.y; mu[2] += t.z; mu[3] += t.w; }
      }
    }
#pragma unroll
    for (int b = 0; b < B; ++b) packed(cx[b]);
    // ---- variance about the mean, sums of u = g w and of u (x - mu)
    float q[B], su[B], sd[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      q[b] = su[b] = sd[b] = 0.f;
      if (b >= here) continue;
      mu[b] = mean(mu[b]);
      const f32x2 neg = splat2(-mu[b]);
      f32x2 q2 = pack2(0.f, 0.f), u2 = q2, d2 = q2;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const f32x2 d = add2(unpack(word(cx[b], j)), neg), u = mul2(g_pair(b, j), w2[j]);
        q2 = fma2(d, d, q2); u2 = add2(u2, u); d2 = fma2(u, d, d2);
      }
      unpack2(q2, lo, hi); q[b] = has ? lo + hi : 0.f;
      unpack2(u2, lo, hi); su[b] = lo + hi;                    // (zero beyond the row's end: g and w are)
      unpack2(d2, lo, hi); sd[b] = lo + hi;
    }
    const float rq = sum_rows(q, lane), ru = sum_rows(su, lane), rd = sum_rows(sd, lane);
    if (wpr == 1) {
#pragma unroll
      for (int b = 0; b < B; ++b) { q[b] = __shfl_sync(0xffffffffu, rq, b); su[b] = __shfl_sync(0xffffffffu, ru, b); sd[b] = __shfl_sync(0xffffffffu, rd, b); }
    } else {
      if (lane < B) {
        float* t = reinterpret_cast<float*>(&sums[3 * (warp - group * wpr)]) + lane;
        t[0] = rq; t[4] = ru; t[8] = rd;
      }
      meet();
#pragma unroll
      for (int b = 0; b < B; ++b) q[b] = su[b] = sd[b] = 0.f;
      for (int k = 0; k < wpr; ++k) {
        const float4 t0 = sums[3 * k], t1 = sums[3 * k + 1], t2 = sums[3 * k + 2];
        q[0] += t0.x; su[0] += t1.x; sd[0] += t2.x;
        if constexpr (B == 4) {
          q[1] += t0.y; q[2] += t0.z; q[3] += t0.w;
          su[1] += t1.y; su[2] += t1.z; su[3] += t1.w;
          sd[1] += t2.y; sd[2] += t2.z; sd[3] += t2.w;
        }
      }
    }
#pragma unroll
    for (int b = 0; b < B; ++b) { packed(cx[b]); packed(cg[b]); }
    // ---- dX = beta_x rstd (u - mean(u) - xhat mean(u xhat)), column sums
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int64_t row = row0 + b * stride;
      if (b >= here) continue;
      const float rstd = rsqrtf(mean(q[b]) + a.eps), k = a.beta_x * rstd;
      const f32x2 rstd2 = splat2(rstd), neg = splat2(-mu[b]), k2 = splat2(k), c0 = splat2(-k * (su[b] * inv_n)),
                  c1 = splat2(-k * (sd[b] * rstd * inv_n));
      float d[8];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const f32x2 g2 = g_pair(b, j), xh = mul2(add2(unpack(word(cx[b], j)), neg), rstd2);     // (exact where the mean is far above the spread)
        sw[j] = fma2(g2, xh, sw[j]);
        sc[j] = add2(sc[j], g2);
        unpack2(fma2(xh, c1, fma2(mul2(g2, w2[j]), k2, c0)), d[2 * j], d[2 * j + 1]);
      }
      if (OUT >= kLnAny) {
        if (has) ln_store8<OUT == kLnAnyCopy>(a, row, col, true, d);
      } else if (has) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = XBF ? pack_bf16x2(d[2 * j], d[2 * j + 1]) : pack_f16x2(d[2 * j], d[2 * j + 1]);
        *reinterpret_cast<uint4*>(static_cast<char*>(a.out) + (row * a.out_ld + col) * 2) = make_uint4(w[0], w[1], w[2], w[3]);
        if (OUT != kLnSame) {
#pragma unroll
          for (int j = 0; j < 4; ++j) { const float2 t = XBF ? unpack_bf16x2(w[j]) : unpack_f16x2(w[j]); d[2 * j] = t.x; d[2 * j + 1] = t.y; }
          constexpr bool E5 = OUT == kLnSameE5;
          *reinterpret_cast<uint2*>(static_cast<char*>(a.q) + row * a.q_ld + col) =
              make_uint2(cvt_fp8x4<E5>(d[0], d[1], d[2], d[3]), cvt_fp8x4<E5>(d[4], d[5], d[6], d[7]));
        }
      }
    }
  }
  // ---- combine the CTA's row groups in their order; one partial row (G xhat sums, then G sums) per CTA
  if (has) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      *reinterpret_cast<f32x2*>(comb + (size_t)(2 * group) * a.cols + col + 2 * j) = sw[j];
      *reinterpret_cast<f32x2*>(comb + (size_t)(2 * group + 1) * a.cols + col + 2 * j) = sc[j];
    }
  }
  __syncthreads();
  float* dst = a.partial + (size_t)blockIdx.x * 2 * a.cols;
  for (int j = threadIdx.x; j < 2 * a.cols; j += blockDim.x) {
    float t = 0.f;
    for (int g = 0; g < groups; ++g) t += comb[(size_t)g * 2 * a.cols + j];
    dst[j] = t;
  }
}

// dw_j = beta * sum over CTAs of partial[cta][0][j], dc_j likewise from partial[cta][1][j].
// One CTA per 32 columns of the 2 * cols sums: 32 groups of 32 threads each add every 32nd partial row
// in order (four independent partial sums per thread, combined in a fixed order), then the groups are
// added in order.
constexpr int kLnReduceGroups = 32;
__global__ void __launch_bounds__(32 * kLnReduceGroups) ln_bwd_reduce_kernel(const float* partial, int nparts, int cols, float beta,
                                                                             void* dw, int dw_dt, void* dc, int dc_dt) {
  __shared__ float acc[kLnReduceGroups][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int j = blockIdx.x * 32 + tx;               // index into [2][cols]
  float s4[4] = {0.f, 0.f, 0.f, 0.f};
  const int zero = ptx::grid_wait_previous();
  if (j < 2 * cols) {
    int p = ty + zero;
    for (; p + 3 * kLnReduceGroups < nparts; p += 4 * kLnReduceGroups) {
#pragma unroll
      for (int u = 0; u < 4; ++u) s4[u] += partial[(size_t)(p + u * kLnReduceGroups) * 2 * cols + j];
    }
#pragma unroll
    for (int u = 0; u < 3; ++u)                     // at most three rows are left for this group
      if (p + u * kLnReduceGroups < nparts) s4[u] += partial[(size_t)(p + u * kLnReduceGroups) * 2 * cols + j];
  }
  acc[ty][tx] = (s4[0] + s4[1]) + (s4[2] + s4[3]);
  __syncthreads();
  if (ty == 0 && j < 2 * cols) {
    float t = 0.f;
#pragma unroll
    for (int q = 0; q < kLnReduceGroups; ++q) t += acc[q][tx];
    t *= beta;
    if (j < cols) store_one(dw, dw_dt, j, t);
    else store_one(dc, dc_dt, j - cols, t);
  }
}

static bool ln_rows_aligned(const us_mat* m) {
  return reinterpret_cast<uintptr_t>(m->ptr) % 16 == 0 && (m->ld * dtype_size(m->dtype)) % 16 == 0;
}
// Eight codes of an FP8 copy are stored at once.
static bool copy_rows_aligned(const us_mat* q) { return !q || (reinterpret_cast<uintptr_t>(q->ptr) % 8 == 0 && q->ld % 8 == 0); }
static bool is_float_in(int dt) { return dt == US_F32 || dt == US_BF16 || dt == US_F16; }

static us_status check_matrix(const us_mat* m, const us_mat* like, bool input) {
  if (!m || m->rows < 0 || m->cols < 0 || m->ld < m->cols) return US_ERR_INVALID_ARG;
  if (like && (m->rows != like->rows || m->cols != like->cols)) return US_ERR_INVALID_ARG;
  if (m->rows * m->cols > 0 && !m->ptr) return US_ERR_INVALID_ARG;
  if (m->cols > 0x7ffffff0) return US_ERR_INVALID_ARG;
  if (input ? !is_float_in(m->dtype) : !(m->dtype >= US_F32 && m->dtype <= US_E5M2)) return US_ERR_UNSUPPORTED;
  if (m->ptr && reinterpret_cast<uintptr_t>(m->ptr) % dtype_size(m->dtype)) return US_ERR_ALIGNMENT;
  return US_OK;
}
// The FP8 copy of a result that is not FP8 itself.
static us_status check_copy(const us_mat* q, const us_mat* of) {
  if (!q) return US_OK;
  const us_status s = check_matrix(q, of, false);
  if (s != US_OK) return s;
  return (q->dtype == US_E4M3 || q->dtype == US_E5M2) && is_float_in(of->dtype) ? US_OK : US_ERR_UNSUPPORTED;
}
// A parameter vector: 1 x cols.
static us_status check_vector(const us_mat* v, int64_t cols, bool input) {
  if (!v || v->rows != 1 || v->cols != cols || v->ld < v->cols) return US_ERR_INVALID_ARG;
  if (cols > 0 && !v->ptr) return US_ERR_INVALID_ARG;
  if (input ? !is_float_in(v->dtype) : !(v->dtype == US_F32 || v->dtype == US_BF16 || v->dtype == US_F16)) return US_ERR_UNSUPPORTED;
  if (v->ptr && reinterpret_cast<uintptr_t>(v->ptr) % dtype_size(v->dtype)) return US_ERR_ALIGNMENT;
  return US_OK;
}

// CTAs of a backward kernel: `rows_each` rows in flight per CTA, at most `per_sm` CTAs per SM.
static int ln_bwd_grid(int64_t rows, int rows_each = kLnWarps, int per_sm = 2) {
  const int sms = host::sm_count();
  if (sms <= 0) return 0;
  const int64_t want = (rows + rows_each - 1) / rows_each;
  const int64_t cap = (int64_t)sms * per_sm;
  return (int)(want < cap ? want : cap);
}

constexpr int kLnFastWarps = 4, kLnFastPerSm = 3;   // of ln_bwd16_kernel
// Rows of partial sums that a workspace holds, whichever kernel the call takes: a CTA writes one.
static int ln_bwd_partials(int64_t rows) { return std::max(ln_bwd_grid(rows), ln_bwd_grid(rows, kLnFastWarps, kLnFastPerSm)); }

template <bool COPY>
static us_status ln_fwd_launch(const LnArgs& a, cudaStream_t st) {
  const int64_t grid64 = (a.rows + kLnWarps - 1) / kLnWarps;
  if (grid64 > 0x7fffffff) return US_ERR_INVALID_ARG;
  const int grid = (int)grid64, nch = (a.cols + 255) / 256;
  if (a.vec_ok && (a.x_dt == US_BF16 || a.x_dt == US_F16) && nch <= 8) {
    const int sms = host::sm_count();
    if (sms <= 0) return US_ERR_CUDA;
    // resident CTAs, warps walk the rows; three an SM where their registers fit (BF16, two -> three: 8192 x 1024 9.8 -> 9.4 us, 8192 x 256
    // 4.6 -> 4.2, 32768 x 128 10.5 -> 9.0, 32768 x 1024 28.3 -> 28.2; up to 1000 rows, which are no more CTAs than SMs, equal)
    const int most = (nch <= 4 ? 3 : 2) * sms, pgrid = grid < most ? grid : most;
    const size_t smem = (size_t)2 * a.cols * sizeof(float);
    if (nch <= 1) return host::launch(ln_fwd16_kernel<1, COPY>, nullptr, pgrid, kLnThreads, smem, 1, st, a);
    if (nch <= 2) return host::launch(ln_fwd16_kernel<2, COPY>, nullptr, pgrid, kLnThreads, smem, 1, st, a);
    if (nch <= 4) return host::launch(ln_fwd16_kernel<4, COPY>, nullptr, pgrid, kLnThreads, smem, 1, st, a);
    return host::launch(ln_fwd16_kernel<8, COPY>, nullptr, pgrid, kLnThreads, smem, 1, st, a);
  }
  if (nch <= 1) ln_fwd_kernel<1, COPY><<<grid, kLnThreads, 0, st>>>(a);
  else if (nch <= 2) ln_fwd_kernel<2, COPY><<<grid, kLnThreads, 0, st>>>(a);
  else if (nch <= 4) ln_fwd_kernel<4, COPY><<<grid, kLnThreads, 0, st>>>(a);
  else if (nch <= 8) ln_fwd_kernel<8, COPY><<<grid, kLnThreads, 0, st>>>(a);
  else ln_fwd_kernel<0, COPY><<<grid, kLnThreads, 0, st>>>(a);
  return cudaGetLastError() == cudaSuccess ? US_OK : US_ERR_CUDA;
}

static us_status ln_fwd(const us_mat* X, const us_mat* w, const us_mat* c, float eps, const us_mat* Y, const us_mat* Yq, void* stream) {
  us_status s = check_matrix(X, nullptr, true);
  if (s == US_OK) s = check_matrix(Y, X, false);
  if (s == US_OK) s = check_vector(w, X->cols, true);
  if (s == US_OK) s = check_vector(c, X->cols, true);
  if (s == US_OK) s = check_copy(Yq, Y);
  if (s != US_OK) return s;
  if (!(eps >= 0.f)) return US_ERR_INVALID_ARG;
  if (X->rows == 0 || X->cols == 0) return US_OK;
  LnArgs a{};
  a.x = X->ptr; a.x_dt = X->dtype; a.x_ld = X->ld;
  a.w = w->ptr; a.w_dt = w->dtype; a.c = c->ptr; a.c_dt = c->dtype;
  a.out = Y->ptr; a.out_dt = Y->dtype; a.out_ld = Y->ld;
  if (Yq) { a.q = Yq->ptr; a.q_dt = Yq->dtype; a.q_ld = Yq->ld; }
  a.rows = X->rows; a.cols = (int)X->cols; a.eps = eps; a.beta_x = 1.f;
  a.vec_ok = ln_rows_aligned(X) && ln_rows_aligned(Y) && ln_rows_aligned(w) && ln_rows_aligned(c) && copy_rows_aligned(Yq) && X->cols % 8 == 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return Yq ? ln_fwd_launch<true>(a, st) : ln_fwd_launch<false>(a, st);
}

template <bool COPY>
static us_status ln_bwd_launch(const LnArgs& a, int grid, float beta_wc, const us_mat* dw, const us_mat* dc, cudaStream_t st) {
  const int nch = (a.cols + 255) / 256;
  int nparts = grid;
  // With no rows the first kernel still runs (one CTA) and writes zero partials, so dw = dc = 0.
  const bool rows16 = a.vec_ok && (a.x_dt == US_BF16 || a.x_dt == US_F16);
  // Large 16-bit cases (X and G no longer stay in L2), a warp per row with a ring of bulk copies, which keeps more of memory busy: from 16 M
  // elements on, with 513 to 1024 columns, whose CTAs hold two rows, from 14 M, up to 768 of them, six warps, from 7.5 M.  us, rows among warps / warp per
  // row, BF16: 10000 x 640 18.0 / 18.0, 12288 x 640 20.5 / 19.9, 14000 x 768 21.7 / 22.1, 20000 x 768 34.0 / 30.4, 26000 x 640 41.3 / 34.7; 14000 x 1024
  // 27.5 / 28.5, 16384 x 896 29.0 / 28.1, 16384 x 1024 32.1 / 31.0; 26000 x 512 24.1 / 25.8, 65536 x 512 56.5 / 53.4; a float32 gradient
  // 32768 x 1024 66 / 89, rows of at most 256 131072 x 256 48 / 75.
  const int64_t ring_from = nch == 2 ? 32 : nch == 3 ? 15 : 28;          // in half millions of elements
  if (rows16 && a.g_dt == a.x_dt && nch > 1 && nch <= 4 && a.rows * a.cols >= ring_from << 19) {
    nparts = ln_bwd_grid(a.rows, kLnFastWarps, kLnFastPerSm);
    const size_t smem = ((size_t)(nch <= 2 ? 2 : 4) * 256 + (size_t)kLnFastWarps * a.cols) * sizeof(float) + (size_t)kLnFastWarps * kLnStages * (a.cols * 4 + 8);
    const bool xbf = a.x_dt == US_BF16;
    void (*fn)(const LnArgs) = nch <= 2 ? (xbf ? ln_bwd16_kernel<2, true, COPY> : ln_bwd16_kernel<2, false, COPY>)
                                        : (xbf ? ln_bwd16_kernel<4, true, COPY> : ln_bwd16_kernel<4, false, COPY>);
    if (smem > 48 * 1024 && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return host::failed();
    const us_status launched = host::launch(fn, nullptr, nparts, 32 * kLnFastWarps, smem, 1, st, a);
    if (launched != US_OK) return launched;
  } else if (rows16 && nch <= kLnWarps && (a.g_dt == a.x_dt || a.g_dt == US_F32)) {
    const int groups = kLnWarps / nch;
    // Rows per group: four, fewer where that would be few CTAs, each of which is a partial row that the second kernel adds (us with 4 / 2 / 1: 1000 x
    // 384 5.4 / 5.4 / 6.2, 4096 x 256 5.6 / 6.2 / 6.6; with 2 / 1: 300 x 384 5.3 / 4.6, 600 x 256 4.8 / 4.2, 1200 x 256 4.9 / 5.1), and never more CTAs
    // than the workspace has partial rows (which binds few long rows: 16 x 2048 6.3 us with a CTA a row, 6.7 with one for four).
    const int64_t turns = (a.rows + kLnBatch * groups - 1) / (kLnBatch * groups);
    nparts = std::min(ln_bwd_grid(a.rows > 0 ? a.rows : 1, (turns >= 64 ? 4 : turns >= 32 ? 2 : 1) * groups, kLnCtasPerSm), ln_bwd_partials(a.rows > 0 ? a.rows : 1));
    const size_t smem = ((size_t)16 * nch * groups + (size_t)2 * groups * a.cols) * sizeof(float);
    const bool g32 = a.g_dt == US_F32, xbf = a.x_dt == US_BF16, one = (int64_t)nparts * groups >= a.rows;      // (a row for each group: no turns of four)
    const int out = a.out_dt != a.x_dt ? (COPY ? kLnAnyCopy : kLnAny) : !COPY ? kLnSame : a.q_dt == US_E5M2 ? kLnSameE5 : kLnSameE4;
    void (*fn)(const LnArgs, const int) = nullptr;
#define US_LN_PICK(OUT)                                                                            \
  fn = one ? (g32 ? (xbf ? ln_bwd_rows_kernel<true, true, OUT, 1> : ln_bwd_rows_kernel<true, false, OUT, 1>)                       \
                  : (xbf ? ln_bwd_rows_kernel<false, true, OUT, 1> : ln_bwd_rows_kernel<false, false, OUT, 1>))                    \
           : (g32 ? (xbf ? ln_bwd_rows_kernel<true, true, OUT, kLnBatch> : ln_bwd_rows_kernel<true, false, OUT, kLnBatch>)         \
                  : (xbf ? ln_bwd_rows_kernel<false, true, OUT, kLnBatch> : ln_bwd_rows_kernel<false, false, OUT, kLnBatch>))
    if constexpr (COPY) {
      if (out == kLnAnyCopy) US_LN_PICK(kLnAnyCopy);
      else if (out == kLnSameE5) US_LN_PICK(kLnSameE5);
      else US_LN_PICK(kLnSameE4);
    } else {
      if (out == kLnAny) US_LN_PICK(kLnAny);
      else US_LN_PICK(kLnSame);
    }
#undef US_LN_PICK
    const us_status launched = host::launch(fn, nullptr, nparts, 32 * nch * groups, smem, 1, st, a, nch);
    if (launched != US_OK) return launched;
  } else if (nch <= 4) {
    const size_t smem = (size_t)kLnWarps * a.cols * sizeof(float);
    if (nch <= 1) ln_bwd_kernel<1, COPY><<<grid, kLnThreads, smem, st>>>(a);
    else if (nch <= 2) ln_bwd_kernel<2, COPY><<<grid, kLnThreads, smem, st>>>(a);
    else ln_bwd_kernel<4, COPY><<<grid, kLnThreads, smem, st>>>(a);
  } else {
    const size_t smem = (size_t)4 * 2 * a.cols * sizeof(float);
    if (cudaFuncSetAttribute(ln_bwd_kernel<0, COPY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
      return host::failed();
    ln_bwd_kernel<0, COPY><<<grid, 128, smem, st>>>(a);
  }
  if (cudaGetLastError() != cudaSuccess) return US_ERR_CUDA;
  const int rgrid = (2 * a.cols + 31) / 32;
  return host::launch(ln_bwd_reduce_kernel, nullptr, rgrid, 32 * kLnReduceGroups, 0, 1, st, static_cast<const float*>(a.partial), nparts, a.cols, beta_wc, dw->ptr,
                      dw->dtype, dc->ptr, dc->dtype);
}

static us_status ln_bwd(const us_mat* X, const us_mat* w, const us_mat* G, float eps, float beta_x, float beta_wc, const us_mat* dX,
                        const us_mat* dXq, const us_mat* dw, const us_mat* dc, void* ws, size_t ws_bytes, void* stream) {
  us_status s = check_matrix(X, nullptr, true);
  if (s == US_OK) s = check_matrix(G, X, true);
  if (s == US_OK) s = check_matrix(dX, X, false);
  if (s == US_OK) s = check_vector(w, X->cols, true);
  if (s == US_OK) s = check_vector(dw, X->cols, false);
  if (s == US_OK) s = check_vector(dc, X->cols, false);
  if (s == US_OK) s = check_copy(dXq, dX);
  if (s != US_OK) return s;
  if (!(eps >= 0.f)) return US_ERR_INVALID_ARG;
  if (X->cols > kLnMaxBwdCols) return US_ERR_UNSUPPORTED;
  if (X->cols == 0) return US_OK;
  const int grid = ln_bwd_grid(X->rows > 0 ? X->rows : 1);
  if (grid <= 0) return US_ERR_CUDA;
  if (!ws || ws_bytes < ::us_layer_norm_bwd_workspace_bytes(X->rows > 0 ? X->rows : 1, X->cols)) return US_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(ws) % 16) return US_ERR_ALIGNMENT;
  LnArgs a{};
  a.x = X->ptr; a.x_dt = X->dtype; a.x_ld = X->ld;
  a.g = G->ptr; a.g_dt = G->dtype; a.g_ld = G->ld;
  a.w = w->ptr; a.w_dt = w->dtype;
  a.out = dX->ptr; a.out_dt = dX->dtype; a.out_ld = dX->ld;
  if (dXq) { a.q = dXq->ptr; a.q_dt = dXq->dtype; a.q_ld = dXq->ld; }
  a.partial = static_cast<float*>(ws);
  a.rows = X->rows; a.cols = (int)X->cols; a.eps = eps; a.beta_x = beta_x;
  a.vec_ok = ln_rows_aligned(X) && ln_rows_aligned(G) && ln_rows_aligned(dX) && ln_rows_aligned(w) &&
             copy_rows_aligned(dXq) && X->cols % 8 == 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return dXq ? ln_bwd_launch<true>(a, grid, beta_wc, dw, dc, st) : ln_bwd_launch<false>(a, grid, beta_wc, dw, dc, st);
}

}  // namespace us

using namespace us;

extern "C" size_t us_layer_norm_bwd_workspace_bytes(int64_t rows, int64_t cols) {
  if (rows <= 0 || cols <= 0) return 0;
  const int grid = ln_bwd_partials(rows);
  return (size_t)(grid > 0 ? grid : 1) * 2 * (size_t)cols * sizeof(float);
}

extern "C" us_status us_layer_norm_fwd(const us_mat* X, const us_mat* w, const us_mat* c, float eps, const us_mat* Y,
                                       void* stream) {
  return ln_fwd(X, w, c, eps, Y, nullptr, stream);
}
extern "C" us_status us_layer_norm_fwd_cast(const us_mat* X, const us_mat* w, const us_mat* c, float eps, const us_mat* Y,
                                            const us_mat* Yq, void* stream) {
  return Yq ? ln_fwd(X, w, c, eps, Y, Yq, stream) : US_ERR_INVALID_ARG;
}
extern "C" us_status us_layer_norm_bwd(const us_mat* X, const us_mat* w, const us_mat* G, float eps, float beta_x,
                                       float beta_wc, const us_mat* dX, const us_mat* dw, const us_mat* dc, void* ws,
                                       size_t ws_bytes, void* stream) {
  return ln_bwd(X, w, G, eps, beta_x, beta_wc, dX, nullptr, dw, dc, ws, ws_bytes, stream);
}
extern "C" us_status us_layer_norm_bwd_cast(const us_mat* X, const us_mat* w, const us_mat* G, float eps, float beta_x,
                                            float beta_wc, const us_mat* dX, const us_mat* dXq, const us_mat* dw, const us_mat* dc,
                                            void* ws, size_t ws_bytes, void* stream) {
  return dXq ? ln_bwd(X, w, G, eps, beta_x, beta_wc, dX, dXq, dw, dc, ws, ws_bytes, stream) : US_ERR_INVALID_ARG;
}
