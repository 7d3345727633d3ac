// Feed-forward sublayer of BF16 passes with few packed tokens, both projections in one kernel.
//
// As two kernels it was 1.4 us of work, a kernel boundary and 1.2 us more, and the second one's CTAs, for which the first one's left no registers, began to
// fetch their weights only once those had gone: 5.7 us a layer of a 512-wide model.  Here a CTA owns 64 hidden features: its warps split the
// input features for W1 (64 each), exchange their partial sums through shared memory, and then split the output features for W2 (64 each), whose
// contraction is over the CTA's own 64 hidden features: the hidden activations never leave the SM.  Both weight slices (128 KB for d = 512) are in
// registers before the dependency wait.  What remains is one round trip for the activations, two short rows of MMAs and one exchange.
// The price are d_ffn / 64 partial sums for the LayerNorm behind it (layernorm_parts_kernel: 0.3 us more than with four).  29 tokens, 512 wide: 1.5 us
// after the wait, 3.0 us a layer with the boundary behind it.  The kernels around it take 0.2 to 0.5 us longer than before for a reason that
// is not known (neither shares of shared memory, nor its grid, nor cold instruction caches), so that a decode iteration gains 4 us of the 14.
#pragma once

#include "attention_few.cuh"

namespace ad {
namespace few {

constexpr int FFN_SLICE = 64;            // hidden features per CTA
constexpr int FFN_MAX_PARTS = 32;
constexpr int FFN_MAX_ROWS = 160 * 32;   // most rows of partial sums: what the LayerNorm has to read outgrows the kernel that was saved
inline bool ffn_few_fits(int d, int F, int M_cap) {
  return d % 128 == 0 && d <= 64 * MAX_WARPS && F % FFN_SLICE == 0 && F / FFN_SLICE <= FFN_MAX_PARTS && (long)M_cap * (F / FFN_SLICE) <= FFN_MAX_ROWS;
}

struct FfnFewParams {
  const int* M_ptr;
  const bf16* x;         // [M_cap, d]
  const bf16 *w1, *w2;   // [F, d], [d, F]
  const float* b1;       // [F]
  float* out;            // [F / 64][M_cap, d] partial sums (no bias)
  size_t stride;         // M_cap * d
  int d, F;
};

// grid = (groups of 16-token tiles, F / 64), block = 32 * (d / 64): CTA (i, s) takes the tiles i, i + gridDim.x, ... for hidden features 64 s ..
__global__ void __launch_bounds__(32 * MAX_WARPS, 1)
ffn_few_kernel(const FfnFewParams p) {
  __shared__ __align__(16) float part[MAX_WARPS * AQ * O_LD];
  __shared__ __align__(16) bf16 hs[AQ * K_LD];
  trace_mark(TR_GEMM + EPI_ACT, 0);
  pdl_launch();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int nw = blockDim.x >> 5, nthreads = blockDim.x;
  const int slice = warp * 64, h0 = blockIdx.y * FFN_SLICE, d = p.d;
  const int M = plan_load(p.M_ptr);
  int m0 = blockIdx.x * AQ;
  if (m0 >= M) {                               // (one CTA always waits, see early exits in ad_common.cuh)
    if (blockIdx.x == 0 && blockIdx.y == 0) pdl_wait();
    return;
  }
  uint4 w1f[8][2], w2f[8][2];
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int c = 0; c < 2; ++c) w1f[j][c] = __ldg(reinterpret_cast<const uint4*>(p.w1 + (size_t)(h0 + 8 * j + g) * d + slice + 8 * t + 32 * c));
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int c = 0; c < 2; ++c) w2f[j][c] = __ldg(reinterpret_cast<const uint4*>(p.w2 + (size_t)(slice + 8 * j + g) * p.F + h0 + 8 * t + 32 * c));
  const int bc = (tid & 15) * 4;               // this thread's hidden features in the exchange
  const float4 bias = *reinterpret_cast<const float4*>(p.b1 + h0 + bc);
  pdl_wait();
  trace_mark(TR_GEMM + EPI_ACT, 1);
  auto load = [&](int m, uint4 (&x)[2][2]) {   // rows beyond the last token repeat it; never stored
    const bf16* x0 = p.x + (size_t)min(m + g, M - 1) * d + slice + 8 * t;
    const bf16* x1 = p.x + (size_t)min(m + g + 8, M - 1) * d + slice + 8 * t;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      x[c][0] = *reinterpret_cast<const uint4*>(x0 + 32 * c);
      x[c][1] = *reinterpret_cast<const uint4*>(x1 + 32 * c);
    }
  };
  auto multiply = [&](const uint4 (&a)[2][2], const uint4 (&w)[8][2], float (&acc)[8][4]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) { acc[j][0] = 0.f; acc[j][1] = 0.f; acc[j][2] = 0.f; acc[j][3] = 0.f; }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int j = 0; j < 8; ++j) mma16816(acc[j], a[c][0].x, a[c][1].x, a[c][0].y, a[c][1].y, w[j][c].x, w[j][c].y);
#pragma unroll
      for (int j = 0; j < 8; ++j) mma16816(acc[j], a[c][0].z, a[c][1].z, a[c][0].w, a[c][1].w, w[j][c].z, w[j][c].w);
    }
  };
  uint4 xa[2][2];
  load(m0, xa);
  for (; m0 < M; m0 += AQ * gridDim.x) {
    float acc[8][4];
    multiply(xa, w1f, acc);
    if (m0 + AQ * (int)gridDim.x < M) load(m0 + AQ * gridDim.x, xa);       // the next tile's, under this one
    float* pw = part + warp * AQ * O_LD;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      *reinterpret_cast<float2*>(pw + g * O_LD + 8 * j + 2 * t) = make_float2(acc[j][0], acc[j][1]);
      *reinterpret_cast<float2*>(pw + (g + 8) * O_LD + 8 * j + 2 * t) = make_float2(acc[j][2], acc[j][3]);
    }
    __syncthreads();
    for (int r = tid >> 4; r < AQ; r += nthreads >> 4) {
      float4 v = *reinterpret_cast<const float4*>(part + r * O_LD + bc);
#pragma unroll
      for (int w = 1; w < MAX_WARPS; ++w)
        if (w < nw) {
          const float4 o = *reinterpret_cast<const float4*>(part + (w * AQ + r) * O_LD + bc);
          v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
        }
      uint2 u;
      u.x = pack2(fmaxf(v.x + bias.x, 0.f), fmaxf(v.y + bias.y, 0.f));
      u.y = pack2(fmaxf(v.z + bias.z, 0.f), fmaxf(v.w + bias.w, 0.f));
      *reinterpret_cast<uint2*>(hs + r * K_LD + bc) = u;
    }
    __syncthreads();
    uint4 ha[2][2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      ha[c][0] = *reinterpret_cast<const uint4*>(hs + g * K_LD + 32 * c + 8 * t);
      ha[c][1] = *reinterpret_cast<const uint4*>(hs + (g + 8) * K_LD + 32 * c + 8 * t);
    }
    multiply(ha, w2f, acc);
    float* dst = p.out + (size_t)blockIdx.y * p.stride + (size_t)m0 * d + slice + 2 * t;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (m0 + g < M) *reinterpret_cast<float2*>(dst + (size_t)g * d + 8 * j) = make_float2(acc[j][0], acc[j][1]);
      if (m0 + g + 8 < M) *reinterpret_cast<float2*>(dst + (size_t)(g + 8) * d + 8 * j) = make_float2(acc[j][2], acc[j][3]);
    }
  }
  trace_mark(TR_GEMM + EPI_ACT, 2);
}

}  // namespace few
}  // namespace ad
