// BF16 projections of passes with few packed tokens (up to a hundred or so), on warp-level MMAs with the weights held in
// registers.
//
// With so few tokens a projection moves 1-8 MB of weights that sit in L2 and does next to no arithmetic; what it costs is
// latency: the tcgen05 kernel (gemm_tc.cuh) needs 2.3-4 us for one after its dependency wait (TMA round trip, MMA issue,
// tensor-memory read-out, transposition, stores).  Here a CTA owns 16 output features and its eight warps split K between
// them, so that a warp's share of the weights is a handful of 16-byte loads per lane that are issued BEFORE the dependency
// wait (weights never change).  After the wait a CTA does one round trip for its activations, a few dozen MMAs, one
// exchange through shared memory (the warps' partial sums, added in warp order) and the stores.
//
// The contraction index is permuted identically for both operands (a lane's 16-byte piece holds eight consecutive K
// elements, which serve as the fragments of two k16 steps), so no ldmatrix and no shared-memory staging is needed.
#pragma once

#include "ad_common.cuh"

namespace ad {
namespace few {

constexpr int THREADS = 256;
constexpr int WARPS = 8;
constexpr int FEAT = 16;          // output features per CTA = MMA M
constexpr int W_FEAT = 32;        // ... of the form for wide slices of K (gemm_few_wide_kernel)
constexpr int RED_LD = 20;        // floats per token row of a warp's partial sums: conflict-free, 16-byte aligned
constexpr int MAX_TOKENS = 128;   // most packed tokens of a pass that these kernels take ...
constexpr int INNER_TOKENS = 64;  // ... where its capacity is larger: one round
constexpr int MAX_CHUNKS = 4;     // 32-wide K chunks per warp: K per CTA = 256 .. 1024

// D (16 x 8, FP32) += A (16 x 16, BF16, row-major) * B (16 x 8, BF16, column-major).  Not volatile: free to be scheduled.
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Tokens of one round trip: 64 while a warp's slice of K is 64 wide, 32 beyond (register budget of two CTAs per SM).
__host__ __device__ constexpr int round_tokens(int nch) { return nch <= 2 ? 64 : 32; }

// K split of a projection with N output features: the smallest power of two that leaves at most 1024 of K to a CTA, more
// while the grid stays within 128 CTAs and the split is wanted (consumer adds partial sums up).  0: shape not supported.
inline int split_for(int N, int K, bool may_split, int max_split) {
  if (N % W_FEAT || K % 256) return 0;
  int s = 1;
  while (K / s > 256 * MAX_CHUNKS || (may_split && (N / FEAT) * s * 2 <= 128 && K % (512 * s) == 0 && K / (2 * s) >= 512)) {
    s *= 2;
    if (K % (256 * s)) return 0;
  }
  if (s > 1 && (!may_split || s > max_split)) return 0;
  return s;
}

// First projection of a pass: its operand is the embedding of the planned tokens, x = emb[token] * sqrt(d) + PE[position],
// computed where it is used; the CTAs also share the writing of the FP32 residual stream y.
struct EmbedParams {
  const bf16* emb;
  const float* pe;
  float scale;
  const int *tok_id, *tok_pos;
  float* y;
};
// Eight consecutive elements of x, rounded like a stored operand.
__device__ __forceinline__ uint4 embed8(const EmbedParams& ep, int tok, int pos, int K, int k) {
  const uint4 e = __ldg(reinterpret_cast<const uint4*>(ep.emb + (size_t)tok * K + k));
  const float4 p0 = __ldg(reinterpret_cast<const float4*>(ep.pe + (size_t)pos * K + k));
  const float4 p1 = __ldg(reinterpret_cast<const float4*>(ep.pe + (size_t)pos * K + k + 4));
  const float pp[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
  const uint32_t w[4] = {e.x, e.y, e.z, e.w};
  uint32_t r[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float a = __uint_as_float(w[i] << 16) * ep.scale + pp[2 * i];
    const float b = __uint_as_float(w[i] & 0xffff0000u) * ep.scale + pp[2 * i + 1];
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    r[i] = *reinterpret_cast<const uint32_t*>(&h);
  }
  return make_uint4(r[0], r[1], r[2], r[3]);
}

// Four output features n .. n + 3 of token m: bias, activation, store.  slot: the token's K/V row (EPI_SCATTER).
template <int EPI>
__device__ __forceinline__ void few_store(const GemmParams& p, int kz, int M, int m, int n, float4 v, float4 bias, int slot) {
  if (EPI == EPI_F32) {
    *reinterpret_cast<float4*>(p.out_f32 + ((size_t)kz * M + m) * p.N + n) = v;
    return;
  }
  v.x += bias.x; v.y += bias.y; v.z += bias.z; v.w += bias.w;
  if (EPI == EPI_ACT && p.relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
  bf16* dst;
  if (EPI == EPI_ACT) {
    dst = reinterpret_cast<bf16*>(p.out_act) + (size_t)m * p.N + n;
  } else {
    const int seg = n / p.seg_width, col = n - seg * p.seg_width;
    char* base = p.seg_pair_stride ? static_cast<char*>(p.dst[seg & 1]) + (size_t)(seg >> 1) * p.seg_pair_stride
                                   : static_cast<char*>(p.dst[seg]);
    dst = reinterpret_cast<bf16*>(base) + (size_t)(seg < p.n_direct ? m : slot) * p.seg_width + col;
  }
  __nv_bfloat162 h0 = __floats2bfloat162_rn(v.x, v.y), h1 = __floats2bfloat162_rn(v.z, v.w);
  uint2 u;
  u.x = *reinterpret_cast<unsigned int*>(&h0);
  u.y = *reinterpret_cast<unsigned int*>(&h1);
  *reinterpret_cast<uint2*>(dst) = u;
}
// The embedding as FP32 residual stream, tokens first, first + step, ...
__device__ __forceinline__ void few_embed_y(const GemmParams& p, const EmbedParams& ep, int M, int first, int step) {
  const int groups = p.K >> 2;
  const size_t K = (size_t)p.K;
  for (int m = first; m < M; m += step) {
    const int tok = plan_load(ep.tok_id + m), pos = plan_load(ep.tok_pos + m);
    for (int i = threadIdx.x; i < groups; i += THREADS) {
      const uint2 e = __ldg(reinterpret_cast<const uint2*>(ep.emb + (size_t)tok * K + 4 * i));
      const float4 pp = __ldg(reinterpret_cast<const float4*>(ep.pe + (size_t)pos * K + 4 * i));
      float4 v;
      v.x = __uint_as_float(e.x << 16) * ep.scale + pp.x; v.y = __uint_as_float(e.x & 0xffff0000u) * ep.scale + pp.y;
      v.z = __uint_as_float(e.y << 16) * ep.scale + pp.z; v.w = __uint_as_float(e.y & 0xffff0000u) * ep.scale + pp.w;
      *reinterpret_cast<float4*>(ep.y + (size_t)m * K + 4 * i) = v;
    }
  }
}

// Body of the kernel for the CTA of features 16 bx .. 16 bx + 15 and K part kz (K / ksplit = 256 * NCH).
// EPI_F32: partial sums [ksplit][M, N] (no bias); EPI_ACT: bias (+ ReLU) -> BF16; EPI_SCATTER: q / K / V rows.
// EMB: the operand is the embedding (ep), X is not read; nothing depends on the predecessor until the first store.
// red: shared memory, [WARPS][round_tokens(NCH)][RED_LD] floats.
__host__ __device__ constexpr size_t red_bytes(int nch) { return sizeof(float) * WARPS * (nch <= 2 ? 64 : 32) * RED_LD; }

template <int EPI, int NCH, bool EMB>
__device__ __forceinline__ void few_body(const bf16* __restrict__ W, const bf16* X, const GemmParams& p, const EmbedParams& ep, int bx,
                                         int kz, int M, float* red_mem) {
  constexpr int TPR = round_tokens(NCH);
  constexpr int NT = TPR / 8;
  float (*red)[TPR][RED_LD] = reinterpret_cast<float (*)[TPR][RED_LD]>(red_mem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int n0 = bx * FEAT;
  const int kbase = kz * (256 * NCH) + warp * (32 * NCH) + 8 * t;
  const size_t K = (size_t)p.K;
  uint4 wa[NCH][2];
#pragma unroll
  for (int c = 0; c < NCH; ++c) {
    wa[c][0] = weight_load_once(W + (size_t)(n0 + g) * K + kbase + 32 * c);
    wa[c][1] = weight_load_once(W + (size_t)(n0 + g + 8) * K + kbase + 32 * c);
  }
  const int of = (tid & 3) * 4, ot = tid >> 2;               // this thread's output: four features of one token per round
  float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
  if (EPI != EPI_F32) bias = *reinterpret_cast<const float4*>(p.bias + n0 + of);
  int slot = 0;
  if (EPI == EPI_SCATTER && ot < M) slot = plan_load(p.slot + ot);
  if (!EMB) pdl_wait();
  trace_mark(TR_GEMM + EPI, 1);
  for (int t0 = 0; t0 < M; t0 += TPR) {
    float acc[NT][4];
    uint4 xb[NT][NCH];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      if (t0 + 8 * nt < M) {
        if (EMB) {
          const int m = min(t0 + 8 * nt + g, M - 1);
          const int tok = plan_load(ep.tok_id + m), pos = plan_load(ep.tok_pos + m);
#pragma unroll
          for (int c = 0; c < NCH; ++c) xb[nt][c] = embed8(ep, tok, pos, p.K, kbase + 32 * c);
        } else {
          const bf16* xr = X + (size_t)min(t0 + 8 * nt + g, p.M_cap - 1) * K + kbase;
#pragma unroll
          for (int c = 0; c < NCH; ++c) xb[nt][c] = *reinterpret_cast<const uint4*>(xr + 32 * c);
        }
      }
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) { acc[nt][0] = 0.f; acc[nt][1] = 0.f; acc[nt][2] = 0.f; acc[nt][3] = 0.f; }
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
        if (t0 + 8 * nt < M) mma16816(acc[nt], wa[c][0].x, wa[c][1].x, wa[c][0].y, wa[c][1].y, xb[nt][c].x, xb[nt][c].y);
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
        if (t0 + 8 * nt < M) mma16816(acc[nt], wa[c][0].z, wa[c][1].z, wa[c][0].w, wa[c][1].w, xb[nt][c].z, xb[nt][c].w);
    }
    if (t0 > 0) __syncthreads();                             // the previous round has been read out
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      if (t0 + 8 * nt < M) {
        float* r0 = &red[warp][8 * nt + 2 * t][g];
        r0[0] = acc[nt][0]; r0[RED_LD] = acc[nt][1];
        r0[8] = acc[nt][2]; r0[RED_LD + 8] = acc[nt][3];
      }
    }
    __syncthreads();
    if (EMB && t0 == 0) pdl_wait();
    const int m = t0 + ot;
    if (ot < TPR && m < M) {
      float4 v = *reinterpret_cast<const float4*>(&red[0][ot][of]);
#pragma unroll
      for (int w = 1; w < WARPS; ++w) {
        const float4 o = *reinterpret_cast<const float4*>(&red[w][ot][of]);
        v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
      }
      if (EPI == EPI_SCATTER && t0 > 0) slot = plan_load(p.slot + m);
      few_store<EPI>(p, kz, M, m, n0 + of, v, bias, slot);
    }
  }
  if (EMB) {
    if (M <= 0) pdl_wait();                                  // (a grid without work still ends after its predecessor)
    few_embed_y(p, ep, M, bx, p.N / FEAT);
  }
}

// grid = (N / 16, ksplit); block = 256.  NCH = 1, 2.
template <int EPI, int NCH, bool EMB>
__global__ void __launch_bounds__(THREADS, 2)
gemm_few_kernel(const bf16* __restrict__ W, const bf16* X, const GemmParams p, const EmbedParams ep) {
  __shared__ __align__(16) float red[red_bytes(NCH) / sizeof(float)];
  trace_mark(TR_GEMM + EPI, 0);
  pdl_launch();
  few_body<EPI, NCH, EMB>(W, X, p, ep, blockIdx.x, blockIdx.y, plan_load(p.M_ptr), red);
  trace_mark(TR_GEMM + EPI, 2);
}

// The same for wider slices of K (768 and 1024 per CTA), where 16 features per CTA leave the kernel bound by the activations it
// re-reads (90 tokens of a 768-wide model: 192 CTAs x 138 KB, three dependent rounds, 4.9 us after the wait): 32 features per
// CTA halve that traffic, one CTA per SM has the registers for the next round's activations to be in flight under this one.
// DECODER: decoder passes read their weights past L1 and bring those of kernels further on into L2 (p.next, where they need it).  Encoder passes,
// whose weights are read once a call, do neither: calls of four layers, 768 wide, in the decoder's form -> in their own, us: 1 x 97 tokens
// 170 -> 163, 4 x 17 129 -> 125, 7 x 16 162 -> 155.  The other way round (weights through L1, prefetch code only where there is something to
// prefetch) a decode call of the 1024-wide model takes 3720 us instead of 3653, of the 768-wide one 1476 instead of 1460.
// grid = (N / 32, ksplit); block = 256.  NCH = 3, 4.
constexpr int W_TOK = 32;
constexpr int W_LD = W_FEAT + 4;
template <int EPI, int NCH, bool EMB, bool DECODER>
__global__ void __launch_bounds__(THREADS, 1)
gemm_few_wide_kernel(const bf16* __restrict__ W, const bf16* X, const GemmParams p, const EmbedParams ep) {
  constexpr int NT = W_TOK / 8;
  __shared__ __align__(16) float red[WARPS][W_TOK][W_LD];
  trace_mark(TR_GEMM + EPI, 0);
  pdl_launch();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int n0 = blockIdx.x * W_FEAT, kz = blockIdx.y;
  const int kbase = kz * (256 * NCH) + warp * (32 * NCH) + 8 * t;
  const size_t K = (size_t)p.K;
  auto weights = [](const bf16* w) { return DECODER ? weight_load_once(w) : __ldg(reinterpret_cast<const uint4*>(w)); };
  uint4 wa[2][NCH][2];
#pragma unroll
  for (int f = 0; f < 2; ++f)
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      wa[f][c][0] = weights(W + (size_t)(n0 + 16 * f + g) * K + kbase + 32 * c);
      wa[f][c][1] = weights(W + (size_t)(n0 + 16 * f + g + 8) * K + kbase + 32 * c);
    }
  if (DECODER && tid == THREADS - 1) prefetch_share(p.next, blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y);
  const int of = (tid & 7) * 4, ot = tid >> 3;               // this thread's output: four features of one token per round
  float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
  if (EPI != EPI_F32) bias = *reinterpret_cast<const float4*>(p.bias + n0 + of);
  const int M = plan_load(p.M_ptr);
  int slot = 0;
  if (EPI == EPI_SCATTER && ot < M) slot = plan_load(p.slot + ot);
  auto load = [&](int t0, uint4 (&xb)[NT][NCH]) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      if (t0 + 8 * nt < M) {
        const int m = min(t0 + 8 * nt + g, M - 1);
        if (EMB) {
          const int tok = plan_load(ep.tok_id + m), pos = plan_load(ep.tok_pos + m);
#pragma unroll
          for (int c = 0; c < NCH; ++c) xb[nt][c] = embed8(ep, tok, pos, p.K, kbase + 32 * c);
        } else {
#pragma unroll
          for (int c = 0; c < NCH; ++c) xb[nt][c] = *reinterpret_cast<const uint4*>(X + (size_t)m * K + kbase + 32 * c);
        }
      }
    }
  };
  if (!EMB) pdl_wait();
  trace_mark(TR_GEMM + EPI, 1);
  uint4 xb[NT][NCH], xn[NT][NCH];
  load(0, xb);
  for (int t0 = 0; t0 < M; t0 += W_TOK) {
    if (t0 + W_TOK < M) load(t0 + W_TOK, xn);
    float acc[2][NT][4];
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) { acc[f][nt][0] = 0.f; acc[f][nt][1] = 0.f; acc[f][nt][2] = 0.f; acc[f][nt][3] = 0.f; }
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
#pragma unroll
      for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
          mma16816(acc[f][nt], wa[f][c][0].x, wa[f][c][1].x, wa[f][c][0].y, wa[f][c][1].y, xb[nt][c].x, xb[nt][c].y);
#pragma unroll
      for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
          mma16816(acc[f][nt], wa[f][c][0].z, wa[f][c][1].z, wa[f][c][0].w, wa[f][c][1].w, xb[nt][c].z, xb[nt][c].w);
    }
    if (t0 > 0) __syncthreads();                             // the previous round has been read out
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        float* r0 = &red[warp][8 * nt + 2 * t][16 * f + g];
        r0[0] = acc[f][nt][0]; r0[W_LD] = acc[f][nt][1];
        r0[8] = acc[f][nt][2]; r0[W_LD + 8] = acc[f][nt][3];
      }
    __syncthreads();
    if (EMB && t0 == 0) pdl_wait();
    const int m = t0 + ot;
    if (m < M) {
      float4 v = *reinterpret_cast<const float4*>(&red[0][ot][of]);
#pragma unroll
      for (int w = 1; w < WARPS; ++w) {
        const float4 o = *reinterpret_cast<const float4*>(&red[w][ot][of]);
        v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
      }
      if (EPI == EPI_SCATTER && t0 > 0) slot = plan_load(p.slot + m);
      few_store<EPI>(p, kz, M, m, n0 + of, v, bias, slot);
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int c = 0; c < NCH; ++c) xb[nt][c] = xn[nt][c];
  }
  if (EMB) {
    if (M <= 0) pdl_wait();                                  // (a grid without work still ends after its predecessor)
    few_embed_y(p, ep, M, blockIdx.x, gridDim.x);
  }
  trace_mark(TR_GEMM + EPI, 2);
}

}  // namespace few
}  // namespace ad
