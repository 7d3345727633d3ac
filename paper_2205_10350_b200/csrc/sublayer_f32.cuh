// Sublayers of FP32 passes of up to a thousand packed tokens, models 128 or 256 wide: attention with its output projection and, for the cross-attention, the
// query projection, and the feed-forward sublayer with both of its projections, one kernel each.
//
// As kernels of their own the projections are 2.1 us a piece, most of it boundary and round trips: eleven kernels a decoder layer.  With these it is
// seven: QKV | attention + Wo | LayerNorm | Wq + attention + Wo | LayerNorm | W1 + W2 | LayerNorm.  A CTA owns a head (or a slice of the hidden features) and 16
// tokens; its shares of both weight matrices are in registers before the dependency wait, and what it computes in between stays in shared memory.
// What bounds them: one memory round trip, three to five barriers and, at 16 tokens, 512 to 1024 multiply-adds per thread.  Whole calls, sentences of 16 to 30
// tokens, before -> after, us: 128 wide, 2 + 2 layers, batch 1 608 -> 551, batch 6 1155 -> 776, batch 32 1909 -> 1433, batch 5 with drafter 2022 -> 1240; 256 wide, 3 + 3 layers,
// batch 1 1612 -> 1020, batch 6 2892 -> 1740, batch 24 4834 -> 2977.
// All sums are FP32 multiply-adds.  The output projection leaves one partial sum per head (slice) for the LayerNorm to add (pairwise: see add_partials).
#pragma once

#include "attention.cuh"

namespace ad {
namespace sub32 {

enum Kind { SELF, CROSS, FFN };
constexpr int TOK = 16;           // tokens per CTA: two per warp in the attention
constexpr int KEYS = 64;          // keys per shared-memory tile
constexpr int THREADS = 256;
constexpr int MAX_TOKENS = 1024;  // largest capacity of a pass that takes these kernels

struct Params {
  AttnParams a;        // attention: q (SELF), k, v, scale, q_bias, segments; wo as float in w_out
  const float* x;      // [M_cap, D] input of the first projection (CROSS, FFN)
  const float* w_in;   // CROSS: Wq [D, D]; FFN: W1 [F, D]
  const float* b_in;   // CROSS: bq; FFN: b1
  const float* w_out;  // Wo [D, D] or W2 [D, F]
  float* out;          // [heads or slices][M_cap, D] partial sums (no bias)
  size_t stride;       // M_cap * D
  int K2;              // row length of w_out: D or F
};

// Shared memory in floats: rows of the tiles are 16-byte aligned and four words apart modulo 32 (conflict-free 16-byte reads of 8 rows).
template <int D, int S>
struct Layout {
  static constexpr int LD = S + 4;
  static constexpr int XS = 0, RED = XS + TOK * D, HS = RED + TOK * THREADS, OS = HS + TOK * LD, KS = OS + TOK * LD, VS = KS + KEYS * LD, PS = VS + KEYS * LD,
                       FLOATS = PS + TOK * KEYS;
};

// Products in four running sums, which keeps the chains of additions, and with them the rounding, as short as in the kernels that split K between half-warps.  Error of
// the scores against 64 bits, two layers, rms, with those kernels / one running sum / four: 128 wide, batch 1 x 17 4.31e-8 / 4.33e-8 / 4.26e-8, 256 wide, batch 4 x 30 7.25e-8 /
// 7.23e-8 / 7.17e-8.  In one sum a call takes 3 % less at 128 wide and up to 3 % more at 256.
__device__ __forceinline__ void fma4(float4& s, float4 a, float4 b) {
  s.x = fmaf(a.x, b.x, s.x); s.y = fmaf(a.y, b.y, s.y); s.z = fmaf(a.z, b.z, s.z); s.w = fmaf(a.w, b.w, s.w);
}
__device__ __forceinline__ float sum4(float4 s) { return (s.x + s.y) + (s.z + s.w); }

// S: width of a head, or of a slice of hidden features.  grid = (B * qchunks, heads), or (groups, F / S): a group per tile of 16 tokens or, with LOOP, group i takes the
// tiles i, i + groups, ... (a form of its own: with the weights live throughout, 119 registers instead of 90, a call of 128 wide, batch 1 takes 0.4 % longer).
// block = 256; dynamic shared memory Layout<D, S>::FLOATS floats (FFN: OS).
template <Kind KIND, int D, int S, bool LOOP>
__global__ void __launch_bounds__(THREADS)
sublayer_f32_kernel(const Params p) {
  typedef Layout<D, S> L;
  constexpr int PARTS = THREADS / S, KP = D / PARTS;        // parts of the first projection's contraction
  constexpr int GROUPS = THREADS / D;                       // tokens side by side in the second projection
  extern __shared__ __align__(16) float sub_smem[];
  float *xs = sub_smem + L::XS, *red = sub_smem + L::RED, *hs = sub_smem + L::HS, *os = KIND == FFN ? hs : sub_smem + L::OS;
  float *ks = sub_smem + L::KS, *vs = sub_smem + L::VS, *ps = sub_smem + L::PS;
  pdl_launch();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, h = blockIdx.y;
  int m0, nt, kbase = 0, row_nk = 0, M = 0;
  if (KIND == FFN) {
    m0 = blockIdx.x * TOK;
    M = plan_load(p.a.M_ptr);
    nt = min(TOK, M - m0);
  } else {
    const int b = blockIdx.x / p.a.qchunks, i0 = (blockIdx.x - b * p.a.qchunks) * TOK;
    nt = min(TOK, plan_load(p.a.seg_len + b) - i0);
    m0 = plan_load(p.a.seg_off + b) + i0;
    kbase = plan_load(p.a.key_base + b); row_nk = plan_load(p.a.nkeys_row + b);
  }
  if (nt <= 0) {                                            // (one CTA always waits, see early exits in ad_common.cuh)
    if ((blockIdx.x | blockIdx.y) == 0) pdl_wait();
    return;
  }
  // weights
  const int f = tid % S, part = tid / S, n = tid % D, group = tid / D;
  float4 w1[KIND == SELF ? 1 : KP / 4], w2[S / 4];
  float bias = 0.f;
  if (KIND != SELF) {
#pragma unroll
    for (int i = 0; i < KP / 4; ++i) w1[KIND == SELF ? 0 : i] = __ldg(reinterpret_cast<const float4*>(p.w_in + (size_t)(h * S + f) * D + part * KP + 4 * i));
    bias = p.b_in[h * S + f];
  }
#pragma unroll
  for (int i = 0; i < S / 4; ++i) w2[i] = __ldg(reinterpret_cast<const float4*>(p.w_out + (size_t)n * p.K2 + h * S + 4 * i));
  const float *kk = reinterpret_cast<const float*>(p.a.k), *vv = reinterpret_cast<const float*>(p.a.v);
  auto fetch_keys = [&](int j0) {                           // keys j0 .. j0 + 63 of the row and their values; zeros beyond the last
    for (int idx = tid; idx < KEYS * (S / 4); idx += THREADS) {
      const int j = idx / (S / 4), c = (idx % (S / 4)) * 4;
      const bool there = j0 + j < row_nk;
      const size_t off = (size_t)(kbase + (there ? j0 + j : 0)) * D + h * S + c;
      cp16(ks + j * L::LD + c, kk + off, there);
      cp16(vs + j * L::LD + c, vv + off, there);
    }
  };
  if (KIND == CROSS) fetch_keys(0);                         // the encoder's: older than the plan
  int nk[2] = {0, 0};
  if (KIND != FFN)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int r = warp + 8 * u;
      if (r < nt) nk[u] = p.a.nkeys_tok ? min(plan_load(p.a.nkeys_tok + m0 + r), row_nk) : row_nk;
    }
  pdl_wait();
  if (KIND == SELF) {
    fetch_keys(0);
    const float* q = reinterpret_cast<const float*>(p.a.q);
    for (int idx = tid; idx < nt * S; idx += THREADS) hs[(idx / S) * L::LD + idx % S] = q[(size_t)(m0 + idx / S) * D + h * S + idx % S] * p.a.scale;
  }
  auto fetch_x = [&](int m, int n) {                        // n tokens' input
    for (int idx = tid; idx < n * (D / 4); idx += THREADS) {
      const int r = idx / (D / 4), c = (idx % (D / 4)) * 4;
      cp16(xs + r * D + c, p.x + (size_t)(m + r) * D + c, true);
    }
  };
  if (KIND != SELF) fetch_x(m0, nt);
  asm volatile("cp.async.commit_group;" ::: "memory");
  int m_next, n_next;
  do {
    m_next = m0 + TOK * (int)gridDim.x;
    n_next = LOOP ? min(TOK, M - m_next) : 0;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (KIND != SELF) {
      // first projection: every part's share of the tokens' S features, then their sum
#pragma unroll 4
      for (int r = 0; r < nt; ++r) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < KP / 4; ++i) fma4(s, w1[KIND == SELF ? 0 : i], *reinterpret_cast<const float4*>(xs + r * D + part * KP + 4 * i));
        red[(part * TOK + r) * S + f] = sum4(s);
      }
      __syncthreads();
      if (LOOP && n_next > 0) {                      // the next tile's input, under the rest of this one
        fetch_x(m_next, n_next);
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
      for (int r = part; r < nt; r += PARTS) {
        float s = red[r * S + f];
#pragma unroll
        for (int q = 1; q < PARTS; ++q) s += red[(q * TOK + r) * S + f];
        s += bias;
        hs[r * L::LD + f] = KIND == FFN ? fmaxf(s, 0.f) : s * p.a.scale;
      }
      __syncthreads();
    }
    if (KIND != FFN) {
      // attention: two queries per warp, keys lane and lane + 32 of every tile, running maximum and sum
      float mx[2] = {-INFINITY, -INFINITY}, den[2] = {0.f, 0.f}, acc[2][S / 32];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int c = 0; c < S / 32; ++c) acc[u][c] = 0.f;
      for (int j0 = 0; j0 < row_nk; j0 += KEYS) {
        if (j0 > 0) {
          __syncthreads();                                    // the previous tile has been read
          fetch_keys(j0);
          asm volatile("cp.async.commit_group;" ::: "memory");
          asm volatile("cp.async.wait_group 0;" ::: "memory");
          __syncthreads();
        }
        float s[2][2];
        float4 s4[2][2];
#pragma unroll
        for (int u = 0; u < 2; ++u) s4[u][0] = s4[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int c = 0; c < S; c += 4) {
          const float4 k0 = *reinterpret_cast<const float4*>(ks + lane * L::LD + c), k1 = *reinterpret_cast<const float4*>(ks + (lane + 32) * L::LD + c);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const float4 q = *reinterpret_cast<const float4*>(hs + (warp + 8 * u) * L::LD + c);
            fma4(s4[u][0], q, k0);
            fma4(s4[u][1], q, k1);
          }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) { s[u][0] = sum4(s4[u][0]); s[u][1] = sum4(s4[u][1]); }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          float p0 = 0.f, p1 = 0.f, corr = 1.f;
          if (nk[u] > j0) {                                   // warp-uniform; otherwise the query sees no key of this tile
            const float a0 = j0 + lane < nk[u] ? s[u][0] : -INFINITY, a1 = j0 + lane + 32 < nk[u] ? s[u][1] : -INFINITY;
            float top = fmaxf(a0, a1);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
            const float now = fmaxf(mx[u], top);              // finite: key j0 is visible
            corr = expf(mx[u] - now);                         // exp(-inf) = 0 on the first tile
            p0 = expf(a0 - now); p1 = expf(a1 - now);
            float sum = p0 + p1;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            den[u] = den[u] * corr + sum;
            mx[u] = now;
          }
          ps[(warp + 8 * u) * KEYS + lane] = p0;
          ps[(warp + 8 * u) * KEYS + lane + 32] = p1;
#pragma unroll
          for (int c = 0; c < S / 32; ++c) acc[u][c] *= corr;
        }
        __syncwarp();
        const int jn = min(KEYS, row_nk - j0);
#pragma unroll 2
        for (int j = 0; j < jn; j += 4) {                     // (keys beyond the last are zeros with probability 0)
          const float4 pa = *reinterpret_cast<const float4*>(ps + warp * KEYS + j), pb = *reinterpret_cast<const float4*>(ps + (warp + 8) * KEYS + j);
#pragma unroll
          for (int c = 0; c < S / 32; ++c) {
            const float* v = vs + j * L::LD + lane + 32 * c;
            const float v0 = v[0], v1 = v[L::LD], v2 = v[2 * L::LD], v3 = v[3 * L::LD];
            acc[0][c] = fmaf(pa.x, v0, acc[0][c]); acc[0][c] = fmaf(pa.y, v1, acc[0][c]); acc[0][c] = fmaf(pa.z, v2, acc[0][c]); acc[0][c] = fmaf(pa.w, v3, acc[0][c]);
            acc[1][c] = fmaf(pb.x, v0, acc[1][c]); acc[1][c] = fmaf(pb.y, v1, acc[1][c]); acc[1][c] = fmaf(pb.z, v2, acc[1][c]); acc[1][c] = fmaf(pb.w, v3, acc[1][c]);
          }
        }
        __syncwarp();
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float inv = nk[u] > 0 ? 1.f / den[u] : 0.f;
#pragma unroll
        for (int c = 0; c < S / 32; ++c) os[(warp + 8 * u) * L::LD + lane + 32 * c] = acc[u][c] * inv;
      }
      __syncthreads();
    }
    // second projection: this thread's output feature of every GROUPS-th token
    float* dst = p.out + (size_t)h * p.stride + (size_t)m0 * D + n;
#pragma unroll 4
    for (int r = group; r < nt; r += GROUPS) {
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < S / 4; ++i) fma4(s, w2[i], *reinterpret_cast<const float4*>(os + r * L::LD + 4 * i));
      dst[(size_t)r * D] = sum4(s);
    }
    m0 = m_next; nt = n_next;
  } while (LOOP && nt > 0);
}

}  // namespace sub32
}  // namespace ad
