// FP32 projection GEMMs on the FP32 pipes (FFMA), for models whose weights are FP32 and whose scores have to match an FP32
// definition to 1e-3: no TF32, no reduced-precision operands.  Same D^T[n, m] orientation and the same epilogues as the
// tensor-core kernels.
//
// Two kernels.  gemm_f32_kernel: tiles of 64 or 128 features x 16 or 32 tokens, both operands copied asynchronously to shared memory
// as they lie (no transposition: a thread multiplies its outputs by four consecutive k at a time).  gemm_f32_few_kernel:
// passes of few tokens, where that kernel's walk along K is all latency: 16 features per CTA, K dealt to 16 half-warps,
// weights in registers before the dependency wait.
#pragma once

#include "ad_common.cuh"
#include "gemm_tc.cuh"   // warp_argmax

namespace ad {
namespace simt {

constexpr int KT = 32;            // k per stage
constexpr int LDK = KT + 4;       // rows 144 bytes apart: conflict-free 16-byte reads of consecutive rows
constexpr int STAGES = 4;
constexpr int ARGMAX_FEAT = 128;  // features per tile of the arg-max epilogue: the layout of the partial arrays

// Tiles of FEAT features x 4 TJ tokens, four warps per 64 features.
template <int FEAT, int TJ>
constexpr size_t smem_bytes() {
  constexpr size_t ring = sizeof(float) * (size_t)STAGES * (FEAT + 4 * TJ) * LDK, sums = sizeof(float) * (size_t)(FEAT / 16) * 8 * TJ * 33;
  return ring > sums ? ring : sums;
}

__device__ __forceinline__ void cp4(void* s, const void* g, bool there) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(s))), "l"(g),
               "r"(there ? 4 : 0) : "memory");
}

// One output row of the non-arg-max epilogues.
template <int EPI>
__device__ __forceinline__ void store_out(const GemmParams& p, int n, int m, float v) {
  if (EPI == EPI_F32) {
    p.out_f32[(size_t)m * p.N + n] = v;
  } else if (EPI == EPI_ACT) {
    reinterpret_cast<float*>(p.out_act)[(size_t)m * p.N + n] = p.relu ? fmaxf(v, 0.f) : v;
  } else {
    const int s = n / p.seg_width, c = n - s * p.seg_width;
    const int row = s < p.n_direct ? m : plan_load(p.slot + m);
    char* base = p.seg_pair_stride ? static_cast<char*>(p.dst[s & 1]) + (size_t)(s >> 1) * p.seg_pair_stride : static_cast<char*>(p.dst[s]);
    reinterpret_cast<float*>(base)[(size_t)row * p.seg_width + c] = v;
  }
}

// A warp covers 64 features x 4 TJ tokens, 8 x TJ outputs per lane; four warps per 64 features take every fourth quad of k and
// their sums meet in shared memory at the end.  What bounds it: instruction issue.  Shared memory is the next limit: a 16-byte
// load of eight different rows costs a warp four wavefronts, one that four rows serve two, so a lane's tile of 8 x 8 spends 48
// on 256 FFMA instructions of a warp (64 SM cycles); 8 x 4 spends 40 on 128.  With the loads of a step in front of its
// multiply-adds a warp issued in 47 % of its cycles, fetching ahead (below) in 60 %: 333 x 512 x 2048 48 -> 38 us on one warp per
// scheduler (2048 -> 512 features); 700 x 1024 x 4096 177 -> 148 us.
// grid = (ceil(N / FEAT), ceil(M_cap / (4 TJ))); block = 2 FEAT; dynamic smem smem_bytes<FEAT, TJ>().  x: [M_cap, K], w: [N, K].
// vec: K is a multiple of four and both operands are 16-byte aligned.
constexpr int GROUPS = 4;
constexpr int SUM_LD = 33;
template <int EPI, int FEAT, int TJ>
__global__ void __launch_bounds__(2 * FEAT, FEAT == 64 ? 3 : 1)
gemm_f32_kernel(const float* __restrict__ w, const float* x, const GemmParams p, const int vec) {
  constexpr int THREADS = 2 * FEAT;
  constexpr int RSTEP = THREADS / (KT / 4);            // rows between a thread's 16-byte copies: FEAT / RSTEP of W, then of x
  constexpr int TOK = 4 * TJ;
  constexpr int NW = FEAT / RSTEP, NX = (TOK + RSTEP - 1) / RSTEP;
  extern __shared__ __align__(16) float simt_smem[];   // [STAGES][FEAT + TOK][LDK], later [warps][64][SUM_LD] partial sums
  const int M = p.M_ptr ? plan_load(p.M_ptr) : p.M_host;
  const int t0 = blockIdx.y * TOK, n0 = blockIdx.x * FEAT;
  pdl_launch();
  if (t0 >= M && (blockIdx.x | blockIdx.y) > 0) return;
  pdl_wait();
  if (t0 >= M) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = warp % GROUPS, half = warp / GROUPS;               // share of k; 64-feature part of the tile
  const int tx = lane & 7, ty = lane >> 3;                           // features tx + 8 i, tokens ty + 4 j
  const int K = p.K, nk = (K + KT - 1) / KT;
  const int fr = tid / (KT / 4), fc = (tid % (KT / 4)) * 4;          // first row and k of this thread's 16-byte copies
  const float *wsrc = w + (size_t)(n0 + fr) * K + fc, *xsrc = x + (size_t)(t0 + fr) * K + fc;
  auto fetch = [&](int kt) {
    float* dst = simt_smem + (size_t)(kt % STAGES) * (FEAT + TOK) * LDK;
    const int k0 = kt * KT;
    if (kt < nk) {
      if (vec) {
        const bool in_k = k0 + fc < K;
#pragma unroll
        for (int i = 0; i < NW; ++i) {
          const bool there = in_k && n0 + fr + RSTEP * i < p.N;
          cp16(dst + (fr + RSTEP * i) * LDK + fc, there ? wsrc + (size_t)(RSTEP * i) * K + k0 : w, there);
        }
#pragma unroll
        for (int i = 0; i < NX; ++i) {
          if (TOK % RSTEP && fr + RSTEP * i >= TOK) break;
          const bool there = in_k && t0 + fr + RSTEP * i < M;
          cp16(dst + (FEAT + fr + RSTEP * i) * LDK + fc, there ? xsrc + (size_t)(RSTEP * i) * K + k0 : x, there);
        }
      } else {
        for (int idx = tid; idx < (FEAT + TOK) * KT; idx += THREADS) {
          const int r = idx / KT, c = idx % KT;
          const bool is_w = r < FEAT;
          const int row = is_w ? n0 + r : t0 + r - FEAT;
          const bool there = row < (is_w ? p.N : M) && k0 + c < K;
          cp4(dst + r * LDK + c, (is_w ? w : x) + (there ? (size_t)row * K + k0 + c : 0), there);
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[8][TJ];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < TJ; ++j) acc[i][j] = 0.f;
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) fetch(s);
  // One step: 16 k of a stage, four per warp.  A row of W is fetched one row ahead of its use and the tokens' pieces one step ahead,
  // so that no multiply-add waits for shared memory.
  const float* const wbase = simt_smem + (half * 64 + tx) * LDK + 4 * grp;
  const float* const xbase = simt_smem + (FEAT + ty) * LDK + 4 * grp;
  constexpr int STAGE = (FEAT + TOK) * LDK;
  float4 a, b[TJ], bn[TJ];
  auto step = [&](float4 (&bc)[TJ], float4 (&bnext)[TJ], int at, int next) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float4 an = *reinterpret_cast<const float4*>(i < 7 ? wbase + at + (i + 1) * 8 * LDK : wbase + next);
      if (i < TJ) bnext[i] = *reinterpret_cast<const float4*>(xbase + next + i * 4 * LDK);
#pragma unroll
      for (int j = 0; j < TJ; ++j) acc[i][j] = fmaf(a.x, bc[j].x, acc[i][j]);
#pragma unroll
      for (int j = 0; j < TJ; ++j) acc[i][j] = fmaf(a.y, bc[j].y, acc[i][j]);
#pragma unroll
      for (int j = 0; j < TJ; ++j) acc[i][j] = fmaf(a.z, bc[j].z, acc[i][j]);
#pragma unroll
      for (int j = 0; j < TJ; ++j) acc[i][j] = fmaf(a.w, bc[j].w, acc[i][j]);
      a = an;
    }
  };
  static_assert(KT == 8 * GROUPS && TJ <= 8, "two steps per stage");
  asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
  __syncthreads();
  a = *reinterpret_cast<const float4*>(wbase);
#pragma unroll
  for (int j = 0; j < TJ; ++j) b[j] = *reinterpret_cast<const float4*>(xbase + j * 4 * LDK);
  int at = 0;
  for (int kt = 0; kt < nk; ++kt) {
    step(b, bn, at, at + 4 * GROUPS);
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 3) : "memory");
    __syncthreads();                                    // stage kt + 1 has landed, stage kt - 1 is free
    fetch(kt + STAGES - 1);
    const int next = at == (STAGES - 1) * STAGE ? 0 : at + STAGE;
    step(bn, b, at + 4 * GROUPS, next);                 // (after the last stage: pieces that nobody uses)
    at = next;
  }
  // the groups' sums meet in shared memory
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  float* sums = simt_smem + (size_t)warp * 8 * TJ * SUM_LD + lane;
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < TJ; ++j) sums[(i * TJ + j) * SUM_LD] = acc[i][j];
  __syncthreads();
  auto sum_of = [&](int f, int tok) {                   // output (feature f, token tok) of the tile
    const float* q = simt_smem + (size_t)(f / 64) * GROUPS * 8 * TJ * SUM_LD + ((f % 64) / 8 * TJ + tok / 4) * SUM_LD + (tok % 4) * 8 + f % 8;
    float v = q[0];
#pragma unroll
    for (int g = 1; g < GROUPS; ++g) v += q[(size_t)g * 8 * TJ * SUM_LD];
    return v;
  };
  if (EPI == EPI_ARGMAX) {
    for (int tok = warp; tok < TOK && t0 + tok < M; tok += THREADS / 32) {       // a warp per token; lowest id on ties
      const int m = t0 + tok;
      float v = -INFINITY;
      int id = 0x7fffffff, cnt = 0;
      const float dval = p.draft_val ? p.draft_val[m] : 0.f;
      const int did = p.draft_val ? p.draft_id[m] : -1;
#pragma unroll
      for (int f = lane; f < FEAT; f += 32) {
        const int n = n0 + f;
        if (n < p.N) {
          const float s = sum_of(f, tok);
          if (s > v) { v = s; id = n; }
          if (id == 0x7fffffff) id = n;                              // (the lowest one where no score compares above -inf)
          if (p.draft_val && n != did && s > dval) ++cnt;           // other features that score strictly higher
        }
      }
      tc::warp_argmax(v, id);
      if (p.draft_val) cnt = __reduce_add_sync(0xffffffffu, cnt);
      if (lane == 0) {
        const size_t o = (size_t)m * gridDim.x + blockIdx.x;
        p.part_val[o] = v;
        p.part_idx[o] = id;
        if (p.draft_val) p.part_cnt[o] = cnt;
      }
    }
  } else {
    // output (token, feature): neighbouring threads take neighbouring features
    for (int idx = tid; idx < FEAT * TOK; idx += THREADS) {
      const int f = idx % FEAT, tok = idx / FEAT, n = n0 + f, m = t0 + tok;
      if (n < p.N && m < M) store_out<EPI>(p, n, m, sum_of(f, tok) + (p.bias ? p.bias[n] : 0.f));
    }
  }
}

// ---- few tokens ------------------------------------------------------------------------------------------
constexpr int F_FEAT = 16;        // features per CTA
constexpr int F_TOK = 16;         // tokens per round
constexpr int F_PARTS = 16;       // half-warps of the CTA = parts of K
constexpr int F_MAX_K = 512;

inline bool few_fits(int N, int K) { return N % F_FEAT == 0 && K % 64 == 0 && K <= F_MAX_K; }

// grid = N / 16, block = 256; K / 16 = 4 * NQ consecutive k per half-warp.  Lane: feature lane % 16.
template <int EPI, int NQ>
__global__ void __launch_bounds__(256)
gemm_f32_few_kernel(const float* __restrict__ w, const float* x, const GemmParams p) {
  constexpr int K = 64 * NQ;
  __shared__ __align__(16) float xs[F_TOK][K];
  __shared__ float red[F_PARTS][F_TOK][F_FEAT];
  pdl_launch();
  const int tid = threadIdx.x, f = tid & 15, part = tid >> 4, n0 = blockIdx.x * F_FEAT;
  float4 wr[NQ];
#pragma unroll
  for (int i = 0; i < NQ; ++i) wr[i] = __ldg(reinterpret_cast<const float4*>(w + (size_t)(n0 + f) * K + part * 4 * NQ + 4 * i));
  const float bias = p.bias ? p.bias[n0 + f] : 0.f;
  const int M = plan_load(p.M_ptr);
  pdl_wait();
  for (int t0 = 0; t0 < M; t0 += F_TOK) {
    if (t0 > 0) __syncthreads();
    for (int idx = tid; idx < F_TOK * (K / 4); idx += 256) {
      const int r = idx / (K / 4), c = (idx % (K / 4)) * 4;
      if (t0 + r < M) cp16(&xs[r][c], x + (size_t)(t0 + r) * K + c, true);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const int nt = min(F_TOK, M - t0);
#pragma unroll 4
    for (int r = 0; r < nt; ++r) {
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < NQ; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(&xs[r][part * 4 * NQ + 4 * i]);
        s = fmaf(wr[i].x, v.x, s); s = fmaf(wr[i].y, v.y, s); s = fmaf(wr[i].z, v.z, s); s = fmaf(wr[i].w, v.w, s);
      }
      red[part][r][f] = s;
    }
    __syncthreads();
    const int r = tid >> 4;                             // one output per thread
    if (r < nt) {
      float s = red[0][r][f];
#pragma unroll
      for (int q = 1; q < F_PARTS; ++q) s += red[q][r][f];
      store_out<EPI>(p, n0 + f, t0 + r, s + bias);
    }
  }
}

}  // namespace simt
}  // namespace ad
