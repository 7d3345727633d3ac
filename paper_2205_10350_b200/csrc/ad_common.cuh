// Shared device-side definitions of the verification-step kernels (sm_100a).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/aggressive_decoding.h"

namespace ad {

typedef __nv_bfloat16 bf16;

// ---------------------------------------------------------------------------------------------
// Scalar conversion helpers: activations between kernels are float (FP32 models) or bf16.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(bf16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f32<bf16>(float v) { return __float2bfloat16_rn(v); }

// ---------------------------------------------------------------------------------------------
// One pass over a packed set of token rows.  A "pass" is the verification block forward, the
// drafter forward or the encoder forward; rows of the batch contribute seg_len[b] consecutive
// packed tokens starting at seg_off[b].
// ---------------------------------------------------------------------------------------------
struct PassPlan {
  int* M;          // [1] total packed tokens of this pass
  int* seg_off;    // [B] first packed token of row b
  int* seg_len;    // [B] tokens of row b (0 = row idle)
  int* key_base;   // [B] slot index of self-attention key 0 of row b
  int* row_nk;     // [B] largest number of self-attention keys any token of row b sees
  int* tok_row;    // [Mmax] batch row of packed token m
  int* tok_pos;    // [Mmax] position fed to the positional table
  int* tok_id;     // [Mmax] input token id
  int* kv_slot;    // [Mmax] slot that receives this token's self-attention key/value
  int* att_n;      // [Mmax] number of self-attention keys the token may see (from key_base)
};

// Epilogue selector of the two GEMM kernels.
enum Epi : int {
  EPI_F32 = 0,      // out_f32[m][n] = acc (+ bias) (+ resid[m][n])
  EPI_ACT = 1,      // out_act[m][n] = act(acc + bias), optional ReLU
  EPI_SCATTER = 2,  // feature n belongs to segment n / seg_width; segment s goes to dst[s] at row
                    //   (s < n_direct ? m : slot[m]), column n % seg_width.  With seg_pair_stride != 0 there may be any
                    //   number of segments: segment s goes to dst[s & 1] + (s >> 1) * seg_pair_stride bytes (key / value
                    //   buffers of consecutive layers)
  EPI_ARGMAX = 3    // per (feature tile, token) running (max, lowest id) partials
};

// Launch geometry of the tensor-core projection kernel (gemm_tc.cuh) for M packed tokens: token tile and K split.  Evaluated
// on the device from the M the plan holds, by the projection and by whoever adds its partial sums up, so that a pass always
// runs at the geometry of the tokens it has, not at that of its capacity.
//
// Token tile: up to 64 tokens one tile; beyond that the kernels are latency-bound and smaller tiles win -- more CTAs, a
// shorter epilogue each -- until the grids outgrow the SMs.  Measured per verification step, builds that differ in the tile alone
// (512 wide: base model, capacity 256 for the first line, 2048 for the others; 1024 wide: big model, capacity 1024):
//   512 wide, 200 / 240 tokens: 32-token tiles 212 / 224 us, 64: 220 / 226, 128: 238 / 248, 16: 224 / 232;
//   320 / 512 / 800 / 1024 tokens: 64-token tiles 293 / 309 / 344 / 363 us, 128: 340 / 351 / 379 / 388, 32: 334 / 362 / 435 / 455;
//   2048 tokens: 128-token tiles 490 us, 64: 519, 256: 586 (256 is taken once it alone gives two CTAs per SM).
// The line at 1024 is the narrow models': 1024 wide, 128-token tiles already win there (648 us, 64: 717), and 64 at 200 (386, 32: 404).
// 65 to 128 tokens inside a larger capacity: 32-token tiles too, while they are one wave of CTAs.  Verified blocks of 68 / 100 / 128 tokens of 200, 64-token tiles -> 32:
// 768 wide 269 / 279 / 282 us -> 261 / 272 / 276, 1024 wide 305 / 318 / 324 -> 304 / 317 / 320; 512 wide, 72 / 96 / 128 tokens of 256, 182 / 186 / 193 -> 170 / 173 / 186 (the 16-feature
// form of the few-token kernel in two rounds 191 / 202 / 212).  With more CTAs than SMs each of them reads its weights once more for nothing: arg-max over
// a vocabulary of 16000, 512 wide, 100 tokens 10.3 -> 13.8 us, 65 tokens 10.9 -> 12.2; of 18816, 1024 wide, 12.5 -> 18.7; 8192, 768 wide, 8.2 -> 9.7.
// Passes that never have more than 128 tokens take the few-token kernels and the rule is only asked for what those do not cover.
// A projection whose feature tiles alone outnumber the SMs (the vocabulary) fills them with one token tile, and every further one
// reads its weights again: one 128-token tile up to 128 tokens (90 tokens x 50265 x 768: 19.5 us with two of 64), then tiles of 128
// (400 x 768 x 50265: 56 us, 76 with 64-token tiles), of 256 beyond 1536 tokens, where L2 traffic bounds it (2048: 114 against 119 us).
// K split (projections whose consumer adds partial sums up): as many CTAs as there are SMs at most, 112 for a single token tile
// (the big model's 25-token pass lost 4 % with 128 one-K-block CTAs).
struct GeoRule {
  int N, K;
  int max_tile;      // largest token tile that has a tensor map
  int max_split;     // 1: no split
  int sms;
  int few_split;     // > 0: passes of at most few_tokens tokens run on the few-token kernel (gemm_few.cuh) with this K split
  int few_tokens;
  int fixed_tile;    // > 0: M is known on the host, which evaluated the rule already (operator-level calls); no split
};
struct Geo {
  int tile, ksplit;
  bool few;
};
__host__ __device__ inline Geo geometry(const GeoRule& r, int M) {
  Geo g;
  g.few = r.few_split > 0 && M <= r.few_tokens;
  if (r.fixed_tile > 0) { g.tile = r.fixed_tile; g.ksplit = 1; return g; }
  if (g.few) { g.tile = 0; g.ksplit = r.few_split; return g; }
  const int nf = (r.N + 127) / 128;
  if (M <= 64) {
    g.tile = 16;
    while (g.tile < M) g.tile *= 2;
  } else if (nf >= r.sms) {
    g.tile = M <= 1536 ? 128 : 256;
  } else if (M <= 256) {
    g.tile = M > 128 || nf * ((M + 31) / 32) <= r.sms ? 32 : 64;
  } else if (M <= 1024) {
    g.tile = 64;
  } else {
    g.tile = nf * ((M + 255) / 256) >= 2 * r.sms ? 256 : 128;
  }
  if (g.tile > r.max_tile) g.tile = r.max_tile;
  const int tiles = nf * ((M + g.tile - 1) / g.tile), kb = r.K / 64, cap = M <= 64 ? 112 : r.sms;
  g.ksplit = 1;
  while (g.ksplit * 2 <= r.max_split && tiles * g.ksplit * 2 <= cap && kb % (g.ksplit * 2) == 0) g.ksplit *= 2;
  return g;
}
// Partial sums [nsplit][.., N] of a projection: how many there are and how far apart, for whoever adds them up.
struct Partials {
  const float* ptr;
  int nsplit;        // > 0: fixed, `stride` floats apart; 0: by rule and the pass's token count M, M * N floats apart
  size_t stride;
  GeoRule rule;
};
__device__ __forceinline__ void resolve_partials(const Partials& q, int M, int& nsplit, size_t& stride) {
  nsplit = q.nsplit > 0 ? q.nsplit : geometry(q.rule, M).ksplit;
  stride = q.nsplit > 0 ? q.stride : (size_t)M * q.rule.N;
}

// Weights that kernels further down the chain will read, to be brought into L2 (see prefetch_share).
struct Prefetch {
  const char* ptr[2];
  uint32_t bytes[2];     // multiples of 16 (see prefetch_bytes); 0: nothing
};
// What to prefetch of a matrix: all of it, or nothing of one that would push a quarter of L2 and more out (whose offsets, moreover, might not
// be numbers of 32 bits).
constexpr size_t PF_MAX = (size_t)32 << 20;
__host__ __device__ constexpr uint32_t prefetch_bytes(size_t bytes) { return bytes <= PF_MAX ? (uint32_t)bytes : 0u; }

struct GemmParams {
  int K;                 // contraction length
  int N;                 // output features (rows of W)
  const int* M_ptr;      // device scalar: number of valid packed tokens (null: use M_host)
  int M_host;
  int M_cap;             // capacity of the token dimension of the buffers
  const float* bias;     // [N] or null
  int relu;
  GeoRule rule;          // launch geometry of the tensor-core kernel
  // EPI_F32
  float* out_f32;        // [ksplit][M, N]: partial sums; the consumer adds them up
  // EPI_ACT
  void* out_act;         // [M_cap, N] float or bf16
  // EPI_SCATTER
  void* dst[3];
  size_t seg_pair_stride;
  int seg_width;
  int n_direct;
  const int* slot;       // [M_cap]
  // EPI_ARGMAX
  float* part_val;       // [M_cap, n_tiles]: per token, the best value of every 128-feature tile
  int* part_idx;         // [M_cap, n_tiles]
  // EPI_ARGMAX with the relaxed verification (null: off): per token, the drafted token and its score; the kernel
  // adds, per feature tile, how many OTHER features score strictly higher than the draft
  const float* draft_val;  // [M_cap]
  const int* draft_id;     // [M_cap] (negative: no draft at this position)
  int* part_cnt;           // [M_cap, n_tiles]
  int* status;           // device status word (latches AD_ERR_TIMEOUT), may be null
  Prefetch next;         // few-token kernel for wide slices of K: what to bring into L2
};

// Programmatic dependent launch: a kernel launched with the programmatic-serialization attribute may start
// while its predecessor in the stream is still running.  pdl_wait() blocks until the predecessor grid (and,
// transitively, everything before it) has completed and its writes are visible; everything a kernel does
// before pdl_wait() must touch only data that no kernel ever writes (weights, the kernel's own shared memory).
// pdl_launch() lets the successor begin its own pre-wait part.  Both are no-ops in an ordinary launch.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Plan data.  The kernels that lay a pass out (plan_*, prepare_verify, and the accept kernel when it plans the next block)
// never call pdl_launch(): a kernel behind one of them can only start once it has completed, and every later kernel of the
// pass starts later still.  What they write -- PassPlan, the row state, and with it everything older, such as the encoder's
// keys and values -- may therefore be read BEFORE pdl_wait(), off the critical path.  Read past L1, which may hold the
// previous pass's lines.
__device__ __forceinline__ int plan_load(const int* p) { return __ldcg(p); }
// Early exits.  A CTA that the plan gives no work leaves before pdl_wait(), so that it does not hold an SM's resources
// while the predecessor runs.  One CTA of the grid always waits, work or not: a grid that completed before its predecessor
// would release its own successors too early.

// 16-byte asynchronous copy global -> shared; zeros unless `there` (the source address must be valid all the same).
__device__ __forceinline__ void cp16(void* smem_dst, const void* gmem_src, bool there) {
  const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(gmem_src), "r"(there ? 16 : 0) : "memory");
}

// 16 bytes of weights that one CTA reads once, kept out of L1 (whole calls: batch 1 1133 -> 1124 us, batch 8 3587 -> 3548; not for the
// attention's weights, which the CTAs of a row's other query chunks read again: batch 8 with drafter 7865 -> 8090).
__device__ __forceinline__ uint4 weight_load_once(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// Optional timeline tracing (compile with -DAD_TRACE): thread 0 of CTA (0,0,0) of every kernel stamps the
// global nanosecond timer at entry (phase 0), after the dependency wait (phase 1), at exit (phase 2) and at
// kernel-specific points in between (phases 3..7); the last CTA along x does the same under id + 16.
#ifdef AD_TRACE
__device__ unsigned long long g_trace_buf[1 << 15];
__device__ unsigned int g_trace_n;
__device__ __forceinline__ void trace_mark(int id, int phase) {
  const bool first = blockIdx.x == 0, last = blockIdx.x == gridDim.x - 1 && gridDim.x > 1;
#ifdef AD_TRACE_ALL_EXITS
  // every CTA stamps its exit (under id + 16 unless it is CTA (0,0,0)): shows the tail of a grid
  if (phase == 2 && threadIdx.x == 0 && !(first && blockIdx.y == 0 && blockIdx.z == 0)) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    const unsigned int i = atomicAdd(&g_trace_n, 1u);
    if (i < (1u << 15)) g_trace_buf[i] = (t & 0x00FFFFFFFFFFFFFFull) | ((unsigned long long)((id + 16) * 8 + phase) << 56);
    return;
  }
#endif
  if (threadIdx.x == 0 && (first || last) && blockIdx.y == 0 && blockIdx.z == 0) {
    if (last) id += 16;
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    const unsigned int i = atomicAdd(&g_trace_n, 1u);
    if (i < (1u << 15)) g_trace_buf[i] = (t & 0x00FFFFFFFFFFFFFFull) | ((unsigned long long)(id * 8 + phase) << 56);
  }
}
// The same from whichever thread of CTA 0 calls it (role threads of warp-specialised kernels).
__device__ __forceinline__ void trace_mark_role(int id, int phase) {
  if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    const unsigned int i = atomicAdd(&g_trace_n, 1u);
    if (i < (1u << 15)) g_trace_buf[i] = (t & 0x00FFFFFFFFFFFFFFull) | ((unsigned long long)(id * 8 + phase) << 56);
  }
}
#else
__device__ __forceinline__ void trace_mark(int, int) {}
__device__ __forceinline__ void trace_mark_role(int, int) {}
#endif
enum TraceId { TR_GEMM = 0, TR_ATTN = 8, TR_LN = 9, TR_EMBED = 10, TR_PREPARE = 11, TR_ACCEPT = 12, TR_COMMIT = 13,
               TR_PV_ISSUE = 20, TR_PV_EPI = 21, TR_PV_LOAD = 22 };

// Share i of n of what is to be brought into L2, in pieces that one thread hands to the SM's bulk-copy unit; nothing waits for them.
// To be shared by a hundred CTAs: one CTA alone (the accept kernel was tried) gets no more than its SM's share of the way into L2 and stays
// until all is through.
constexpr uint32_t PF_PIECE = 8192;
__device__ __forceinline__ void prefetch_share(const Prefetch& f, uint32_t i, uint32_t n) {
#pragma unroll
  for (int r = 0; r < 2; ++r)
    for (uint32_t o = i * PF_PIECE; o < f.bytes[r]; o += n * PF_PIECE)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(f.ptr[r] + o), "r"(min(PF_PIECE, f.bytes[r] - o)) : "memory");
}

__device__ __forceinline__ void latch_error(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

}  // namespace ad
