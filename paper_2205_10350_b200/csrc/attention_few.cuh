// Attention of passes with few queries per row (BF16, 64-wide heads), output projection included and, for the
// cross-attention, the query projection as well.
//
// A CTA handles one head and up to 16 queries of one row.  Everything is latency: a few dozen keys, a few thousand
// multiply-adds.  The CTA's warps therefore split whatever there is to split: the contraction of the query projection (64
// input features per warp), the keys (16 per warp and round), the output features of the output projection (64 per warp).
// Models up to 512 wide take d / 64 warps in one CTA; wider ones two CTAs of d / 128 warps (SPLIT = 2), so that both
// projections' weights still fit the registers of eight warps: each CTA of the pair projects the queries over half of the
// input features (the halves meet through distributed shared memory, the pair being a cluster) and the output to half of
// the output features; the attention in between is done by both.  All products are warp-level MMAs on fragments read with 16-byte loads (contraction index permuted
// identically for both operands, see gemm_few.cuh).  Weights, and for the cross-attention the keys and values (written
// by the encoder pass long before), are requested before the dependency wait; plan data is read there too.
//
// The FFMA kernel it replaces for these shapes (attention.cuh: one query per warp, keys staged as FP32) took 4.4 us after
// its dependency wait inside a 40-token step of a 512-wide model, and the cross-attention's query projection was a kernel
// of its own (2.3 us and a kernel boundary).
//
// Probabilities multiply the values as a sum of two BF16 numbers (p = hi + lo), so nothing is lost against FP32
// probabilities; queries and the output that enters the projection are rounded to BF16 exactly where a stored operand
// would be.
#pragma once

#include <type_traits>

#include "attention.cuh"
#include "gemm_few.cuh"

namespace ad {
namespace few {

constexpr int AQ = 16;            // queries per CTA = MMA M
constexpr int AK = 16;            // keys per warp and round
constexpr int K_LD = 96;          // key rows: 192 bytes apart (16-byte fragment loads without bank conflicts)
constexpr int V_LD = 72;          // value rows: 144 bytes apart (ldmatrix without bank conflicts)
constexpr int O_LD = 68;          // floats per row of a warp's partial output
constexpr int MAX_WARPS = 8;      // per CTA

struct FewAttnParams {
  AttnParams a;
  const bf16* x;        // query projection: its input [M_cap, d] (normalised hidden states) ...
  const bf16* wq;       // ... and weights [d, d]; null: the queries are in a.q
  int rounds;           // rounds of keys the capacity may need
  int rows;             // LOOP: rows of the batch
};

constexpr int MAX_ROUNDS = 4;     // rounds of AK keys per warp, all resident at once: 512 keys with eight warps (222 KB)
inline size_t att_few_smem(int warps, int rounds, bool loop_pair) {
  const size_t kv = (size_t)rounds * warps * AK * (K_LD + V_LD) * sizeof(bf16);
  const size_t part = (size_t)warps * AQ * O_LD * sizeof(float);      // partial query projections, later partial outputs
  return kv + part + 2 * (size_t)warps * AQ * sizeof(float) + 2 * (size_t)AQ * K_LD * sizeof(bf16) +
         (loop_pair ? 4 : 2) * (size_t)AQ * 64 * sizeof(float);
}
// CTAs a head's work is split over, and warps per CTA.
inline int att_few_split(int d) { return d > 64 * MAX_WARPS ? 2 : 1; }
inline int att_few_warps(int d) { return d / 64 / att_few_split(d); }

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}

// One item of a looping grid: up to AQ queries of one row.
struct FewItem { int row, m0, nq, kbase, row_nk, nk0, nk1; };
// The items of a pass, row by row.  Lane l of every warp holds rows l * per .. l * per + per - 1: `mine` items in them, `before` in front of
// them, and what the first of these rows needs to be described (with up to 32 rows everything comes from the lanes, in one round trip).
struct FewItems {
  int per, mine, before, total, len, off, base, nk;
  __device__ __forceinline__ static int chunks(int len) { return (len + AQ - 1) / AQ; }
  __device__ __forceinline__ void count(const AttnParams& p, int rows, int lane) {
    per = (rows + 31) >> 5;
    const int r0 = lane * per;
    const bool on = r0 < rows;
    len = on ? plan_load(p.seg_len + r0) : 0;
    off = on ? plan_load(p.seg_off + r0) : 0;
    base = on ? plan_load(p.key_base + r0) : 0;
    nk = on ? plan_load(p.nkeys_row + r0) : 0;
    mine = chunks(len);
    for (int r = r0 + 1; r < min(rows, r0 + per); ++r) mine += chunks(plan_load(p.seg_len + r));
    before = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int a = __shfl_up_sync(0xffffffffu, before, o);
      if (lane >= o) before += a;
    }
    total = __shfl_sync(0xffffffffu, before, 31);
    before -= mine;
  }
  // Item i < total, the same for every lane (nk0, nk1: its row's number of keys).
  __device__ __forceinline__ FewItem find(const AttnParams& p, int i) const {
    const int l = __ffs(__ballot_sync(0xffffffffu, before + mine > i)) - 1;
    int chunk = i - __shfl_sync(0xffffffffu, before, l), n = __shfl_sync(0xffffffffu, len, l), first = __shfl_sync(0xffffffffu, off, l);
    FewItem it;
    it.row = l * per; it.kbase = __shfl_sync(0xffffffffu, base, l); it.row_nk = __shfl_sync(0xffffffffu, nk, l);
    while (chunk >= chunks(n)) {                 // (more than 32 rows: a later one of this lane's)
      chunk -= chunks(n);
      ++it.row;
      n = plan_load(p.seg_len + it.row); first = plan_load(p.seg_off + it.row);
      it.kbase = plan_load(p.key_base + it.row); it.row_nk = plan_load(p.nkeys_row + it.row);
    }
    it.m0 = first + chunk * AQ; it.nq = min(AQ, n - chunk * AQ);
    it.nk0 = it.nk1 = it.row_nk;
    return it;
  }
};

// grid = (B * qchunks * SPLIT, H), qchunks = ceil(longest segment / 16); block = 32 * att_few_warps(d) threads; dynamic smem
// att_few_smem; cluster (SPLIT, 1, 1) when QPROJ and SPLIT == 2.
// LOOP: grid = (groups * SPLIT, H) of any size; the items that the pass has are dealt to the groups in runs, so that a CTA reads its weights
// once and the keys and values of a row once for the queries of it that follow one another.  Taken where the other grid, a CTA for every piece of the
// longest block that a row could have, has more of them than there are SMs, one of which fits each: those came in waves, CTAs without work among them, and every one read
// 64 or 128 KB of weights.  An item costs 2.7 us (128 keys) to 5.1 us (400 keys), the first as well as the following ones: it is a chain of five exchanges
// between the warps with 1.3 us of MMAs in it.  Drafter's pass of 414 tokens, 512 wide, after the wait: self-attention 8.2 -> 7.6 us, cross-attention
// over 400 keys 16.5 -> 12.2.  Whole calls: 768 wide, batch 6 4676 -> 4330 us, batch 8 with drafter 7732 -> 7464; 1024 wide, batch 4 5990 -> 5724, batch 3
// with drafter 7233 -> 6991; 512 wide, batch 16, relaxed 2625 -> 2488.  Straight-line rounds (below) do not fit its registers: they spilled,
// and the cross-attention took 15.3 us.
// SCORES_FIRST: three or four rounds of keys.  Whole calls, round after round -> this: 512 wide, batch 8 with drafter, 400 keys 7858 -> 7780 us;
// 768 wide, batch 4, 300 keys 2478 -> 2460.  With one or two rounds it is slower (batch 1 1132 -> 1139, 768 wide, batch 3, 150 keys 2250 -> 2275).
template <bool QPROJ, int SPLIT, bool SCORES_FIRST, bool LOOP>
__global__ void __launch_bounds__(32 * MAX_WARPS, 1)
attention_few_kernel(const FewAttnParams fp) {
  const AttnParams& p = fp.a;
  extern __shared__ __align__(16) uint8_t few_smem[];
  trace_mark(TR_ATTN, 0);
  pdl_launch();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int nw = blockDim.x >> 5, nthreads = blockDim.x;
  const int rank = SPLIT == 1 ? 0 : blockIdx.x % SPLIT, row_chunk = blockIdx.x / SPLIT;
  const int h = blockIdx.y;
  const int slice = (rank * nw + warp) * 64;      // this warp's input features of the query projection, output features of Wo
  const int d = p.d;
  // weights: rows 8 j + g of this head's query projection / of this warp's 64 output features, 64-wide slices of K
  uint4 wf[8][2], wqf[QPROJ ? 8 : 1][2];
  auto weights = [&]() {
    if (QPROJ) {
      const bf16* wb = fp.wq + (size_t)(h * 64 + g) * d + slice + 8 * t;
  #pragma unroll
      for (int j = 0; j < 8; ++j)
  #pragma unroll
        for (int c = 0; c < 2; ++c) wqf[QPROJ ? j : 0][c] = __ldg(reinterpret_cast<const uint4*>(wb + (size_t)(8 * j) * d + 32 * c));
    }
    const bf16* ob = p.wo + (size_t)(slice + g) * d + h * 64 + 8 * t;
  #pragma unroll
    for (int j = 0; j < 8; ++j)
  #pragma unroll
      for (int c = 0; c < 2; ++c) wf[j][c] = __ldg(reinterpret_cast<const uint4*>(ob + (size_t)(8 * j) * d + 32 * c));
  };
  if (LOOP) weights();          // (before the item is known: every CTA of a grid that fits the device has one but for the smallest passes)
  FewItems items;
  FewItem cur;
  int item = 0, item_end = 1;
  bool have;
  if (LOOP) {
    const int groups = gridDim.x / SPLIT;
    items.count(p, fp.rows, lane);
    item = row_chunk * items.total / groups;
    item_end = (row_chunk + 1) * items.total / groups;
    have = item < item_end;
    if (have) cur = items.find(p, item);
  } else {
    cur.row = row_chunk / p.qchunks;
    const int i0 = (row_chunk - cur.row * p.qchunks) * AQ, seg_len = plan_load(p.seg_len + cur.row);
    have = i0 < seg_len;
    cur.nq = min(AQ, seg_len - i0); cur.m0 = i0;
  }
  // The first CTA always waits: a grid whose CTAs all left here would let its successors run before its predecessor is done.
  if (!have) {
    if (blockIdx.x == 0 && h == 0) pdl_wait();
    return;
  }
  bf16* ks = reinterpret_cast<bf16*>(few_smem) + (size_t)warp * AK * (K_LD + V_LD);   // this warp's keys of a round ...
  bf16* vs = ks + AK * K_LD;                                                          // ... and values
  const int round_stride = nw * AK * (K_LD + V_LD);                                   // elements from one round to the next
  float* part = reinterpret_cast<float*>(few_smem + (size_t)fp.rounds * round_stride * sizeof(bf16));   // [nw][16][O_LD]
  float* pm = part + (size_t)nw * AQ * O_LD;                                          // [nw][16] maxima
  float* pl = pm + nw * AQ;                                                           // [nw][16] sums
  bf16* qs = reinterpret_cast<bf16*>(pl + nw * AQ);                                   // [16][K_LD] queries
  bf16* os = qs + AQ * K_LD;                                                          // [16][K_LD] outputs
  // (the pair's first barrier: a CTA's shared memory may be written once it is known to run)
  if (QPROJ && SPLIT > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  float* const xq0 = reinterpret_cast<float*>(os + AQ * K_LD);                        // [SPLIT][16][64] the pair's query halves; LOOP: two of them
  int xq_turn = 0;              // (the peer may write the next item's while this CTA still reads)

  if (!LOOP) weights();
  if (!LOOP) {
    cur.m0 += plan_load(p.seg_off + cur.row);
    cur.kbase = plan_load(p.key_base + cur.row); cur.row_nk = plan_load(p.nkeys_row + cur.row);
    cur.nk0 = cur.nk1 = cur.row_nk;
  }
  auto own_keys = [&](FewItem& it) {            // queries with their own number of keys (missing queries repeat the last one; never stored)
    if (!p.nkeys_tok) return;
    it.nk0 = min(plan_load(p.nkeys_tok + it.m0 + min(g, it.nq - 1)), it.row_nk);
    it.nk1 = min(plan_load(p.nkeys_tok + it.m0 + min(g + 8, it.nq - 1)), it.row_nk);
  };
  own_keys(cur);
  const bf16* kk = reinterpret_cast<const bf16*>(p.k);
  const bf16* vv = reinterpret_cast<const bf16*>(p.v);
  // this warp's 16 keys of every round, 64 elements each: 128 16-byte pieces, four per lane, for keys and values each
  auto fetch = [&](int kbase, int row_nk) {
    for (int r = 0; r < fp.rounds; ++r) {
      const int key0 = (r * nw + warp) * AK;
      if (key0 >= row_nk) break;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int idx = lane + 32 * i, j = idx >> 3, c = (idx & 7) * 8;
        const bool there = key0 + j < row_nk;
        const size_t off = (size_t)(kbase + (there ? key0 + j : 0)) * d + h * 64 + c;
        cp16(ks + r * round_stride + j * K_LD + c, kk + off, there);
        cp16(vs + r * round_stride + j * V_LD + c, vv + off, there);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (QPROJ) fetch(cur.kbase, cur.row_nk);          // the encoder's keys and values: older than the plan
  pdl_wait();
  trace_mark(TR_ATTN, 1);
  if (!QPROJ) fetch(cur.kbase, cur.row_nk);

  bool more = false, first = true;
  do {
    const int m0 = cur.m0, nq = cur.nq, row_nk = cur.row_nk, nk0 = cur.nk0, nk1 = cur.nk1;
    const int r0 = min(g, nq - 1), r1 = min(g + 8, nq - 1);
    uint4 qa[2][2];               // query fragments: [32-wide chunk of the head][row g / g + 8]
    if (QPROJ) {
      const bf16* x0 = fp.x + (size_t)(m0 + r0) * d + slice + 8 * t;
      const bf16* x1 = fp.x + (size_t)(m0 + r1) * d + slice + 8 * t;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        qa[c][0] = *reinterpret_cast<const uint4*>(x0 + 32 * c);
        qa[c][1] = *reinterpret_cast<const uint4*>(x1 + 32 * c);
      }
      float acc[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j) { acc[j][0] = 0.f; acc[j][1] = 0.f; acc[j][2] = 0.f; acc[j][3] = 0.f; }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int j = 0; j < 8; ++j) mma16816(acc[j], qa[c][0].x, qa[c][1].x, qa[c][0].y, qa[c][1].y, wqf[QPROJ ? j : 0][c].x, wqf[QPROJ ? j : 0][c].y);
#pragma unroll
        for (int j = 0; j < 8; ++j) mma16816(acc[j], qa[c][0].z, qa[c][1].z, qa[c][0].w, qa[c][1].w, wqf[QPROJ ? j : 0][c].z, wqf[QPROJ ? j : 0][c].w);
      }
      trace_mark(TR_ATTN, 3);
      float* const xq = xq0 + xq_turn;
      float* pw = part + (size_t)warp * AQ * O_LD;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        *reinterpret_cast<float2*>(pw + g * O_LD + 8 * j + 2 * t) = make_float2(acc[j][0], acc[j][1]);
        *reinterpret_cast<float2*>(pw + (g + 8) * O_LD + 8 * j + 2 * t) = make_float2(acc[j][2], acc[j][3]);
      }
      __syncthreads();
      if (SPLIT > 1 && first) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
      for (int idx = tid; idx < AQ * 16; idx += nthreads) {
        const int r = idx >> 4, c = (idx & 15) * 4;
        float4 v = SPLIT == 1 ? *reinterpret_cast<const float4*>(p.q_bias + h * 64 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
        for (int w = 0; w < nw; ++w) {
          const float4 o = *reinterpret_cast<const float4*>(part + ((size_t)w * AQ + r) * O_LD + c);
          v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
        }
        if (SPLIT == 1) {
          uint2 u;
          u.x = pack2(v.x, v.y); u.y = pack2(v.z, v.w);
          *reinterpret_cast<uint2*>(qs + r * K_LD + c) = u;
        } else {
          float* mine = xq + (rank * AQ + r) * 64 + c;
          *reinterpret_cast<float4*>(mine) = v;
          uint32_t peer;
          const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(mine));
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(local), "r"(rank ^ 1));
          asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(peer), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
        }
      }
      if (SPLIT > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        for (int idx = tid; idx < AQ * 16; idx += nthreads) {
          const int r = idx >> 4, c = (idx & 15) * 4;
          const float4 bq = *reinterpret_cast<const float4*>(p.q_bias + h * 64 + c);
          const float4 a0 = *reinterpret_cast<const float4*>(xq + r * 64 + c), a1 = *reinterpret_cast<const float4*>(xq + (AQ + r) * 64 + c);
          uint2 u;
          u.x = pack2(bq.x + a0.x + a1.x, bq.y + a0.y + a1.y); u.y = pack2(bq.z + a0.z + a1.z, bq.w + a0.w + a1.w);
          *reinterpret_cast<uint2*>(qs + r * K_LD + c) = u;
        }
      }
      __syncthreads();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        qa[c][0] = *reinterpret_cast<const uint4*>(qs + g * K_LD + 32 * c + 8 * t);
        qa[c][1] = *reinterpret_cast<const uint4*>(qs + (g + 8) * K_LD + 32 * c + 8 * t);
      }
    } else {
      const bf16* q0 = reinterpret_cast<const bf16*>(p.q) + (size_t)(m0 + r0) * d + h * 64 + 8 * t;
      const bf16* q1 = reinterpret_cast<const bf16*>(p.q) + (size_t)(m0 + r1) * d + h * 64 + 8 * t;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        qa[c][0] = *reinterpret_cast<const uint4*>(q0 + 32 * c);
        qa[c][1] = *reinterpret_cast<const uint4*>(q1 + 32 * c);
      }
    }

    trace_mark(TR_ATTN, 4);
    float o[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j) { o[j][0] = 0.f; o[j][1] = 0.f; o[j][2] = 0.f; o[j][3] = 0.f; }
    float mx0 = -INFINITY, mx1 = -INFINITY, den0 = 0.f, den1 = 0.f;      // den: this lane's share of the row sums
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    // 16 keys and up to 16 queries: two groups of eight keys, the two halves of the head side by side
    auto scores = [&](const bf16* kr, float (&s)[2][4]) {
      float s1[2][4];
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) { s[n][e] = 0.f; s1[n][e] = 0.f; }
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const uint4 k0 = *reinterpret_cast<const uint4*>(kr + (g + 8 * n) * K_LD + 8 * t);
        const uint4 k1 = *reinterpret_cast<const uint4*>(kr + (g + 8 * n) * K_LD + 32 + 8 * t);
        mma16816(s[n], qa[0][0].x, qa[0][1].x, qa[0][0].y, qa[0][1].y, k0.x, k0.y);
        mma16816(s1[n], qa[1][0].x, qa[1][1].x, qa[1][0].y, qa[1][1].y, k1.x, k1.y);
        mma16816(s[n], qa[0][0].z, qa[0][1].z, qa[0][0].w, qa[0][1].w, k0.z, k0.w);
        mma16816(s1[n], qa[1][0].z, qa[1][1].z, qa[1][0].w, qa[1][1].w, k1.z, k1.w);
      }
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) s[n][e] += s1[n][e];
    };
    // element e of group n: key key0 + 8 n + 2 t + (e & 1), query row g + 8 (e >> 1)
    auto mask = [&](int key0, float (&s)[2][4], float& t0, float& t1) {
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const int j = key0 + 8 * n + 2 * t;
        s[n][0] = j < nk0 ? s[n][0] * p.scale : -INFINITY;
        s[n][1] = j + 1 < nk0 ? s[n][1] * p.scale : -INFINITY;
        s[n][2] = j < nk1 ? s[n][2] * p.scale : -INFINITY;
        s[n][3] = j + 1 < nk1 ? s[n][3] * p.scale : -INFINITY;
        t0 = fmaxf(t0, fmaxf(s[n][0], s[n][1]));
        t1 = fmaxf(t1, fmaxf(s[n][2], s[n][3]));
      }
    };
    auto quad_max = [&](float& t0, float& t1) {
      t0 = fmaxf(t0, __shfl_xor_sync(0xffffffffu, t0, 1)); t1 = fmaxf(t1, __shfl_xor_sync(0xffffffffu, t1, 1));
      t0 = fmaxf(t0, __shfl_xor_sync(0xffffffffu, t0, 2)); t1 = fmaxf(t1, __shfl_xor_sync(0xffffffffu, t1, 2));
    };
    // probabilities (a query that sees none of the keys: on == false) and their sums, then times the values
    auto weigh = [&](const bf16* vr, const float (&s)[2][4], bool on0, bool on1, float& sum0, float& sum1) {
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const float p0 = on0 ? expf(s[n][0] - mx0) : 0.f, p1 = on0 ? expf(s[n][1] - mx0) : 0.f;
        const float p2 = on1 ? expf(s[n][2] - mx1) : 0.f, p3 = on1 ? expf(s[n][3] - mx1) : 0.f;
        sum0 += p0 + p1; sum1 += p2 + p3;
        split2(p0, p1, hi[2 * n], lo[2 * n]);
        split2(p2, p3, hi[2 * n + 1], lo[2 * n + 1]);
      }
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        uint32_t v[4];
        const uint32_t addr = static_cast<uint32_t>(__cvta_generic_to_shared(vr + (lane & 15) * V_LD + 8 * (j + (lane >> 4))));
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr));
        mma16816(o[j], hi[0], hi[1], hi[2], hi[3], v[0], v[1]);
        mma16816(o[j + 1], hi[0], hi[1], hi[2], hi[3], v[2], v[3]);
        mma16816(o[j], lo[0], lo[1], lo[2], lo[3], v[0], v[1]);
        mma16816(o[j + 1], lo[0], lo[1], lo[2], lo[3], v[2], v[3]);
      }
    };
    if (SCORES_FIRST) {
      // Scores of all rounds first: their MMAs do not depend on one another, and the maximum is known before the first exponential.  Without a
      // branch between the rounds, so that one round's work fills the gaps of another's (768 wide, batch 4, 300 keys, with the merge below:
      // 3983 -> 3954 us a call).
      const bool on0 = nk0 > warp * AK, on1 = nk1 > warp * AK;             // otherwise the query sees none of this warp's keys
      auto all_rounds = [&](auto rounds) {
        constexpr int R = decltype(rounds)::value;
        float s[R][2][4];
        float t0 = -INFINITY, t1 = -INFINITY;
        auto past = [&](int r) { return LOOP && (r * nw + warp) * AK >= row_nk; };
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (past(r)) break;
          scores(ks + r * round_stride, s[r]);
          if (LOOP) mask((r * nw + warp) * AK, s[r], t0, t1);
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (!LOOP) mask((r * nw + warp) * AK, s[r], t0, t1);
        quad_max(t0, t1);
        if (on0) mx0 = t0;
        if (on1) mx1 = t1;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (past(r)) break;
          weigh(vs + r * round_stride, s[r], on0, on1, den0, den1);
        }
      };
      if (LOOP) all_rounds(std::integral_constant<int, MAX_ROUNDS>());
      else switch ((row_nk - warp * AK + AK * nw - 1) / (AK * nw)) {            // rounds in which this warp has keys
        case 4: all_rounds(std::integral_constant<int, 4>()); break;
        case 3: all_rounds(std::integral_constant<int, 3>()); break;
        case 2: all_rounds(std::integral_constant<int, 2>()); break;
        case 1: all_rounds(std::integral_constant<int, 1>()); break;
        default: break;
      }
    } else {
      const bf16 *kr = ks, *vr = vs;
      for (int key0 = warp * AK; key0 < row_nk; key0 += AK * nw, kr += round_stride, vr += round_stride) {
        float s[2][4];
        float t0 = -INFINITY, t1 = -INFINITY;
        scores(kr, s);
        mask(key0, s, t0, t1);
        quad_max(t0, t1);
        const bool on0 = nk0 > key0, on1 = nk1 > key0;                     // otherwise the query sees none of these keys
        const float n0 = on0 ? fmaxf(mx0, t0) : mx0, n1 = on1 ? fmaxf(mx1, t1) : mx1;
        const float c0 = on0 ? expf(mx0 - n0) : 1.f, c1 = on1 ? expf(mx1 - n1) : 1.f;     // exp(-inf) = 0 at first
        mx0 = n0; mx1 = n1;
        den0 *= c0; den1 *= c1;
#pragma unroll
        for (int j = 0; j < 8; ++j) { o[j][0] *= c0; o[j][1] *= c0; o[j][2] *= c1; o[j][3] *= c1; }
        weigh(vr, s, on0, on1, den0, den1);
      }
    }
    if (LOOP) {
      more = item + 1 < item_end;
      if (more) {
        const int row = cur.row;
        cur = items.find(p, ++item);
        own_keys(cur);
        if (cur.row != row) {       // (the keys and values are this warp's own)
          __syncwarp();
          fetch(cur.kbase, cur.row_nk);
        }
      }
    }
    // merge the warps that had keys
    trace_mark(TR_ATTN, 5);
    const int na = min(nw, (row_nk + AK - 1) / AK);
    den0 += __shfl_xor_sync(0xffffffffu, den0, 1); den1 += __shfl_xor_sync(0xffffffffu, den1, 1);
    den0 += __shfl_xor_sync(0xffffffffu, den0, 2); den1 += __shfl_xor_sync(0xffffffffu, den1, 2);
    if (warp < na) {              // (the partial query projections in `part` were read before the last barrier)
      float* pw = part + (size_t)warp * AQ * O_LD;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        *reinterpret_cast<float2*>(pw + g * O_LD + 8 * j + 2 * t) = make_float2(o[j][0], o[j][1]);
        *reinterpret_cast<float2*>(pw + (g + 8) * O_LD + 8 * j + 2 * t) = make_float2(o[j][2], o[j][3]);
      }
      if (t == 0) {
        pm[warp * AQ + g] = mx0; pm[warp * AQ + g + 8] = mx1;
        pl[warp * AQ + g] = den0; pl[warp * AQ + g + 8] = den1;
      }
    }
    __syncthreads();
    // At most `most` warps, whose shares are read all at once: in a loop over the warps each cost a round trip to shared memory and an exponential
    // (whole calls, with the scores' two halves side by side: 512 wide, batch 1 1214 -> 1206 us; 768 wide, batch 3, 150 keys 2116 -> 2096).
    auto merge = [&](auto most) {
      constexpr int W = decltype(most)::value;
      for (int idx = tid; idx < AQ * 16; idx += nthreads) {
        const int r = idx >> 4, c = (idx & 15) * 4;
        float wm[W], wl[W];
        float4 x[W];
#pragma unroll
        for (int w = 0; w < W; ++w) wm[w] = w < na ? pm[w * AQ + r] : -INFINITY;
#pragma unroll
        for (int w = 0; w < W; ++w) {
          wl[w] = w < na ? pl[w * AQ + r] : 0.f;
          x[w] = w < na ? *reinterpret_cast<const float4*>(part + ((size_t)w * AQ + r) * O_LD + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float m = -INFINITY;
#pragma unroll
        for (int w = 0; w < W; ++w) m = fmaxf(m, wm[w]);
        float den = 0.f;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const float f = w < na ? expf(wm[w] - m) : 0.f;                  // a warp whose keys were all masked: exp(-inf) = 0
          den += wl[w] * f;
          v.x += x[w].x * f; v.y += x[w].y * f; v.z += x[w].z * f; v.w += x[w].w * f;
        }
        const float inv = 1.f / den;
        uint2 u;
        u.x = pack2(v.x * inv, v.y * inv); u.y = pack2(v.z * inv, v.w * inv);
        *reinterpret_cast<uint2*>(os + r * K_LD + c) = u;
      }
    };
    if (na <= 2) merge(std::integral_constant<int, 2>());
    else if (na <= 4) merge(std::integral_constant<int, 4>());
    else merge(std::integral_constant<int, MAX_WARPS>());
    __syncthreads();
    trace_mark(TR_ATTN, 6);
    // output projection: 16 queries x this warp's 64 features, K = this head's 64 dimensions
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      qa[c][0] = *reinterpret_cast<const uint4*>(os + g * K_LD + 32 * c + 8 * t);
      qa[c][1] = *reinterpret_cast<const uint4*>(os + (g + 8) * K_LD + 32 * c + 8 * t);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) { o[j][0] = 0.f; o[j][1] = 0.f; o[j][2] = 0.f; o[j][3] = 0.f; }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int j = 0; j < 8; ++j) mma16816(o[j], qa[c][0].x, qa[c][1].x, qa[c][0].y, qa[c][1].y, wf[j][c].x, wf[j][c].y);
#pragma unroll
      for (int j = 0; j < 8; ++j) mma16816(o[j], qa[c][0].z, qa[c][1].z, qa[c][0].w, qa[c][1].w, wf[j][c].z, wf[j][c].w);
    }
    trace_mark(TR_ATTN, 7);
    float* dst = p.o_part + (size_t)h * p.o_stride + (size_t)m0 * d + slice + 2 * t;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (g < nq) *reinterpret_cast<float2*>(dst + (size_t)g * d + 8 * j) = make_float2(o[j][0], o[j][1]);
      if (g + 8 < nq) *reinterpret_cast<float2*>(dst + (size_t)(g + 8) * d + 8 * j) = make_float2(o[j][2], o[j][3]);
    }
    first = false;
    if (LOOP && SPLIT > 1) xq_turn ^= SPLIT * AQ * 64;
  } while (LOOP && more);
  trace_mark(TR_ATTN, 2);
}

}  // namespace few
}  // namespace ad
