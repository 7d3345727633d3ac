// Attention for many queries, or over hundreds of keys, on the tensor cores (BF16, head dimension 64).
//
// Same operation and masking rules as attention_kernel (attention.cuh).  The tiles of one (row, head) pair are small (at most
// 64 queries x 64 keys x 64 dims per step), far below the 128-row atoms of the tcgen05 path and not worth a round trip through
// tensor memory, so the products run as warp-level m16n8k16 MMAs on register fragments: S = Q K^T, online softmax on the
// accumulator fragments, P (rounded to BF16, or as a sum of two BF16 numbers) reused in place as the A operand of O += P V, with V
// read through transposing ldmatrix loads.  Key fragments are read 16 bytes at a time, the contraction index permuted identically for both operands
// (see gemm_few.cuh).  Keys and values that are older than the plan (cross-attention: the encoder wrote them) are requested
// before the dependency wait.
#pragma once

#include "attention.cuh"

namespace ad {

constexpr int AM_Q = 64;        // queries per CTA with one key group
constexpr int AM_KT = 64;       // keys per shared-memory tile

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);   // .x = lo (low half), .y = hi
  return *reinterpret_cast<uint32_t*>(&h);
}
template <bool SPLIT_P>
__device__ __forceinline__ float exp_p(float x) { return SPLIT_P ? expf(x) : __expf(x); }
// K/V tiles in shared memory.
constexpr int AL_KLD = 96;             // key rows 192 bytes apart: conflict-free 16-byte fragment loads
constexpr int AL_VLD = 72;             // value rows 144 bytes apart: conflict-free ldmatrix
constexpr int AL_TILE_BYTES = AM_KT * (AL_KLD + AL_VLD) * 2;   // 21 504

// One 64-key tile of K and V into `dst`; keys from row_nk on are written as zeros.
template <int THREADS>
__device__ __forceinline__ void fetch_kv_tile(uint8_t* dst, const bf16* k, const bf16* v, int first_key, int row_nk, int d, int tid) {
  bf16* kd = reinterpret_cast<bf16*>(dst);
#pragma unroll
  for (int i = 0; i < AM_KT * 8 / THREADS; ++i) {
    const int idx = tid + THREADS * i, j = idx >> 3, c = (idx & 7) * 8;
    const bool there = first_key + j < row_nk;
    const size_t off = (size_t)(there ? first_key + j : 0) * d + c;
    cp16(kd + j * AL_KLD + c, k + off, there);
    cp16(kd + AM_KT * AL_KLD + j * AL_VLD + c, v + off, there);
  }
}

// Running state of 16 queries of a warp: output fragments, maxima, this lane's share of the row sums.
struct AttnState {
  float o[8][4];
  float mx0, mx1, den0, den1;
};
__device__ __forceinline__ void attn_init(AttnState& a) {
#pragma unroll
  for (int t = 0; t < 8; ++t) { a.o[t][0] = 0.f; a.o[t][1] = 0.f; a.o[t][2] = 0.f; a.o[t][3] = 0.f; }
  a.mx0 = a.mx1 = -INFINITY;
  a.den0 = a.den1 = 0.f;
}
// KS keys (rows of ks / vs; the first is key jw of the row) for 16 queries whose two of this lane see nk0 / nk1 keys.
// SPLIT_P: probabilities from expf, multiplied as a sum of two BF16 numbers; otherwise from __expf, rounded to BF16.
template <int KS, bool SPLIT_P>
__device__ __forceinline__ void attn_keys(AttnState& a, const uint4 (&qa)[2][2], const bf16* ks, const bf16* vs, int jw, int nk0, int nk1,
                                          float scale, int lane) {
  const int g = lane >> 2, tq = lane & 3;
  constexpr int NT = KS / 8;
  // S = Q K^T (consecutive MMAs go to different accumulators and do not wait for one another)
  float s[NT][4];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) { s[nt][0] = 0.f; s[nt][1] = 0.f; s[nt][2] = 0.f; s[nt][3] = 0.f; }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    uint4 kf[NT];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) kf[nt] = *reinterpret_cast<const uint4*>(ks + (nt * 8 + g) * AL_KLD + 32 * c + 8 * tq);
    const uint32_t a0[4] = {qa[c][0].x, qa[c][1].x, qa[c][0].y, qa[c][1].y}, a1[4] = {qa[c][0].z, qa[c][1].z, qa[c][0].w, qa[c][1].w};
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(s[nt], a0, kf[nt].x, kf[nt].y);
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(s[nt], a1, kf[nt].z, kf[nt].w);
  }
  // mask, scale, online softmax; element e of group nt is key jw + nt * 8 + tq * 2 + (e & 1), query row e >> 1
  if (jw + KS > nk0 || jw + KS > nk1) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const int j = jw + nt * 8 + tq * 2;
      if (j >= nk0) s[nt][0] = -INFINITY;
      if (j + 1 >= nk0) s[nt][1] = -INFINITY;
      if (j >= nk1) s[nt][2] = -INFINITY;
      if (j + 1 >= nk1) s[nt][3] = -INFINITY;
    }
  }
  float t0 = -INFINITY, t1 = -INFINITY;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    s[nt][0] *= scale; s[nt][1] *= scale; s[nt][2] *= scale; s[nt][3] *= scale;
    t0 = fmaxf(t0, fmaxf(s[nt][0], s[nt][1]));
    t1 = fmaxf(t1, fmaxf(s[nt][2], s[nt][3]));
  }
  t0 = fmaxf(t0, __shfl_xor_sync(0xffffffffu, t0, 1)); t0 = fmaxf(t0, __shfl_xor_sync(0xffffffffu, t0, 2));
  t1 = fmaxf(t1, __shfl_xor_sync(0xffffffffu, t1, 1)); t1 = fmaxf(t1, __shfl_xor_sync(0xffffffffu, t1, 2));
  const bool on0 = nk0 > jw, on1 = nk1 > jw;         // otherwise none of these keys is visible to the query
  const float m0n = on0 ? fmaxf(a.mx0, t0) : a.mx0, m1n = on1 ? fmaxf(a.mx1, t1) : a.mx1;
  const float corr0 = on0 ? exp_p<SPLIT_P>(a.mx0 - m0n) : 1.f, corr1 = on1 ? exp_p<SPLIT_P>(a.mx1 - m1n) : 1.f;   // exp(-inf) = 0 at first
  a.mx0 = m0n; a.mx1 = m1n;
  const float e0 = on0 ? m0n : 0.f, e1 = on1 ? m1n : 0.f;           // (all scores are -inf when the query sees no key here)
  float sum0 = 0.f, sum1 = 0.f;
  uint32_t pa[KS / 16][4], pl[SPLIT_P ? KS / 16 : 1][4];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const float p0 = exp_p<SPLIT_P>(s[nt][0] - e0), p1 = exp_p<SPLIT_P>(s[nt][1] - e0);
    const float p2 = exp_p<SPLIT_P>(s[nt][2] - e1), p3 = exp_p<SPLIT_P>(s[nt][3] - e1);
    sum0 += p0 + p1; sum1 += p2 + p3;
    // accumulator fragments of two neighbouring key groups are exactly one A fragment of 16 keys
    const int i = (nt & 1) * 2;
    if (SPLIT_P) {
      split2(p0, p1, pa[nt >> 1][i], pl[SPLIT_P ? nt >> 1 : 0][i]);
      split2(p2, p3, pa[nt >> 1][i + 1], pl[SPLIT_P ? nt >> 1 : 0][i + 1]);
    } else {
      pa[nt >> 1][i] = pack_bf16(p0, p1);
      pa[nt >> 1][i + 1] = pack_bf16(p2, p3);
    }
  }
  a.den0 = a.den0 * corr0 + sum0;
  a.den1 = a.den1 * corr1 + sum1;
#pragma unroll
  for (int dt = 0; dt < 8; ++dt) { a.o[dt][0] *= corr0; a.o[dt][1] *= corr0; a.o[dt][2] *= corr1; a.o[dt][3] *= corr1; }
#pragma unroll
  for (int tt = 0; tt < KS / 16; ++tt) {
#pragma unroll
    for (int dt = 0; dt < 8; dt += 2) {              // lanes 0..15 address the keys of column group dt, 16..31 those of dt + 1
      uint32_t v0, v1, v2, v3;
      const uint32_t addr = static_cast<uint32_t>(__cvta_generic_to_shared(vs + (tt * 16 + (lane & 15)) * AL_VLD + (dt + (lane >> 4)) * 8));
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(v0), "=r"(v1), "=r"(v2), "=r"(v3) : "r"(addr));
      mma_bf16_16816(a.o[dt], pa[tt], v0, v1);
      mma_bf16_16816(a.o[dt + 1], pa[tt], v2, v3);
      if (SPLIT_P) {
        mma_bf16_16816(a.o[dt], pl[SPLIT_P ? tt : 0], v0, v1);
        mma_bf16_16816(a.o[dt + 1], pl[SPLIT_P ? tt : 0], v2, v3);
      }
    }
  }
}

// ---- many queries -----------------------------------------------------------------------------------------
// NG = number of key groups.  With NG = 1 the CTA's four warps take 16 queries each (64 queries per CTA) and walk the row's
// tiles, the next one being copied under the arithmetic of this one.  When rows have few queries, or when 64-query CTAs would
// leave SMs idle, NG = 2 or 4 warps share a 16-query tile instead (32 or 16 queries per CTA) and split the keys of every tile
// between them; their running maxima, sums and outputs are merged at the end.
// grid = (B * qchunks, H), qchunks = ceil(longest segment / queries per CTA); block = 128 threads.
template <int NG, bool SPLIT_P>
__global__ void __launch_bounds__(128, 3)
attention_mma_kernel(const AttnParams p, const int kv_old) {
  constexpr int DH = 64;
  constexpr int QT = 4 / NG;            // 16-query tiles per CTA
  constexpr int KS = AM_KT / NG;        // keys of a tile that one warp handles
  __shared__ __align__(16) uint8_t kv[2][AL_TILE_BYTES];

  trace_mark(TR_ATTN, 0);
  pdl_launch();
  const int b = blockIdx.x / p.qchunks;
  const int chunk = blockIdx.x % p.qchunks;
  const int h = blockIdx.y;
  const int seg_len = plan_load(p.seg_len + b);
  const int i0 = chunk * (16 * QT);
  if (i0 >= seg_len) {
    if ((blockIdx.x | blockIdx.y) == 0) pdl_wait();
    return;
  }
  const int seg_off = plan_load(p.seg_off + b);
  const int kbase = plan_load(p.key_base + b);
  const int row_nk = plan_load(p.nkeys_row + b);
  int q_nsplit = 0;
  size_t q_stride = 0;
  if (p.q_part.ptr) resolve_partials(p.q_part, plan_load(p.M_ptr), q_nsplit, q_stride);
  const int nq = min(16 * QT, seg_len - i0);
  const int m0 = seg_off + i0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tq = lane & 3;           // fragment row (0..7) and column pair (0..3) of this lane
  const int qtile = warp % QT, grp = warp / QT;     // this warp's query tile and key group
  const bool active = qtile * 16 < nq;              // otherwise the warp only helps loading
  const int d = p.d;
  const bf16* q = reinterpret_cast<const bf16*>(p.q);
  const bf16* kk = reinterpret_cast<const bf16*>(p.k) + (size_t)kbase * d + h * DH;
  const bf16* vv = reinterpret_cast<const bf16*>(p.v) + (size_t)kbase * d + h * DH;
  const int n_tiles = (row_nk + AM_KT - 1) / AM_KT;
  auto fetch = [&](int tile) {
    if (tile < n_tiles) fetch_kv_tile<128>(kv[tile & 1], kk, vv, tile * AM_KT, row_nk, d, tid);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (kv_old) { fetch(0); fetch(1); }
  // this lane's two queries (fragment rows g and g + 8 of the warp's 16) and their visible-key counts
  const int r0 = qtile * 16 + g, r1 = r0 + 8;
  int nk0 = 0, nk1 = 0;
  if (r0 < nq) nk0 = p.nkeys_tok ? min(plan_load(p.nkeys_tok + m0 + r0), row_nk) : row_nk;
  if (r1 < nq) nk1 = p.nkeys_tok ? min(plan_load(p.nkeys_tok + m0 + r1), row_nk) : row_nk;
  pdl_wait();
  trace_mark(TR_ATTN, 1);
  if (!kv_old) { fetch(0); fetch(1); }
  // Q as A fragments: eight consecutive elements of the head per lane, 32-wide chunk and row
  uint4 qa[2][2];
  {
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int r = e ? r1 : r0, col = h * DH + 32 * c + 8 * tq;
        qa[c][e] = zero;
        if (r < nq) {
          if (!p.q_part.ptr) {
            qa[c][e] = *reinterpret_cast<const uint4*>(q + (size_t)(m0 + r) * d + col);
          } else {      // split-K partial sums of the projection (+ bias), rounded like stored queries
            float acc[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = p.q_bias ? p.q_bias[col + i] : 0.f;
            for (int sp = 0; sp < q_nsplit; ++sp) {
              float part[8];
              load8(p.q_part.ptr + sp * q_stride + (size_t)(m0 + r) * d + col, part);
#pragma unroll
              for (int i = 0; i < 8; ++i) acc[i] += part[i];
            }
            qa[c][e] = make_uint4(pack_bf16(acc[0], acc[1]), pack_bf16(acc[2], acc[3]), pack_bf16(acc[4], acc[5]), pack_bf16(acc[6], acc[7]));
          }
        }
      }
    }
  }
  AttnState a;
  attn_init(a);
  for (int t = 0; t < n_tiles; ++t) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();                                 // everybody's copies of tile t have landed
    const int jw = t * AM_KT + grp * KS;             // first key of this warp's share of the tile
    const bf16* ks = reinterpret_cast<const bf16*>(kv[t & 1]);
    if (active && jw < row_nk) attn_keys<KS, SPLIT_P>(a, qa, ks + grp * KS * AL_KLD, ks + AM_KT * AL_KLD + grp * KS * AL_VLD, jw, nk0, nk1, p.scale, lane);
    __syncthreads();                                 // tile t is fully consumed
    fetch(t + 2);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");

  float den0 = a.den0, den1 = a.den1, mx0 = a.mx0, mx1 = a.mx1;
  den0 += __shfl_xor_sync(0xffffffffu, den0, 1); den0 += __shfl_xor_sync(0xffffffffu, den0, 2);
  den1 += __shfl_xor_sync(0xffffffffu, den1, 1); den1 += __shfl_xor_sync(0xffffffffu, den1, 2);
  float (&o)[8][4] = a.o;
  if (NG > 1) {
    // Merge the key groups of a query tile.  Every lane of a group > 0 leaves its fragment (32 outputs, two
    // maxima, two sums) in the tile memory, value-major so that lanes hit different banks; the lane with the
    // same number in group 0 folds them in.
    float* rec = reinterpret_cast<float*>(&kv[0][0]);        // [36][128]
    __syncthreads();                                       // all tile reads are done
    if (grp > 0) {
#pragma unroll
      for (int dt = 0; dt < DH / 8; ++dt)
#pragma unroll
        for (int e = 0; e < 4; ++e) rec[(dt * 4 + e) * 128 + tid] = o[dt][e];
      rec[32 * 128 + tid] = mx0; rec[33 * 128 + tid] = mx1;
      rec[34 * 128 + tid] = den0; rec[35 * 128 + tid] = den1;
    }
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int g2 = 1; g2 < NG; ++g2) {
      const int src = (g2 * QT + qtile) * 32 + lane;       // same query tile, same lane, key group g2
      const float om0 = rec[32 * 128 + src], om1 = rec[33 * 128 + src];
      const float n0 = fmaxf(mx0, om0), n1 = fmaxf(mx1, om1);
      // a row that saw no key at all keeps maximum -inf on both sides: factors 0, nothing to add
      const float a0 = n0 == -INFINITY ? 0.f : exp_p<SPLIT_P>(mx0 - n0), b0 = n0 == -INFINITY ? 0.f : exp_p<SPLIT_P>(om0 - n0);
      const float a1 = n1 == -INFINITY ? 0.f : exp_p<SPLIT_P>(mx1 - n1), b1 = n1 == -INFINITY ? 0.f : exp_p<SPLIT_P>(om1 - n1);
      den0 = den0 * a0 + rec[34 * 128 + src] * b0;
      den1 = den1 * a1 + rec[35 * 128 + src] * b1;
#pragma unroll
      for (int dt = 0; dt < DH / 8; ++dt) {
        o[dt][0] = o[dt][0] * a0 + rec[(dt * 4 + 0) * 128 + src] * b0;
        o[dt][1] = o[dt][1] * a0 + rec[(dt * 4 + 1) * 128 + src] * b0;
        o[dt][2] = o[dt][2] * a1 + rec[(dt * 4 + 2) * 128 + src] * b1;
        o[dt][3] = o[dt][3] * a1 + rec[(dt * 4 + 3) * 128 + src] * b1;
      }
      mx0 = n0; mx1 = n1;
    }
  }
  bf16* out = reinterpret_cast<bf16*>(p.out);
  if (r0 < nq && nk0 > 0) {
    const float inv = 1.f / den0;
    bf16* dst = out + (size_t)(m0 + r0) * d + h * DH + tq * 2;
#pragma unroll
    for (int dt = 0; dt < DH / 8; ++dt) *reinterpret_cast<uint32_t*>(dst + dt * 8) = pack_bf16(o[dt][0] * inv, o[dt][1] * inv);
  }
  if (r1 < nq && nk1 > 0) {
    const float inv = 1.f / den1;
    bf16* dst = out + (size_t)(m0 + r1) * d + h * DH + tq * 2;
#pragma unroll
    for (int dt = 0; dt < DH / 8; ++dt) *reinterpret_cast<uint32_t*>(dst + dt * 8) = pack_bf16(o[dt][2] * inv, o[dt][3] * inv);
  }
  trace_mark(TR_ATTN, 2);
}

// ---- rows with hundreds of keys ------------------------------------------------------------------------
// In the kernel above a warp walks all K/V tiles of its row one after the other; with 400 keys that is seven tiles of
// dependent-latency-bound instructions.  Here the KEYS are spread over warps instead: a CTA holds QT 16-query tiles x NW key
// warps; warp (qtile, kw) handles the whole 64-key tiles kw, kw + NW, ... of the row for its 16 queries, and the NW partial
// results (running maximum, sum, output) of a query tile are merged through shared memory at the end.
// All tiles of a row are resident at once (up to AL_MAX_SLOTS, in rounds beyond that), and when the keys are older than the
// plan (cross-attention: the encoder wrote them) they are copied before the dependency wait, off the critical path.  
//
// What bounds it: with few queries latency (one round trip for the queries, two tiles per warp, one merge), with an encoder
// pass's thousands the warp instructions of the softmax.  The cross-attention of 8 rows x 25 queries over 400 keys took
// 6.1-6.9 us after the wait with the kernel before (whole tiles per warp too, 4-byte key fragments, keys after the wait: 8 us).
//
// grid = (B * qchunks, H), qchunks = ceil(longest segment / (16 QT)); block = 32 QT NW threads; dynamic shared memory =
// slots * AL_TILE_BYTES + 16 QT rows of queries (att_long_smem).
constexpr int AL_MAX_SLOTS = 9;
constexpr int AL_RECORD = 36;          // floats per thread in the merge
inline int att_long_slots(int max_keys, int threads) {
  const int tiles = (max_keys + AM_KT - 1) / AM_KT, merge = (AL_RECORD * threads * 4 + AL_TILE_BYTES - 1) / AL_TILE_BYTES;
  return tiles < merge ? merge : (tiles > AL_MAX_SLOTS ? AL_MAX_SLOTS : tiles);
}
inline size_t att_long_smem(int slots, int qt) { return (size_t)slots * AL_TILE_BYTES + (size_t)16 * qt * AL_KLD * 2; }

template <int QT, int NW>
__global__ void __launch_bounds__(32 * QT * NW)
attention_long_kernel(const AttnParams p, const int slots, const int kv_old) {
  constexpr int DH = 64;
  constexpr int THREADS = 32 * QT * NW;
  extern __shared__ __align__(16) uint8_t am_smem[];

  trace_mark(TR_ATTN, 0);
  pdl_launch();
  const int b = blockIdx.x / p.qchunks;
  const int chunk = blockIdx.x % p.qchunks;
  const int h = blockIdx.y;
  const int seg_len = plan_load(p.seg_len + b);
  const int i0 = chunk * (16 * QT);
  if (i0 >= seg_len) {
    if ((blockIdx.x | blockIdx.y) == 0) pdl_wait();
    return;
  }
  const int seg_off = plan_load(p.seg_off + b);
  const int kbase = plan_load(p.key_base + b);
  const int row_nk = plan_load(p.nkeys_row + b);
  int q_nsplit = 0;
  size_t q_stride = 0;
  if (p.q_part.ptr) resolve_partials(p.q_part, plan_load(p.M_ptr), q_nsplit, q_stride);
  const int nq = min(16 * QT, seg_len - i0);
  const int m0 = seg_off + i0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tq = lane & 3;           // fragment row (0..7) and column pair (0..3) of this lane
  const int qtile = warp % QT, kw = warp / QT;      // this warp's query tile and key warp
  const bool active = qtile * 16 < nq;              // otherwise the warp only helps loading
  const int d = p.d;
  const bf16* q = reinterpret_cast<const bf16*>(p.q);
  const bf16* kk = reinterpret_cast<const bf16*>(p.k) + (size_t)kbase * d + h * DH;
  const bf16* vv = reinterpret_cast<const bf16*>(p.v) + (size_t)kbase * d + h * DH;
  const int n_tiles = (row_nk + AM_KT - 1) / AM_KT;

  auto fetch_round = [&](int first_tile) {
    for (int tl = 0; tl < min(slots, n_tiles - first_tile); ++tl)
      fetch_kv_tile<THREADS>(am_smem + (size_t)tl * AL_TILE_BYTES, kk, vv, (first_tile + tl) * AM_KT, row_nk, d, tid);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (kv_old) fetch_round(0);
  // this lane's two queries (fragment rows g and g + 8 of the warp's 16) and their visible-key counts
  const int r0 = qtile * 16 + g, r1 = r0 + 8;
  int nk0 = 0, nk1 = 0;
  if (r0 < nq) nk0 = p.nkeys_tok ? min(plan_load(p.nkeys_tok + m0 + r0), row_nk) : row_nk;
  if (r1 < nq) nk1 = p.nkeys_tok ? min(plan_load(p.nkeys_tok + m0 + r1), row_nk) : row_nk;
  pdl_wait();
  trace_mark(TR_ATTN, 1);
  if (!kv_old) fetch_round(0);

  // Queries as A fragments.  Those that come as split-K partial sums of their projection are summed (+ bias) and rounded like
  // stored ones by the whole CTA, every thread issuing all partial loads of its elements at once: one memory round trip.
  uint4 qa[2][2];                                    // [32-wide chunk of the head][row g / g + 8]
  bf16* qs = reinterpret_cast<bf16*>(am_smem + (size_t)slots * AL_TILE_BYTES);   // [16 QT][AL_KLD]
  if (p.q_part.ptr) {
    for (int idx = tid; idx < 16 * QT * (DH / 2); idx += THREADS) {
      const int r = idx / (DH / 2), c2 = (idx - r * (DH / 2)) * 2;
      float2 acc = make_float2(0.f, 0.f);
      if (r < nq) {
        const int c = h * DH + c2;
        if (p.q_bias) acc = *reinterpret_cast<const float2*>(p.q_bias + c);
        const float* src = p.q_part.ptr + (size_t)(m0 + r) * d + c;
        float2 part[ATT_MAX_QSPLIT];
#pragma unroll
        for (int sp = 0; sp < ATT_MAX_QSPLIT; ++sp)
          part[sp] = sp < q_nsplit ? *reinterpret_cast<const float2*>(src + sp * q_stride) : make_float2(0.f, 0.f);
#pragma unroll
        for (int sp = 0; sp < ATT_MAX_QSPLIT; ++sp) { acc.x += part[sp].x; acc.y += part[sp].y; }
      }
      *reinterpret_cast<uint32_t*>(qs + r * AL_KLD + c2) = pack_bf16(acc.x, acc.y);
    }
  } else {
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    const bf16* q0 = q + (size_t)(m0 + r0) * d + h * DH + 8 * tq;
    const bf16* q1 = q + (size_t)(m0 + r1) * d + h * DH + 8 * tq;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      qa[c][0] = r0 < nq ? *reinterpret_cast<const uint4*>(q0 + 32 * c) : zero;
      qa[c][1] = r1 < nq ? *reinterpret_cast<const uint4*>(q1 + 32 * c) : zero;
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();                                   // first round of tiles and the staged queries are in place
  trace_mark(TR_ATTN, 3);
  if (p.q_part.ptr) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      qa[c][0] = *reinterpret_cast<const uint4*>(qs + r0 * AL_KLD + 32 * c + 8 * tq);
      qa[c][1] = *reinterpret_cast<const uint4*>(qs + r1 * AL_KLD + 32 * c + 8 * tq);
    }
  }

  AttnState a;
  attn_init(a);
  for (int first = 0; first < n_tiles; first += slots) {
    if (first > 0) {
      __syncthreads();                               // the previous round is fully consumed
      fetch_round(first);
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();                               // everybody's copies have landed
    }
    for (int tl = kw; active && tl < min(slots, n_tiles - first); tl += NW) {
      const int jw = (first + tl) * AM_KT;           // first key of this tile
      const bf16* ks = reinterpret_cast<const bf16*>(am_smem + (size_t)tl * AL_TILE_BYTES);
      attn_keys<AM_KT, false>(a, qa, ks, ks + AM_KT * AL_KLD, jw, nk0, nk1, p.scale, lane);
    }
  }

  float den0 = a.den0, den1 = a.den1, mx0 = a.mx0, mx1 = a.mx1;
  float (&o)[8][4] = a.o;
  den0 += __shfl_xor_sync(0xffffffffu, den0, 1); den0 += __shfl_xor_sync(0xffffffffu, den0, 2);
  den1 += __shfl_xor_sync(0xffffffffu, den1, 1); den1 += __shfl_xor_sync(0xffffffffu, den1, 2);
  // Merge the key warps of a query tile.  Every lane leaves its fragment (32 outputs, two maxima, two sums) in the tile
  // memory, value-major so that lanes hit different banks.  The merge itself is spread over the key warps as well: key
  // warp kw folds the NW records for the output columns 8 dt .. 8 dt + 7 with dt = kw, kw + NW, ... and stores them
  // (folding everything in key warp 0 took longer than the attention itself).  (AL_RECORD * THREADS floats fit the slots.)
  float* rec = reinterpret_cast<float*>(am_smem);          // [36][THREADS]
  trace_mark(TR_ATTN, 4);
  __syncthreads();                                         // all tile reads are done
#pragma unroll
  for (int dt = 0; dt < DH / 8; ++dt)
#pragma unroll
    for (int e = 0; e < 4; ++e) rec[(dt * 4 + e) * THREADS + tid] = o[dt][e];
  rec[32 * THREADS + tid] = mx0; rec[33 * THREADS + tid] = mx1;
  rec[34 * THREADS + tid] = den0; rec[35 * THREADS + tid] = den1;
  __syncthreads();
  trace_mark(TR_ATTN, 5);
  if (!active) return;
  float n0 = -INFINITY, n1 = -INFINITY;
#pragma unroll
  for (int g2 = 0; g2 < NW; ++g2) {
    const int src = (g2 * QT + qtile) * 32 + lane;         // same query tile, same lane, key warp g2
    n0 = fmaxf(n0, rec[32 * THREADS + src]);
    n1 = fmaxf(n1, rec[33 * THREADS + src]);
  }
  float f0[NW], f1[NW], dsum0 = 0.f, dsum1 = 0.f;
#pragma unroll
  for (int g2 = 0; g2 < NW; ++g2) {
    const int src = (g2 * QT + qtile) * 32 + lane;
    // a key warp that saw no visible key keeps maximum -inf: factor 0 (also when no warp saw any)
    const float om0 = rec[32 * THREADS + src], om1 = rec[33 * THREADS + src];
    f0[g2] = om0 == -INFINITY ? 0.f : __expf(om0 - n0);
    f1[g2] = om1 == -INFINITY ? 0.f : __expf(om1 - n1);
    dsum0 += rec[34 * THREADS + src] * f0[g2];
    dsum1 += rec[35 * THREADS + src] * f1[g2];
  }
  bf16* out = reinterpret_cast<bf16*>(p.out);
  const float inv0 = 1.f / dsum0, inv1 = 1.f / dsum1;
  for (int dt = kw; dt < DH / 8; dt += NW) {
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
    for (int g2 = 0; g2 < NW; ++g2) {
      const int src = (g2 * QT + qtile) * 32 + lane;
      a0 += rec[(dt * 4 + 0) * THREADS + src] * f0[g2];
      a1 += rec[(dt * 4 + 1) * THREADS + src] * f0[g2];
      a2 += rec[(dt * 4 + 2) * THREADS + src] * f1[g2];
      a3 += rec[(dt * 4 + 3) * THREADS + src] * f1[g2];
    }
    if (r0 < nq && nk0 > 0)
      *reinterpret_cast<uint32_t*>(out + (size_t)(m0 + r0) * d + h * DH + tq * 2 + dt * 8) = pack_bf16(a0 * inv0, a1 * inv0);
    if (r1 < nq && nk1 > 0)
      *reinterpret_cast<uint32_t*>(out + (size_t)(m0 + r1) * d + h * DH + tq * 2 + dt * 8) = pack_bf16(a2 * inv1, a3 * inv1);
  }
  trace_mark(TR_ATTN, 2);
}


}  // namespace ad
