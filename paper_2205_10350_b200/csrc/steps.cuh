// The small kernels around the GEMMs and attention: block planning (which tokens are fed at which
// positions), embedding, LayerNorm, the arg-max reduction with the draft compare / first-mismatch decision,
// the commit (cache-length advance / rollback), the input-guided draft policy of Algorithm 1, and the
// planning of the drafter and encoder passes.
#pragma once

#include <type_traits>

#include <cuda_device_runtime_api.h>

#include "ad_common.cuh"

namespace ad {

// Per-row decoding state and per-call block buffers, all resident in the workspace.
struct DevState {
  int* len;        // [B] accepted-prefix length = cached positions
  int* last;       // [B] last accepted token ([BOS] at the start)
  int* fin;        // [B] 1 once [EOS] was accepted or the row's cap was reached
  int* maxlen;     // [B] per-row output cap
  int* srclen;     // [B]
  int* src;        // [B, max_src]
  int* out_ids;    // [B, max_tgt]
  int* drafts;     // [B, kmax]
  int* pred;       // [B, kmax] greedy choices of the last verification
  int* n_acc;      // [B] accepted count of the last verification (0 = nothing to commit)
  int* stat_it;    // [B] iterations the row took part in
  int* stat_acc;   // [B] tokens accepted
  int* stat_off;   // [B] block sizes offered
  int* loop_it;    // [0] iterations with at least one active row, [1] rows-done counter of the accept kernel, [2] iterations of the device-side loop,
                   // [3] their limit, [4] the kernels they launched
  int* status;     // [1] latched device error
  int* all_fin;    // [1] 1 when every row is finished
  int* words;      // [4] what a call may change from one time to the next and a captured graph must not: block-size cap, valid entries of
                   // an override row, beta and tau (float bits) of the relaxed verification
  int* cross_base; // [B] = b * max_src
  int* gidx;       // [B * kmax] drafter: packed token holding mask position i of row b
  int* enc_slot;   // [B * max_src] encoder: cross-K/V slot of packed source token m
  int* user_k;     // [B] staging of caller-provided k
  int* user_drafts;// [B, kmax]
  unsigned int* sync_ctr;  // [128 x 32] per-stage arrival counters of the persistent decoder pass (one per 128-byte line);
                           // every planning kernel that precedes such a pass clears them
};

enum DraftSource : int {
  SRC_USER = 0,      // drafts and k come from the caller (ad_verify_block)
  SRC_OVERRIDE = 1,  // k = min(cap, remaining); drafts = position-aligned stream
  SRC_POLICY = 2,    // Algorithm 1: suffix match on the source
  SRC_SIZES = 3,     // k = min(cap, remaining); drafts left untouched (the drafter fills them)
  SRC_KEEP = 4       // k and drafts as they are (after the drafter); optional override on top
};

struct Dims {
  int B, max_src, max_tgt, kmax;
  int bos, pad, eos, mask;
  int vocab;
};

// Token ids that reach an embedding lookup come from the caller (source, drafts, override stream, forced tokens).
// An id outside [0, vocab) is never used as an index: it is replaced and AD_ERR_ARG is latched.
__device__ __forceinline__ bool id_in_vocab(int id, const Dims& dm) { return id >= 0 && id < dm.vocab; }

// ---------------------------------------------------------------------------------------------
// Suffix match of Algorithm 1, line 3, for one row, executed by one warp.
// o_0 = [BOS], o_t = out[t-1]; x_0 = [BOS], x_t = src[t-1], t <= n.  For q = 0, 1, ... counts the end
// positions i with o[j-q..j] == x[i-q..i]; a unique one is the match, none means no match, several means
// a longer suffix is tried.  Returns i or -1 (same value in every lane).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ int tok_o(const int* out, int t, int bos) { return t == 0 ? bos : out[t - 1]; }

__device__ int warp_suffix_match(const int* out, int j, const int* src, int n, int bos, int lane) {
  for (int q = 0; q <= j; ++q) {
    int count = 0, where = -1;
    for (int i0 = q; i0 <= n; i0 += 32) {
      const int i = i0 + lane;
      bool ok = i <= n;
      for (int t = 0; ok && t <= q; ++t) ok = tok_o(out, j - t, bos) == tok_o(src, i - t, bos);
      const unsigned bal = __ballot_sync(0xffffffffu, ok);
      if (bal) { count += __popc(bal); where = i0 + 31 - __clz(bal); }
    }
    if (count == 1) return where;
    if (count == 0) return -1;
  }
  return -1;
}

// ---------------------------------------------------------------------------------------------
// Chooses every row's block (size and drafted tokens) and lays the block tokens out as packed rows.
// Decoder inputs of row b are (last accepted token, drafts[0..k-2]) at positions len .. len+k-1
// (Eq. 6 / Eq. 7); a negative draft that would be fed is replaced by [PAD].
// Executed by ALL threads of one CTA (any multiple of 32 threads); s_k / s_off: shared arrays of 256 / 257 ints.
// (Inside a decode loop the accept kernel does this for the next iteration, see accept.cuh.)
// ---------------------------------------------------------------------------------------------
struct NextBlock {
  int source;                  // DraftSource
  const int* override_stream;
  int override_stride;
};

__device__ __forceinline__ void plan_verify_block(const DevState& st, const PassPlan& plan, const Dims& dm, const NextBlock& nb,
                                                  int* s_k, int* s_off) {
  const int tid = threadIdx.x, nthreads = blockDim.x, warp = tid >> 5, lane = tid & 31, nwarps = nthreads >> 5;
  const int B = dm.B, source = nb.source, k_cap = __ldcg(st.words), override_len = __ldcg(st.words + 1);
  const int* override_stream = nb.override_stream;
  const int override_stride = nb.override_stride;

  if (source == SRC_POLICY) {
    for (int b = warp; b < B; b += nwarps) {
      int k = 0;
      const int len = __ldcg(st.len + b);
      if (!__ldcg(st.fin + b) && len < st.maxlen[b]) {
        const int n = st.srclen[b];
        const int* src = st.src + (size_t)b * dm.max_src;
        const int i = warp_suffix_match(st.out_ids + (size_t)b * dm.max_tgt, len, src, n, dm.bos, lane);
        int* dr = st.drafts + (size_t)b * dm.kmax;
        if (i >= 0) {
          // draft = x_{i+1..n} followed by the [PAD] slot that matches nothing
          k = n - i + 1;
          k = min(k, min(k_cap, st.maxlen[b] - len));
          for (int t = lane; t < k; t += 32) dr[t] = (i + 1 + t <= n) ? src[i + t] : -1;
        } else {
          k = 1;
          if (lane == 0) dr[0] = -1;
        }
      }
      if (lane == 0) s_k[b] = k;
    }
  } else {
    for (int b = tid; b < B; b += nthreads) {
      int k;
      const int len = __ldcg(st.len + b);
      if (source == SRC_USER) {
        k = st.user_k[b];
        if (k < 0 || k > dm.kmax || len + k > dm.max_tgt) { latch_error(st.status, AD_ERR_ARG); k = 0; }
      } else if (source == SRC_KEEP) {
        k = plan.seg_len[b];
      } else {
        k = (__ldcg(st.fin + b) || len >= st.maxlen[b]) ? 0 : min(k_cap, st.maxlen[b] - len);
      }
      s_k[b] = k;
    }
  }
  __syncthreads();
  if (tid == 0) {
    int acc = 0;
    for (int b = 0; b < B; ++b) { s_off[b] = acc; acc += s_k[b]; }
    s_off[B] = acc;
    *plan.M = acc;
    st.loop_it[1] = 0;   // rows-done counter of the accept kernel: every iteration starts from zero
  }
  if (tid < 128) st.sync_ctr[tid * 32] = 0u;
  __syncthreads();
  for (int b = warp; b < B; b += nwarps) {
    const int k = s_k[b], off = s_off[b], len = __ldcg(st.len + b);
    int* dr = st.drafts + (size_t)b * dm.kmax;
    if (lane == 0) {
      plan.seg_off[b] = off;
      plan.seg_len[b] = k;
      plan.key_base[b] = b * dm.max_tgt;
      plan.row_nk[b] = len + k;
    }
    for (int i = lane; i < k; i += 32) {
      if (source == SRC_USER) dr[i] = st.user_drafts[(size_t)b * dm.kmax + i];
      if (override_stream && (source == SRC_OVERRIDE || source == SRC_KEEP))
        dr[i] = (len + i < override_len) ? override_stream[(size_t)b * override_stride + len + i] : -1;
      // a caller-provided draft beyond the vocabulary becomes a slot that matches nothing (negative = sentinel is legal)
      if (dr[i] >= dm.vocab) { latch_error(st.status, AD_ERR_ARG); dr[i] = -1; }
    }
    __syncwarp();
    for (int i = lane; i < k; i += 32) {
      const int m = off + i;
      int tok = (i == 0) ? __ldcg(st.last + b) : dr[i - 1];
      if (tok < 0 || tok >= dm.vocab) tok = dm.pad;
      plan.tok_row[m] = b;
      plan.tok_pos[m] = len + i;
      plan.tok_id[m] = tok;
      plan.kv_slot[m] = b * dm.max_tgt + len + i;
      plan.att_n[m] = len + i + 1;
    }
  }
}

// A decode loop whose body comes in several forms (each for at most so many tokens): picks the first one that holds the pass that has been planned.
struct BodyPick {
  static constexpr int BODIES = 3;
  unsigned long long node;   // 0: there is one form
  int cap[BODIES - 1];
};
__device__ __forceinline__ void pick_body(const BodyPick& p, int tokens) {
  if (p.node) cudaGraphSetConditional(p.node, tokens <= p.cap[0] ? 0u : tokens <= p.cap[1] ? 1u : 2u);
}

// grid = 1, block = 256.
__global__ void __launch_bounds__(256)
prepare_verify_kernel(DevState st, PassPlan plan, Dims dm, int source, const int* override_stream, int override_stride, BodyPick pick) {
  trace_mark(TR_PREPARE, 0);
  pdl_wait();                  // (no pdl_launch: see plan data in ad_common.cuh)
  trace_mark(TR_PREPARE, 1);
  __shared__ int s_k[256];
  __shared__ int s_off[257];
  NextBlock nb;
  nb.source = source; nb.override_stream = override_stream; nb.override_stride = override_stride;
  plan_verify_block(st, plan, dm, nb, s_k, s_off);
  if (threadIdx.x == 0) pick_body(pick, s_off[dm.B]);
  __threadfence();
}

// ---------------------------------------------------------------------------------------------
// Drafter pass (Section 3.2.1): row b feeds ([BOS], accepted tokens, k x [MASK]) at positions 0 .. len+k
// with no cache and unmasked attention.  blk is the verification plan holding k per row.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
plan_draft_kernel(DevState st, PassPlan blk, PassPlan plan, Dims dm) {
  pdl_wait();                  // (no pdl_launch: see plan data in ad_common.cuh)
  __shared__ int s_off[257];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int B = dm.B;
  if (tid == 0) {
    int acc = 0;
    for (int b = 0; b < B; ++b) {
      s_off[b] = acc;
      const int k = blk.seg_len[b];
      acc += k > 0 ? st.len[b] + 1 + k : 0;
    }
    s_off[B] = acc;
    *plan.M = acc;
  }
  if (tid < 128) st.sync_ctr[tid * 32] = 0u;
  __syncthreads();
  for (int b = warp; b < B; b += 8) {
    const int k = blk.seg_len[b], len = st.len[b], off = s_off[b];
    const int n = k > 0 ? len + 1 + k : 0;
    if (lane == 0) { plan.seg_off[b] = off; plan.seg_len[b] = n; plan.key_base[b] = off; plan.row_nk[b] = n; }
    for (int i = lane; i < n; i += 32) {
      const int m = off + i;
      plan.tok_row[m] = b;
      plan.tok_pos[m] = i;
      int tok = (i == 0) ? dm.bos : (i <= len ? st.out_ids[(size_t)b * dm.max_tgt + i - 1] : dm.mask);
      if (!id_in_vocab(tok, dm)) { latch_error(st.status, AD_ERR_ARG); tok = dm.pad; }
      plan.tok_id[m] = tok;
      plan.kv_slot[m] = m;
      plan.att_n[m] = n;
    }
    for (int i = lane; i < k; i += 32) st.gidx[blk.seg_off[b] + i] = off + len + 1 + i;
  }
  __threadfence();
}

// ---------------------------------------------------------------------------------------------
// Encoder pass: row b feeds its src_len[b] source tokens (padding is simply not packed, and the per-row
// key counts keep it out of every attention).  Also resets the decoding state of every row.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
plan_encode_kernel(DevState st, PassPlan plan, Dims dm, const int* maxlen) {
  pdl_wait();                  // (no pdl_launch: see plan data in ad_common.cuh)
  __shared__ int s_off[257];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int B = dm.B;
  // a device-resident src_len is checked here (the host cannot see it): out-of-range lengths are clamped
  for (int b = tid; b < B; b += 256) {
    const int n = st.srclen[b];
    if (n < 1 || n > dm.max_src) { latch_error(st.status, AD_ERR_ARG); st.srclen[b] = max(1, min(n, dm.max_src)); }
  }
  __syncthreads();
  if (tid == 0) {
    int acc = 0;
    for (int b = 0; b < B; ++b) { s_off[b] = acc; acc += st.srclen[b]; }
    *plan.M = acc;
    *st.loop_it = 0;
    st.loop_it[2] = 0;
    st.loop_it[4] = 0;
    *st.all_fin = 0;
  }
  for (int b = tid; b < B; b += 256) {
    st.len[b] = 0; st.last[b] = dm.bos; st.fin[b] = 0; st.n_acc[b] = 0;
    int ml = maxlen ? maxlen[b] : dm.max_tgt;
    if (ml < 1 || ml > dm.max_tgt) { latch_error(st.status, AD_ERR_ARG); ml = max(1, min(ml, dm.max_tgt)); }
    st.maxlen[b] = ml;
    st.stat_it[b] = 0; st.stat_acc[b] = 0; st.stat_off[b] = 0;
    st.cross_base[b] = b * dm.max_src;
  }
  __syncthreads();
  for (int b = warp; b < B; b += 8) {
    const int n = st.srclen[b], off = s_off[b];
    if (lane == 0) { plan.seg_off[b] = off; plan.seg_len[b] = n; plan.key_base[b] = off; plan.row_nk[b] = n; }
    for (int i = lane; i < n; i += 32) {
      const int m = off + i;
      plan.tok_row[m] = b;
      plan.tok_pos[m] = i;
      int id = st.src[(size_t)b * dm.max_src + i];
      if (!id_in_vocab(id, dm)) { latch_error(st.status, AD_ERR_ARG); id = dm.pad; st.src[(size_t)b * dm.max_src + i] = id; }
      plan.tok_id[m] = id;
      plan.kv_slot[m] = m;
      plan.att_n[m] = n;
      st.enc_slot[m] = b * dm.max_src + i;
    }
  }
  __threadfence();
}

// Inputs of a call into the workspace: sources, lengths, and for ad_generate per-row caps, the draft-override stream, the
// iteration limit of the device-side loop and the words (see DevState).  The arrays are device memory or the handle's mapped pinned staging area, which is
// read in place: one launch instead of a copy per array.  Null pointers: that input is not part of the call.
// grid = B, block = 128.
struct ImportParams {
  const int* src;
  const int* src_len;
  const int* maxlen;
  const int* ovr;
  int src_stride, src_width, ovr_stride, ovr_width, limit;   // limit > 0: a call of ad_generate
  int4 words;
};
__global__ void __launch_bounds__(128)
import_kernel(DevState st, Dims dm, ImportParams p, int* maxlen_out, int* ovr_out) {
  pdl_launch();
  pdl_wait();
  const int b = blockIdx.x, tid = threadIdx.x;
  for (int i = tid; i < p.src_width; i += 128) st.src[(size_t)b * dm.max_src + i] = p.src[(size_t)b * p.src_stride + i];
  if (p.ovr)
    for (int i = tid; i < p.ovr_width; i += 128) ovr_out[(size_t)b * dm.max_tgt + i] = p.ovr[(size_t)b * p.ovr_stride + i];
  if (tid == 0) {
    st.srclen[b] = p.src_len[b];
    if (p.maxlen) maxlen_out[b] = p.maxlen[b];
    if (b == 0 && p.limit > 0) {
      st.loop_it[3] = p.limit;
      *reinterpret_cast<int4*>(st.words) = p.words;
    }
  }
}

// The words alone, for the block-level calls.  One thread.
__global__ void set_words_kernel(DevState st, int4 words) {
  pdl_launch();
  pdl_wait();
  *reinterpret_cast<int4*>(st.words) = words;
}

// ---------------------------------------------------------------------------------------------
// y = emb[token] * sqrt(d) + PE[pos]  ->  FP32 residual stream and the GEMM-operand copy.
// grid = M_cap, block = 128.
// ---------------------------------------------------------------------------------------------
template <typename WT, typename ActT>
__global__ void __launch_bounds__(128)
embed_kernel(PassPlan plan, const WT* __restrict__ emb, const float* __restrict__ pe, int d, float scale,
             float* __restrict__ y, ActT* __restrict__ yb) {
  trace_mark(TR_EMBED, 0);
  pdl_launch();
  pdl_wait();
  trace_mark(TR_EMBED, 1);
  const int m = blockIdx.x;
  if (m >= *plan.M) return;
  const int id = plan.tok_id[m], pos = plan.tok_pos[m];
  for (int i = threadIdx.x; i < d; i += blockDim.x) {
    const float v = to_f32(emb[(size_t)id * d + i]) * scale + pe[(size_t)pos * d + i];
    y[(size_t)m * d + i] = v;
    yb[(size_t)m * d + i] = from_f32<ActT>(v);
  }
}

__device__ __forceinline__ void load4(const float* p, float (&v)[4]) {
  const float4 f = *reinterpret_cast<const float4*>(p);
  v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
}
__device__ __forceinline__ void load4(const bf16* p, float (&v)[4]) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  v[0] = __uint_as_float(u.x << 16); v[1] = __uint_as_float(u.x & 0xffff0000u);
  v[2] = __uint_as_float(u.y << 16); v[3] = __uint_as_float(u.y & 0xffff0000u);
}
__device__ __forceinline__ void store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(bf16* p, float4 v) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  uint2 u;
  u.x = *reinterpret_cast<unsigned int*>(&a);
  u.y = *reinterpret_cast<unsigned int*>(&b);
  *reinterpret_cast<uint2*>(p) = u;
}

// ---------------------------------------------------------------------------------------------
// Residual + LayerNorm:  x = sum_s pre[s][m, :] + bias + resid[m, :];  y = LN(x) (biased variance).
// pre holds the partial sums of the preceding projection (Partials: at most 16).  y may alias resid.  d % 4 == 0, d <= 1024.
// ---------------------------------------------------------------------------------------------
struct LnParams {
  const int* M_ptr;
  Partials pre;
  const float *bias, *resid, *g, *bta;   // bias, resid may be null
  int d;
  float eps;
  float* y;
};

// Sum over the THREADS threads of a group: the CTA (half < 0), or one half of it.
template <int THREADS>
__device__ __forceinline__ void group_sync(int half) {
  if (half < 0) __syncthreads();
  else if (half == 0) asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
  else asm volatile("bar.sync 2, %0;" ::"n"(THREADS) : "memory");
}
template <int THREADS>
__device__ __forceinline__ float group_sum(float v, float* red, int tid, int half) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if ((tid & 31) == 0) red[tid >> 5] = v;      // two calls in turn use two buffers: no barrier in front
  group_sync<THREADS>(half);
  float t = 0.f;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) t += red[w];
  return t;
}

// Gains and biases of one thread's four features: weights, fetched while the previous kernel is still running.
struct LnWeights { float4 g, b, c; };
__device__ __forceinline__ LnWeights ln_weights(const LnParams& p, int gi) {
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  const bool on = gi < (p.d >> 2);
  LnWeights w;
  w.g = on ? reinterpret_cast<const float4*>(p.g)[gi] : zero4;
  w.b = on ? reinterpret_cast<const float4*>(p.bta)[gi] : zero4;
  w.c = on && p.bias ? reinterpret_cast<const float4*>(p.bias)[gi] : zero4;
  return w;
}

// Normalisation of a token whose features a group of THREADS threads holds, four each at off (`on`: this thread has some).
template <typename ActT, int THREADS>
__device__ __forceinline__ void ln_finish(const LnParams& p, const LnWeights& w, size_t off, bool on, float4 v, ActT* yb, float* red, int tid, int half) {
  const float mean = group_sum<THREADS>(v.x + v.y + v.z + v.w, red, tid, half) / (float)p.d;
  float vs = 0.f;
  if (on) {
    const float a = v.x - mean, b = v.y - mean, c = v.z - mean, e = v.w - mean;
    vs = a * a + b * b + c * c + e * e;
  }
  const float inv = rsqrtf(group_sum<THREADS>(vs, red + THREADS / 32, tid, half) / (float)p.d + p.eps);
  if (on) {
    float4 o;
    o.x = w.g.x * ((v.x - mean) * inv) + w.b.x;
    o.y = w.g.y * ((v.y - mean) * inv) + w.b.y;
    o.z = w.g.z * ((v.z - mean) * inv) + w.b.z;
    o.w = w.g.w * ((v.w - mean) * inv) + w.b.w;
    store4(p.y + off * 4, o);
    store4(yb + off * 4, o);
  }
}

__device__ __forceinline__ void add4(float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; }
// v += all partial sums.  FP32 models: pairwise among themselves first.  They are small beside the residual in v, at whose magnitude each of up to 32 additions
// would round.  Scores of two layers, error against 64 bits, rms: 128 wide, 4 x 30 tokens, one after the other 5.7e-8, pairwise 4.3e-8 (projections in kernels of
// their own, one sum: 4.3e-8); 256 wide 9.4e-8, 7.2e-8 (7.3e-8), 32 sums 8.8e-8, 7.0e-8 (7.5e-8).
template <typename ActT, int P>
__device__ __forceinline__ void add_partials(float4& v, float4 (&part)[P]) {
  if constexpr (std::is_same<ActT, float>::value) {
#pragma unroll
    for (int n = P / 2; n > 0; n /= 2)
#pragma unroll
      for (int i = 0; i < n; ++i) add4(part[i], part[i + n]);
    add4(v, part[0]);
  } else {
#pragma unroll
    for (int sp = 0; sp < P; ++sp) add4(v, part[sp]);
  }
}

// Token m by a group of THREADS threads, four features per thread (d <= 4 * THREADS): the residual and all partial sums of a thread
// (P of them at most) are requested at once, so that the kernel costs one memory round trip.  (Two groups of features per thread took
// 2.8 us instead of 1.5 us per launch on a 1024-wide model with 16 partials; 9 to 16 partials in two turns of eight, with 64
// registers: whole calls 768 wide +2.5 %, 1024 wide +3 %.)
template <typename ActT, int THREADS, int P>
__device__ __forceinline__ void ln_token(const LnParams& p, const LnWeights& w, int m, int nsplit, size_t stride, ActT* yb, float* red,
                                         int tid, int half) {
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  const int groups = p.d >> 2;
  const size_t off = (size_t)m * groups + tid;
  const bool on = tid < groups;
  float4 v = zero4;
  if (on) {
    const float4* pre = reinterpret_cast<const float4*>(p.pre.ptr) + off;
    const size_t step = stride >> 2;               // (stride is a multiple of d, d of 4)
    float4 part[P];
#pragma unroll
    for (int sp = 0; sp < P; ++sp, pre += step) part[sp] = sp < nsplit ? *pre : zero4;
    const float4 r = p.resid ? reinterpret_cast<const float4*>(p.resid)[off] : zero4;
    v = make_float4(w.c.x + r.x, w.c.y + r.y, w.c.z + r.z, w.c.w + r.w);
    add_partials<ActT, P>(v, part);
  }
  ln_finish<ActT, THREADS>(p, w, off, on, v, yb, red, tid, half);
}
// One CTA per token.  grid = M_cap, block = THREADS (128 for d <= 512, else 256).
// What bounds it: one memory round trip (1.0-1.3 us), and what it keeps from the projection behind it, whose CTAs (32 K registers and up to
// 200 KB of shared memory each) want to be on the SM before this kernel's wait is over.  With room for 16 partial sums whatever their number
// (96 registers) the CTAs of a few hundred tokens filled the register files; now 48 or 64 for up to 4 or 8, 96 only for more (12 and 16
// heads).  Whole calls: 768 wide, batch 16 5090 -> 4805 us; 512 wide, batch 24 with drafter 6310 -> 6000, batch 32 5385 -> 5170; batch 1
// 1177 -> 1135.  With a tail loop for sums beyond P, which no pass has, it was 128 registers and 0.3 to 0.6 % of every decode call more.
template <typename ActT, int THREADS, int P>
__global__ void __launch_bounds__(THREADS, (P <= 4 ? 1280 : P <= 8 ? 1024 : 512) / THREADS)
layernorm_kernel(const LnParams p, ActT* __restrict__ yb) {
  __shared__ float red[2 * (THREADS / 32)];
  trace_mark(TR_LN, 0);
  pdl_launch();
  const int m = blockIdx.x, M = plan_load(p.M_ptr);
  const LnWeights w = ln_weights(p, threadIdx.x);
  if (m >= M && m > 0) return;                     // CTA 0 always waits (see early exits in ad_common.cuh)
  int nsplit;
  size_t stride;
  resolve_partials(p.pre, M, nsplit, stride);
  pdl_wait();
  trace_mark(TR_LN, 1);
  if (m >= M) return;
  ln_token<ActT, THREADS, P>(p, w, m, nsplit, stride, yb, red, threadIdx.x, -1);
  trace_mark(TR_LN, 2);
}

// 17 to 32 partial sums, d <= 512: two halves of a CTA add up to 16 each.  One CTA per token; grid = M_cap, block = 256.  What bounds it is the 64 KB that
// a token's sums are (512 wide): half a microsecond on one SM.
template <typename ActT>
__global__ void __launch_bounds__(256, 2)
layernorm_parts_kernel(const LnParams p, ActT* __restrict__ yb) {
  __shared__ float red[2 * 4];
  __shared__ __align__(16) float4 other[128];
  trace_mark(TR_LN, 0);
  pdl_launch();
  const int m = blockIdx.x, M = plan_load(p.M_ptr), half = threadIdx.x >> 7, tid = threadIdx.x & 127;
  const LnWeights w = ln_weights(p, tid);
  if (m >= M && m > 0) return;                     // CTA 0 always waits (see early exits in ad_common.cuh)
  pdl_wait();
  trace_mark(TR_LN, 1);
  if (m >= M) return;
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  const size_t off = (size_t)m * (p.d >> 2) + tid, step = p.pre.stride >> 2;
  const bool on = tid < (p.d >> 2);
  float4 v = zero4, base = zero4;                  // (FP32: the residual is added last, see add_partials)
  if (on) {
    const int n = p.pre.nsplit, first = half * 16;
    const float4* pre = reinterpret_cast<const float4*>(p.pre.ptr) + off + first * step;
    float4 part[16];
#pragma unroll
    for (int sp = 0; sp < 16; ++sp, pre += step) part[sp] = first + sp < n ? *pre : zero4;
    if (half == 0) {
      const float4 r = p.resid ? reinterpret_cast<const float4*>(p.resid)[off] : zero4;
      base = make_float4(w.c.x + r.x, w.c.y + r.y, w.c.z + r.z, w.c.w + r.w);
    }
    if (!std::is_same<ActT, float>::value) v = base;
    add_partials<ActT, 16>(v, part);
  }
  if (half == 1) other[tid] = v;
  __syncthreads();
  if (half == 1) return;
  add4(v, other[tid]);
  if (std::is_same<ActT, float>::value) add4(v, base);
  ln_finish<ActT, 128>(p, w, off, on, v, yb, red, tid, 0);
  trace_mark(TR_LN, 2);
}

// Passes that may hold many tokens: two tokens (one for d > 512) per CTA and turn.  grid: at most four CTAs per SM, which loop (a grid sized
// for the capacity cost 5 us per launch in waves of CTAs without work); block = 256.
template <typename ActT, int THREADS, int P>
__global__ void __launch_bounds__(256, P <= 8 ? 4 : 2)
layernorm_many_kernel(const LnParams p, ActT* __restrict__ yb) {
  constexpr int TOKENS = 256 / THREADS;
  __shared__ float red[TOKENS][2 * (THREADS / 32)];
  trace_mark(TR_LN, 0);
  pdl_launch();
  const int M = plan_load(p.M_ptr);
  int m = blockIdx.x * TOKENS;
  if (m >= M && blockIdx.x > 0) return;
  const int half = TOKENS == 1 ? 0 : threadIdx.x / THREADS, tid = threadIdx.x % THREADS;
  const LnWeights w = ln_weights(p, tid);
  int nsplit;
  size_t stride;
  resolve_partials(p.pre, M, nsplit, stride);
  pdl_wait();
  trace_mark(TR_LN, 1);
  for (m += half; m < M; m += gridDim.x * TOKENS) ln_token<ActT, THREADS, P>(p, w, m, nsplit, stride, yb, red[half], tid, TOKENS == 1 ? -1 : half);
  trace_mark(TR_LN, 2);
}

// dst[j, :] = src[gidx[j], :] for j < *M_ptr.  grid = M_cap, block = 128.
template <typename ActT>
__global__ void __launch_bounds__(128)
gather_rows_kernel(const int* __restrict__ M_ptr, const int* __restrict__ gidx, const ActT* __restrict__ src,
                   ActT* __restrict__ dst, int d) {
  pdl_launch();
  const int j = blockIdx.x;
  const bool have = j < plan_load(M_ptr);
  if (!have && j > 0) return;
  const int s = have ? plan_load(gidx + j) : 0;
  pdl_wait();
  if (!have) return;
  for (int i = threadIdx.x; i < d; i += blockDim.x) dst[(size_t)j * d + i] = src[(size_t)s * d + i];
}

// ---------------------------------------------------------------------------------------------
// Commit of one row (Algorithm 1 lines 6-7): n > 0 appends pred[0..n) to the row's output, advances the cache
// length, sets the last token and the finished flag; n < 0 rolls |n| committed tokens back; n = 0 discards
// the block.  Executed by one warp.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void commit_row(const DevState& st, const PassPlan& blk, const Dims& dm, int b, int n,
                                           int nacc, int lane) {
  int len = st.len[b];
  if (n > nacc || (n < 0 && -n > len)) {
    if (lane == 0) latch_error(st.status, AD_ERR_ARG);
    n = 0;
  }
  __syncwarp();
  if (n > 0) {
    const int* pred = st.pred + (size_t)b * dm.kmax;
    int* out = st.out_ids + (size_t)b * dm.max_tgt;
    for (int i = lane; i < n; i += 32) out[len + i] = pred[i];
    if (lane == 0) {
      const int last = pred[n - 1];
      len += n;
      st.len[b] = len;
      st.last[b] = last;
      if (last == dm.eos || len >= st.maxlen[b]) st.fin[b] = 1;
      st.stat_acc[b] += n;
    }
  } else if (n < 0 && lane == 0) {
    len += n;
    st.len[b] = len;
    st.last[b] = len > 0 ? st.out_ids[(size_t)b * dm.max_tgt + len - 1] : dm.bos;
    st.fin[b] = 0;
  }
  if (lane == 0) {
    if (nacc > 0) {
      st.stat_it[b] += 1;
      st.stat_off[b] += blk.seg_len[b];
    }
    st.n_acc[b] = 0;
  }
}

// Hands the latched status word to the host (mapped memory) and clears it.  One thread.
__device__ __forceinline__ void export_status(const DevState& st, int* status_out) {
  *status_out = atomicExch(st.status, 0);
}
__global__ void export_status_kernel(DevState st, int* status_out) {
  pdl_launch();
  pdl_wait();
  if (threadIdx.x == 0) export_status(st, status_out);
}

// After every row has been committed: loop counter and the "all rows finished" word.  One thread.
__device__ __forceinline__ void finish_iteration(const DevState& st, const Dims& dm, bool any_active) {
  int all = 1;
  for (int b = 0; b < dm.B; ++b) all &= (__ldcg(st.fin + b) != 0);
  if (any_active) *st.loop_it += 1;
  *st.all_fin = all;
}

// ---------------------------------------------------------------------------------------------
// Relaxed verification (Section 3.2.3): score of every block position's drafted token,
// draft_val[m] = x[m, :] . emb[draft, :], and its id (negative: sentinel, never kept).  The projection kernel
// then counts, per position, the other tokens that score strictly higher (Eq. 8), and the accept kernel applies
// Eq. 8 and Eq. 9.  One warp per packed token; grid = ceil(M_cap / 8), block = 256.
// ---------------------------------------------------------------------------------------------
template <typename WT, typename ActT>
__global__ void __launch_bounds__(256)
draft_score_kernel(DevState st, PassPlan blk, Dims dm, const WT* __restrict__ emb, const ActT* __restrict__ x, int d,
                   float* __restrict__ draft_val, int* __restrict__ draft_id) {
  pdl_launch();
  pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = blockIdx.x * 8 + warp;
  if (m >= *blk.M) return;
  const int b = blk.tok_row[m];
  int id = st.drafts[(size_t)b * dm.kmax + (m - blk.seg_off[b])];
  if (id >= dm.vocab) id = -1;
  float acc = 0.f;
  if (id >= 0)
    for (int i = lane; i < d; i += 32) acc = fmaf(to_f32(x[(size_t)m * d + i]), to_f32(emb[(size_t)id * d + i]), acc);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) { draft_val[m] = acc; draft_id[m] = id; }
}

// ---------------------------------------------------------------------------------------------
// Commit as a call of its own (ad_commit): cache-length advance or rollback.  n_in == null commits n_acc.
// grid = 1, block = 256 (one warp per row at a time).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
commit_kernel(DevState st, PassPlan blk, Dims dm, const int* n_in, int* status_out) {
  __shared__ int s_active;
  trace_mark(TR_COMMIT, 0);
  pdl_launch();
  pdl_wait();
  trace_mark(TR_COMMIT, 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) s_active = 0;
  __syncthreads();
  for (int b = warp; b < dm.B; b += 8) {
    const int nacc = st.n_acc[b];
    const int n = n_in ? n_in[b] : nacc;
    __syncwarp();
    commit_row(st, blk, dm, b, n, nacc, lane);
    if (lane == 0 && nacc > 0) atomicOr(&s_active, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    finish_iteration(st, dm, s_active != 0);
    if (status_out) export_status(st, status_out);
  }
}

// Teacher-forced commit: the caller supplies the accepted tokens.  grid = 1, block = 256.
__global__ void __launch_bounds__(256)
force_commit_kernel(DevState st, PassPlan blk, Dims dm, const int* tokens, const int* n_in, int* status_out) {
  pdl_launch();
  pdl_wait();
  for (int b = threadIdx.x; b < dm.B; b += 256) {
    const int n = n_in[b], k = blk.seg_len[b];
    const int* tk = tokens + (size_t)b * dm.kmax;
    const int* dr = st.drafts + (size_t)b * dm.kmax;
    bool ok = n >= 0 && n <= k;
    for (int i = 0; ok && i + 1 < n; ++i) ok = tk[i] == dr[i];
    for (int i = 0; ok && i < n; ++i) ok = id_in_vocab(tk[i], dm);      // the last one is fed to the next block
    if (!ok) { latch_error(st.status, AD_ERR_ARG); continue; }
    if (n > 0) {
      int len = st.len[b];
      int* out = st.out_ids + (size_t)b * dm.max_tgt;
      for (int i = 0; i < n; ++i) out[len + i] = tk[i];
      len += n;
      st.len[b] = len;
      st.last[b] = tk[n - 1];
      if (tk[n - 1] == dm.eos || len >= st.maxlen[b]) st.fin[b] = 1;
    }
    st.n_acc[b] = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0 && status_out) export_status(st, status_out);
}

// Copies the block results to caller-visible arrays (device pointers).  grid = B, block = 64.
__global__ void export_block_kernel(DevState st, Dims dm, int* argmax_out, int* n_out, int* drafts_out, int* k_out,
                                    PassPlan blk) {
  pdl_launch();
  pdl_wait();
  const int b = blockIdx.x;
  if (argmax_out)
    for (int i = threadIdx.x; i < dm.kmax; i += blockDim.x) argmax_out[(size_t)b * dm.kmax + i] = st.pred[(size_t)b * dm.kmax + i];
  if (drafts_out)
    for (int i = threadIdx.x; i < dm.kmax; i += blockDim.x) drafts_out[(size_t)b * dm.kmax + i] = st.drafts[(size_t)b * dm.kmax + i];
  if (threadIdx.x == 0) {
    if (n_out) n_out[b] = st.n_acc[b];
    if (k_out) k_out[b] = blk.seg_len[b];
  }
}

// The same into mapped host memory, for calls with host-resident arrays: block[0] = status word (cleared),
// block[4 .. 4 + B) = n_accepted (drafts: block sizes), then [B, kmax] ids.  grid = B, block = 64.
__global__ void export_host_kernel(DevState st, Dims dm, PassPlan blk, int drafts, int* block) {
  pdl_launch();
  pdl_wait();
  const int b = blockIdx.x;
  const int* ids = (drafts ? st.drafts : st.pred) + (size_t)b * dm.kmax;
  for (int i = threadIdx.x; i < dm.kmax; i += blockDim.x) block[4 + dm.B + (size_t)b * dm.kmax + i] = ids[i];
  if (threadIdx.x == 0) {
    block[4 + b] = drafts ? blk.seg_len[b] : st.n_acc[b];
    if (b == 0) export_status(st, block);
  }
}

// End of ad_generate: everything the host needs, gathered into one block (device pointer of pinned, mapped host memory
// or a device buffer), so that the call ends with ONE synchronisation and no further copies:
//   block[0] = iterations the device-side loop ran, block[1] = latched status word (cleared here),
//   block[2] = iterations with an active row, block[3] = kernels that the device-side loop launched,
//   block[4 + 4 b ..] = {row iterations, accepted, offered, output length} of row b,
//   block[4 + 4 B + b * max_tgt ..] = output ids of row b (only when out_dev is null: host-resident results).
// out_dev / out_len_dev (device pointers, may be null): the caller's result arrays when they live on the device.
// grid = B, block = 128.
__global__ void __launch_bounds__(128)
finalize_generate_kernel(DevState st, Dims dm, int* out_dev, int out_stride, int* out_len_dev, int* block) {
  pdl_launch();
  pdl_wait();
  const int b = blockIdx.x, tid = threadIdx.x;
  const int len = st.len[b];
  if (tid == 0) {
    if (b == 0) {
      block[0] = st.loop_it[2];
      block[1] = *st.status;
      *st.status = 0;
      block[2] = st.loop_it[0];
      block[3] = st.loop_it[4];
    }
    int* row = block + 4 + 4 * b;
    row[0] = st.stat_it[b]; row[1] = st.stat_acc[b]; row[2] = st.stat_off[b]; row[3] = len;
    if (out_len_dev) out_len_dev[b] = len;
  }
  const int* src = st.out_ids + (size_t)b * dm.max_tgt;
  if (out_dev) {
    const int w = min(out_stride, dm.max_tgt);
    for (int i = tid; i < w; i += 128) out_dev[(size_t)b * out_stride + i] = src[i];
  } else {
    int* dst = block + 4 + 4 * dm.B + (size_t)b * dm.max_tgt;
    for (int i = tid; i < dm.max_tgt; i += 128) dst[i] = src[i];
  }
}

// FP32 copy of an activation buffer (debug).  grid-stride.
template <typename ActT>
__global__ void to_f32_kernel(const ActT* __restrict__ src, float* __restrict__ dst, size_t n) {
  pdl_launch();
  pdl_wait();
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = to_f32(src[i]);
}

}  // namespace ad
