// End of a projection: final arg-max over its per-tile partials, the accept decision, and -- inside a decode loop -- the
// commit, the choice of the next block and the layout of the pass that verifies it, all in one kernel.
#pragma once

#include <type_traits>

#include "gemm_tc.cuh"   // float_key
#include "steps.cuh"

namespace ad {

// What the accept kernel prepares for the pass behind it (source < 0: nothing).
struct NextPass {
  static constexpr int BODIES = BodyPick::BODIES;
  typedef BodyPick Pick;
  int source;            // SRC_POLICY / SRC_OVERRIDE: plan the next verification block after the commit;
                         // SRC_SIZES: plan the drafter's pass after the commit (block sizes, then its tokens);
                         // SRC_KEEP (drafter's choices): plan the verification of the block just drafted
  const int* override_stream;
  int override_stride;
  PassPlan draft;        // SRC_SIZES: plan of the drafter's pass
  Pick pick;
  int launches;          // kernels of this iteration
};

constexpr int ACC_THREADS = 1024;
constexpr int ACC_SRC = 512;            // source tokens kept in shared memory for the suffix match

// Suffix match of Algorithm 1, line 3 (see warp_suffix_match) by the whole CTA: every thread looks at the end positions
// tid, tid + 1024, ... of the source.  o(t): output token t (o(0) = [BOS]); x: source tokens; *where: shared word.
template <typename OutTok>
__device__ __forceinline__ int cta_suffix_match(OutTok o, int j, const int* x, int n, int bos, int* where) {
  int found = -1;
  for (int q = 0; q <= j; ++q) {
    int count = 0;
    for (int i0 = q; i0 <= n; i0 += ACC_THREADS) {
      const int i = i0 + (int)threadIdx.x;
      bool ok = i <= n;
      for (int t = 0; ok && t <= q; ++t) ok = o(j - t) == (i - t == 0 ? bos : x[i - t - 1]);
      if (ok) *where = i;
      count += __syncthreads_count(ok);
    }
    if (count == 1) { found = *where; break; }
    if (count == 0) break;
    __syncthreads();
  }
  return found;
}

// Arg-max over the tiles of H block positions (i0, i0 + 32, ...) by one warp, the lowest id on ties; U tiles per lane and
// position in flight.  COUNT: also the sum of the tiles' counts.  decide(position, maximum, id, count) runs in lane 0.
template <int H, int U, bool COUNT, typename F>
__device__ __forceinline__ void scan_tiles(const float* __restrict__ val, const int* __restrict__ id, const int* __restrict__ cnt, int off, int i0,
                                           int k, int n_tiles, int lane, F decide) {
  float v[H];
  int idx[H], higher[H];
#pragma unroll
  for (int h = 0; h < H; ++h) { v[h] = -INFINITY; idx[h] = 0x7fffffff; higher[h] = 0; }
  for (int t0 = 0; t0 < n_tiles; t0 += 32 * U) {
    float pv[H][U];
    int pi[H][U], pc[H][COUNT ? U : 1];
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const int i = i0 + 32 * h;
      const size_t row = (size_t)(off + i) * n_tiles;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int t = t0 + 32 * u + lane;
        const bool on = i < k && t < n_tiles;
        pv[h][u] = on ? val[row + t] : -INFINITY;
        pi[h][u] = on ? id[row + t] : 0x7fffffff;
        if (COUNT) pc[h][u] = on ? cnt[row + t] : 0;
      }
    }
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (pv[h][u] > v[h] || (pv[h][u] == v[h] && pi[h][u] < idx[h])) { v[h] = pv[h][u]; idx[h] = pi[h][u]; }   // (-inf included)
        if (COUNT) higher[h] += pc[h][u];
      }
  }
#pragma unroll
  for (int h = 0; h < H; ++h) {
    if (i0 + 32 * h >= k) break;
    const unsigned int key = tc::float_key(v[h] + 0.f);      // (-0 and +0 are equal scores)
    const unsigned int best = __reduce_max_sync(0xffffffffu, key);
    const unsigned int lowest = __reduce_min_sync(0xffffffffu, key == best ? (unsigned int)idx[h] : 0x7fffffffu);
    if (COUNT) higher[h] = __reduce_add_sync(0xffffffffu, higher[h]);
    if (lane == 0) decide(i0 + 32 * h, tc::key_float(best), (int)lowest, higher[h]);
  }
}

// The decision for one row:
//   c = first block position whose greedy choice differs from the draft (Section 3.1.1; definition of c in Section 3.2),
//   n = c + 1 (the bifurcation token is kept), n = k when nothing differs, cut at the first accepted [EOS].
// relaxed_on: relaxed verification of Section 3.2.3 -- a position keeps its drafted token when fewer than beta other tokens
//   score strictly higher (Eq. 8: the draft is within the top beta) and the best score exceeds the draft's by at most tau
//   (Eq. 9; differences of log-likelihoods are differences of scores); otherwise the greedy choice.  beta and tau: st.words.
// to_drafts: the choices are the row's drafts and nothing is compared.
// auto_commit (decode loop): n is committed at once (Algorithm 1 lines 6-7); what concerns one row alone (suffix match, drafts,
//   sizes) is done by the row's own CTA.  The loop counters, the all-finished word and, with next.source >= 0, the layout of the
//   pass behind this kernel need all rows; how these meet is the kernel's form:
//   ACC_ONE        there is one row;
//   ACC_CLUSTERED  2 to ACC_CLUSTER rows of a decode loop, as many as the device places as one cluster: each CTA tells the others its next
//                  block's size through distributed shared memory and lays its own row out, row 0's updates the loop words;
//   ACC_ROWS       through global memory: the last CTA to finish (done_ctr: rows done in the low half, active rows in the high
//                  half; left at zero) reads what the others wrote, updates the loop words and lays out all rows (3.3 us and 1.8 us: an
//                  iteration takes 2.2 us longer than with a cluster with 4 rows, 3 us with 8).
//   (Calls that commit nothing need no other row and run as one of the first and the last.)
//
// What bounds it: a chain of dependent memory round trips, so whatever older kernels wrote (row state, drafts, source) is
// read before the dependency wait, and from the partials to the next plan everything stays in shared memory: one round trip
// for the partials (plus the hand-over between CTAs when B > 1).
// Batch 1, 40-token blocks: 11.4 us with the state, the match and the plan in global memory.
// grid = B, block = 1024; ACC_CLUSTERED: cluster (B, 1, 1).
constexpr int ACC_CLUSTER = 16;
enum AcceptForm { ACC_ONE, ACC_CLUSTERED, ACC_ROWS };
template <AcceptForm FORM>
__global__ void __launch_bounds__(ACC_THREADS)
argmax_accept_kernel(DevState st, PassPlan blk, Dims dm, const float* __restrict__ part_val, const int* __restrict__ part_idx,
                     int n_tiles, int to_drafts, int auto_commit, unsigned int* done_ctr, unsigned long long cond, int relaxed_on,
                     const float* __restrict__ draft_val, const int* __restrict__ draft_id,
                     const int* __restrict__ part_cnt, NextPass next) {
  constexpr bool CLUSTER = FORM == ACC_CLUSTERED;
  __shared__ int s_dr[256], s_pred[256], s_src[ACC_SRC];
  __shared__ int s_k[256], s_off[256], s_boff[256], s_len[256];
  __shared__ int s_next[256], s_row[CLUSTER ? ACC_CLUSTER : 1];   // the next block's drafts; per row: 1 finished, 2 took part
  __shared__ int s_n, s_last_cta, s_where;
  if (CLUSTER) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");      // (a CTA's shared memory may be written once it is known to run)
  trace_mark(TR_ACCEPT, 0);
  if (next.source < 0) pdl_launch();     // a kernel that plans never does (see plan data in ad_common.cuh)
  const int b = blockIdx.x, B = dm.B;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // ---- what older kernels wrote ----
  const int k = plan_load(blk.seg_len + b), off = plan_load(blk.seg_off + b);
  const int len = plan_load(st.len + b), maxlen = plan_load(st.maxlen + b), old_last = plan_load(st.last + b);
  const int old_fin = plan_load(st.fin + b);
  const int4 words = __ldcg(reinterpret_cast<const int4*>(st.words));
  const int k_cap = words.x, override_len = words.y, beta = words.z;
  const float tau = __int_as_float(words.w);
  // the first thread's row counters, the last one's loop counters
  const bool counts = tid == 0 || (tid == ACC_THREADS - 1 && auto_commit);
  const int ctr0 = counts ? plan_load(tid == 0 ? st.stat_acc + b : st.loop_it) : 0;
  const int ctr1 = counts ? plan_load(tid == 0 ? st.stat_it + b : st.loop_it + 2) : 0;
  const int ctr2 = counts ? plan_load(tid == 0 ? st.stat_off + b : st.loop_it + 3) : 0;
  if (!to_drafts && tid < k) s_dr[tid] = plan_load(st.drafts + (size_t)b * dm.kmax + tid);     // k <= kmax <= 256
  int n_src = 0;
  const int* x = st.src + (size_t)b * dm.max_src;
  if (next.source == SRC_POLICY) {
    n_src = plan_load(st.srclen + b);
    if (n_src <= ACC_SRC) {
      for (int i = tid; i < n_src; i += ACC_THREADS) s_src[i] = plan_load(x + i);
      x = s_src;
    }
  }
  pdl_wait();
  trace_mark(TR_ACCEPT, 1);

  // ---- arg-max over the tiles of every block position: a warp per position, the lowest id wins ties ----
  const bool relaxed = relaxed_on && !to_drafts;
  int* pred = (to_drafts ? st.drafts : st.pred) + (size_t)b * dm.kmax;
  auto decide = [&](int i, float v, int idx, int higher) {      // lane 0 of the position's warp
    int choice = idx < dm.vocab ? idx : 0;                        // a position without any ordered score (NaN) still gets an id that exists
    if (relaxed) {
      const int did = draft_id[off + i];
      if (did >= 0 && higher <= beta - 1 && v - draft_val[off + i] <= tau) choice = did;
    }
    s_pred[i] = choice;
    if (!(to_drafts && next.source == SRC_KEEP)) pred[i] = choice;
  };
  if (relaxed) {
    for (int i = warp; i < k; i += ACC_THREADS / 32) scan_tiles<1, 8, true>(part_val, part_idx, part_cnt, off, i, k, n_tiles, lane, decide);
  } else if (k <= ACC_THREADS / 32) {
    if (warp < k) scan_tiles<1, 16, false>(part_val, part_idx, part_cnt, off, warp, k, n_tiles, lane, decide);
  } else {
    for (int i = warp; i < k; i += 2 * (ACC_THREADS / 32)) scan_tiles<2, 8, false>(part_val, part_idx, part_cnt, off, i, k, n_tiles, lane, decide);
  }
  __syncthreads();

  if (to_drafts) {
    if (next.source != SRC_KEEP) return;
    // the drafted block becomes the verification block of this row: its place among the packed tokens is known already
    int dr = -1;
    if (tid < k) {
      dr = s_pred[tid];
      if (next.override_stream) dr = len + tid < override_len ? next.override_stream[(size_t)b * next.override_stride + len + tid] : -1;
      if (dr >= dm.vocab) { latch_error(st.status, AD_ERR_ARG); dr = -1; }
      s_dr[tid] = dr;
      st.drafts[(size_t)b * dm.kmax + tid] = dr;
    }
    __syncthreads();
    if (tid < k) {
      int tok = tid == 0 ? old_last : s_dr[tid - 1];
      if (tok < 0 || tok >= dm.vocab) tok = dm.pad;
      const int m = off + tid;
      blk.tok_row[m] = b; blk.tok_pos[m] = len + tid; blk.tok_id[m] = tok;
      blk.kv_slot[m] = b * dm.max_tgt + len + tid; blk.att_n[m] = len + tid + 1;
    }
    if (tid == 0) {
      blk.key_base[b] = b * dm.max_tgt; blk.row_nk[b] = len + k;
      if (b == 0) st.loop_it[1] = 0;
    }
    __threadfence();
    trace_mark(TR_ACCEPT, 2);
    return;
  }

  // ---- the decision ----
  trace_mark(TR_ACCEPT, 3);
  int n = k;                               // (every warp for itself)
  for (int i0 = 0; i0 < k; i0 += 32) {
    const int i = i0 + lane;
    const unsigned bal = __ballot_sync(0xffffffffu, i < k && (s_dr[i] < 0 || s_pred[i] != s_dr[i]));
    if (bal) { n = i0 + __ffs(bal); break; }
  }
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane;
    const unsigned bal = __ballot_sync(0xffffffffu, i < n && s_pred[i] == dm.eos);
    if (bal) { n = i0 + __ffs(bal); break; }
  }
  if (!auto_commit) {
    if (tid == 0) st.n_acc[b] = n;
    return;
  }

  // ---- commit ----
  trace_mark(TR_ACCEPT, 4);
  const int len1 = len + n, last1 = n > 0 ? s_pred[n - 1] : old_last;
  const int fin1 = old_fin || (n > 0 && (last1 == dm.eos || len1 >= maxlen));
  if (tid < n) st.out_ids[(size_t)b * dm.max_tgt + len + tid] = s_pred[tid];
  if (tid == 0) {
    st.n_acc[b] = 0;
    if (n > 0) {
      st.len[b] = len1; st.last[b] = last1; st.fin[b] = fin1;
      st.stat_acc[b] = ctr0 + n; st.stat_it[b] = ctr1 + 1; st.stat_off[b] = ctr2 + k;
    }
  }
  // ---- this row's next block ----
  int k1 = 0;
  if (next.source >= 0) {
    const bool live = !fin1 && len1 < maxlen;
    if (next.source == SRC_POLICY) {
      if (live) {
        const int* old_out = st.out_ids + (size_t)b * dm.max_tgt;
        auto o = [&](int t) { return t == 0 ? dm.bos : (t - 1 >= len ? s_pred[t - 1 - len] : __ldcg(old_out + t - 1)); };
        const int i = cta_suffix_match(o, len1, x, n_src, dm.bos, &s_where);
        // draft = x_{i+1..n} followed by the [PAD] slot that matches nothing; a plain step without a match
        k1 = i >= 0 ? min(n_src - i + 1, min(k_cap, maxlen - len1)) : 1;
        if (tid < k1) s_next[tid] = (i >= 0 && i + 1 + tid <= n_src) ? x[i + tid] : -1;
      }
    } else {
      k1 = live ? min(k_cap, maxlen - len1) : 0;
      if (next.source == SRC_OVERRIDE && tid < k1)
        s_next[tid] = len1 + tid < override_len ? next.override_stream[(size_t)b * next.override_stride + len1 + tid] : -1;
    }
    if (next.source != SRC_SIZES && tid < k1) {
      int dr = s_next[tid];
      // a caller-provided draft beyond the vocabulary becomes a slot that matches nothing (negative = sentinel is legal)
      if (dr >= dm.vocab) { latch_error(st.status, AD_ERR_ARG); dr = -1; s_next[tid] = dr; }
      st.drafts[(size_t)b * dm.kmax + tid] = dr;
    }
    if (tid == 0) {
      blk.seg_len[b] = k1; blk.key_base[b] = b * dm.max_tgt; blk.row_nk[b] = len1 + k1;
      if (!CLUSTER) { s_k[b] = k1; s_len[b] = len1; }
    }
  }
  // ---- what the rows have to tell one another; without a cluster the last row to get here sees all of them ----
  trace_mark(TR_ACCEPT, 5);
  bool all_fin = fin1 != 0, any_active = n > 0;
  if (CLUSTER) {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (tid < B) {
      auto tell = [&](int* mine, int v) {
        uint32_t a;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(mine))), "r"(tid));
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
      };
      tell(s_k + b, k1); tell(s_len + b, len1); tell(s_row + b, (fin1 ? 1 : 0) | (n > 0 ? 2 : 0));
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    const int row = lane < B ? s_row[lane] : 1;
    all_fin = __all_sync(0xffffffffu, row & 1);
    any_active = __any_sync(0xffffffffu, row & 2);
  } else {
    __syncthreads();
  }
  if (FORM == ACC_ROWS) {
    if (tid == 0) {
      __threadfence();
      const unsigned int t = atomicAdd(done_ctr, n > 0 ? 0x10001u : 1u);
      s_last_cta = (t & 0xffffu) == (unsigned)B - 1 ? 1 : 0;
      if (s_last_cta) { __threadfence(); s_n = ((t >> 16) + (n > 0 ? 1u : 0u)) != 0; }
    }
    __syncthreads();
    if (!s_last_cta) return;
    any_active = s_n != 0;
    int f = 1;
    if (tid < B) {
      f = __ldcg(st.fin + tid);
      if (next.source >= 0) { s_k[tid] = __ldcg(blk.seg_len + tid); s_len[tid] = __ldcg(st.len + tid); }
    }
    all_fin = __syncthreads_and(f) != 0;
  }
  if (tid == ACC_THREADS - 1 && (!CLUSTER || b == 0)) {            // (not a thread of the warp that adds up many rows' offsets)
    *done_ctr = 0;
    if (any_active) *st.loop_it = ctr0 + 1;
    *st.all_fin = all_fin;
    if (cond) {
      // the iteration runs inside a device-side `while` graph node, which repeats while its condition is non-zero: cleared
      // when every row has finished or, as a bound that does not depend on the data, at the limit the host stored
      st.loop_it[2] = ctr1 + 1;
      atomicAdd(st.loop_it + 4, next.launches);
      cudaGraphSetConditional(cond, (all_fin || ctr1 + 1 >= ctr2) ? 0u : 1u);
    }
  }
  if (next.source < 0) return;
  // ---- layout of the pass behind this kernel ----
  trace_mark(TR_ACCEPT, 6);
  const bool draft_pass = next.source == SRC_SIZES;
  // drafter's tokens of a row: [BOS], accepted tokens, k x [MASK]
  auto draft_tokens = [&](int r) { return s_k[r] > 0 ? s_len[r] + 1 + s_k[r] : 0; };
  // tokens of row r from o0 on (block offset boff), by the lanes of a group; alone: the row is this CTA's own
  auto lay_out = [&](int r, int o0, int boff, int first, int step, auto alone) {
    constexpr bool ALONE = decltype(alone)::value;
    const int lr = s_len[r], kr = s_k[r];
    if (draft_pass) {
      const int nr = draft_tokens(r);
      const PassPlan& pl = next.draft;
      if (first == 0) { pl.seg_off[r] = o0; pl.seg_len[r] = nr; pl.key_base[r] = o0; pl.row_nk[r] = nr; }
      for (int i = first; i < nr; i += step) {
        const int m = o0 + i;
        int tok = i == 0 ? dm.bos : i > lr ? dm.mask : ALONE && i > len ? s_pred[i - 1 - len] : __ldcg(st.out_ids + (size_t)r * dm.max_tgt + i - 1);
        if (!id_in_vocab(tok, dm)) { latch_error(st.status, AD_ERR_ARG); tok = dm.pad; }
        pl.tok_row[m] = r; pl.tok_pos[m] = i; pl.tok_id[m] = tok; pl.kv_slot[m] = m; pl.att_n[m] = nr;
      }
      for (int i = first; i < kr; i += step) st.gidx[boff + i] = o0 + lr + 1 + i;
    } else {
      const int* dr = st.drafts + (size_t)r * dm.kmax;
      for (int i = first; i < kr; i += step) {
        const int m = o0 + i;
        int tok = ALONE ? (i == 0 ? last1 : s_next[i - 1]) : (i == 0 ? __ldcg(st.last + r) : __ldcg(dr + i - 1));
        if (tok < 0 || tok >= dm.vocab) tok = dm.pad;
        blk.tok_row[m] = r; blk.tok_pos[m] = lr + i; blk.tok_id[m] = tok;
        blk.kv_slot[m] = r * dm.max_tgt + lr + i; blk.att_n[m] = lr + i + 1;
      }
    }
  };
  if constexpr (FORM != ACC_ROWS) {
    // (at most 16 rows: every warp adds up those in front of its own)
    const int kr = lane < B ? s_k[lane] : 0, dr = lane < B && draft_pass ? draft_tokens(lane) : 0;
    const int boff = __reduce_add_sync(0xffffffffu, lane < b ? kr : 0), all = __reduce_add_sync(0xffffffffu, kr);
    const int doff = __reduce_add_sync(0xffffffffu, lane < b ? dr : 0), dall = __reduce_add_sync(0xffffffffu, dr);
    const int o0 = draft_pass ? doff : boff;
    if (tid == 0) {
      blk.seg_off[b] = boff;
      if (b == 0) {
        *blk.M = all;
        if (draft_pass) *next.draft.M = dall;
        pick_body(next.pick, all);
      }
    }
    lay_out(b, o0, boff, tid, ACC_THREADS, std::true_type());
  } else {
    if (warp == 0) {                       // offsets: an exclusive scan over the rows
      int base = 0, dbase = 0;
      for (int b0 = 0; b0 < B; b0 += 32) {
        const int r = b0 + lane, kr = r < B ? s_k[r] : 0;
        const int dr = r < B ? draft_tokens(r) : 0;
        int sum = kr, dsum = dr;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int a = __shfl_up_sync(0xffffffffu, sum, o), c = __shfl_up_sync(0xffffffffu, dsum, o);
          if (lane >= o) { sum += a; dsum += c; }
        }
        if (r < B) {
          blk.seg_off[r] = base + sum - kr;
          s_off[r] = draft_pass ? dbase + dsum - dr : base + sum - kr;
          s_boff[r] = base + sum - kr;
        }
        base += __shfl_sync(0xffffffffu, sum, 31);
        dbase += __shfl_sync(0xffffffffu, dsum, 31);
      }
      if (lane == 0) {
        *blk.M = base;
        if (draft_pass) *next.draft.M = dbase;
        pick_body(next.pick, base);
      }
    }
    __syncthreads();
    for (int r = warp; r < B; r += ACC_THREADS / 32) lay_out(r, s_off[r], s_boff[r], lane, 32, std::false_type());
  }
  __threadfence();
  trace_mark(TR_ACCEPT, 2);
}

}  // namespace ad
