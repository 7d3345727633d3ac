// Output projection fused with the per-tile arg-max for passes with many tokens (hundreds to thousands of packed rows): a
// persistent, warp-specialised tcgen05 GEMM on pairs of SMs (cta_group::2), token-stationary for K <= 512.
//
// Unlike gemm_tc.cuh (weights on the MMA's M side so that a handful of tokens still fill an instruction), the tokens are the M
// side here: D[token, vocabulary row] = sum_k X[token, k] * E[row, k], one token per tensor-memory lane and one vocabulary row
// per column.  The arg-max over vocabulary rows is then a scan over a thread's own columns: no exchange between lanes, no
// shared memory, no barrier.
//
// A pair of CTAs (a cluster on two neighbouring SMs) works on 256 tokens x 256 vocabulary rows at a time: each CTA holds its 128
// tokens (128 x K BF16, resident in shared memory as long as the token tile stays) and loads HALF of the vocabulary
// rows; the paired MMA reads both halves from both shared memories, so a K block brings 16 KB into each SM instead of the 32 KB that
// one CTA per token tile needs.  2048 tokens x 32000 x 512, call behind call: one CTA per token tile 61 us, pairs 64.5 us while the
// MMAs were issued from a branch on the lane number, 49.7 us (1350 TFLOP/s) issued from a converged warp; 600 tokens 25.5 -> 23.7 us.
// A single call between two events takes 57.8 us (1161 TFLOP/s), 600 tokens 31.
// What bounds it now: 0.4 us per K block against 0.27 us of MMA time, plus 6 us to fill, read the last step out and tear down.
//
// K > 512 (STREAM): the token tile no longer fits beside a ring, so its K blocks travel through the ring with the vocabulary's, 32 KB
// a stage.  One CTA per 128 x 128 tile, as these widths ran before, is bound by the tiles' way through L2 (11.7 TB/s).  One call between two
// events: 2048 tokens x 32000 x 1024 137 -> 90 us (1488 TFLOP/s), 600 x 768 x 50265 65 -> 47 us, 200 x 768 x 50265 31 -> 25 us; call behind
// call 129 -> 91, 59 -> 42 and 25 -> 19 us.  Up to 512 the resident form stays 2 to 4 % ahead.
//
// The range of (token tile, 128-row vocabulary tile) units is dealt to the pairs in contiguous pieces, the vocabulary tile
// running fastest; a pair takes two units a step, one where its piece or the vocabulary ends (the MMA is then 128 columns wide
// and each CTA loads 64 rows).  Roles in each CTA (576 threads):
//   warps 8 .. 8+S-1, one lane: producers of the vocabulary ring, one stage each (boxes of 64 rows); inside a pass the weights
//                             never change and are requested before the dependency wait;
//   warps 8+S .. 14, 16, 17, one lane: load the resident token tile whenever the range moves on to the next one, K blocks dealt to them (one
//                             thread's copies run one after the other), a barrier per K block so that the MMAs follow the copies;
//   warp 15, one lane (first CTA of the pair): MMA issuer; the accumulators of both CTAs alternate between two 256-column halves of
//                             tensor memory, so the K loop of step i + 1 runs while step i is read out;
//   warps 0-7:                read-out: warp w owns the 32 tokens of lane quadrant w % 4 of its CTA and the 128 columns w / 4 of
//                             the half, i.e. one 128-row vocabulary tile of the partial arrays; each thread scans its columns in
//                             ascending row order (strict comparison: lowest id wins ties) and writes the token's (maximum,
//                             id[, rows scoring above the draft]) for that tile.
// Barriers that the issuer waits on live in the first CTA (the second CTA's copies and readers signal them remotely); those it
// signals are signalled in both CTAs by one multicast commit.  Every mbarrier wait is bounded in time; a wait that runs out
// latches AD_ERR_TIMEOUT, raises the CTA's abort flag and every role leaves its loop.  Nobody waits at a barrier of all threads
// inside the loops.
#pragma once

#include <type_traits>

#include "gemm_tc.cuh"

namespace ad {
namespace tc {

constexpr int P_THREADS = 576;
constexpr int P_TOK = 128;                       // tokens per CTA; MMA M = 256
constexpr int P_VOC = 256;                       // vocabulary rows per step = MMA N
constexpr int P_MAX_KB = 8;                      // K <= 512: the token tile stays in shared memory
constexpr int P_MAX_STAGES = 6;
constexpr int P_BOX = 64;                        // rows per vocabulary box
constexpr int P_BOX_BYTES = P_BOX * BLOCK_K * 2;    // 8 KiB
constexpr int P_A_KB_BYTES = P_TOK * BLOCK_K * 2;   // 16 KiB: one K block of the resident token tile
constexpr int P_B_STAGE_BYTES = 2 * P_BOX_BYTES;    // 16 KiB: this CTA's half of a step's vocabulary rows
constexpr int P_READ_WARPS = 8;

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Address, in the cluster's shared window, of the same object in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
  return a;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// Bounded wait of a converged warp as mbar_wait_warp, ordering what follows behind arrivals from the whole cluster.
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, int* status) {
  for (int i = 0; i < 64; ++i)
    if (__all_sync(0xffffffffu, mbar_try_wait_cluster(bar, parity))) return true;
  const unsigned long long t0 = global_ns();
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (__all_sync(0xffffffffu, mbar_try_wait_cluster(bar, parity))) return true;
    if (__any_sync(0xffffffffu, global_ns() - t0 > WAIT_BUDGET_NS)) break;
  }
  latch_error(status, AD_ERR_TIMEOUT);
  return false;
}
// Tile copy into this CTA's shared memory that signals a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t cluster_bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(cluster_bar)
      : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The barrier at this address in both CTAs tracks completion of every paired MMA issued so far.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"((uint16_t)3)
               : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Shared memory a launch needs for kb K blocks and `stages` ring stages.
inline size_t vocab_pair_smem(int kb, int stages) {
  return (size_t)(kb <= P_MAX_KB ? kb : stages) * P_A_KB_BYTES + (size_t)stages * P_B_STAGE_BYTES + 1024;
}

// grid = 2 x pairs; cluster (2, 1, 1); block = 576 threads; dynamic smem = vocab_pair_smem(K / 64, stages).
// map_x: box of 128 token rows x 64; map_w: box of 64 vocabulary rows x 64.  p.bias must be null.
template <bool STREAM>
__global__ void __launch_bounds__(P_THREADS, 1)
vocab_argmax_pair_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x, const GemmParams p,
                         const int stages) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_full[P_MAX_STAGES];      // first CTA's: both CTAs' rows of a stage have landed
  __shared__ __align__(8) uint64_t bar_empty[P_MAX_STAGES];     // both: the stage has been consumed
  __shared__ __align__(8) uint64_t a_full[P_MAX_KB];            // first CTA's: both CTAs' tokens of a K block have landed
  __shared__ __align__(8) uint64_t a_empty;                     // both
  __shared__ __align__(8) uint64_t acc_full[2];                 // both
  __shared__ __align__(8) uint64_t acc_empty[2];                // first CTA's: read out by both CTAs
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int KB = p.K / BLOCK_K;
  const uint32_t a_base = (smem_u32(smem_raw) + 1023u) & ~1023u;      // resident token tile: KB blocks of 16 KiB
  const uint32_t b_base = STREAM ? a_base + P_A_KB_BYTES : a_base + (uint32_t)(KB * P_A_KB_BYTES);     // ring
  constexpr uint32_t STAGE_BYTES = STREAM ? P_A_KB_BYTES + P_B_STAGE_BYTES : P_B_STAGE_BYTES;
  constexpr uint32_t TMEM_COLS = 2 * P_VOC;

  if (threadIdx.x == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_w)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_x)) : "memory");
    for (int s = 0; s < stages; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int kb = 0; kb < KB && !STREAM; ++kb) mbar_init(smem_u32(&a_full[kb]), 1);
    mbar_init(smem_u32(&a_empty), 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&acc_full[b]), 1);
      mbar_init(smem_u32(&acc_empty[b]), 2 * P_READ_WARPS);
    }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 15) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();                             // barriers of both CTAs are initialised, tensor memory of both is allocated
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_acc = tmem_base_slot;
  pdl_launch();
  const int M = p.M_ptr ? plan_load(p.M_ptr) : p.M_host;

  const int n_vt = (p.N + BLOCK_N_FEAT - 1) / BLOCK_N_FEAT;    // 128-row tiles: the layout of the partial arrays
  const int n_tt = (M + 2 * P_TOK - 1) / (2 * P_TOK);          // 256-token tiles that hold tokens
  const long long n_units = (long long)n_tt * n_vt;
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int u_lo = (int)((n_units * pair) / n_pairs);
  const int u_hi = (int)((n_units * (pair + 1)) / n_pairs);
  // the steps of the piece: from unit u, `width` (1 or 2) vocabulary tiles of token tile t
  struct Step { int t, vt, width; };
  auto step_at = [&](int u) {
    Step s;
    s.t = u / n_vt;
    s.vt = u - s.t * n_vt;
    s.width = (u + 1 < u_hi && s.vt + 1 < n_vt) ? 2 : 1;
    return s;
  };
  volatile int* abort_v = &abort_flag;

  if (warp >= 8 && warp < 8 + stages) {
    // ---- ring producers: producer pw owns stage pw and the K blocks pw, pw + S, ... of the pair's whole sequence ----
    {
      if (!p.M_ptr) pdl_wait();                            // operator-level call: the matrix may have just been written
      const int pw = warp - 8;
      const uint32_t full = smem_u32(&bar_full[pw]), empty = smem_u32(&bar_empty[pw]), full0 = cluster_addr(full, 0);
      const uint32_t dst = b_base + (uint32_t)pw * STAGE_BYTES;
      int u = u_lo, first_kb = 0;                          // the step at unit u starts with K block number first_kb of the sequence
      bool ok = true;
      for (int g = pw; ok && u < u_hi;) {
        const Step st = step_at(u);
        // this CTA's rows: one of the two tiles, or half of the only one
        const int row = st.vt * BLOCK_N_FEAT + (int)rank * (st.width * P_BOX);
        for (; g < first_kb + KB; g += stages) {
          const uint32_t round = (uint32_t)(g / stages);
          if (round > 0 && !mbar_wait_warp(empty, (round - 1) & 1u, p.status)) { *abort_v = 1; ok = false; break; }
          if (*abort_v) { ok = false; break; }
          const int kb = g - first_kb;
          // rows beyond the vocabulary are filled with zeros and still count their bytes
          if (elect_one()) {
            if (rank == 0) mbar_expect_tx(full, (uint32_t)(2 * st.width * P_BOX_BYTES + (STREAM ? 2 * P_A_KB_BYTES : 0)));
            tma_load_2d_pair(dst, &map_w, kb * BLOCK_K, row, full0);
            if (st.width == 2) tma_load_2d_pair(dst + P_BOX_BYTES, &map_w, kb * BLOCK_K, row + P_BOX, full0);
          }
          if (STREAM) {
            if (g == pw) pdl_wait();
            if (elect_one()) tma_load_2d_pair(dst - P_A_KB_BYTES, &map_x, kb * BLOCK_K, (2 * st.t + (int)rank) * P_TOK, full0);
          }
          __syncwarp();
        }
        first_kb += KB;
        u += st.width;
      }
    }
  } else if ((warp >= 8 + stages && warp < 15) || warp > 15) {
    // ---- the resident token tile: loader l of n takes K blocks l, l + n, ... ----
    if (!STREAM) {
      const int l = warp > 15 ? warp - 16 : 2 + warp - 8 - stages, n = 9 - stages;
      pdl_wait();
      int cur_t = -1;
      uint32_t uses = 0;
      for (int u = u_lo; u < u_hi;) {
        const Step st = step_at(u);
        u += st.width;
        if (st.t == cur_t) continue;
        // the MMAs of the previous token tile must have read it for the last time
        if (uses > 0 && !mbar_wait_warp(smem_u32(&a_empty), (uses - 1) & 1u, p.status)) { *abort_v = 1; break; }
        if (*abort_v) break;
        for (int kb = l; kb < KB; kb += n) {
          const uint32_t full = smem_u32(&a_full[kb]);
          if (elect_one()) {
            if (rank == 0) mbar_expect_tx(full, (uint32_t)(2 * P_A_KB_BYTES));
            tma_load_2d_pair(a_base + (uint32_t)(kb * P_A_KB_BYTES), &map_x, kb * BLOCK_K, (2 * st.t + (int)rank) * P_TOK, cluster_addr(full, 0));
          }
          __syncwarp();
        }
        cur_t = st.t;
        ++uses;
      }
    }
  } else if (warp == 15) {
    // ---- MMA issuer ----
    if (rank == 0) {
      const uint32_t idesc2 = make_idesc(2 * P_TOK, P_VOC), idesc1 = make_idesc(2 * P_TOK, BLOCK_N_FEAT);
      const uint64_t desc_a0 = make_smem_desc(a_base);
      const uint64_t desc_b0 = make_smem_desc(b_base);
      const uint64_t a_step = (uint64_t)(P_A_KB_BYTES >> 4), b_step = (uint64_t)(STAGE_BYTES >> 4);
      bool ok = true;
      int cur_t = -1, it = 0, s = 0;
      uint32_t uses = 0, phase = 0;                        // ring position of the next K block
      // the K loop of one step; FRESH: first step of a token tile, whose K blocks arrive one by one.  (The issuing thread's own
      // instructions matter: ring position by counting, no division.)
      auto k_loop = [&](uint32_t acc, uint32_t idesc, auto fresh) {
        uint64_t desc_a = desc_a0;
        uint32_t accumulate = 0;
        for (int kb = 0; kb < KB; ++kb) {
          if (!STREAM && decltype(fresh)::value && !mbar_wait_cluster(smem_u32(&a_full[kb]), (uses - 1) & 1u, p.status)) return false;
          if (!mbar_wait_cluster(smem_u32(&bar_full[s]), phase, p.status)) return false;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t desc_b = desc_b0 + b_step * (uint64_t)s;
          if (STREAM) desc_a = desc_a0 + b_step * (uint64_t)s;
          if (elect_one()) {
#pragma unroll
            for (int k4 = 0; k4 < BLOCK_K / UMMA_K; ++k4) umma_bf16_pair(acc, desc_a + 2 * k4, desc_b + 2 * k4, idesc, k4 == 0 ? accumulate : 1u);
            umma_commit_pair(smem_u32(&bar_empty[s]));
          }
          __syncwarp();
          accumulate = 1u;
          if (!STREAM) desc_a += a_step;
          if (++s == stages) { s = 0; phase ^= 1u; }
        }
        return true;
      };
      for (int u = u_lo; u < u_hi && ok; ++it) {
        const Step st = step_at(u);
        u += st.width;
        const int b = it & 1;
        const bool fresh = st.t != cur_t;
        if (fresh) { cur_t = st.t; ++uses; }
        // the half must have been read out (step it - 2)
        if (it >= 2) ok = mbar_wait_cluster(smem_u32(&acc_empty[b]), (uint32_t)((it >> 1) - 1) & 1u, p.status);
        if (!ok || *abort_v) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc = tmem_acc + (uint32_t)(b * P_VOC), idesc = st.width == 2 ? idesc2 : idesc1;
        if (lane == 0) trace_mark_role(TR_PV_ISSUE, 0);
        ok = fresh ? k_loop(acc, idesc, std::true_type{}) : k_loop(acc, idesc, std::false_type{});
        if (!ok) break;
        const bool last_of_tile = u < u_hi && u / n_vt != st.t;
        if (elect_one()) {
          umma_commit_pair(smem_u32(&acc_full[b]));
          // last step of this token tile: once these MMAs are done the resident tiles may be replaced
          if (last_of_tile) umma_commit_pair(smem_u32(&a_empty));
        }
        __syncwarp();
        if (lane == 0) trace_mark_role(TR_PV_ISSUE, 1);
      }
      if (!ok && lane == 0) {   // nobody in this CTA must be left waiting for an accumulator that will not come
        *abort_v = 1;
        mbar_arrive(smem_u32(&acc_full[0]));
        mbar_arrive(smem_u32(&acc_full[1]));
      }
    }
  } else if (warp < P_READ_WARPS) {
    // ---- read-out: warps 0-7 ----
    const int quad = warp & 3, grp = warp >> 2;
    const bool relaxed = p.draft_val != nullptr;
    const uint32_t empty0 = cluster_addr(smem_u32(&acc_empty[0]), 0), empty1 = cluster_addr(smem_u32(&acc_empty[1]), 0);
    int cur_t = -1, did = -1, it = 0;
    float dval = 0.f;
    pdl_wait();
    for (int u = u_lo; u < u_hi; ++it) {
      const Step st = step_at(u);
      u += st.width;
      const int b = it & 1, t = st.t;
      const int tok = (2 * t + (int)rank) * P_TOK + quad * 32 + lane;   // this thread's token
      const int vt = st.vt + grp;                                // this warp's 128-row tile of the partial arrays
      if (relaxed && t != cur_t) {
        dval = tok < M ? p.draft_val[tok] : 0.f;
        did = tok < M ? p.draft_id[tok] : -1;
      }
      cur_t = t;
      if (!mbar_wait(smem_u32(&acc_full[b]), (uint32_t)(it >> 1) & 1u, p.status)) { *abort_v = 1; break; }
      if (*abort_v) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (threadIdx.x == 0) trace_mark_role(TR_PV_EPI, 0);
      const uint32_t taddr = tmem_acc + (static_cast<uint32_t>(quad * 32) << 16) + (uint32_t)(b * P_VOC + grp * BLOCK_N_FEAT);
      const int n_base = vt * BLOCK_N_FEAT;
      float best = -INFINITY;
      int best_n = n_base, cnt = 0;
      const bool mine = grp < st.width;                          // (a step of one tile has no second half)
      if (mine) {
        for (int c = 0; c < BLOCK_N_FEAT; c += 16) {
          float acc[16];
          tmem_ld16(taddr + static_cast<uint32_t>(c), acc);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int n = n_base + c + j;
            const float val = n < p.N ? acc[j] : -INFINITY;     // rows beyond the vocabulary were zero-filled
            if (relaxed) cnt += (n != did && val > dval) ? 1 : 0;
            if (val > best) { best = val; best_n = n; }
          }
        }
      }
      // this warp has read its share of the half: hand it back to the issuer
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(b ? empty1 : empty0);
      if (threadIdx.x == 0) trace_mark_role(TR_PV_EPI, 1);
      if (mine && tok < M) {
        const size_t o = (size_t)tok * n_vt + vt;
        p.part_val[o] = best;
        p.part_idx[o] = best_n;
        if (relaxed) p.part_cnt[o] = cnt;
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();                             // nobody of the pair reads or signals the other's memory any more
  if (warp == 15) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_acc), "r"(TMEM_COLS) : "memory");
  }
}

}  // namespace tc
}  // namespace ad
