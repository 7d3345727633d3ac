// Host side of the verification-step library: handle, workspace layout, kernel sequencing, CUDA-graph
// replay of the decode loop, and the extern "C" entry points declared in include/aggressive_decoding.h.
#include <limits.h>
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <string>
#include <tuple>
#include <type_traits>
#include <vector>

#include "accept.cuh"
#include "ad_common.cuh"
#include "attention.cuh"
#include "attention_few.cuh"
#include "attention_mma.cuh"
#include "ffn_few.cuh"
#include "gemm_few.cuh"
#include "gemm_simt.cuh"
#include "gemm_tc.cuh"
#include "gemm_tc_pair.cuh"
#include "grid_sync.cuh"
#include "mega.cuh"
#include "steps.cuh"
#include "sublayer_f32.cuh"

using namespace ad;

namespace {

enum PassKind { PK_VERIFY = 0, PK_DRAFT = 1, PK_ENCODE = 2, PK_COUNT = 3 };

struct Mat {
  const void* ptr = nullptr;
  int N = 0, K = 0;
  CUtensorMap map;
  CUtensorMap map64;     // embedding matrix only: boxes of 64 rows
};
struct ActBuf {
  void* ptr = nullptr;
  int cols = 0;
  // one map per pass kind and token tile: box rows 16, 32, 64, 128, 256 (index log2(rows) - 4), up to the pass's own tile
  tc::TileMaps map[PK_COUNT];
  const CUtensorMap& map_for(int pk, int tile) const {
    int i = 0;
    while ((16 << i) < tile && i < 4) ++i;
    return map[pk].m[i];
  }
};
struct EncLayer {
  Mat wqkv, wo, w1, w2;
  const float *bqkv, *bo, *ln1g, *ln1b, *b1, *b2, *ln2g, *ln2b;
};
struct DecLayer {
  Mat wqkv, wo, cq, ckv, co, w1, w2;
  const float *bqkv, *bo, *ln1g, *ln1b, *cbq, *cbkv, *cbo, *ln2g, *ln2b, *b1, *b2, *ln3g, *ln3b;
};
struct Model {
  bool present = false;
  Mat emb;
  std::vector<EncLayer> enc;
  std::vector<DecLayer> dec;
  void* kenc = nullptr;   // [n_dec][B * max_src][d] cross-attention keys
  void* venc = nullptr;
  // the decoder layers' cross-attention key/value projections gathered into one [n_dec * 2d, d] matrix (and their
  // biases into one vector) at ad_create, so that ad_encode projects the encoder memory for all layers in one launch
  Mat ckv_all;
  void* ckv_pack = nullptr;
  float* cbkv_pack = nullptr;
};
// Passes of at most this many packed tokens run their projections on the few-token kernel (gemm_few.cuh).
constexpr int kFewTokens = few::MAX_TOKENS;
// Encoder passes of at most this many have the embedding in their first projection; beyond, the projection's CTAs, each of which computes all of it
// (its loads are three times the operand), take longer than a kernel in front of them.  Encoder calls of four layers, in the projection -> a kernel:
// 512 wide, 1 x 80 tokens 111 -> 108 us, 2 x 50 116 -> 111, 4 x 32 121 -> 116; 768 wide, 1 x 97 161 -> 157; 1024 wide, 1 x 128 200 -> 190.
constexpr int kFusedEmbed = 64;

struct PassCfg {
  int M_cap = 0;     // packed-token capacity of this pass kind
  int ntile = 16;    // tokens per GEMM tile
  int seg_max = 0;   // longest segment of one row
  int max_split = 1; // largest split-K factor this pass may use (sizes the partial-sum buffer)
  int few_cap = few::MAX_TOKENS;   // capacities up to which every pass runs its projections on the few-token kernels; 0: one of several layouts, picked
                                   // by the tokens that are there, and not the first (see LoopBodies)
  PassPlan plan;
  // Most pieces of up to q tokens of one row that a pass over `rows` rows can have.
  long pieces(int rows, int q) const { return std::min((long)rows * ((seg_max + q - 1) / q), (long)std::min(rows, M_cap) + M_cap / q); }
};

// Launch shape of the tensor-core projection kernel (see tc_shape); ksplit: the most partial sums of any token count.
struct TcShape { int ctas, budget, smem, ksplit; };

// A second set of activation buffers (encoder-pass sized) for work that runs on the side stream.
struct ActSet {
  float *y = nullptr, *pre = nullptr, *pre2 = nullptr;
  ActBuf yb, abuf, hbuf;
  void *qbuf = nullptr, *ktmp = nullptr, *vtmp = nullptr;
};

NextPass no_next_pass() {
  NextPass n = {};
  n.source = -1;
  return n;
}

thread_local std::string g_create_error;

// Switches of a handle, read from the environment when it is created.
struct Switches {
  bool graph_calls = true;      // AD_NO_ENCODE_GRAPH=1: launch the kernels of the block-level calls and of the encoder directly
  bool two_stream_encode = true;   // AD_NO_CONCURRENT_ENCODERS=1: the drafter's encoder after the verifier's, on one stream
  bool devloop = true;          // AD_NO_DEVLOOP=1: one graph replay per iteration with host polling instead of a device-side loop
  bool fuse_attn_proj = true;   // AD_NO_ATTN_PROJ=1: attention and its output projection always as separate kernels
  bool fuse_plan = true;        // AD_NO_FUSED_PLAN=1: plan in kernels of their own in every iteration
  bool few_body = true;         // AD_NO_FEW_BODY=1: one body for every iteration of a device-side loop
  int accept_cluster = ACC_CLUSTER;   // AD_ACCEPT_CLUSTER=n: rows of a loop meet in a cluster up to n of them (0: always through global memory)
  // AD_MEGA=1: run eligible decoder passes (BF16, 64-wide heads, at most 64 packed tokens) as ONE persistent kernel
  // instead of the kernel chain.  Off by default: measured on a B200 it is slower than the chain at every shape tried
  // (base model: 342 / 360 / 424 / 462 us per verification step for blocks of 1 / 16 / 40 / 64 tokens against 214 / 223 /
  // 247 / 258 us; big model, 25 tokens: 537 against 323 us), because a stage that hands its result to other SMs through
  // L2 costs about 7 us there (operand staging 1.3-3 us, MMA hand-over 0.6, tensor-memory read-out 0.3, cluster hand-shake
  // 0.8-1.2, reduction and epilogue 1-1.7, release 0.5, propagation 0.7) against about 3.7 us per kernel of the chain.
  bool mega = false;
};

}  // namespace

struct ad_handle {
  ad_model_cfg cfg;
  cudaStream_t stream = nullptr;
  Switches sw;
  bool bf16 = false;
  size_t esz = 4;            // bytes per activation / weight element
  Model ar, nar;
  PassCfg pass[PK_COUNT];
  int M_all = 0;
  Dims dims;
  DevState st;
  // activations
  float *y = nullptr, *pre = nullptr;
  float* pre2 = nullptr;     // per-head partial sums of an output projection fused into the attention kernel
  ActBuf yb, abuf, hbuf, xg;
  void *qbuf = nullptr, *ktmp = nullptr, *vtmp = nullptr, *kself = nullptr, *vself = nullptr;
  ActBuf encmem;             // the verifier's encoder memory
  float* part_val = nullptr;
  int* part_idx = nullptr;
  int* part_cnt = nullptr;   // relaxed verification: per tile and token, other tokens scoring above the draft
  float* draft_val = nullptr;
  int* draft_id = nullptr;
  // The drafter's encoder does not depend on the verifier's: it runs on a side stream with its own activations.
  ActSet side;
  cudaStream_t side_stream = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  int beta = 0;              // 0: exact-match verification; >= 1: relaxed verification (Section 3.2.3)
  float tau = 0.f;
  int n_vtiles = 0;
  int accept_rows = 0;       // rows of a loop up to which the accept kernel is one cluster
  float* pe = nullptr;
  int max_pos = 0;
  int* ovr = nullptr;        // [B, max_tgt] staged draft-override stream
  int* host_flag = nullptr;  // pinned, mapped host memory: [0..15] flag words, then the upload area (sources, lengths, caps,
                             // override stream) and the result block of ad_generate
  int* host_flag_dev = nullptr;   // the same memory as the device sees it
  int* up_src = nullptr;     // pinned staging of host-resident inputs
  int* up_len = nullptr;
  int* up_max = nullptr;
  int* up_ovr = nullptr;
  int* up_ids = nullptr;     // drafts or forced tokens [B, kmax]
  int* up_n = nullptr;       // block sizes or commit counts [B]
  int* in_max = nullptr;     // per-row caps of ad_generate as imported
  int* dev_view(int* host) const { return host_flag_dev + (host - host_flag); }
  int* down = nullptr;       // result block of finalize_generate_kernel (host view) ...
  int* down_dev = nullptr;   // ... and its device view
  // st.words as the calls enqueued so far leave them, and whether a caller has recorded calls into a graph of its own (whose replays
  // set the words again at times that the handle does not see).
  int4 words = {0, 0, 0, 0};
  bool foreign_graphs = false;
  // Decode loop: the accept kernel of one pass plans the pass behind it; next_pass is what the accept kernel being enqueued
  // shall plan (source < 0: nothing).
  NextPass next_pass = no_next_pass();
  bool profiling = false;    // ad_debug_profile_verify: an event in front of every launch
  std::vector<std::pair<std::string, cudaEvent_t>> prof;
  // state
  int B = 0;                 // batch of the last ad_encode
  bool encoded = false;
  int last_vocab_which = -1;
  std::string err;
  struct GraphEntry {
    cudaGraphExec_t exec;   // null: the form has been called once, directly
    int launches;        // kernels per replay (a device-side loop counts its own)
    bool device_loop;    // whole-call graph ...
    int once;            // ... and its kernels outside the loop
    long last_use;
  };
  long graph_uses = 0;
  std::map<std::string, GraphEntry> graphs;
  std::map<std::tuple<int, int, int, int, int, int, int, int, int>, TcShape> tc_shapes;   // see cached_shape
  cudaEvent_t ev0 = nullptr, ev1 = nullptr, ev2 = nullptr;
  int launches = 0;          // kernels launched by the last ad_generate (direct) or per graph replay
  // Persistent decoder pass (one kernel for the decoder stack + projection): per pass kind, whether it applies and its
  // fixed arguments; device-resident tables of tensor maps (per model) and of per-layer pointers (per pass kind).
  struct MegaPass { bool on = false; mega::Params p; };
  MegaPass mega[PK_COUNT];
  int mega_cs = 0, mega_nc = 0;
  size_t mega_smem = 0;
  CUtensorMap* mega_maps[2] = {nullptr, nullptr};          // [0] verifier, [1] drafter
  mega::LayerPtrs* mega_layers[2] = {nullptr, nullptr};    // [0] verification pass, [1] drafter pass
  float* mega_stats[2] = {nullptr, nullptr};
  unsigned long long* mega_timeline = nullptr;
  unsigned long long cond_handle = 0;   // non-zero only while the body of a device-side `while` node is captured
  NextPass::Pick pick = {};             // set only while a loop whose body comes in several forms is captured
  int body_launches = 0;                // h->launches where the body being captured begins
};

namespace {

#define AD_CUDA(h, call)                                                                      \
  do {                                                                                        \
    cudaError_t e__ = (call);                                                                 \
    if (e__ != cudaSuccess) {                                                                 \
      (h)->err = std::string(#call) + ": " + cudaGetErrorString(e__);                         \
      return AD_ERR_CUDA;                                                                     \
    }                                                                                         \
  } while (0)

int fail(ad_handle* h, int code, const std::string& msg) {
  if (h) h->err = msg; else g_create_error = msg;
  return code;
}

// Counts a kernel launch of this library and, while a profiling pass is active, drops an event in front of it (the
// time between two consecutive events is then the device time of the kernel launched after the first one).
void note_launch(ad_handle* h, const char* what) {
  h->launches++;
  if (h->profiling) {
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) == cudaSuccess) {
      cudaEventRecord(e, h->stream);
      h->prof.emplace_back(what, e);
    }
  }
}

// ---- TMA descriptor encoding through the driver entry point (no link-time dependency on libcuda) ----
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// Row-major bf16 [rows, cols]; box = 64 columns (one 128-byte swizzle row) x box_rows.
bool make_map(CUtensorMap* m, const void* base, int rows, int cols, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1u, 1u};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

int pow2ceil(int v) { int p = 1; while (p < v) p <<= 1; return p; }
int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }
size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// ---- workspace layout: one bump allocation pass, run with base = null to size it ----
struct Bump {
  char* base;
  size_t off = 0;
  explicit Bump(void* b) : base(static_cast<char*>(b)) {}
  void* take(size_t bytes, size_t align = 1024) {
    off = align_up(off, align);
    void* p = base ? base + off : nullptr;
    off += bytes;
    return p;
  }
};

void plan_take(Bump& bp, PassPlan& pl, int B, int M_cap) {
  pl.M = (int*)bp.take(sizeof(int) * 4, 256);
  pl.seg_off = (int*)bp.take(sizeof(int) * B, 256);
  pl.seg_len = (int*)bp.take(sizeof(int) * B, 256);
  pl.key_base = (int*)bp.take(sizeof(int) * B, 256);
  pl.row_nk = (int*)bp.take(sizeof(int) * B, 256);
  pl.tok_row = (int*)bp.take(sizeof(int) * M_cap, 256);
  pl.tok_pos = (int*)bp.take(sizeof(int) * M_cap, 256);
  pl.tok_id = (int*)bp.take(sizeof(int) * M_cap, 256);
  pl.kv_slot = (int*)bp.take(sizeof(int) * M_cap, 256);
  pl.att_n = (int*)bp.take(sizeof(int) * M_cap, 256);
}

void pass_shapes(const ad_model_cfg& c, PassCfg* pass, int* M_all) {
  const int B = c.max_batch;
  pass[PK_VERIFY].seg_max = c.kmax;
  pass[PK_DRAFT].seg_max = c.max_tgt + 1;
  pass[PK_ENCODE].seg_max = c.max_src;
  int all = 0;
  for (int k = 0; k < PK_COUNT; ++k) {
    pass[k].M_cap = B * pass[k].seg_max;
    pass[k].ntile = clampi(pow2ceil(pass[k].M_cap), 16, 256);
    pass[k].max_split = 16;
    if (pass[k].M_cap > all) all = pass[k].M_cap;
  }
  if (!c.has_drafter) { /* the drafter pass is never run; keep its shapes for sizing simplicity */ }
  *M_all = all;
}

// FP32 sublayers of few tokens (sublayer_f32.cuh): the model widths they are built for, and the width of their slices of hidden features of the feed-forward
// sublayer (0: not covered).
bool f32_sublayer_width(int d) { return d == 128 || d == 256; }
int f32_ffn_slice(int F) { return F % 32 == 0 && F / 32 <= 16 ? 32 : F % 64 == 0 && F / 64 <= 32 ? 64 : 0; }

// Floats of the partial sums of a projection with d output features over at most M tokens: a split projection has at most one
// CTA per SM, each with at most 128 x 128 outputs (few-token kernel: at most 16 parts of 128 tokens).
int num_sms();
size_t partial_elems(const ad_model_cfg& c, int M) {
  const int d = c.d_model;
  const size_t all = (size_t)M * d;
  // the feed-forward kernels of few tokens: a part per slice of hidden features
  size_t ffn = 0;
  if (c.dtype != AD_DTYPE_BF16) {
    if (f32_sublayer_width(d) && f32_ffn_slice(c.d_ffn) > 0) ffn = (size_t)(c.d_ffn / f32_ffn_slice(c.d_ffn)) * std::min(M, sub32::MAX_TOKENS) * d;
  } else if (few::ffn_few_fits(d, c.d_ffn, 1)) {
    ffn = std::min((size_t)(c.d_ffn / few::FFN_SLICE) * M, (size_t)few::FFN_MAX_ROWS) * d;
  }
  return std::max(std::max(all, ffn), std::min(16 * all, std::max((size_t)num_sms() * 128 * 128, (size_t)16 * few::MAX_TOKENS * d)));
}

// Floats of the partial output projections, one per head, that some attention kernels leave (0: none of this model does).  The FP32 ones stop at
// sub32::MAX_TOKENS tokens, whatever the handle can hold.
size_t head_partial_elems(const ad_model_cfg& c, int M) {
  if (c.n_heads > 16) return 0;
  const size_t row = (size_t)c.n_heads * c.d_model;
  return c.dtype == AD_DTYPE_BF16 ? row * M : f32_sublayer_width(c.d_model) ? row * std::min(M, sub32::MAX_TOKENS) : 0;
}

size_t layout(ad_handle* h, void* base) {
  const ad_model_cfg& c = h->cfg;
  const int B = c.max_batch, d = c.d_model, F = c.d_ffn;
  const size_t e = h->esz;
  Bump bp(base);
  pass_shapes(c, h->pass, &h->M_all);
  const int M_all = h->M_all, Mv = h->pass[PK_VERIFY].M_cap;
  const int M_tmp = std::max(h->pass[PK_DRAFT].M_cap, h->pass[PK_ENCODE].M_cap);
  h->y = (float*)bp.take(sizeof(float) * (size_t)M_all * d);
  h->pre = (float*)bp.take(sizeof(float) * partial_elems(c, M_all));
  if (const size_t n = head_partial_elems(c, M_all)) h->pre2 = (float*)bp.take(sizeof(float) * n);
  h->yb.ptr = bp.take(e * (size_t)M_all * d); h->yb.cols = d;
  h->abuf.ptr = bp.take(e * (size_t)M_all * d); h->abuf.cols = d;
  h->hbuf.ptr = bp.take(e * (size_t)M_all * F); h->hbuf.cols = F;
  h->xg.ptr = bp.take(e * (size_t)M_all * d); h->xg.cols = d;
  h->qbuf = bp.take(e * (size_t)M_all * d);
  h->ktmp = bp.take(e * (size_t)M_tmp * d);
  h->vtmp = bp.take(e * (size_t)M_tmp * d);
  h->encmem.ptr = bp.take(e * (size_t)h->pass[PK_ENCODE].M_cap * d); h->encmem.cols = d;
  const size_t self_sz = e * (size_t)c.n_dec * B * c.max_tgt * d;
  h->kself = bp.take(self_sz);
  h->vself = bp.take(self_sz);
  const size_t cross_sz = e * (size_t)c.n_dec * B * c.max_src * d;
  h->ar.kenc = bp.take(cross_sz);
  h->ar.venc = bp.take(cross_sz);
  if (c.has_drafter) {
    h->nar.kenc = bp.take(cross_sz);
    h->nar.venc = bp.take(cross_sz);
  }
  if (c.has_drafter) {
    const int Me = h->pass[PK_ENCODE].M_cap;
    ActSet& sd = h->side;
    sd.y = (float*)bp.take(sizeof(float) * (size_t)Me * d);
    sd.pre = (float*)bp.take(sizeof(float) * partial_elems(c, Me));
    if (const size_t n = head_partial_elems(c, Me)) sd.pre2 = (float*)bp.take(sizeof(float) * n);
    sd.yb.ptr = bp.take(e * (size_t)Me * d); sd.yb.cols = d;
    sd.abuf.ptr = bp.take(e * (size_t)Me * d); sd.abuf.cols = d;
    sd.hbuf.ptr = bp.take(e * (size_t)Me * F); sd.hbuf.cols = F;
    sd.qbuf = bp.take(e * (size_t)Me * d);
    sd.ktmp = bp.take(e * (size_t)Me * d);
    sd.vtmp = bp.take(e * (size_t)Me * d);
  }
  {
    const size_t pack = e * (size_t)c.n_dec * 2 * d * d, bpack = sizeof(float) * (size_t)c.n_dec * 2 * d;
    h->ar.ckv_pack = bp.take(pack); h->ar.cbkv_pack = (float*)bp.take(bpack);
    if (c.has_drafter) { h->nar.ckv_pack = bp.take(pack); h->nar.cbkv_pack = (float*)bp.take(bpack); }
  }
  h->n_vtiles = (c.vocab + 127) / 128;
  h->part_val = (float*)bp.take(sizeof(float) * (size_t)h->n_vtiles * Mv);
  h->part_idx = (int*)bp.take(sizeof(int) * (size_t)h->n_vtiles * Mv);
  h->part_cnt = (int*)bp.take(sizeof(int) * (size_t)h->n_vtiles * Mv);
  h->draft_val = (float*)bp.take(sizeof(float) * (size_t)Mv);
  h->draft_id = (int*)bp.take(sizeof(int) * (size_t)Mv);
  h->max_pos = std::max(c.max_src, c.max_tgt + 1);
  h->pe = (float*)bp.take(sizeof(float) * (size_t)h->max_pos * d);
  h->ovr = (int*)bp.take(sizeof(int) * (size_t)B * c.max_tgt);
  h->in_max = (int*)bp.take(sizeof(int) * (size_t)B, 256);
  for (int i = 0; i < 2; ++i) {
    h->mega_maps[i] = (CUtensorMap*)bp.take(sizeof(CUtensorMap) * (size_t)(6 * c.n_dec + 1));
    h->mega_layers[i] = (mega::LayerPtrs*)bp.take(sizeof(mega::LayerPtrs) * (size_t)c.n_dec);
    h->mega_stats[i] = (float*)bp.take(sizeof(float) * 2 * (size_t)(d / 128 + 1) * M_all);
  }
  h->mega_timeline = (unsigned long long*)bp.take(sizeof(unsigned long long) * 2 * (size_t)(mega::ST_PER_LAYER * c.n_dec + 1));
  for (int k = 0; k < PK_COUNT; ++k) plan_take(bp, h->pass[k].plan, B, h->pass[k].M_cap);
  DevState& s = h->st;
  auto ints = [&](size_t n) { return (int*)bp.take(sizeof(int) * n, 256); };
  s.len = ints(B); s.last = ints(B); s.fin = ints(B); s.maxlen = ints(B); s.srclen = ints(B);
  s.src = ints((size_t)B * c.max_src);
  s.out_ids = ints((size_t)B * c.max_tgt);
  s.drafts = ints((size_t)B * c.kmax); s.pred = ints((size_t)B * c.kmax); s.n_acc = ints(B);
  s.stat_it = ints(B); s.stat_acc = ints(B); s.stat_off = ints(B);
  s.loop_it = ints(8); s.status = ints(4); s.all_fin = ints(4); s.words = ints(4);
  s.sync_ctr = (unsigned int*)ints((size_t)mega::SYNC_COUNTERS * mega::SYNC_STRIDE);
  s.cross_base = ints(B);
  s.gidx = ints((size_t)B * c.kmax);
  s.enc_slot = ints((size_t)B * c.max_src);
  s.user_k = ints(B); s.user_drafts = ints((size_t)B * c.kmax);
  return align_up(bp.off, 1024);
}

int check_cfg(const ad_model_cfg* c, std::string* why) {
  auto bad = [&](const char* m) { *why = m; return AD_ERR_ARG; };
  if (!c) return bad("cfg is null");
  if (c->d_model <= 0 || c->n_heads <= 0 || c->d_model % c->n_heads) return bad("d_model must be a positive multiple of n_heads");
  const int dh = c->d_model / c->n_heads;
  if (dh != 32 && dh != 64) return bad("head dimension must be 32 or 64");
  if (c->d_model > 1024) return bad("d_model must be at most 1024");
  if (c->d_ffn <= 0 || c->vocab <= 4 || c->n_enc < 1 || c->n_dec < 1) return bad("bad model sizes");
  if (c->dtype != AD_DTYPE_FP32 && c->dtype != AD_DTYPE_BF16) return bad("dtype must be AD_DTYPE_FP32 or AD_DTYPE_BF16");
  if (c->dtype == AD_DTYPE_BF16 && (c->d_model % 128 || c->d_ffn % 64)) return bad("BF16 needs d_model to be a multiple of 128 and d_ffn a multiple of 64");
  // (biases and gains are read 16 bytes at a time, and the vectors behind a b1 begin where it ends)
  if (c->dtype == AD_DTYPE_FP32 && c->d_ffn % 4) return bad("FP32 needs d_ffn to be a multiple of 4");
  if (c->max_batch < 1 || c->max_batch > 256) return bad("max_batch must be 1..256");
  if (c->max_src < 1 || c->max_tgt < 1) return bad("max_src and max_tgt must be positive");
  if (c->kmax < 1 || c->kmax > 256 || c->kmax > c->max_tgt) return bad("kmax must be 1..min(256, max_tgt)");
  const int ids[4] = {c->bos, c->pad, c->eos, c->mask};
  for (int i = 0; i < 4; ++i) if (ids[i] < 0 || ids[i] >= c->vocab) return bad("special token id outside the vocabulary");
  if (!(c->ln_eps >= 0.f)) return bad("ln_eps must be non-negative");
  return AD_OK;
}

void weight_counts(const ad_model_cfg& c, size_t* mat, size_t* vec) {
  const size_t d = c.d_model, F = c.d_ffn, V = c.vocab;
  *mat = V * d + (size_t)c.n_enc * (3 * d * d + d * d + 2 * d * F) + (size_t)c.n_dec * (3 * d * d + d * d + d * d + 2 * d * d + d * d + 2 * d * F);
  *vec = (size_t)c.n_enc * (3 * d + d + 2 * d + F + d + 2 * d) + (size_t)c.n_dec * (3 * d + d + 2 * d + d + 2 * d + d + 2 * d + F + d + 2 * d);
}

int bind_model(ad_handle* h, Model& m, const ad_model_weights& w) {
  const ad_model_cfg& c = h->cfg;
  const int d = c.d_model, F = c.d_ffn;
  if (!w.matrices || !w.vectors) return fail(h, AD_ERR_ARG, "weight pointers are null");
  if (reinterpret_cast<uintptr_t>(w.vectors) % 16) return fail(h, AD_ERR_ARG, "weight vectors must be 16-byte aligned");
  if (reinterpret_cast<uintptr_t>(w.matrices) % 256) return fail(h, AD_ERR_ARG, "weight matrices must be 256-byte aligned");
  const char* mp = static_cast<const char*>(w.matrices);
  const float* vp = w.vectors;
  bool ok = true;
  auto mat = [&](Mat& t, int N, int K) {
    t.ptr = mp; t.N = N; t.K = K;
    mp += (size_t)N * K * h->esz;
    if (h->bf16) ok = ok && make_map(&t.map, t.ptr, N, K, tc::BLOCK_N_FEAT);
  };
  auto vec = [&](const float*& t, int n) { t = vp; vp += n; };
  mat(m.emb, c.vocab, d);
  if (h->bf16) ok = ok && make_map(&m.emb.map64, m.emb.ptr, c.vocab, d, tc::P_BOX);
  m.enc.resize(c.n_enc);
  m.dec.resize(c.n_dec);
  for (auto& L : m.enc) {
    mat(L.wqkv, 3 * d, d); mat(L.wo, d, d); mat(L.w1, F, d); mat(L.w2, d, F);
    vec(L.bqkv, 3 * d); vec(L.bo, d); vec(L.ln1g, d); vec(L.ln1b, d); vec(L.b1, F); vec(L.b2, d); vec(L.ln2g, d); vec(L.ln2b, d);
  }
  for (auto& L : m.dec) {
    mat(L.wqkv, 3 * d, d); mat(L.wo, d, d); mat(L.cq, d, d); mat(L.ckv, 2 * d, d); mat(L.co, d, d); mat(L.w1, F, d); mat(L.w2, d, F);
    vec(L.bqkv, 3 * d); vec(L.bo, d); vec(L.ln1g, d); vec(L.ln1b, d); vec(L.cbq, d); vec(L.cbkv, 2 * d); vec(L.cbo, d);
    vec(L.ln2g, d); vec(L.ln2b, d); vec(L.b1, F); vec(L.b2, d); vec(L.ln3g, d); vec(L.ln3b, d);
  }
  if (!ok) return fail(h, AD_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight matrix");
  m.present = true;
  return AD_OK;
}

// ---- kernel launch helpers -----------------------------------------------------------------------

// AD_NO_PDL=1 in the environment turns programmatic dependent launch off; a thread that times every launch turns it off for itself.
bool env_is_1(const char* name) {
  const char* e = getenv(name);
  return e && e[0] == '1';
}
thread_local bool t_serialise_launches = false;
bool use_pdl() {
  static const bool off = env_is_1("AD_NO_PDL");
  return !off && !t_serialise_launches;
}

// Launches `kernel` so that it may begin while its predecessor in the stream still runs (the kernels
// themselves wait with griddepcontrol.wait before touching anything a predecessor writes).
// shared_share: share of an SM's memory to prefer as shared memory, in percent (negative: the runtime's choice).
template <typename... KArgs, typename... Args>
cudaError_t launch_shared(int shared_share, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n_attr = 0;
  if (use_pdl()) {
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (shared_share >= 0) {
    attr[n_attr].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[n_attr++].val.sharedMemCarveout = shared_share;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n_attr;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(std::forward<Args>(args))...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  return launch_shared(-1, kernel, grid, block, smem, st, std::forward<Args>(args)...);
}

// Per-device caches (a process may hold handles on several GPUs): SM count, and which kernels already had their
// dynamic shared-memory limit raised on that device (the attribute is per device, not per process).
constexpr int kMaxDevices = 64;
int current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
  return dev;
}
int num_sms() {
  static int n[kMaxDevices] = {};
  const int dev = current_device();
  if (!n[dev]) {
    cudaDeviceGetAttribute(&n[dev], cudaDevAttrMultiProcessorCount, dev);
    if (n[dev] <= 0) n[dev] = 148;
  }
  return n[dev];
}

// Share of an SM's memory that leaves room for one CTA of smem_bytes and not for two.  Left to itself the runtime makes room for two, and
// the CTAs of a small grid share SMs while others stand by (weights and activations of both then queue for one L1).
int one_cta_share(size_t smem_bytes) { return (int)((smem_bytes + 1024) * 100 / (228 * 1024)) + 1; }

// Dynamic shared memory of a pass of M tokens: the ring doubles as the epilogue's transposition buffer (up to 128 rows of 132 floats)
// and the few-token partial sums.
int tc_smem_need(const GeoRule& r, int M, int budget) {
  const Geo g = geometry(r, M);
  const int need = g.few ? (int)few::red_bytes(2)
                         : std::max(tc::ring_stages(g.tile, (r.K / tc::BLOCK_K + g.ksplit - 1) / g.ksplit, budget) * (tc::A_STAGE_BYTES + g.tile * tc::BLOCK_K * 2),
                                    std::min(g.tile, 128) * 132 * 4);
  return need + 1024;
}
// Launch shape of the tensor-core projection kernel for passes of at most M_cap tokens: the most CTAs any token count asks for
// and the shared memory of its ring.  Up to one CTA per SM: ~200 KB, so that the ring is as deep as it can be; with more CTAs
// half of that, so that two CTAs share an SM: up to twice the SM count the whole grid is then resident at once, beyond that
// one CTA's prologue and epilogue overlap the other's K loop.
TcShape tc_shape(const GeoRule& r, int M_cap, bool exact) {
  TcShape sh = {1, 0, 0, 1};
  auto each = [&](auto f) {
    if (exact) { f(M_cap); return; }
    for (int M = 1; M <= M_cap; M += M < 2048 ? 1 : 64) f(M);
    f(M_cap);
  };
  each([&](int M) { sh.ctas = std::max(sh.ctas, tc::geometry_ctas(r, M)); sh.ksplit = std::max(sh.ksplit, geometry(r, M).ksplit); });
  sh.budget = (sh.ctas > num_sms() ? 100 : 200) * 1024;
  each([&](int M) { sh.smem = std::max(sh.smem, tc_smem_need(r, M, sh.budget)); });
  return sh;
}

template <int EPI, int NCH>
cudaError_t launch_tc_n(cudaStream_t st, const CUtensorMap& mw, const tc::TileMaps& mx, const GemmParams& p, const TcShape& sh, const void* w,
                        const void* x) {
  static bool attr_set[kMaxDevices] = {};
  const int dev = current_device();
  if (!attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(tc::gemm_tc_kernel<EPI, NCH>, cudaFuncAttributeMaxDynamicSharedMemorySize, 204 * 1024);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  const int nf = (p.N + tc::BLOCK_N_FEAT - 1) / tc::BLOCK_N_FEAT;
  return launch_k(tc::gemm_tc_kernel<EPI, NCH>, dim3(nf, (sh.ctas + nf - 1) / nf), dim3(tc::THREADS), sh.smem, st, mw, mx, p, sh.budget, (const bf16*)w, (const bf16*)x);
}
template <int EPI>
cudaError_t launch_tc(cudaStream_t st, const CUtensorMap& mw, const tc::TileMaps& mx, const GemmParams& p, const TcShape& sh, const void* w = nullptr,
                      const void* x = nullptr) {
  if (EPI != EPI_ARGMAX && p.rule.few_split > 0) {
    switch (p.K / p.rule.few_split / 256) {
      case 1: return launch_tc_n<EPI, EPI == EPI_ARGMAX ? 0 : 1>(st, mw, mx, p, sh, w, x);
      case 2: return launch_tc_n<EPI, EPI == EPI_ARGMAX ? 0 : 2>(st, mw, mx, p, sh, w, x);
      case 3: return launch_tc_n<EPI, EPI == EPI_ARGMAX ? 0 : 3>(st, mw, mx, p, sh, w, x);
      default: return launch_tc_n<EPI, EPI == EPI_ARGMAX ? 0 : 4>(st, mw, mx, p, sh, w, x);
    }
  }
  return launch_tc_n<EPI, 0>(st, mw, mx, p, sh, w, x);
}

// Projection + arg-max over many tokens: the persistent kernel on pairs of SMs beyond 128 tokens (a pair's tile is 256), once there
// is at least one (128 token x 256 vocabulary row) piece of work per SM; up to 128 tokens one tile per CTA is faster (100 tokens x
// 50265 x 768: 18 us against 23).  AD_NO_PERSISTENT_VOCAB=1 keeps the one-tile-per-CTA kernel.
bool vocab_goes_persistent(int K, int N, int M_cap, const float* bias) {
  static const bool enabled = [] { const char* e = getenv("AD_NO_PERSISTENT_VOCAB"); return !(e && e[0] == '1'); }();
  if (!enabled || bias || K % tc::BLOCK_K || M_cap <= tc::P_TOK) return false;
  return (long)((N + tc::P_VOC - 1) / tc::P_VOC) * ((M_cap + tc::P_TOK - 1) / tc::P_TOK) >= (long)num_sms();
}
// mw64: the matrix' map with a 64-row box; mx128: the token operand's with a 128-row box.
template <bool STREAM>
cudaError_t launch_vocab_pair(cudaStream_t st, const CUtensorMap& mw64, const CUtensorMap& mx128, const GemmParams& p, int M_cap) {
  static bool attr_set[kMaxDevices] = {};
  const int dev = current_device();
  constexpr int kSmemLimit = 227 * 1024 - 512;   // the kernel's static shared memory is a few hundred bytes
  if (!attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(tc::vocab_argmax_pair_kernel<STREAM>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  const int kb = p.K / tc::BLOCK_K;
  const int stages = STREAM ? tc::P_MAX_STAGES : clampi((kSmemLimit - 1024 - kb * tc::P_A_KB_BYTES) / tc::P_B_STAGE_BYTES, 1, tc::P_MAX_STAGES);
  const long units = (long)((p.N + tc::BLOCK_N_FEAT - 1) / tc::BLOCK_N_FEAT) * ((M_cap + 2 * tc::P_TOK - 1) / (2 * tc::P_TOK));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (int)std::min<long>(units, num_sms() / 2)); cfg.blockDim = dim3(tc::P_THREADS);
  cfg.dynamicSmemBytes = tc::vocab_pair_smem(kb, stages); cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = use_pdl() ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, tc::vocab_argmax_pair_kernel<STREAM>, mw64, mx128, p, stages);
}
cudaError_t launch_vocab_persistent(cudaStream_t st, const CUtensorMap& mw64, const CUtensorMap& mx128, const GemmParams& p, int M_cap) {
  return p.K / tc::BLOCK_K > tc::P_MAX_KB ? launch_vocab_pair<true>(st, mw64, mx128, p, M_cap) : launch_vocab_pair<false>(st, mw64, mx128, p, M_cap);
}

// Projection of a pass with few tokens (gemm_few.cuh).  ksplit: few::split_for of the shape, non-zero.
template <int EPI, bool EMB = false>
cudaError_t launch_few(cudaStream_t st, const Mat& W, const void* x, const GemmParams& p, int ksplit, bool decoder, const few::EmbedParams& ep = {}) {
  const dim3 grid(p.N / few::FEAT, ksplit);
  const bf16 *w = (const bf16*)W.ptr, *xp = (const bf16*)x;
  const dim3 wgrid(p.N / few::W_FEAT, ksplit);
  // One CTA of the 16-feature forms an SM where there are no more CTAs than SMs.  Whole calls, the runtime's choice -> this: 512 wide,
  // batch 1 1124 -> 1075 us, batch 2 with drafter 4360 -> 3950, batch 8 3560 -> 3520; 12+2, batch 1 960 -> 906.  Room for two again: 1120,
  // 4300, 3530, 961.  Larger grids would take turns: encoder calls of four layers, 512 wide, batch 1, 25 tokens: 89.1 us with one CTA an SM
  // for the 384 CTAs of the cross-attention's keys and values, 87.1 with the runtime's choice; feed-forward width 4096 (256 CTAs) 93.7, 86.7.
  const int share = (long)grid.x * grid.y <= num_sms() ? one_cta_share(few::red_bytes(2)) : -1;
  switch (p.K / ksplit / 256) {
    case 1: return launch_shared(share, few::gemm_few_kernel<EPI, 1, EMB>, grid, dim3(few::THREADS), 0, st, w, xp, p, ep);
    case 2: return launch_shared(share, few::gemm_few_kernel<EPI, 2, EMB>, grid, dim3(few::THREADS), 0, st, w, xp, p, ep);
    case 3:
      return launch_k(decoder ? few::gemm_few_wide_kernel<EPI, 3, EMB, true> : few::gemm_few_wide_kernel<EPI, 3, EMB, false>, wgrid,
                      dim3(few::THREADS), 0, st, w, xp, p, ep);
    default:
      return launch_k(decoder ? few::gemm_few_wide_kernel<EPI, 4, EMB, true> : few::gemm_few_wide_kernel<EPI, 4, EMB, false>, wgrid,
                      dim3(few::THREADS), 0, st, w, xp, p, ep);
  }
}

// Geometry rule of a projection of pass pc.  split: its consumer adds partial sums up.
GeoRule geo_rule(const PassCfg& pc, int epi, int N, int K, bool split, bool has_bias) {
  GeoRule r = {N, K, pc.ntile, split ? pc.max_split : 1, num_sms(), 0, 0, 0};
  if (epi == EPI_F32 ? split : (epi != EPI_ARGMAX && has_bias)) r.few_split = few::split_for(N, K, split, pc.max_split);
  if (r.few_split > 0) {
    // (within a larger capacity a pass of few tokens runs the 16-feature form inside the tensor-core kernel)
    r.few_tokens = pc.M_cap <= pc.few_cap ? pc.few_cap : few::INNER_TOKENS;
  }
  return r;
}
// Whether every projection of such a shape in pass pc runs on the few-token kernel.
bool always_few(const PassCfg& pc, const GeoRule& r) { return r.few_split > 0 && pc.M_cap <= r.few_tokens; }

template <int EPI, int TJ>
cudaError_t launch_simt_tile(cudaStream_t st, const void* w, const void* x, const GemmParams& p, int M_cap) {
  constexpr int FEAT = EPI == EPI_ARGMAX ? simt::ARGMAX_FEAT : 64;
  constexpr size_t smem = simt::smem_bytes<FEAT, TJ>();
  static bool attr_set[kMaxDevices] = {};
  const int dev = current_device();
  if (!attr_set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(simt::gemm_f32_kernel<EPI, FEAT, TJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  const int vec = p.K % 4 == 0 && (reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(x)) % 16 == 0;
  const dim3 grid((p.N + FEAT - 1) / FEAT, (M_cap + 4 * TJ - 1) / (4 * TJ));
  return launch_k(simt::gemm_f32_kernel<EPI, FEAT, TJ>, grid, dim3(2 * FEAT), smem, st, (const float*)w, (const float*)x, p, vec);
}
// FP32 projection in tiles of 32 tokens, or of 16 where the fullest SM then has less to do: a small tile takes two thirds of a
// large one's time (7 x 1536 x 512: 9.6 us against 13; 100 x 1024 x 4096: 50 against 73; with the same number of tiles for an SM
// as before there is nothing to gain: 40 x 4096 x 1024 23 against 22).
template <int EPI>
cudaError_t launch_simt(cudaStream_t st, const void* w, const void* x, const GemmParams& p, int M_cap) {
  const int feat = EPI == EPI_ARGMAX ? simt::ARGMAX_FEAT : 64, sms = num_sms();
  auto per_sm = [&](int tokens) { return ((long)((p.N + feat - 1) / feat) * ((M_cap + tokens - 1) / tokens) + sms - 1) / sms; };
  return 2 * per_sm(16) <= 3 * per_sm(32) ? launch_simt_tile<EPI, 4>(st, w, x, p, M_cap) : launch_simt_tile<EPI, 8>(st, w, x, p, M_cap);
}
// The few-token FP32 kernel: passes of at most kFewTokens tokens, shapes it covers.
bool f32_few(const PassCfg& pc, int epi, int N, int K) { return pc.M_cap <= kFewTokens && epi != EPI_ARGMAX && simt::few_fits(N, K); }
// The FP32 kernels of a sublayer (this one and the attention with one query per warp) keep to one CTA an SM whatever their grid: where only
// one of two neighbours does, the change from one share to the other costs more than a second CTA gains.  Whole calls, both at one CTA an
// SM -> the attention at the runtime's choice once it has more CTAs than SMs: 128 wide, batch 32 2264 -> 2458 us; 256 wide, batch 12
// 3223 -> 3530; 512 wide, batch 6 3692 -> 3775, 12 4955 -> 5460, 24 6754 -> 6910.
template <int EPI, int NQ>
cudaError_t launch_simt_few_n(cudaStream_t st, const Mat& W, const void* x, const GemmParams& p) {
  const int share = one_cta_share(sizeof(float) * simt::F_TOK * (64 * NQ + simt::F_PARTS * simt::F_FEAT));
  return launch_shared(share, simt::gemm_f32_few_kernel<EPI, NQ>, dim3(p.N / simt::F_FEAT), dim3(256), 0, st, (const float*)W.ptr, (const float*)x, p);
}
template <int EPI>
cudaError_t launch_simt_few(cudaStream_t st, const Mat& W, const void* x, const GemmParams& p) {
  switch (p.K / 64) {
    case 1: return launch_simt_few_n<EPI, 1>(st, W, x, p);
    case 2: return launch_simt_few_n<EPI, 2>(st, W, x, p);
    case 3: return launch_simt_few_n<EPI, 3>(st, W, x, p);
    case 4: return launch_simt_few_n<EPI, 4>(st, W, x, p);
    case 5: return launch_simt_few_n<EPI, 5>(st, W, x, p);
    case 6: return launch_simt_few_n<EPI, 6>(st, W, x, p);
    case 7: return launch_simt_few_n<EPI, 7>(st, W, x, p);
    default: return launch_simt_few_n<EPI, 8>(st, W, x, p);
  }
}

// Launch shape of a rule, worked out once per handle.  The key is everything the shape follows from: projections of equal N and K may
// still differ in their rule (a vocabulary as large as the feed-forward width never takes the few-token kernel, FFN1 does).
const TcShape& cached_shape(ad_handle* h, const GeoRule& r, int M_cap) {
  const auto key = std::make_tuple(r.N, r.K, r.max_tile, r.max_split, r.sms, r.few_split, r.few_tokens, r.fixed_tile, M_cap);
  auto it = h->tc_shapes.find(key);
  if (it == h->tc_shapes.end()) it = h->tc_shapes.emplace(key, tc_shape(r, M_cap, false)).first;
  return it->second;
}

// Whether a decoder pass reads more weights than stay in L2 (126 MB, shared with everything else) from one pass to the next.  Its kernels
// then fetch them from HBM, and can begin to when an SM has room for them, one kernel ahead at most: the feed-forward projections, 128 CTAs
// that fill an SM's registers each, waited 1.2 us for theirs.  So the QKV projection of a layer, three to four kernels ahead, brings
// the layer's feed-forward weights into L2, its first feed-forward projection the next layer's attention weights (both in the form for wide slices of K
// alone: models up to 512 wide prefetch nothing).  Whole calls: 1024 wide
// (242 MB a pass), batch 4 greedy 7730 -> 7580 us, batch 1 with drafter 3810 -> 3760; 768 wide (176 MB) 2287 -> 2267.  The embedding matrix
// fetched ahead in the last layers, or the first layer's weights at the end of the vocabulary kernel, gained nothing or lost it again.
bool weights_stream(const ad_handle* h) {
  const ad_model_cfg& c = h->cfg;
  const size_t d = c.d_model;
  return h->bf16 && h->esz * ((size_t)c.n_dec * (6 * d * d + 2 * d * c.d_ffn) + (size_t)c.vocab * d) > (size_t)100 << 20;
}
Prefetch attention_weights(const ad_handle* h, const Model& m, int l) {
  Prefetch f = {};
  if (!weights_stream(h) || l >= h->cfg.n_dec) return f;
  const size_t dd = h->esz * h->cfg.d_model * h->cfg.d_model;
  f.ptr[0] = (const char*)m.dec[l].wqkv.ptr; f.bytes[0] = prefetch_bytes(5 * dd);      // wqkv, wo, cq: one behind the other
  f.ptr[1] = (const char*)m.dec[l].co.ptr; f.bytes[1] = prefetch_bytes(dd);
  return f;
}
Prefetch ffn_weights(const ad_handle* h, const Model& m, int l) {
  Prefetch f = {};
  if (!weights_stream(h)) return f;
  const uint32_t df = prefetch_bytes(h->esz * h->cfg.d_model * h->cfg.d_ffn);
  f.ptr[0] = (const char*)m.dec[l].w1.ptr; f.bytes[0] = df;
  f.ptr[1] = (const char*)m.dec[l].w2.ptr; f.bytes[1] = df;
  return f;
}

// embed_of: the operand is the embedding of pass pk's tokens (first projection of a pass, few-token kernel only).
// split: the result is partial sums that the consumer adds up (EPI_F32).
int gemm(ad_handle* h, int epi, const Mat& W, const ActBuf& X, int pk, const int* M_ptr, int M_cap, GemmParams p, const Model* embed_of = nullptr,
         bool split = false) {
  p.K = W.K; p.N = W.N; p.M_ptr = M_ptr; p.M_cap = M_cap; p.status = h->st.status;
  cudaError_t e;
  {
    static const char* epi_name[4] = {"gemm_f32_partials", "gemm_act", "gemm_scatter", "gemm_vocab_argmax"};
    char nm[64];
    snprintf(nm, sizeof(nm), "%s N%d K%d", epi_name[epi & 3], W.N, W.K);
    note_launch(h, nm);
  }
  PassCfg& pc = h->pass[pk];
  if (h->bf16) p.rule = geo_rule(pc, epi, W.N, W.K, split, p.bias != nullptr);
  if (h->bf16 && always_few(pc, p.rule)) {
    const int split = p.rule.few_split;
    const bool decoder = pk != PK_ENCODE;
    switch (epi) {
      case EPI_F32: e = launch_few<EPI_F32>(h->stream, W, X.ptr, p, split, decoder); break;
      case EPI_ACT: e = launch_few<EPI_ACT>(h->stream, W, X.ptr, p, split, decoder); break;
      default:
        if (embed_of) {
          const few::EmbedParams ep = {(const bf16*)embed_of->emb.ptr, h->pe, sqrtf((float)W.K), pc.plan.tok_id, pc.plan.tok_pos, h->y};
          e = launch_few<EPI_SCATTER, true>(h->stream, W, X.ptr, p, split, decoder, ep);
        } else {
          e = launch_few<EPI_SCATTER>(h->stream, W, X.ptr, p, split, decoder);
        }
        break;
    }
  } else if (h->bf16 && epi == EPI_ARGMAX && pc.ntile == 256 && vocab_goes_persistent(W.K, W.N, M_cap, p.bias)) {
    // (a pass with a 256-token tile also has the 128-row map of its token operand)
    e = launch_vocab_persistent(h->stream, W.map64, X.map_for(pk, tc::P_TOK), p, M_cap);
  } else if (h->bf16) {
    const TcShape& sh = cached_shape(h, p.rule, M_cap);
    switch (epi) {
      case EPI_F32: e = launch_tc<EPI_F32>(h->stream, W.map, X.map[pk], p, sh, W.ptr, X.ptr); break;
      case EPI_ACT: e = launch_tc<EPI_ACT>(h->stream, W.map, X.map[pk], p, sh, W.ptr, X.ptr); break;
      case EPI_SCATTER: e = launch_tc<EPI_SCATTER>(h->stream, W.map, X.map[pk], p, sh, W.ptr, X.ptr); break;
      default: e = launch_tc<EPI_ARGMAX>(h->stream, W.map, X.map[pk], p, sh); break;
    }
  } else if (p.M_ptr && f32_few(h->pass[pk], epi, W.N, W.K)) {
    switch (epi) {
      case EPI_F32: e = launch_simt_few<EPI_F32>(h->stream, W, X.ptr, p); break;
      case EPI_ACT: e = launch_simt_few<EPI_ACT>(h->stream, W, X.ptr, p); break;
      default: e = launch_simt_few<EPI_SCATTER>(h->stream, W, X.ptr, p); break;
    }
  } else {
    switch (epi) {
      case EPI_F32: e = launch_simt<EPI_F32>(h->stream, W.ptr, X.ptr, p, M_cap); break;
      case EPI_ACT: e = launch_simt<EPI_ACT>(h->stream, W.ptr, X.ptr, p, M_cap); break;
      case EPI_SCATTER: e = launch_simt<EPI_SCATTER>(h->stream, W.ptr, X.ptr, p, M_cap); break;
      default: e = launch_simt<EPI_ARGMAX>(h->stream, W.ptr, X.ptr, p, M_cap); break;
    }
  }
  if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("GEMM launch: ") + cudaGetErrorString(e));
  return AD_OK;
}

template <typename T, int D, int Q, bool FUSE = false, int MINB = 1>
cudaError_t launch_attention(dim3 grid, dim3 block, cudaStream_t st, const AttnParams& p) {
  constexpr size_t smem = att_smem_bytes<D, Q>();
  static bool attr_set[kMaxDevices] = {};
  const int dev = current_device();
  if (!attr_set[dev] && smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(attention_kernel<T, D, Q, FUSE, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  attr_set[dev] = true;
  const int share = std::is_same<T, float>::value && Q == 1 ? one_cta_share(smem + sizeof(bf16) * ATT_WARPS * 96) : -1;
  return launch_shared(share, attention_kernel<T, D, Q, FUSE, MINB>, grid, block, smem, st, p);
}

// Whether a verification pass has, at its capacity, work for at most three waves (beyond 512 wide four) of the few-query kernel's CTAs (attention_few.cuh).
bool within_few_waves(const ad_handle* h, const PassCfg& pc) {
  const int split = few::att_few_split(h->cfg.d_model);
  return pc.pieces(h->cfg.max_batch, few::AQ) * h->cfg.n_heads * split <= (split > 1 ? 4L : 3L) * num_sms();
}
// Whether the grid of the FFMA kernel, a CTA for every eight queries that a row could have, is too large for it.  It counts CTAs without work as well, in layouts for few tokens
// most of them: 13 to 24 rows of one token in blocks of up to 64, 768 wide, counted by the work there can be (FFMA kernel) -> by the grid (MMA), four layers, 178 -> 138, 308 -> 149 us.
bool many_queries(const ad_handle* h, const PassCfg& pc, int rows) {
  return (long)rows * ((pc.seg_max + 7) / 8) * h->cfg.n_heads > 3L * num_sms();
}

int attention(ad_handle* h, const PassCfg& pc, const void* q, const void* k, const void* v, void* out,
              const int* key_base, const int* nkeys_tok, const int* nkeys_row, int max_keys,
              const float* q_bias = nullptr, const Partials* q_part = nullptr, const Mat* wo = nullptr, bool* fused = nullptr, bool kv_old = false) {
  const ad_model_cfg& c = h->cfg;
  AttnParams p;
  p.q = q; p.k = k; p.v = v; p.out = out;
  p.q_part = q_part ? *q_part : Partials{}; p.M_ptr = pc.plan.M; p.q_bias = q_bias;
  p.seg_off = pc.plan.seg_off; p.seg_len = pc.plan.seg_len;
  p.key_base = key_base; p.nkeys_tok = nkeys_tok; p.nkeys_row = nkeys_row;
  p.d = c.d_model;
  // one query per warp while the grid stays within a couple of waves, eight when there are many queries
  const int dh = c.d_model / c.n_heads;
  const bool many = many_queries(h, pc, h->dims.B);
  p.scale = 1.0f / sqrtf((float)dh);
  // Tensor-core kernels when there are thousands of queries or rows may hold hundreds of keys (max_keys: the capacity, known on
  // the host); the FFMA kernel spreads few queries and few keys over more CTAs.
  // An encoder's rows are all queries: between the two it keeps the FFMA kernel, which has the output projection in it, only for rows of one
  // key tile in at most one and a half waves of its CTAs (two for rows of at most eight, half of an MMA tile).  Calls of four layers, FFMA -> MMA, us:
  // 768 wide 8 x 8 tokens 113 -> 120, 2 x 64 171 -> 176, 4 x 17 127 -> 138, but 4 x 48 153 -> 146, 2 x 90 171 -> 147, 1 x 200 274 -> 173; 1024 wide
  // 3 x 50 215 -> 184, 1 x 150 273 -> 190; 512 wide 5 x 81 190 -> 146, 16 x 17 143 -> 128, 32 x 8 125 -> 129.
  const long ffma_ctas = (long)h->dims.B * ((pc.seg_max + 7) / 8) * c.n_heads;
  const bool encode_mma = &pc == &h->pass[PK_ENCODE] && (pc.seg_max > ATT_KT || 2 * ffma_ctas > (pc.seg_max <= 8 ? 4 : 3) * (long)num_sms());
  if (h->bf16 && dh == 64 && (many || encode_mma || max_keys >= 256) && !(max_keys >= 256 && pc.seg_max <= 128)) {
    // What the FFMA kernel would do with FP32 probabilities keeps them (two BF16 numbers each; 0 to 5 us of such a call more than with one):
    // memory of one layer dominated by its attention, 27 sizes of 256 to 1024 wide: error against 64 bits within 0.03 % of the FFMA kernel's,
    // 0.3 to 1.8 % above it with probabilities rounded to BF16.
    // So do layouts for few tokens whose grid alone is many, and verification passes within the most waves that the few-query kernel takes (see attention_is_few).
    const bool many_work = pc.pieces(h->dims.B, 8) * c.n_heads > 3L * num_sms();
    const bool split_p = (!many_work || (&pc == &h->pass[PK_VERIFY] && within_few_waves(h, pc))) && max_keys < 256;
    // Warps share a 16-query tile and split the keys (2 or 4 key groups) when rows have few queries; two groups also while
    // 64-query CTAs would not give every SM two.
    const long full = (long)h->dims.B * ((pc.seg_max + AM_Q - 1) / AM_Q) * c.n_heads;
    const int ng = pc.seg_max <= 16 ? 4 : (pc.seg_max <= 32 || (full < 2 * num_sms() && max_keys > AM_KT) ? 2 : 1);
    const int qcta = AM_Q / ng;
    p.qchunks = (pc.seg_max + qcta - 1) / qcta;
    note_launch(h, "attention_mma");
    const dim3 mgrid(h->dims.B * p.qchunks, c.n_heads);
    auto pick = [&](auto split) {
      constexpr bool S = decltype(split)::value;
      return ng == 4 ? attention_mma_kernel<4, S> : (ng == 2 ? attention_mma_kernel<2, S> : attention_mma_kernel<1, S>);
    };
    auto* kernel = split_p ? pick(std::true_type()) : pick(std::false_type());
    const cudaError_t em = launch_k(kernel, mgrid, dim3(128), 0, h->stream, p, kv_old ? 1 : 0);
    if (em != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("attention launch: ") + cudaGetErrorString(em));
    return AD_OK;
  }
  if (h->bf16 && dh == 64 && max_keys >= 256) {
    // few queries per row over hundreds of keys: the keys are spread over the warps of a CTA (whole 64-key tiles per warp), 1 or
    // 2 query tiles of 16 per CTA
    const int qt = pc.seg_max <= 16 ? 1 : 2;
    const int threads = 32 * qt * 8, slots = att_long_slots(max_keys, threads);
    p.qchunks = (pc.seg_max + 16 * qt - 1) / (16 * qt);
    note_launch(h, "attention_long");
    const dim3 mgrid(h->dims.B * p.qchunks, c.n_heads);
    const size_t smem = att_long_smem(slots, qt);
    static bool attr_set[kMaxDevices] = {};
    const int dev = current_device();
    cudaError_t em = cudaSuccess;
    if (!attr_set[dev]) {
      for (auto* kernel : {attention_long_kernel<1, 8>, attention_long_kernel<2, 8>})
        if (em == cudaSuccess) em = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)att_long_smem(AL_MAX_SLOTS, 2));
      if (em != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("attention attribute: ") + cudaGetErrorString(em));
      attr_set[dev] = true;
    }
    auto* kernel = qt == 1 ? attention_long_kernel<1, 8> : attention_long_kernel<2, 8>;
    em = launch_k(kernel, mgrid, dim3(threads), smem, h->stream, p, slots, kv_old ? 1 : 0);
    if (em != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("attention launch: ") + cudaGetErrorString(em));
    return AD_OK;
  }
  const int qpw = many ? 8 : 1;
  p.qchunks = (pc.seg_max + 8 * qpw - 1) / (8 * qpw);
  dim3 grid(h->dims.B * p.qchunks, c.n_heads);
  const dim3 block(256);
  cudaError_t e;
#define AD_ATT(T, D, Q) launch_attention<T, D, Q>(grid, block, h->stream, p)
  // few queries, 64-wide heads: the output projection rides along (one partial sum per head for the LayerNorm kernel)
  const bool fuse = h->sw.fuse_attn_proj && wo && fused && h->pre2 && h->bf16 && dh == 64 && !many && c.n_heads <= pc.max_split &&
                    c.n_heads <= 16 && c.d_model % 128 == 0;
  if (fused) *fused = fuse;
  note_launch(h, fuse ? "attention+out_proj" : "attention");
  if (fuse) {
    p.wo = (const bf16*)wo->ptr; p.o_part = h->pre2; p.o_stride = (size_t)pc.M_cap * c.d_model;
    // more CTAs than SMs: the two-CTAs-per-SM build, so that the grid is still one wave
    e = (long)grid.x * grid.y > num_sms() ? launch_attention<bf16, 64, 1, true, 2>(grid, block, h->stream, p)
                                           : launch_attention<bf16, 64, 1, true, 1>(grid, block, h->stream, p);
  } else if (h->bf16) {
    if (dh == 64) e = AD_ATT(bf16, 64, 1);         // (many queries: the MMA kernels above)
    else e = many ? AD_ATT(bf16, 32, 8) : AD_ATT(bf16, 32, 1);
  } else {
    if (dh == 64) e = many ? AD_ATT(float, 64, 8) : AD_ATT(float, 64, 1);
    else e = many ? AD_ATT(float, 32, 8) : AD_ATT(float, 32, 1);
  }
#undef AD_ATT
  if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("attention launch: ") + cudaGetErrorString(e));
  return AD_OK;
}

// Whether the few-query kernel (attention_few.cuh) serves an attention of pass pk: BF16, 64-wide heads, the keys within four rounds
// of its warps, and work for a few waves of CTAs at most, counted by what the pass could hold (rows that have ended, shorter blocks and a
// drafter's prefix that has not grown leave less).  A wave costs 4 to 7 us, the projections that
// are kernels of their own otherwise 12 us a layer, so a verification pass may need three waves at capacity, a drafter's pass (on
// average half of its capacity) four.  Per decode iteration, one wave allowed -> this rule: base model, batch 12, blocks of 30:
// 214 -> 174 us; batch 24, 12: 237 -> 196; batch 20, 1: 188 -> 160; batch of 5 with drafter 442 -> 373; 1024 wide, batch 2, 40: 272 -> 226;
// batch 3 with drafter 662 -> 600.  Beyond: base batch 32 x 64 (seven waves) 270 -> 315, 1024 wide batch 16 x 1 (four) 239 -> 284.  Wide
// models with fewer than eight queries a row stay at one wave: their CTAs read two weight slices each for a tile that is mostly padding
// (768 wide, batch 12, 1: 202 against 210).  Looping grids, waves 2 / 2.5 / 3 / 3.5 / 4 / 4.5, whole calls: 512 wide, batch 20 5068 / 5046 / 5073 / 5147 / 5350 / 5443,
// batch 16, relaxed 2379 / 2375 / 2482 / 2483 / 2481 / 2480.
// Beyond 512 wide the few-query kernel is taken up to four waves only where the FFMA kernel would run instead, and not for blocks of eight, which fill that kernel's CTAs.
// Full blocks of 130 source tokens, four layers, between three and four waves, few-query kernel / the other one, us: FFMA 768 wide 11 x 18 274 / 351, 1024 wide 8 x 18 298 / 380,
// 768 wide 20 x 8 261 / 248; MMA 768 wide 8 x 48 293 / 243, 11 x 30 292 / 239, 20 x 10 277 / 233, 1024 wide 6 x 48 369 / 281, 8 x 30 324 / 276, 16 x 10 308 / 261.
// With 256 keys or more, where the other kernels round the probabilities, four.
// Layouts that the tokens pick hold as many as they are made for, and with 384 and 512 wide models two and a half waves are the line there; the MMA kernel
// beyond keeps FP32's probabilities up to three waves, as this one does (split_p in attention).  It does so for fewer than 256 keys, with more the line stays at three waves.
// A layout that has to hold whatever comes (device arrays) is mostly emptier than its capacity: verified blocks, two and a half waves for it as well -> three, 512 wide,
// rows x tokens of a capacity of 12 x 64: 12 x 4 218 -> 181 us, 12 x 20 262 -> 256, 12 x 45 319 -> 305, 12 x 64 330 -> 355.  Whole calls, probabilities rounded to BF16 in that
// band -> not: 512 wide, relaxed, 12 x 64 2007 -> 2015, 16 x 40 2001 -> 2029, 24 x 30 2492 -> 2504, 300 source tokens, 12 x 60 (three waves) 2327 -> 2375.
// An encoder's rows are as long as they are announced, and there is one projection to gain: one and a half.  Calls of four layers, 512 wide,
// kernel without it -> with it, us: 3 x 112 tokens 143 -> 137, 4 x 96 143 -> 134, 5 x 75 144 -> 137, 8 x 48 140 -> 132, 24 x 16 139 -> 131.  One wave
// beyond 512 wide (768 wide 2 x 90 147 -> 156, 3 x 64 147 -> 152), for rows of at most eight (512 wide 24 x 8 116 -> 118, 24 x 4 122 -> 125; 256 wide
// the CTAs are small and gain: 40 x 8 111 -> 105) and with 256 keys or more (1 x 304 140 -> 147).
bool attention_is_few(const ad_handle* h, int pk, int max_keys) {
  const ad_model_cfg& c = h->cfg;
  const PassCfg& pc = h->pass[pk];
  if (!h->sw.fuse_attn_proj || !h->bf16 || !h->pre2 || c.d_model != c.n_heads * 64 || c.d_model % 128 || c.d_model > 128 * few::MAX_WARPS) return false;
  const int split = few::att_few_split(c.d_model);
  if (max_keys > few::MAX_ROUNDS * few::AK * few::att_few_warps(c.d_model)) return false;
  // (in half waves)
  const bool one_wave = pk == PK_ENCODE ? split > 1 || max_keys >= 256 || (pc.seg_max <= 8 && c.d_model > 256) : split > 1 && pc.seg_max < 8;
  const bool wide_four = split > 1 && (std::max(c.max_src, c.max_tgt) >= 256 || (pc.seg_max > 8 && !many_queries(h, pc, c.max_batch)));
  const bool half_less = pc.few_cap == 0 && split == 1 && few::att_few_warps(c.d_model) > 4 && std::max(c.max_src, c.max_tgt) < 256;
  const int waves = one_wave ? 2 : pk == PK_ENCODE ? 3 : pk == PK_DRAFT || wide_four ? 8 : half_less ? 5 : 6;
  return 2 * pc.pieces(c.max_batch, few::AQ) * c.n_heads * split <= (long)waves * num_sms();
}

// Forms of the few-query kernel: query projection + 2 (pair of CTAs) + 4 (three or four rounds of keys) + 8 (looping grid).
typedef void (*AttentionFewKernel)(const few::FewAttnParams);
const AttentionFewKernel kAttentionFew[16] = {
    few::attention_few_kernel<false, 1, false, false>, few::attention_few_kernel<true, 1, false, false>,
    few::attention_few_kernel<false, 2, false, false>, few::attention_few_kernel<true, 2, false, false>,
    few::attention_few_kernel<false, 1, true, false>,  few::attention_few_kernel<true, 1, true, false>,
    few::attention_few_kernel<false, 2, true, false>,  few::attention_few_kernel<true, 2, true, false>,
    few::attention_few_kernel<false, 1, false, true>,  few::attention_few_kernel<true, 1, false, true>,
    few::attention_few_kernel<false, 2, false, true>,  few::attention_few_kernel<true, 2, false, true>,
    few::attention_few_kernel<false, 1, true, true>,   few::attention_few_kernel<true, 1, true, true>,
    few::attention_few_kernel<false, 2, true, true>,   few::attention_few_kernel<true, 2, true, true>};

// Attention with its output projection (partial sums per head in pre2) and, with wq, the query projection of x = yb.
int attention_few(ad_handle* h, const PassCfg& pc, const void* k, const void* v, const int* key_base, const int* nkeys_tok,
                  const int* nkeys_row, int max_keys, const Mat& wo, const Mat* wq = nullptr, const float* q_bias = nullptr) {
  const ad_model_cfg& c = h->cfg;
  few::FewAttnParams fp = {};
  AttnParams& p = fp.a;
  p.q = h->qbuf; p.k = k; p.v = v; p.q_bias = q_bias;
  p.seg_off = pc.plan.seg_off; p.seg_len = pc.plan.seg_len;
  p.key_base = key_base; p.nkeys_tok = nkeys_tok; p.nkeys_row = nkeys_row;
  p.d = c.d_model; p.scale = 0.125f;
  p.qchunks = (pc.seg_max + few::AQ - 1) / few::AQ;
  p.wo = (const bf16*)wo.ptr; p.o_part = h->pre2; p.o_stride = (size_t)pc.M_cap * c.d_model;
  if (wq) { fp.x = (const bf16*)h->yb.ptr; fp.wq = (const bf16*)wq->ptr; }
  const int split = few::att_few_split(c.d_model), warps = few::att_few_warps(c.d_model);
  static bool attr_set[kMaxDevices] = {};
  const int dev = current_device();
  cudaError_t e = cudaSuccess;
  if (!attr_set[dev]) {
    const int most = (int)few::att_few_smem(few::MAX_WARPS, few::MAX_ROUNDS, true);
    for (auto* kernel : kAttentionFew)
      if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("attention attribute: ") + cudaGetErrorString(e));
    attr_set[dev] = true;
  }
  note_launch(h, wq ? "q_proj+attention+out_proj" : "attention+out_proj");
  cudaLaunchConfig_t cfg = {};
  // A loop in place of a grid of more than one wave, even of one that has no work for most of its CTAs: a layout for 64 tokens of 14 rows with blocks of up
  // to 64, 512 wide, launched 448 CTAs, an SM each, for at most 144 with work (verified blocks of 14 / 28 / 56 tokens 167 / 173 / 187 us, as a loop 156 / 160 / 176).
  // (CTAs of up to four warps fit an SM twice and keep their waves: 256 wide, encoder calls of four layers, 10 x 60 tokens 114 -> 125 us as a loop)
  const long items = pc.pieces(h->dims.B, few::AQ), ctas = (long)h->dims.B * p.qchunks * c.n_heads * split;
  const bool loop = ctas > num_sms() && warps > 4 && c.n_heads * split <= num_sms();
  fp.rows = h->dims.B;
  const int groups = loop ? (int)std::min(items, (long)num_sms() / (c.n_heads * split)) : h->dims.B * p.qchunks;
  cfg.gridDim = dim3(groups * split, c.n_heads); cfg.blockDim = dim3(32 * warps);
  fp.rounds = (max_keys + few::AK * warps - 1) / (few::AK * warps);
  cfg.dynamicSmemBytes = few::att_few_smem(warps, fp.rounds, loop && wq && split > 1); cfg.stream = h->stream;
  cudaLaunchAttribute attr[2];
  int n_attr = 0;
  if (use_pdl()) {
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (wq && split > 1) {
    attr[n_attr].id = cudaLaunchAttributeClusterDimension;
    attr[n_attr].val.clusterDim.x = split; attr[n_attr].val.clusterDim.y = 1; attr[n_attr++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr; cfg.numAttrs = n_attr;
  auto* kernel = kAttentionFew[(wq ? 1 : 0) + (split - 1) * 2 + (fp.rounds > 2 ? 4 : 0) + (loop ? 8 : 0)];
  e = cudaLaunchKernelEx(&cfg, kernel, fp);
  if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("attention launch: ") + cudaGetErrorString(e));
  return AD_OK;
}

// y = LN(sum of the partial projections + bias + y); the GEMM-operand copy goes to `out` (default yb).
int layernorm(ad_handle* h, const PassCfg& pc, const Partials& pre, const float* bias, const float* g, const float* b,
              const ActBuf* out = nullptr) {
  const int d = h->cfg.d_model;
  const LnParams p = {pc.plan.M, pre, bias, h->y, g, b, d, h->cfg.ln_eps, h->y};
  // P, the partial sums in flight, from the most that any token count of the pass brings (it sets the registers, see layernorm_kernel)
  const int most = pre.nsplit > 0 ? pre.nsplit : cached_shape(h, pre.rule, pc.M_cap).ksplit;
  if (most > 32 || (most > 16 && d > 512)) return fail(h, AD_ERR_ARG, "layernorm: too many partial sums");
  char name[40];
  snprintf(name, sizeof(name), "residual+layernorm P%d", most);
  note_launch(h, name);
  auto go_n = [&](auto* yb, auto threads, auto parts) -> cudaError_t {
    using ActT = std::remove_pointer_t<decltype(yb)>;
    constexpr int T = decltype(threads)::value, P = decltype(parts)::value, per_cta = 256 / T;
    // (up to six tokens an SM a CTA each: batch of 8 with drafter, 648 tokens: 7910 us a call, 7930 with CTAs that loop)
    if (pc.M_cap > 6 * num_sms())
      return launch_k(layernorm_many_kernel<ActT, T, P>, dim3(std::min(4 * num_sms(), (pc.M_cap + per_cta - 1) / per_cta)), dim3(256), 0, h->stream, p, yb);
    return launch_k(layernorm_kernel<ActT, T, P>, dim3(pc.M_cap), dim3(T), 0, h->stream, p, yb);
  };
  auto go_t = [&](auto* yb, auto threads) -> cudaError_t {
    if (most <= 4) return go_n(yb, threads, std::integral_constant<int, 4>());
    if (most <= 8) return go_n(yb, threads, std::integral_constant<int, 8>());
    return go_n(yb, threads, std::integral_constant<int, 16>());
  };
  auto go = [&](auto* yb) -> cudaError_t {
    return d > 512 ? go_t(yb, std::integral_constant<int, 256>()) : go_t(yb, std::integral_constant<int, 128>());
  };
  void* yb = out ? out->ptr : h->yb.ptr;
  if (most > 16) {
    if (h->bf16) AD_CUDA(h, launch_k(layernorm_parts_kernel<bf16>, dim3(pc.M_cap), dim3(256), 0, h->stream, p, (bf16*)yb));
    else AD_CUDA(h, launch_k(layernorm_parts_kernel<float>, dim3(pc.M_cap), dim3(256), 0, h->stream, p, (float*)yb));
    return AD_OK;
  }
  const cudaError_t e = h->bf16 ? go((bf16*)yb) : go((float*)yb);
  if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("layernorm launch: ") + cudaGetErrorString(e));
  return AD_OK;
}
// Partial output projections of the attention kernels that carry it: one per head.
Partials head_partials(const ad_handle* h, const PassCfg& pc) {
  Partials q = {};
  q.ptr = h->pre2; q.nsplit = h->cfg.n_heads; q.stride = (size_t)pc.M_cap * h->cfg.d_model;
  return q;
}

// Projection whose consumer adds partial sums up (residual + LayerNorm, or the attention's queries); bias left to it.
int gemm_to_partials(ad_handle* h, const Mat& W, const ActBuf& X, int pk, Partials* out) {
  PassCfg& pc = h->pass[pk];
  GemmParams o = {};
  o.out_f32 = h->pre;
  *out = Partials{};
  out->ptr = h->pre;
  if (h->bf16) out->rule = geo_rule(pc, EPI_F32, W.N, W.K, true, false);
  else out->nsplit = 1;
  return gemm(h, EPI_F32, W, X, pk, pc.plan.M, pc.M_cap, o, nullptr, true);
}

int embed(ad_handle* h, const PassCfg& pc, const Model& m) {
  const int d = h->cfg.d_model;
  const float sc = sqrtf((float)d);
  note_launch(h, "embed");
  cudaError_t e;
  if (h->bf16) e = launch_k(embed_kernel<bf16, bf16>, dim3(pc.M_cap), dim3(128), 0, h->stream, pc.plan, (const bf16*)m.emb.ptr, (const float*)h->pe, d, sc, h->y, (bf16*)h->yb.ptr);
  else e = launch_k(embed_kernel<float, float>, dim3(pc.M_cap), dim3(128), 0, h->stream, pc.plan, (const float*)m.emb.ptr, (const float*)h->pe, d, sc, h->y, (float*)h->yb.ptr);
  if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("embed launch: ") + cudaGetErrorString(e));
  return AD_OK;
}

// ---- FP32 sublayers of few tokens (sublayer_f32.cuh) ----
// Whether the sublayers of pass pc run on these kernels: what they cover, up to five waves of CTAs of the attention at capacity.  256 wide, 3 + 3 layers, whole calls, the
// projections' own kernels -> these: batch 24 (2.6 waves) 4834 -> 2977 us, 32 (3.5) 5430 -> 3457; full blocks of 1024 tokens (3.5 waves), four layers 689 -> 633.
bool f32_sublayers(const ad_handle* h, const PassCfg& pc) {
  const ad_model_cfg& c = h->cfg;
  return !h->bf16 && h->pre2 && h->sw.fuse_attn_proj && pc.M_cap <= sub32::MAX_TOKENS && pc.pieces(c.max_batch, sub32::TOK) * c.n_heads <= 5L * num_sms();
}
template <sub32::Kind KIND, int D, int S, bool LOOP>
cudaError_t launch_sublayer_f32_n(cudaStream_t st, dim3 grid, const sub32::Params& p) {
  typedef sub32::Layout<D, S> L;
  constexpr size_t smem = sizeof(float) * (KIND == sub32::FFN ? L::OS : L::FLOATS);
  static bool attr_set[kMaxDevices] = {};
  const int dev = current_device();
  if (!attr_set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(sub32::sublayer_f32_kernel<KIND, D, S, LOOP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  // (one CTA an SM, like the projections around it; with the runtime's choice 256 wide, batch 6 1740 -> 1820 us a call, 128 wide, batch 6 776 -> 825, batch 32 1433 -> 1545)
  return launch_shared(one_cta_share(smem), sub32::sublayer_f32_kernel<KIND, D, S, LOOP>, grid, dim3(sub32::THREADS), smem, st, p);
}
template <sub32::Kind KIND, bool LOOP = false>
int launch_sublayer_f32(ad_handle* h, dim3 grid, int width, const sub32::Params& p, const char* what) {
  note_launch(h, what);
  const bool d128 = h->cfg.d_model == 128, s32 = width == 32;
  const cudaError_t e = d128 ? (s32 ? launch_sublayer_f32_n<KIND, 128, 32, LOOP>(h->stream, grid, p) : launch_sublayer_f32_n<KIND, 128, 64, LOOP>(h->stream, grid, p))
                             : (s32 ? launch_sublayer_f32_n<KIND, 256, 32, LOOP>(h->stream, grid, p) : launch_sublayer_f32_n<KIND, 256, 64, LOOP>(h->stream, grid, p));
  if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("sublayer launch: ") + cudaGetErrorString(e));
  return AD_OK;
}
// Attention with its output projection (partial sums per head in pre2) and, with wq, the query projection of x = yb.
int attention_f32(ad_handle* h, const PassCfg& pc, const void* k, const void* v, const int* key_base, const int* nkeys_tok, const int* nkeys_row,
                  const Mat& wo, const Mat* wq = nullptr, const float* q_bias = nullptr) {
  const int d = h->cfg.d_model, dh = d / h->cfg.n_heads;
  sub32::Params p = {};
  p.a.q = h->qbuf; p.a.k = k; p.a.v = v;
  p.a.seg_off = pc.plan.seg_off; p.a.seg_len = pc.plan.seg_len; p.a.key_base = key_base; p.a.nkeys_tok = nkeys_tok; p.a.nkeys_row = nkeys_row;
  p.a.qchunks = (pc.seg_max + sub32::TOK - 1) / sub32::TOK; p.a.scale = 1.0f / sqrtf((float)dh);
  p.x = (const float*)h->yb.ptr; p.b_in = q_bias; p.w_in = wq ? (const float*)wq->ptr : nullptr;
  p.w_out = (const float*)wo.ptr; p.out = h->pre2; p.stride = (size_t)pc.M_cap * d; p.K2 = d;
  const dim3 grid(h->dims.B * p.a.qchunks, h->cfg.n_heads);
  return wq ? launch_sublayer_f32<sub32::CROSS>(h, grid, dh, p, "q_proj+attention+out_proj") : launch_sublayer_f32<sub32::SELF>(h, grid, dh, p, "attention+out_proj");
}

#define AD_TRY(x) do { int rc__ = (x); if (rc__ != AD_OK) return rc__; } while (0)

// Embedding of a pass's tokens: a kernel of its own, unless the pass's first projection computes it (null: it is done).
int embed_or_defer(ad_handle* h, int pk, const Model& m, const Mat& first, const Model** deferred) {
  const bool fits = pk != PK_ENCODE || h->pass[pk].M_cap <= kFusedEmbed;
  *deferred = h->bf16 && fits && always_few(h->pass[pk], geo_rule(h->pass[pk], EPI_SCATTER, first.N, first.K, false, true)) ? &m : nullptr;
  return *deferred ? AD_OK : embed(h, h->pass[pk], m);
}

// Self-attention sublayer + FFN shared by the encoder and decoder layers.
int self_attention_sublayer(ad_handle* h, int pk, const Mat& wqkv, const float* bqkv, const Mat& wo, const float* bo,
                            const float* lng, const float* lnb, void* kbuf, void* vbuf, const Model* embed_of = nullptr, const Prefetch& next = {}) {
  PassCfg& pc = h->pass[pk];
  GemmParams p = {};
  p.next = next;
  p.bias = bqkv; p.dst[0] = h->qbuf; p.dst[1] = kbuf; p.dst[2] = vbuf; p.seg_width = h->cfg.d_model; p.n_direct = 1;
  p.slot = pc.plan.kv_slot;
  AD_TRY(gemm(h, EPI_SCATTER, wqkv, h->yb, pk, pc.plan.M, pc.M_cap, p, embed_of));
  bool fused = false;
  const int max_keys = pk == PK_VERIFY ? h->dims.max_tgt : pc.seg_max;
  if (attention_is_few(h, pk, max_keys)) {
    AD_TRY(attention_few(h, pc, kbuf, vbuf, pc.plan.key_base, pc.plan.att_n, pc.plan.row_nk, max_keys, wo));
    return layernorm(h, pc, head_partials(h, pc), bo, lng, lnb);
  }
  if (f32_sublayers(h, pc)) {
    AD_TRY(attention_f32(h, pc, kbuf, vbuf, pc.plan.key_base, pc.plan.att_n, pc.plan.row_nk, wo));
    return layernorm(h, pc, head_partials(h, pc), bo, lng, lnb);
  }
  AD_TRY(attention(h, pc, h->qbuf, kbuf, vbuf, h->abuf.ptr, pc.plan.key_base, pc.plan.att_n, pc.plan.row_nk, max_keys, nullptr, nullptr, &wo, &fused));
  if (fused) return layernorm(h, pc, head_partials(h, pc), bo, lng, lnb);
  Partials ps;
  AD_TRY(gemm_to_partials(h, wo, h->abuf, pk, &ps));
  return layernorm(h, pc, ps, bo, lng, lnb);
}

int ffn_sublayer(ad_handle* h, int pk, const Mat& w1, const float* b1, const Mat& w2, const float* b2, const float* lng,
                 const float* lnb, const ActBuf* out = nullptr, const Prefetch& next = {}) {
  PassCfg& pc = h->pass[pk];
  const int d = h->cfg.d_model, F = h->cfg.d_ffn;
  // Passes of few tokens, up to 512 wide: both projections in one kernel (wider models would bring 48 partial sums and more).  Whole
  // calls, two kernels -> this: 512 wide, batch 1 1201 -> 1168 us, batch 16 token by token 4880 -> 4742, batch 3, relaxed, 75 tokens 1597 -> 1535, batch 2 with
  // drafter 2689 -> 2605; encoder calls of four layers, 1 x 64 tokens 92 -> 85, 2 x 50 112 -> 100, 4 x 32 117 -> 103, 1 x 140 112 -> 109, 1 x 200 118 -> 122; 256 wide (16
  // partial sums) 2 x 60 100 -> 80, 4 x 60 104 -> 92.
  if (h->bf16 && few::ffn_few_fits(d, F, pc.M_cap)) {
    const few::FfnFewParams p = {pc.plan.M, (const bf16*)h->yb.ptr, (const bf16*)w1.ptr, (const bf16*)w2.ptr, b1, h->pre, (size_t)pc.M_cap * d, d, F};
    Partials ps = {};
    ps.ptr = h->pre; ps.nsplit = F / few::FFN_SLICE; ps.stride = p.stride;
    const int slices = F / few::FFN_SLICE, groups = std::min((pc.M_cap + few::AQ - 1) / few::AQ, std::max(1, num_sms() / slices));
    note_launch(h, "ffn");
    AD_CUDA(h, launch_k(few::ffn_few_kernel, dim3(groups, slices), dim3(d / 2), 0, h->stream, p));
    return layernorm(h, pc, ps, b2, lng, lnb, out);
  }
  if (f32_sublayers(h, pc) && f32_ffn_slice(F) > 0) {
    const int slice = f32_ffn_slice(F);
    sub32::Params p = {};
    p.a.M_ptr = pc.plan.M;
    p.x = (const float*)h->yb.ptr; p.w_in = (const float*)w1.ptr; p.b_in = b1; p.w_out = (const float*)w2.ptr;
    p.out = h->pre; p.stride = (size_t)pc.M_cap * d; p.K2 = F;
    // One wave of CTAs, which keep their weights from tile to tile.  With a CTA per tile, one an SM, every wave read them again: passes of 1024 tokens (four layers), the
    // projections' own kernels -> a CTA per tile -> this: 256 wide, feed-forward width 1024 662 -> 670 -> 579 us, 2048 914 -> 979 -> 777, 128 wide, 2048 570 -> 623 -> 459; of 256
    // 400 -> 302 -> 285, 508 -> 379 -> 330, 308 -> 272 -> 229.  Two waves: 597, 790, 470; 303, 349, 243.
    const int slices = F / slice, tiles = (pc.M_cap + sub32::TOK - 1) / sub32::TOK, groups = std::max(1, num_sms() / slices);
    if (tiles <= groups) AD_TRY(launch_sublayer_f32<sub32::FFN>(h, dim3(tiles, slices), slice, p, "ffn"));
    else AD_TRY((launch_sublayer_f32<sub32::FFN, true>(h, dim3(groups, slices), slice, p, "ffn")));
    Partials ps = {};
    ps.ptr = h->pre; ps.nsplit = slices; ps.stride = p.stride;
    return layernorm(h, pc, ps, b2, lng, lnb, out);
  }
  GemmParams a = {};
  a.next = next;
  a.bias = b1; a.relu = 1; a.out_act = h->hbuf.ptr;
  AD_TRY(gemm(h, EPI_ACT, w1, h->yb, pk, pc.plan.M, pc.M_cap, a));
  Partials ps;
  AD_TRY(gemm_to_partials(h, w2, h->hbuf, pk, &ps));
  return layernorm(h, pc, ps, b2, lng, lnb, out);
}


// ---- persistent decoder pass ---------------------------------------------------------------------------------

// Cluster size for the K split of the projections: the K blocks of d_model and of d_ffn must divide evenly.
int mega_cluster_size(const ad_model_cfg& c) {
  for (int cs : {8, 4}) {
    const int kd = c.d_model / 64, kf = c.d_ffn / 64;
    if (kd % cs == 0 && kf % cs == 0) return cs;
  }
  return 0;
}

// Fills the device tables and the fixed kernel arguments of the persistent decoder pass; leaves mega[pk].on false for
// pass kinds (or models, or devices) it does not apply to.  Runs once, from ad_create.
int mega_setup(ad_handle* h) {
  const ad_model_cfg& c = h->cfg;
  if (!h->sw.mega || !h->bf16 || c.d_model / c.n_heads != 64 || c.d_model % 128 || c.d_ffn % 128) return AD_OK;
  if (mega::ST_PER_LAYER * c.n_dec + 1 > mega::SYNC_COUNTERS) return AD_OK;
  const int cs = mega_cluster_size(c);
  if (!cs) return AD_OK;
  // shared memory: alignment slack + weight ring + work area (see the kernel), sized for the larger of the two passes
  int max_optin = 0, dev = current_device();
  cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  int cap = 0;
  for (int pk : {PK_VERIFY, PK_DRAFT})
    if (h->pass[pk].M_cap <= mega::NT_MAX && (pk == PK_VERIFY || c.has_drafter)) cap = std::max(cap, h->pass[pk].M_cap);
  if (cap == 0) return AD_OK;
  const int ntcap = (cap + 15) / 16 * 16;
  const int b_bytes = (std::max(c.d_model, c.d_ffn) / 64 / cs) * ntcap * 128;
  const int red_bytes = ntcap * mega::RED_LD * 4;
  const int work = std::max(std::max(b_bytes + 2 * red_bytes, (c.d_model / 64) * ntcap * 128), mega::ATT_SMEM);
  int ring = (max_optin - 1024 - work - 13 * 1024) / mega::TILE_A;     // 13 KB: the kernel's static control block
  if (ring > mega::MAX_RING) ring = mega::MAX_RING;
  if (ring < 4) return AD_OK;
  const size_t smem = 1024 + (size_t)ring * mega::TILE_A + (size_t)work;
  if (cudaFuncSetAttribute(mega::decoder_pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
    cudaGetLastError();
    return AD_OK;
  }
  // how many clusters the device holds at once
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs * 64); cfg.blockDim = dim3(mega::THREADS); cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  int n_clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&n_clusters, mega::decoder_pass_kernel, &cfg) != cudaSuccess || n_clusters < 2) {
    cudaGetLastError();
    return AD_OK;
  }
  h->mega_cs = cs; h->mega_nc = n_clusters; h->mega_smem = smem;

  const int d = c.d_model, L = c.n_dec;
  const size_t self_layer = (size_t)c.max_tgt * c.max_batch * d * h->esz;
  const size_t cross_layer = (size_t)c.max_src * c.max_batch * d * h->esz;
  for (int which = 0; which < 2; ++which) {          // 0: verification pass (verifier), 1: drafter pass (drafter)
    Model& m = which == 0 ? h->ar : h->nar;
    if (!m.present) continue;
    const int pk = which == 0 ? PK_VERIFY : PK_DRAFT;
    if (h->pass[pk].M_cap > mega::NT_MAX) continue;
    std::vector<CUtensorMap> maps((size_t)6 * L + 1);
    std::vector<mega::LayerPtrs> lp((size_t)L);
    for (int l = 0; l < L; ++l) {
      DecLayer& D = m.dec[l];
      const Mat* mats[6] = {&D.wqkv, &D.wo, &D.cq, &D.co, &D.w1, &D.w2};
      for (int i = 0; i < 6; ++i) maps[(size_t)6 * l + i] = mats[i]->map;
      mega::LayerPtrs& P = lp[l];
      P.bqkv = D.bqkv; P.bo = D.bo; P.ln1g = D.ln1g; P.ln1b = D.ln1b; P.cbq = D.cbq; P.cbo = D.cbo; P.ln2g = D.ln2g; P.ln2b = D.ln2b;
      P.b1 = D.b1; P.b2 = D.b2; P.ln3g = D.ln3g; P.ln3b = D.ln3b;
      P.kself = (bf16*)(which == 0 ? (char*)h->kself + l * self_layer : (char*)h->ktmp);
      P.vself = (bf16*)(which == 0 ? (char*)h->vself + l * self_layer : (char*)h->vtmp);
      P.kenc = (const bf16*)((char*)m.kenc + l * cross_layer);
      P.venc = (const bf16*)((char*)m.venc + l * cross_layer);
    }
    maps[(size_t)6 * L] = m.emb.map;
    AD_CUDA(h, cudaMemcpyAsync(h->mega_maps[which], maps.data(), sizeof(CUtensorMap) * maps.size(), cudaMemcpyHostToDevice, h->stream));
    AD_CUDA(h, cudaMemcpyAsync(h->mega_layers[which], lp.data(), sizeof(mega::LayerPtrs) * lp.size(), cudaMemcpyHostToDevice, h->stream));
    AD_CUDA(h, cudaStreamSynchronize(h->stream));     // the host vectors go out of scope
    mega::Params& p = h->mega[pk].p;
    p = mega::Params{};
    p.d = d; p.H = c.n_heads; p.F = c.d_ffn; p.V = c.vocab; p.L = L;
    p.qchunks = (h->pass[pk].seg_max + 7) / 8;
    p.maps = h->mega_maps[which]; p.layers = h->mega_layers[which];
    p.plan = h->pass[pk].plan;
    p.cross_base = h->st.cross_base; p.srclen = h->st.srclen;
    p.emb = (const bf16*)m.emb.ptr; p.pe = h->pe;
    p.emb_scale = sqrtf((float)d); p.eps = c.ln_eps; p.att_scale = 1.0f / sqrtf(64.f);
    p.x[0] = h->y; p.x[1] = h->pre;
    p.stats[0] = h->mega_stats[0]; p.stats[1] = h->mega_stats[1];
    p.M_cap = h->pass[pk].M_cap;
    p.q = (bf16*)h->qbuf; p.attn = (bf16*)h->abuf.ptr; p.hid = (bf16*)h->hbuf.ptr;
    p.yb_out = (bf16*)(which == 0 ? h->yb.ptr : h->xg.ptr);
    p.vocab_M = which == 0 ? nullptr : h->pass[PK_VERIFY].plan.M;
    p.vocab_rows = which == 0 ? nullptr : h->st.gidx;
    p.part_val = h->part_val; p.part_idx = h->part_idx; p.n_vtiles = h->n_vtiles;
    p.sync_ctr = h->st.sync_ctr; p.status = h->st.status;
    p.ring = ring; p.b_bytes = b_bytes; p.red_bytes = red_bytes;
    p.timeline = nullptr;
    h->mega[pk].on = true;
  }
  return AD_OK;
}

bool mega_applies(const ad_handle* h, int pk) {
  return h->mega[pk].on && !(pk == PK_VERIFY && h->beta >= 1);
}

// One launch: decoder stack of pass pk and the projection's per-tile arg-max partials.
int mega_launch(ad_handle* h, int pk) {
  mega::Params p = h->mega[pk].p;
  p.B = h->dims.B;
  static const bool trace = [] { const char* e = getenv("AD_MEGA_TIMELINE"); return e && e[0] == '1'; }();
  p.timeline = trace ? h->mega_timeline : nullptr;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(h->mega_cs * h->mega_nc); cfg.blockDim = dim3(mega::THREADS);
  cfg.dynamicSmemBytes = h->mega_smem; cfg.stream = h->stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = h->mega_cs; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = use_pdl() ? 2 : 1;
  note_launch(h, "persistent_decoder_pass");
  cudaError_t e = cudaLaunchKernelEx(&cfg, mega::decoder_pass_kernel, p);
  if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("persistent decoder pass launch: ") + cudaGetErrorString(e));
  return AD_OK;
}

// Decoder stack over the packed tokens of pass pk (verification: cached, block-causal; drafter: no cache,
// unmasked).  Leaves the final hidden states in yb.
int decoder_pass(ad_handle* h, int pk, Model& m) {
  const ad_model_cfg& c = h->cfg;
  PassCfg& pc = h->pass[pk];
  const size_t self_layer = (size_t)h->dims.max_tgt * c.max_batch * c.d_model * h->esz;
  const size_t cross_layer = (size_t)c.max_src * c.max_batch * c.d_model * h->esz;
  const Model* defer = nullptr;
  AD_TRY(embed_or_defer(h, pk, m, m.dec[0].wqkv, &defer));
  for (int l = 0; l < c.n_dec; ++l) {
    DecLayer& L = m.dec[l];
    void* kb = pk == PK_VERIFY ? (char*)h->kself + l * self_layer : h->ktmp;
    void* vb = pk == PK_VERIFY ? (char*)h->vself + l * self_layer : h->vtmp;
    AD_TRY(self_attention_sublayer(h, pk, L.wqkv, L.bqkv, L.wo, L.bo, L.ln1g, L.ln1b, kb, vb, l == 0 ? defer : nullptr, ffn_weights(h, m, l)));
    const Prefetch next = attention_weights(h, m, l + 1);
    // Query projection of the cross-attention.  With few tokens a full-K walk per CTA is the slow part of the
    // projection, so it is split along K and the attention kernel adds the partial sums (and the bias) as it
    // loads its queries.
    bool fused_x = false;
    if (attention_is_few(h, pk, c.max_src)) {
      AD_TRY(attention_few(h, pc, (char*)m.kenc + l * cross_layer, (char*)m.venc + l * cross_layer, h->st.cross_base, nullptr, h->st.srclen, c.max_src,
                           L.co, &L.cq, L.cbq));
      AD_TRY(layernorm(h, pc, head_partials(h, pc), L.cbo, L.ln2g, L.ln2b));
      AD_TRY(ffn_sublayer(h, pk, L.w1, L.b1, L.w2, L.b2, L.ln3g, L.ln3b, nullptr, next));
      continue;
    }
    if (f32_sublayers(h, pc)) {
      AD_TRY(attention_f32(h, pc, (char*)m.kenc + l * cross_layer, (char*)m.venc + l * cross_layer, h->st.cross_base, nullptr, h->st.srclen, L.co, &L.cq, L.cbq));
      AD_TRY(layernorm(h, pc, head_partials(h, pc), L.cbo, L.ln2g, L.ln2b));
      AD_TRY(ffn_sublayer(h, pk, L.w1, L.b1, L.w2, L.b2, L.ln3g, L.ln3b, nullptr, next));
      continue;
    }
    if (h->bf16 && pc.M_cap <= 256) {
      Partials qp;
      AD_TRY(gemm_to_partials(h, L.cq, h->yb, pk, &qp));
      AD_TRY(attention(h, pc, nullptr, (char*)m.kenc + l * cross_layer, (char*)m.venc + l * cross_layer, h->abuf.ptr,
                       h->st.cross_base, nullptr, h->st.srclen, c.max_src, L.cbq, &qp, &L.co, &fused_x, true));
    } else {
      GemmParams q = {};
      q.bias = L.cbq; q.out_act = h->qbuf;
      AD_TRY(gemm(h, EPI_ACT, L.cq, h->yb, pk, pc.plan.M, pc.M_cap, q));
      AD_TRY(attention(h, pc, h->qbuf, (char*)m.kenc + l * cross_layer, (char*)m.venc + l * cross_layer, h->abuf.ptr,
                       h->st.cross_base, nullptr, h->st.srclen, c.max_src, nullptr, nullptr, &L.co, &fused_x, true));
    }
    if (fused_x) {
      AD_TRY(layernorm(h, pc, head_partials(h, pc), L.cbo, L.ln2g, L.ln2b));
    } else {
      Partials ps;
      AD_TRY(gemm_to_partials(h, L.co, h->abuf, pk, &ps));
      AD_TRY(layernorm(h, pc, ps, L.cbo, L.ln2g, L.ln2b));
    }
    AD_TRY(ffn_sublayer(h, pk, L.w1, L.b1, L.w2, L.b2, L.ln3g, L.ln3b, nullptr, next));
  }
  return AD_OK;
}

// Encoder stack + per-decoder-layer cross-attention key/value projection of the memory.
int encoder_pass(ad_handle* h, Model& m, bool keep_memory) {
  const ad_model_cfg& c = h->cfg;
  PassCfg& pc = h->pass[PK_ENCODE];
  const size_t cross_layer = (size_t)c.max_src * c.max_batch * c.d_model * h->esz;
  const Model* defer = nullptr;
  AD_TRY(embed_or_defer(h, PK_ENCODE, m, m.enc[0].wqkv, &defer));
  for (int l = 0; l < c.n_enc; ++l) {
    EncLayer& L = m.enc[l];
    AD_TRY(self_attention_sublayer(h, PK_ENCODE, L.wqkv, L.bqkv, L.wo, L.bo, L.ln1g, L.ln1b, h->ktmp, h->vtmp, l == 0 ? defer : nullptr));
    AD_TRY(ffn_sublayer(h, PK_ENCODE, L.w1, L.b1, L.w2, L.b2, L.ln2g, L.ln2b, keep_memory && l + 1 == c.n_enc ? &h->encmem : nullptr));
  }
  // cross-attention keys and values of every decoder layer in one launch (segments 2l / 2l + 1 = layer l's K / V)
  GemmParams p = {};
  p.bias = m.cbkv_pack; p.dst[0] = m.kenc; p.dst[1] = m.venc; p.seg_pair_stride = cross_layer;
  p.seg_width = c.d_model; p.n_direct = 0; p.slot = h->st.enc_slot;
  AD_TRY(gemm(h, EPI_SCATTER, m.ckv_all, keep_memory ? h->encmem : h->yb, PK_ENCODE, pc.plan.M, pc.M_cap, p));
  return AD_OK;
}

// Exchanges the handle's activation buffers and stream with the side set (and back, when called again).
void swap_side(ad_handle* h) {
  ActSet& sd = h->side;
  std::swap(h->y, sd.y); std::swap(h->pre, sd.pre); std::swap(h->pre2, sd.pre2);
  std::swap(h->yb, sd.yb); std::swap(h->abuf, sd.abuf); std::swap(h->hbuf, sd.hbuf);
  std::swap(h->qbuf, sd.qbuf); std::swap(h->ktmp, sd.ktmp); std::swap(h->vtmp, sd.vtmp);
  std::swap(h->stream, h->side_stream);
}

// Most rows, up to `most`, whose accept kernels this device places as one cluster (0: none).  A CTA takes an SM's registers, so a cluster needs
// that many SMs of one GPC, which a partitioned GPU may not have; beyond eight the device has to allow it too.
int accept_cluster_rows(int most) {
  auto* kernel = argmax_accept_kernel<ACC_CLUSTERED>;
  if (most > 8 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    most = 8;
  }
  for (; most > 1; --most) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(most); cfg.blockDim = dim3(ACC_THREADS);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = most; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0) return most;
    cudaGetLastError();
  }
  return 0;
}

// Output projection fused with arg-max over X (yb for the verifier, the gathered mask rows for the drafter),
// then the final reduction and (verifier) the draft compare.
int vocab_stage(ad_handle* h, Model& m, const ActBuf& X, int to_drafts, int auto_commit, bool partials_ready = false) {
  PassCfg& pc = h->pass[PK_VERIFY];
  GemmParams p = {};
  p.part_val = h->part_val; p.part_idx = h->part_idx;
  const bool relaxed = !to_drafts && h->beta >= 1;
  if (relaxed) {     // relaxed verification: the drafts' own scores first, then the projection counts against them
    const int d = h->cfg.d_model;
    note_launch(h, "draft_score");
    const dim3 sgrid((pc.M_cap + 7) / 8);
    if (h->bf16) AD_CUDA(h, launch_k(draft_score_kernel<bf16, bf16>, sgrid, dim3(256), 0, h->stream, h->st, pc.plan, h->dims, (const bf16*)m.emb.ptr, (const bf16*)X.ptr, d, h->draft_val, h->draft_id));
    else AD_CUDA(h, launch_k(draft_score_kernel<float, float>, sgrid, dim3(256), 0, h->stream, h->st, pc.plan, h->dims, (const float*)m.emb.ptr, (const float*)X.ptr, d, h->draft_val, h->draft_id));
    p.draft_val = h->draft_val; p.draft_id = h->draft_id; p.part_cnt = h->part_cnt;
  }
  if (!partials_ready) AD_TRY(gemm(h, EPI_ARGMAX, m.emb, X, PK_VERIFY, pc.plan.M, pc.M_cap, p));
  note_launch(h, "argmax_accept");
  const int B = h->dims.B;
  const bool cluster = auto_commit && !to_drafts && B > 1 && B <= h->accept_rows;
  NextPass next = h->next_pass;
  next.launches = h->launches - h->body_launches;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(B); cfg.blockDim = dim3(ACC_THREADS); cfg.stream = h->stream;
  cudaLaunchAttribute attr[2];
  int n_attr = 0;
  if (use_pdl()) {
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster) {
    attr[n_attr].id = cudaLaunchAttributeClusterDimension;
    attr[n_attr].val.clusterDim.x = B; attr[n_attr].val.clusterDim.y = 1; attr[n_attr++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr; cfg.numAttrs = n_attr;
  auto* kernel = cluster ? argmax_accept_kernel<ACC_CLUSTERED> : B == 1 ? argmax_accept_kernel<ACC_ONE> : argmax_accept_kernel<ACC_ROWS>;
  AD_CUDA(h, cudaLaunchKernelEx(&cfg, kernel, h->st, pc.plan, h->dims, (const float*)h->part_val,
                                (const int*)h->part_idx, h->n_vtiles, to_drafts, auto_commit, (unsigned int*)(h->st.loop_it + 1),
                                auto_commit ? h->cond_handle : 0ull, relaxed ? 1 : 0, (const float*)h->draft_val, (const int*)h->draft_id,
                                (const int*)h->part_cnt, next));
  h->last_vocab_which = to_drafts ? 1 : 0;
  return AD_OK;
}

// user_drafts / user_k: where SRC_USER finds the caller's block (device, or mapped host memory); null: the workspace copies.
int prepare_verify(ad_handle* h, int source, const int* ovr, int* user_drafts = nullptr, int* user_k = nullptr) {
  DevState st = h->st;
  if (user_drafts) { st.user_drafts = user_drafts; st.user_k = user_k; }
  note_launch(h, "prepare_verify");
  AD_CUDA(h, launch_k(prepare_verify_kernel, dim3(1), dim3(256), 0, h->stream, st, h->pass[PK_VERIFY].plan, h->dims, source, ovr,
                      h->cfg.max_tgt, h->pick));
  return AD_OK;
}

// Whether the accept kernels of a decode loop plan the passes behind them (kernel-chain form of the passes only).
bool loop_plans_ahead(const ad_handle* h) { return h->sw.fuse_plan && !h->mega[PK_VERIFY].on && !h->mega[PK_DRAFT].on; }
// The body of a decode loop comes in up to three forms, each laid out for a verification pass of at most cap[i] tokens; an iteration takes the first
// one that holds the tokens planned for it (the choice is a graph node and costs 3.5 us).  A batch begins with hundreds of tokens and ends with a handful, for which
// the kernels and grids that a large capacity asks for are the wrong ones: 512 wide, batch 32, blocks of 64, an iteration of 9 to 128 tokens took 220 to 320 us,
// of a handle made for so few 130 to 180.  First the few-token kernels, up to 64 tokens (96 beyond 512 wide, see geometry); then, where the whole capacity is too
// much for the few-query attention, as many tokens as it takes; then all.  Calls of the input-guided policy, whose blocks are mostly short, keep the
// few-token kernels as their only form up to 128 tokens, others up to 96.  Whole calls, one form -> several: 512 wide, batch 32 4840 -> 4437 us, batch 20 5740 -> 5104,
// batch 12 2678 -> 2590, batch 8 3112 -> 3046, batch 5 with drafter 4440 -> 4300; 768 wide, batch 6 4209 -> 4005, batch 16 4814 -> 4461; 1024 wide, batch 8 5465 -> 5071, with
// drafter 10890 -> 9975.
struct LoopBodies { int n, cap[NextPass::BODIES]; };
// While one lives, pass pk is laid out for at most `cap` tokens (few_cap: see PassCfg).
struct PassLayout {
  ad_handle* h;
  int pk;
  PassCfg kept;
  PassLayout(ad_handle* h, int pk, int cap, int few_cap) : h(h), pk(pk), kept(h->pass[pk]) {
    PassCfg& pc = h->pass[pk];
    pc.M_cap = std::min(pc.M_cap, cap);
    pc.ntile = clampi(pow2ceil(pc.M_cap), 16, 256);
    pc.few_cap = few_cap;
  }
  ~PassLayout() { h->pass[pk] = kept; }
};
PassLayout body_layout(ad_handle* h, const LoopBodies& b, int i) {
  return PassLayout(h, PK_VERIFY, b.cap[i], b.n > 1 && i > 0 ? 0 : kFewTokens);
}
LoopBodies loop_bodies(ad_handle* h, bool policy) {
  const PassCfg& pc = h->pass[PK_VERIFY];
  const int d = h->cfg.d_model, full = pc.M_cap;
  LoopBodies b = {1, {full, 0, 0}};
  const int few = d <= 512 ? 64 : 96;
  if (!h->bf16 || !h->sw.few_body || !loop_plans_ahead(h) || few::split_for(3 * d, d, false, 1) == 0) return b;
  if (full <= (policy ? kFewTokens : 96)) return b;
  b.n = 0;
  b.cap[b.n++] = few;
  auto takes_few = [&](int cap) {
    const PassLayout at(h, PK_VERIFY, cap, 0);
    return attention_is_few(h, PK_VERIFY, h->cfg.max_src);
  };
  if (!takes_few(full)) {
    int cap = few;
    while (cap + 16 < full && takes_few(cap + 16)) cap += 16;
    if (cap > few) b.cap[b.n++] = cap;
  }
  b.cap[b.n++] = full;
  return b;
}

// Draft substep: sizes and drafter plan ...
int plan_draft(ad_handle* h) {
  AD_TRY(prepare_verify(h, SRC_SIZES, nullptr));
  note_launch(h, "plan_draft");
  AD_CUDA(h, launch_k(plan_draft_kernel, dim3(1), dim3(256), 0, h->stream, h->st, h->pass[PK_VERIFY].plan, h->pass[PK_DRAFT].plan, h->dims));
  return AD_OK;
}
// ... then the drafter's decoder, gather of the mask rows, projection + arg-max.
int draft_stage(ad_handle* h) {
  if (mega_applies(h, PK_DRAFT)) {      // decoder stack, gather of the mask rows and projection in one kernel
    AD_TRY(mega_launch(h, PK_DRAFT));
    return vocab_stage(h, h->nar, h->xg, 1, 0, true);
  }
  AD_TRY(decoder_pass(h, PK_DRAFT, h->nar));
  const int d = h->cfg.d_model;
  PassCfg& pv = h->pass[PK_VERIFY];
  note_launch(h, "gather_rows");
  if (h->bf16) AD_CUDA(h, launch_k(gather_rows_kernel<bf16>, dim3(pv.M_cap), dim3(128), 0, h->stream, (const int*)pv.plan.M, (const int*)h->st.gidx, (const bf16*)h->yb.ptr, (bf16*)h->xg.ptr, d));
  else AD_CUDA(h, launch_k(gather_rows_kernel<float>, dim3(pv.M_cap), dim3(128), 0, h->stream, (const int*)pv.plan.M, (const int*)h->st.gidx, (const float*)h->yb.ptr, (float*)h->xg.ptr, d));
  return vocab_stage(h, h->nar, h->xg, 1, 0);
}

int verify_stage(ad_handle* h, int auto_commit) {
  if (mega_applies(h, PK_VERIFY)) {
    AD_TRY(mega_launch(h, PK_VERIFY));
    return vocab_stage(h, h->ar, h->yb, 0, auto_commit, true);
  }
  AD_TRY(decoder_pass(h, PK_VERIFY, h->ar));
  return vocab_stage(h, h->ar, h->yb, 0, auto_commit);
}

int commit_stage(ad_handle* h, const int* n_dev, int* status_out) {
  note_launch(h, "commit_stage");
  AD_CUDA(h, launch_k(commit_kernel, dim3(1), dim3(256), 0, h->stream, h->st, h->pass[PK_VERIFY].plan, h->dims, n_dev, status_out));
  return AD_OK;
}

bool loop_drafts(const ad_gen_opts& o) { return o.mode == AD_MODE_GAD && o.run_drafter; }
int block_source(const ad_gen_opts& o, const int* ovr) { return o.mode == AD_MODE_GAD || ovr ? SRC_OVERRIDE : SRC_POLICY; }

NextPass next_pass(const ad_handle* h, int source, const int* ovr) {
  NextPass n = no_next_pass();
  n.source = source; n.override_stream = ovr; n.override_stride = h->cfg.max_tgt;
  n.draft = h->pass[PK_DRAFT].plan;
  if (source != SRC_KEEP) n.pick = h->pick;
  return n;
}

// First pass of a loop that plans ahead: planned by kernels of their own.
int plan_first_pass(ad_handle* h, const ad_gen_opts& o, const int* ovr) {
  if (loop_drafts(o)) return plan_draft(h);
  return prepare_verify(h, block_source(o, ovr), ovr);
}

// One iteration of the decode loop: draft -> verify -> commit, all on the device.
int loop_iteration(ad_handle* h, const ad_gen_opts& o, const int* ovr) {
  struct Scope {               // whatever way this function is left
    ad_handle* h;
    ~Scope() {
      h->next_pass = no_next_pass();
    }
  } scope{h};
  if (!loop_plans_ahead(h)) {
    if (loop_drafts(o)) {
      AD_TRY(plan_draft(h));
      AD_TRY(draft_stage(h));
      AD_TRY(prepare_verify(h, SRC_KEEP, ovr));
    } else {
      AD_TRY(prepare_verify(h, block_source(o, ovr), ovr));
    }
    return verify_stage(h, 1);   // accept and commit in one kernel
  }
  // this iteration's first pass has been planned already (plan_first_pass, or the previous iteration's accept kernel)
  if (loop_drafts(o)) {
    h->next_pass = next_pass(h, SRC_KEEP, ovr);
    AD_TRY(draft_stage(h));
    h->next_pass = next_pass(h, SRC_SIZES, nullptr);
  } else {
    h->next_pass = next_pass(h, block_source(o, ovr), ovr);
  }
  return verify_stage(h, 1);
}

// Waits for the stream; `status`: the mapped word a kernel before has exported the latched device error to.
int wait_status(ad_handle* h, volatile int* status) {
  AD_CUDA(h, cudaStreamSynchronize(h->stream));
  const int s = *status;
  if (s != 0) return fail(h, s, s == AD_ERR_TIMEOUT ? "a bounded device-side wait ran out" : "device-side argument check failed");
  return AD_OK;
}
int read_status(ad_handle* h) {
  AD_CUDA(h, launch_k(export_status_kernel, dim3(1), dim3(32), 0, h->stream, h->st, h->dev_view(h->host_flag + 2)));
  return wait_status(h, h->host_flag + 2);
}

// Whether the caller is recording the handle's stream.
bool being_captured(const ad_handle* h) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (h->stream != nullptr) cudaStreamIsCapturing(h->stream, &cap);
  return cap != cudaStreamCaptureStatusNone;
}

// Block-level calls: the words that kernels and captured graphs read, set in stream order (calls with device arrays do not wait for
// one another) where they are not what the last call left.
int set_words(ad_handle* h, bool captured, int k_cap, int beta, float tau) {
  int4 w = h->words;
  w.x = k_cap; w.z = beta;
  memcpy(&w.w, &tau, sizeof(tau));
  if (captured) h->foreign_graphs = true;
  if (!h->foreign_graphs && !memcmp(&w, &h->words, sizeof(w))) return AD_OK;
  note_launch(h, "set_words");
  AD_CUDA(h, launch_k(set_words_kernel, dim3(1), dim3(1), 0, h->stream, h->st, w));
  h->words = w;
  return AD_OK;
}

// The handle's entry for `key`, made if there is none.  Forms that a program can make by calling (batch sizes above all) must not
// pile up: beyond four per row of capacity and a few, the one that has not been used for longest goes, once nothing of it runs.
int graph_entry(ad_handle* h, const char* key, ad_handle::GraphEntry** out) {
  auto it = h->graphs.find(key);
  if (it == h->graphs.end()) {
    while (h->graphs.size() >= (size_t)4 * h->cfg.max_batch + 16) {
      auto oldest = std::min_element(h->graphs.begin(), h->graphs.end(), [](const auto& a, const auto& b) { return a.second.last_use < b.second.last_use; });
      if (oldest->second.exec) {
        AD_CUDA(h, cudaStreamSynchronize(h->stream));
        cudaGraphExecDestroy(oldest->second.exec);
      }
      h->graphs.erase(oldest);
    }
    it = h->graphs.emplace(key, ad_handle::GraphEntry{}).first;
  }
  it->second.last_use = ++h->graph_uses;
  *out = &it->second;
  return AD_OK;
}

// Runs `enqueue` (launches on the handle's stream whose arguments depend only on `key`): the first call with this key directly, so that
// a form that is called once does not pay for a capture, later ones as a graph captured by the second.  Directly as well where the
// stream cannot be captured (captured: the caller is recording it) or every launch is being timed.
template <typename F>
int run_captured(ad_handle* h, bool captured, const char* key, F enqueue) {
  if (h->stream == nullptr || captured || !h->sw.graph_calls || h->profiling) return enqueue();
  ad_handle::GraphEntry* entry = nullptr;
  AD_TRY(graph_entry(h, key, &entry));
  if (!entry->exec) {
    if (!entry->launches) {
      const int before = h->launches;
      AD_TRY(enqueue());
      entry->launches = h->launches - before;
      return AD_OK;
    }
    cudaGraph_t g = nullptr;
    const int before = h->launches;
    AD_CUDA(h, cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
    const int rc = enqueue();
    const cudaError_t e = cudaStreamEndCapture(h->stream, &g);
    const int n = h->launches - before;
    h->launches = before;
    if (rc != AD_OK) { if (g) cudaGraphDestroy(g); return rc; }
    if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("graph capture: ") + cudaGetErrorString(e));
    cudaGraphExec_t exec = nullptr;
    const cudaError_t e2 = cudaGraphInstantiate(&exec, g, 0);
    cudaGraphDestroy(g);
    if (e2 != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(e2));
    entry->exec = exec;
    entry->launches = n;
  }
  AD_CUDA(h, cudaGraphLaunch(entry->exec, h->stream));
  h->launches += entry->launches;
  return AD_OK;
}


void drop_graphs(ad_handle* h) {
  for (auto& kv : h->graphs)
    if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
  h->graphs.clear();
}

}  // namespace

// =====================================================================================================
// extern "C"
// =====================================================================================================

extern "C" int ad_weight_counts(const ad_model_cfg* cfg, size_t* matrix_elems, size_t* vector_elems) {
  std::string why;
  if (check_cfg(cfg, &why) != AD_OK || !matrix_elems || !vector_elems) return fail(nullptr, AD_ERR_ARG, why.empty() ? "null output pointer" : why);
  weight_counts(*cfg, matrix_elems, vector_elems);
  return AD_OK;
}

extern "C" int ad_query_workspace(const ad_model_cfg* cfg, size_t* bytes) {
  std::string why;
  if (check_cfg(cfg, &why) != AD_OK || !bytes) return fail(nullptr, AD_ERR_ARG, why.empty() ? "null output pointer" : why);
  ad_handle tmp;
  tmp.cfg = *cfg;
  tmp.bf16 = cfg->dtype == AD_DTYPE_BF16;
  tmp.esz = tmp.bf16 ? 2 : 4;
  *bytes = layout(&tmp, nullptr);
  return AD_OK;
}

extern "C" const char* ad_last_error(const ad_handle* h) { return h ? h->err.c_str() : g_create_error.c_str(); }

extern "C" int ad_create(const ad_model_cfg* cfg, const ad_weights* w, void* workspace, size_t workspace_bytes,
                         void* stream, ad_handle** out) {
  std::string why;
  if (!out) return fail(nullptr, AD_ERR_ARG, "out is null");
  *out = nullptr;
  if (check_cfg(cfg, &why) != AD_OK) return fail(nullptr, AD_ERR_ARG, why);
  if (!w || !workspace) return fail(nullptr, AD_ERR_ARG, "weights or workspace is null");
  if (reinterpret_cast<uintptr_t>(workspace) % 1024) return fail(nullptr, AD_ERR_ARG, "workspace must be 1024-byte aligned");
  int dev = 0, major = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess)
    return fail(nullptr, AD_ERR_CUDA, "no CUDA device");
  if (major != 10) return fail(nullptr, AD_ERR_CUDA, "this library contains sm_100a code only; the current device is not compute capability 10.x");

  ad_handle* h = new ad_handle();
  h->cfg = *cfg;
  h->stream = static_cast<cudaStream_t>(stream);
  h->sw.devloop = !env_is_1("AD_NO_DEVLOOP");
  h->sw.graph_calls = !env_is_1("AD_NO_ENCODE_GRAPH");
  h->sw.two_stream_encode = !env_is_1("AD_NO_CONCURRENT_ENCODERS");
  h->sw.fuse_attn_proj = !env_is_1("AD_NO_ATTN_PROJ");
  h->sw.fuse_plan = !env_is_1("AD_NO_FUSED_PLAN");
  h->sw.few_body = !env_is_1("AD_NO_FEW_BODY");
  h->sw.mega = env_is_1("AD_MEGA");
  if (const char* e = getenv("AD_ACCEPT_CLUSTER")) h->sw.accept_cluster = clampi(atoi(e), 0, ACC_CLUSTER);
  h->bf16 = cfg->dtype == AD_DTYPE_BF16;
  h->esz = h->bf16 ? 2 : 4;
  const size_t need = layout(h, workspace);
  auto bail = [&](int code, const std::string& msg) { g_create_error = msg; delete h; return code; };
  if (need > workspace_bytes) return bail(AD_ERR_CAPACITY, "workspace too small: need " + std::to_string(need) + " bytes");
  h->dims = Dims{cfg->max_batch, cfg->max_src, cfg->max_tgt, cfg->kmax, cfg->bos, cfg->pad, cfg->eos, cfg->mask, cfg->vocab};
  int rc = bind_model(h, h->ar, w->ar);
  if (rc == AD_OK && cfg->has_drafter) rc = bind_model(h, h->nar, w->nar);
  if (rc != AD_OK) return bail(rc, h->err);
  if (h->bf16) {
    bool ok = true;
    ActBuf* bufs[4] = {&h->yb, &h->abuf, &h->hbuf, &h->xg};
    for (ActBuf* b : bufs)
      for (int k = 0; k < PK_COUNT; ++k)
        for (int i = 0; i < 5 && (16 << i) <= h->pass[k].ntile; ++i)
          ok = ok && make_map(&b->map[k].m[i], b->ptr, h->M_all, b->cols, 16 << i);
    for (int i = 0; i < 5 && (16 << i) <= h->pass[PK_ENCODE].ntile; ++i)
      ok = ok && make_map(&h->encmem.map[PK_ENCODE].m[i], h->encmem.ptr, h->pass[PK_ENCODE].M_cap, h->encmem.cols, 16 << i);
    if (cfg->has_drafter) {
      const int Me = h->pass[PK_ENCODE].M_cap, nt = h->pass[PK_ENCODE].ntile;
      ActBuf* sbufs[3] = {&h->side.yb, &h->side.abuf, &h->side.hbuf};
      for (ActBuf* b : sbufs)
        for (int i = 0; i < 5 && (16 << i) <= nt; ++i)
          ok = ok && make_map(&b->map[PK_ENCODE].m[i], b->ptr, Me, b->cols, 16 << i);
    }
    if (!ok) return bail(AD_ERR_CUDA, "cuTensorMapEncodeTiled failed for an activation buffer");
  }
  if (cfg->has_drafter && h->sw.two_stream_encode) {
    if (cudaStreamCreateWithFlags(&h->side_stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming) != cudaSuccess)
      return bail(AD_ERR_CUDA, "creating the side stream failed");
  }
  h->accept_rows = accept_cluster_rows(std::min(cfg->max_batch, h->sw.accept_cluster));
  // Cache, scratch and state start from zero so that no stale bit pattern is ever read as a number.
  if (cudaMemsetAsync(workspace, 0, need, h->stream) != cudaSuccess) return bail(AD_ERR_CUDA, "clearing the workspace failed");
  // Gather the cross-attention key/value projections of all decoder layers (see Model::ckv_all).
  for (Model* mp : {&h->ar, &h->nar}) {
    if (!mp->present) continue;
    const int d = cfg->d_model;
    const size_t one = h->esz * (size_t)2 * d * d;
    bool okc = true;
    for (int l = 0; l < cfg->n_dec; ++l) {
      okc = okc && cudaMemcpyAsync((char*)mp->ckv_pack + l * one, mp->dec[l].ckv.ptr, one, cudaMemcpyDeviceToDevice, h->stream) == cudaSuccess;
      okc = okc && cudaMemcpyAsync(mp->cbkv_pack + (size_t)l * 2 * d, mp->dec[l].cbkv, sizeof(float) * 2 * d, cudaMemcpyDeviceToDevice, h->stream) == cudaSuccess;
    }
    mp->ckv_all.ptr = mp->ckv_pack; mp->ckv_all.N = cfg->n_dec * 2 * d; mp->ckv_all.K = d;
    if (h->bf16) okc = okc && make_map(&mp->ckv_all.map, mp->ckv_pack, mp->ckv_all.N, d, tc::BLOCK_N_FEAT);
    if (!okc) return bail(AD_ERR_CUDA, "gathering the cross-attention key/value projections failed");
  }
  {
    const int rcm = mega_setup(h);
    if (rcm != AD_OK) return bail(rcm, h->err);
  }
  // Sinusoidal positional table PE(p, 2i) = sin(p / 10000^(2i/d)), PE(p, 2i+1) = cos(.), evaluated in double.
  {
    const int d = cfg->d_model;
    std::vector<float> pe((size_t)h->max_pos * d);
    for (int p = 0; p < h->max_pos; ++p)
      for (int i = 0; i < d; i += 2) {
        const double freq = exp(-log(10000.0) * (double)i / (double)d);
        pe[(size_t)p * d + i] = (float)sin(p * freq);
        if (i + 1 < d) pe[(size_t)p * d + i + 1] = (float)cos(p * freq);
      }
    if (cudaMemcpyAsync(h->pe, pe.data(), pe.size() * sizeof(float), cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
        cudaStreamSynchronize(h->stream) != cudaSuccess)
      return bail(AD_ERR_CUDA, "uploading the positional table failed");
  }
  {
    const size_t B = cfg->max_batch;
    const size_t n_up = B * cfg->max_src + 3 * B + B * cfg->max_tgt + B * cfg->kmax, n_down = 4 + 4 * B + B * cfg->max_tgt;
    if (cudaHostAlloc(&h->host_flag, sizeof(int) * (16 + n_up + n_down), cudaHostAllocMapped) != cudaSuccess ||
        cudaHostGetDevicePointer(&h->host_flag_dev, h->host_flag, 0) != cudaSuccess)
      return bail(AD_ERR_CUDA, "allocating pinned host memory failed");
    h->up_src = h->host_flag + 16; h->up_len = h->up_src + B * cfg->max_src; h->up_max = h->up_len + B;
    h->up_ovr = h->up_max + B; h->up_ids = h->up_ovr + B * cfg->max_tgt; h->up_n = h->up_ids + B * cfg->kmax;
    h->down = h->up_n + B;
    h->down_dev = h->host_flag_dev + (h->down - h->host_flag);
  }
  if (cudaEventCreate(&h->ev0) != cudaSuccess || cudaEventCreate(&h->ev1) != cudaSuccess || cudaEventCreate(&h->ev2) != cudaSuccess)
    return bail(AD_ERR_CUDA, "cudaEventCreate failed");
  *out = h;
  return AD_OK;
}

extern "C" int ad_destroy(ad_handle* h) {
  if (!h) return AD_ERR_ARG;
  cudaStreamSynchronize(h->stream);
  drop_graphs(h);
  if (h->host_flag) cudaFreeHost(h->host_flag);
  if (h->ev0) cudaEventDestroy(h->ev0);
  if (h->ev1) cudaEventDestroy(h->ev1);
  if (h->ev2) cudaEventDestroy(h->ev2);
  if (h->ev_fork) cudaEventDestroy(h->ev_fork);
  if (h->ev_join) cudaEventDestroy(h->ev_join);
  if (h->side_stream) { cudaStreamSynchronize(h->side_stream); cudaStreamDestroy(h->side_stream); }
  delete h;
  return AD_OK;
}

extern "C" int ad_set_acceptance(ad_handle* h, int32_t beta, float tau) {
  if (!h) return AD_ERR_ARG;
  if (beta < 0 || !(tau >= 0.f)) return fail(h, AD_ERR_ARG, "beta must be >= 0 and tau >= 0");
  h->beta = beta;
  h->tau = tau;
  return AD_OK;
}

extern "C" int ad_sync(ad_handle* h) {
  if (!h) return AD_ERR_ARG;
  return read_status(h);
}

namespace {

// What ad_encode and ad_generate import.  maxlen / ovr may be null; limit: iteration limit of the device-side loop (0: none).
int import_inputs(ad_handle* h, const int32_t* src, int32_t src_stride, const int32_t* src_len, int32_t B, const int32_t* maxlen,
                  const int32_t* ovr, int ovr_stride, int ovr_width, int limit, int on_host, int4 words = {}) {
  const ad_model_cfg& c = h->cfg;
  ImportParams p = {src, src_len, maxlen, ovr, src_stride, std::min(src_stride, c.max_src), ovr_stride, ovr_width, limit, words};
  if (on_host) {
    // host-resident inputs go through the handle's pinned staging area, which the device reads in place (every host-array
    // call ends synchronised, so the area is free again)
    for (int b = 0; b < B; ++b) memcpy(h->up_src + (size_t)b * c.max_src, src + (size_t)b * src_stride, sizeof(int) * p.src_width);
    memcpy(h->up_len, src_len, sizeof(int) * B);
    p.src = h->dev_view(h->up_src); p.src_len = h->dev_view(h->up_len); p.src_stride = c.max_src;
    if (maxlen) { memcpy(h->up_max, maxlen, sizeof(int) * B); p.maxlen = h->dev_view(h->up_max); }
    if (ovr) {
      for (int b = 0; b < B; ++b) memcpy(h->up_ovr + (size_t)b * c.max_tgt, ovr + (size_t)b * ovr_stride, sizeof(int) * ovr_width);
      p.ovr = h->dev_view(h->up_ovr); p.ovr_stride = c.max_tgt;
    }
  }
  note_launch(h, "import");
  AD_CUDA(h, launch_k(import_kernel, dim3(B), dim3(128), 0, h->stream, h->st, h->dims, p, h->in_max, h->ovr));
  if (limit > 0) h->words = words;
  return AD_OK;
}

// Plan of the encoder pass (which also resets every row's decoding state), then the encoder pass(es).
int encode_stage(ad_handle* h, bool with_maxlen) {
  const ad_model_cfg& c = h->cfg;
  note_launch(h, "plan_encode");
  AD_CUDA(h, launch_k(plan_encode_kernel, dim3(1), dim3(256), 0, h->stream, h->st, h->pass[PK_ENCODE].plan, h->dims,
                      (const int*)(with_maxlen ? h->in_max : nullptr)));
  if (c.has_drafter && h->side_stream) {
    // the two encoders are independent (Section 3.2: separate models): drafter's on the side stream, verifier's here
    AD_CUDA(h, cudaEventRecord(h->ev_fork, h->stream));
    AD_CUDA(h, cudaStreamWaitEvent(h->side_stream, h->ev_fork, 0));
    swap_side(h);
    const int rc_side = encoder_pass(h, h->nar, false);
    cudaError_t e_join = rc_side == AD_OK ? cudaEventRecord(h->ev_join, h->stream) : cudaSuccess;
    swap_side(h);
    if (rc_side != AD_OK) return rc_side;
    AD_CUDA(h, e_join);
    AD_TRY(encoder_pass(h, h->ar, true));
    AD_CUDA(h, cudaStreamWaitEvent(h->stream, h->ev_join, 0));
    return AD_OK;
  }
  AD_TRY(encoder_pass(h, h->ar, true));
  if (c.has_drafter) AD_TRY(encoder_pass(h, h->nar, false));
  return AD_OK;
}

int check_sources(ad_handle* h, const int32_t* src, int32_t src_stride, const int32_t* src_len, int32_t B, int32_t on_host) {
  const ad_model_cfg& c = h->cfg;
  if (!src || !src_len) return fail(h, AD_ERR_ARG, "src or src_len is null");
  if (B < 1 || B > c.max_batch) return fail(h, AD_ERR_CAPACITY, "B outside 1..max_batch");
  if (src_stride < 1) return fail(h, AD_ERR_ARG, "src_stride must be positive");
  if (on_host)
    for (int b = 0; b < B; ++b)
      if (src_len[b] < 1 || src_len[b] > c.max_src || src_len[b] > src_stride)
        return fail(h, src_len[b] > c.max_src ? AD_ERR_CAPACITY : AD_ERR_ARG, "src_len outside 1..min(max_src, src_stride)");
  return AD_OK;
}

}  // namespace

extern "C" int ad_encode(ad_handle* h, const int32_t* src, int32_t src_stride, const int32_t* src_len, int32_t B,
                         int32_t on_host) {
  if (!h) return AD_ERR_ARG;
  AD_TRY(check_sources(h, src, src_stride, src_len, B, on_host));
  // (captured graphs are keyed by the batch size, so a different B simply uses other entries)
  h->B = B;
  h->dims.B = B;
  h->encoded = false;
  AD_TRY(import_inputs(h, src, src_stride, src_len, B, nullptr, nullptr, 0, 0, 0, on_host));
  // The encoder pass reads its inputs from fixed workspace buffers, so on a capturable stream it is one graph
  // per batch size (about fifty launches otherwise paid on the host for every sentence).
  char key[48];
  snprintf(key, sizeof(key), "encode B%d h%d", B, on_host ? 1 : 0);
  AD_TRY(run_captured(h, being_captured(h), key, [&]() -> int {
    AD_TRY(encode_stage(h, false));
    if (on_host) AD_CUDA(h, launch_k(export_status_kernel, dim3(1), dim3(32), 0, h->stream, h->st, h->dev_view(h->host_flag + 2)));
    return AD_OK;
  }));
  h->encoded = true;
  h->last_vocab_which = -1;
  return on_host ? wait_status(h, h->host_flag + 2) : AD_OK;
}

extern "C" int ad_verify_block(ad_handle* h, const int32_t* drafts, const int32_t* k, int32_t* argmax,
                               int32_t* n_accepted, int32_t on_host) {
  if (!h) return AD_ERR_ARG;
  if (!h->encoded) return fail(h, AD_ERR_STATE, "ad_verify_block before ad_encode");
  if (!drafts || !k) return fail(h, AD_ERR_ARG, "drafts or k is null");
  const ad_model_cfg& c = h->cfg;
  const int B = h->B;
  if (on_host)
    for (int b = 0; b < B; ++b)
      if (k[b] < 0 || k[b] > c.kmax) return fail(h, AD_ERR_ARG, "k outside 0..kmax");
  // With host arrays the tokens are known here, and the pass is laid out for so many (see LoopBodies).
  const bool captured = being_captured(h);
  LoopBodies bodies = {1, {h->pass[PK_VERIFY].M_cap}};
  int layout_of = 0;
  if (on_host && !captured) {
    long tokens = 0;
    for (int b = 0; b < B; ++b) tokens += k[b];
    bodies = loop_bodies(h, false);
    while (layout_of + 1 < bodies.n && tokens > bodies.cap[layout_of]) ++layout_of;
  }
  // One graph per batch size, layout and kind of acceptance rule (its beta and tau are words): with host arrays the whole call (the block is read from, and the result
  // written to, mapped host memory), with device arrays everything but the copies from and to the caller's arrays.
  char key[48];
  snprintf(key, sizeof(key), "verify B%d h%d r%d f%d", B, on_host ? 1 : 0, h->beta >= 1 ? 1 : 0, layout_of);
  AD_TRY(set_words(h, captured, h->words.x, h->beta, h->tau));
  if (on_host) {
    memcpy(h->up_ids, drafts, sizeof(int) * (size_t)B * c.kmax);
    memcpy(h->up_n, k, sizeof(int) * B);
  } else {
    AD_CUDA(h, cudaMemcpyAsync(h->st.user_drafts, drafts, sizeof(int) * (size_t)B * c.kmax, cudaMemcpyDeviceToDevice, h->stream));
    AD_CUDA(h, cudaMemcpyAsync(h->st.user_k, k, sizeof(int) * B, cudaMemcpyDeviceToDevice, h->stream));
  }
  AD_TRY(run_captured(h, captured, key, [&]() -> int {
    const PassLayout layout = body_layout(h, bodies, layout_of);
    if (on_host) AD_TRY(prepare_verify(h, SRC_USER, nullptr, h->dev_view(h->up_ids), h->dev_view(h->up_n)));
    else AD_TRY(prepare_verify(h, SRC_USER, nullptr));
    AD_TRY(verify_stage(h, 0));
    if (on_host) {
      note_launch(h, "ad_verify_block");
      AD_CUDA(h, launch_k(export_host_kernel, dim3(B), dim3(64), 0, h->stream, h->st, h->dims, h->pass[PK_VERIFY].plan, 0, h->down_dev));
    }
    return AD_OK;
  }));
  h->last_vocab_which = 0;
  if (on_host) {
    const int rc = wait_status(h, h->down);
    if (rc == AD_ERR_CUDA) return rc;
    if (argmax) memcpy(argmax, h->down + 4 + B, sizeof(int) * (size_t)B * c.kmax);
    if (n_accepted) memcpy(n_accepted, h->down + 4, sizeof(int) * B);
    return rc;
  }
  note_launch(h, "ad_verify_block");
  AD_CUDA(h, launch_k(export_block_kernel, dim3(B), dim3(64), 0, h->stream, h->st, h->dims, argmax, n_accepted, nullptr, nullptr, h->pass[PK_VERIFY].plan));
  return AD_OK;
}

extern "C" int ad_commit(ad_handle* h, const int32_t* n, int32_t on_host) {
  if (!h) return AD_ERR_ARG;
  if (!h->encoded) return fail(h, AD_ERR_STATE, "ad_commit before ad_encode");
  const int* n_dev = n;
  if (n && on_host) {
    memcpy(h->up_n, n, sizeof(int) * h->B);
    n_dev = h->dev_view(h->up_n);
  }
  AD_TRY(commit_stage(h, n_dev, on_host ? h->dev_view(h->host_flag + 2) : nullptr));
  return on_host ? wait_status(h, h->host_flag + 2) : AD_OK;
}

extern "C" int ad_force_commit(ad_handle* h, const int32_t* tokens, const int32_t* n, int32_t on_host) {
  if (!h) return AD_ERR_ARG;
  if (!h->encoded) return fail(h, AD_ERR_STATE, "ad_force_commit before ad_encode");
  if (!tokens || !n) return fail(h, AD_ERR_ARG, "tokens or n is null");
  const int *tok_dev = tokens, *n_dev = n;
  if (on_host) {
    memcpy(h->up_ids, tokens, sizeof(int) * (size_t)h->B * h->cfg.kmax);
    memcpy(h->up_n, n, sizeof(int) * h->B);
    tok_dev = h->dev_view(h->up_ids);
    n_dev = h->dev_view(h->up_n);
  }
  note_launch(h, "ad_force_commit");
  AD_CUDA(h, launch_k(force_commit_kernel, dim3(1), dim3(256), 0, h->stream, h->st, h->pass[PK_VERIFY].plan, h->dims, tok_dev, n_dev,
                      on_host ? h->dev_view(h->host_flag + 2) : nullptr));
  return on_host ? wait_status(h, h->host_flag + 2) : AD_OK;
}

extern "C" int ad_draft_block(ad_handle* h, int32_t k_cap, int32_t* drafts, int32_t* k, int32_t on_host) {
  if (!h) return AD_ERR_ARG;
  if (!h->encoded) return fail(h, AD_ERR_STATE, "ad_draft_block before ad_encode");
  if (!h->cfg.has_drafter) return fail(h, AD_ERR_STATE, "the handle has no drafter model");
  const ad_model_cfg& c = h->cfg;
  if (k_cap < 1 || k_cap > c.kmax) return fail(h, AD_ERR_ARG, "k_cap outside 1..kmax");
  const int B = h->B;
  char key[48];
  snprintf(key, sizeof(key), "draft B%d h%d", B, on_host ? 1 : 0);
  const bool captured = being_captured(h);
  AD_TRY(set_words(h, captured, k_cap, h->beta, h->tau));
  AD_TRY(run_captured(h, captured, key, [&]() -> int {
    AD_TRY(plan_draft(h));
    AD_TRY(draft_stage(h));
    if (on_host) {
      note_launch(h, "ad_draft_block");
      AD_CUDA(h, launch_k(export_host_kernel, dim3(B), dim3(64), 0, h->stream, h->st, h->dims, h->pass[PK_VERIFY].plan, 1, h->down_dev));
    }
    return AD_OK;
  }));
  h->last_vocab_which = 1;
  if (on_host) {
    const int rc = wait_status(h, h->down);
    if (rc == AD_ERR_CUDA) return rc;
    if (drafts) memcpy(drafts, h->down + 4 + B, sizeof(int) * (size_t)B * c.kmax);
    if (k) memcpy(k, h->down + 4, sizeof(int) * B);
    return rc;
  }
  note_launch(h, "ad_draft_block");
  AD_CUDA(h, launch_k(export_block_kernel, dim3(B), dim3(64), 0, h->stream, h->st, h->dims, nullptr, nullptr, drafts, k, h->pass[PK_VERIFY].plan));
  return AD_OK;
}

extern "C" int ad_get_state(ad_handle* h, int32_t* len, int32_t* last_tok, int32_t* finished) {
  if (!h) return AD_ERR_ARG;
  if (h->B < 1) return fail(h, AD_ERR_STATE, "ad_get_state before ad_encode");
  if (len) AD_CUDA(h, cudaMemcpyAsync(len, h->st.len, sizeof(int) * h->B, cudaMemcpyDeviceToHost, h->stream));
  if (last_tok) AD_CUDA(h, cudaMemcpyAsync(last_tok, h->st.last, sizeof(int) * h->B, cudaMemcpyDeviceToHost, h->stream));
  if (finished) AD_CUDA(h, cudaMemcpyAsync(finished, h->st.fin, sizeof(int) * h->B, cudaMemcpyDeviceToHost, h->stream));
  return read_status(h);
}

namespace {

// ad_generate's device work as one graph: encoder pass(es), plan of the first pass, loop (see ad_generate).
bool build_whole_graph(ad_handle* h, const ad_gen_opts& o, const int* ovr, bool capped, const LoopBodies& bodies, ad_handle::GraphEntry* out) {
  const int before = h->launches;
  cudaGraph_t g = nullptr, dummy = nullptr;
  cudaGraphConditionalHandle ch = 0;
  std::vector<cudaGraphNode_t> tail;
  bool ok = cudaGraphCreate(&g, 0) == cudaSuccess && cudaGraphConditionalHandleCreate(&ch, g, 1, cudaGraphCondAssignDefault) == cudaSuccess;
  if (ok && bodies.n > 1) {
    cudaGraphConditionalHandle pick = 0;
    ok = cudaGraphConditionalHandleCreate(&pick, g, 0, cudaGraphCondAssignDefault) == cudaSuccess;
    h->pick.node = (unsigned long long)pick;
    for (int i = 0; i + 1 < NextPass::BODIES; ++i) h->pick.cap[i] = i + 1 < bodies.n ? bodies.cap[i] : INT_MAX;
  }
  if (ok && cudaStreamBeginCaptureToGraph(h->stream, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
    ok = encode_stage(h, capped) == AD_OK;
    ok = ok && cudaEventRecordWithFlags(h->ev1, h->stream, cudaEventRecordExternal) == cudaSuccess;   // an event node: end of the encoders
    if (ok && loop_plans_ahead(h)) ok = plan_first_pass(h, o, ovr) == AD_OK;
    cudaStreamCaptureStatus status;
    const cudaGraphNode_t* deps = nullptr;
    size_t n = 0;
    ok = ok && cudaStreamGetCaptureInfo_v2(h->stream, &status, nullptr, nullptr, &deps, &n) == cudaSuccess;
    if (ok) tail.assign(deps, deps + n);
    ok = cudaStreamEndCapture(h->stream, &dummy) == cudaSuccess && ok;
  } else {
    ok = false;
  }
  out->once = h->launches - before;
  h->launches = before;
  if (ok) {
    cudaGraphNodeParams np = {cudaGraphNodeTypeConditional};
    np.conditional.handle = ch;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    cudaGraphNode_t node;
    ok = cudaGraphAddNode(&node, g, tail.data(), tail.size(), &np) == cudaSuccess;
    const cudaGraph_t body = ok ? np.conditional.phGraph_out[0] : nullptr;
    auto capture_body = [&](cudaGraph_t into) {
      if (cudaStreamBeginCaptureToGraph(h->stream, into, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return false;
      h->cond_handle = (unsigned long long)ch;
      h->body_launches = h->launches;
      bool done = loop_iteration(h, o, ovr) == AD_OK;
      h->cond_handle = 0;
      h->launches = before;
      return cudaStreamEndCapture(h->stream, &dummy) == cudaSuccess && done;
    };
    if (ok && bodies.n > 1) {
      cudaGraphNodeParams sp = {cudaGraphNodeTypeConditional};
      sp.conditional.handle = (cudaGraphConditionalHandle)h->pick.node;
      sp.conditional.type = cudaGraphCondTypeSwitch;
      sp.conditional.size = bodies.n;
      cudaGraphNode_t pick;
      ok = cudaGraphAddNode(&pick, body, nullptr, 0, &sp) == cudaSuccess;
      for (int i = 0; i < bodies.n && ok; ++i) {
        const PassLayout layout = body_layout(h, bodies, i);
        ok = capture_body(sp.conditional.phGraph_out[i]);
      }
    } else if (ok) {
      ok = capture_body(body);
    }
  }
  h->pick = {};
  ok = ok && cudaGraphInstantiate(&out->exec, g, 0) == cudaSuccess;
  if (g) cudaGraphDestroy(g);
  out->device_loop = ok;
  return ok;
}

}  // namespace

extern "C" int ad_generate(ad_handle* h, const int32_t* src, int32_t src_stride, const int32_t* src_len, int32_t B,
                           const ad_gen_opts* opts, int32_t* out, int32_t out_stride, int32_t* out_len,
                           ad_stats* stats, int32_t on_host) {
  if (!h) return AD_ERR_ARG;
  const ad_model_cfg& c = h->cfg;
  if (!opts || !out || !out_len) return fail(h, AD_ERR_ARG, "opts, out or out_len is null");
  if (opts->mode != AD_MODE_IAD && opts->mode != AD_MODE_GAD) return fail(h, AD_ERR_ARG, "unknown mode");
  if (opts->k < 1 || opts->k > c.kmax) return fail(h, AD_ERR_ARG, "k outside 1..kmax");
  if (opts->mode == AD_MODE_GAD && opts->run_drafter && !c.has_drafter) return fail(h, AD_ERR_STATE, "GAD with run_drafter needs a drafter model");
  if (opts->mode == AD_MODE_GAD && !opts->run_drafter && !opts->draft_override) return fail(h, AD_ERR_ARG, "GAD without the drafter needs draft_override");
  if (opts->draft_override && opts->override_stride < 1) return fail(h, AD_ERR_ARG, "override_stride must be positive");
  if (out_stride < 1) return fail(h, AD_ERR_ARG, "out_stride must be positive");
  if (B < 1 || B > c.max_batch) return fail(h, AD_ERR_CAPACITY, "B outside 1..max_batch");
  // host-visible per-row caps are checked before any device work, so a rejected call leaves the handle untouched
  int max_iters = c.max_tgt;
  if (opts->max_len && on_host) {
    max_iters = 1;
    for (int b = 0; b < B; ++b) {
      if (opts->max_len[b] < 1 || opts->max_len[b] > c.max_tgt) return fail(h, AD_ERR_ARG, "max_len outside 1..max_tgt");
      if (opts->max_len[b] > max_iters) max_iters = opts->max_len[b];
    }
  }

  AD_TRY(check_sources(h, src, src_stride, src_len, B, on_host));
  AD_CUDA(h, cudaEventRecord(h->ev0, h->stream));
  h->launches = 0;
  h->B = B;
  h->dims.B = B;
  h->encoded = false;
  const int ovr_len = opts->draft_override ? std::min(opts->override_stride, c.max_tgt) : 0;   // valid leading entries of an override row
  const int* ovr = opts->draft_override ? h->ovr : nullptr;
  // (the data-independent bound on the iteration count of the device-side loop and the words travel with the inputs)
  int4 words = {opts->k, ovr_len, h->beta, 0};
  memcpy(&words.w, &h->tau, sizeof(h->tau));
  AD_TRY(import_inputs(h, src, src_stride, src_len, B, opts->max_len, opts->draft_override, opts->override_stride, ovr_len, max_iters + 1, on_host,
                       words));
  const bool capped = opts->max_len != nullptr;

  cudaGraphExec_t exec = nullptr;
  int per_iter_launches = 0;
  bool device_loop = false;
  if (opts->use_graph && h->stream != nullptr) {   // the legacy default stream cannot be captured
    char key[64];           // (block-size cap, override width, beta and tau are words)
    snprintf(key, sizeof(key), "B%d m%d o%d d%d c%d r%d", B, opts->mode, ovr ? 1 : 0, opts->run_drafter ? 1 : 0, capped ? 1 : 0, h->beta >= 1 ? 1 : 0);
    ad_handle::GraphEntry* kept = nullptr;
    AD_TRY(graph_entry(h, key, &kept));
    if (!kept->exec) {
      ad_handle::GraphEntry entry = {};
      // First choice: the whole call as one graph -- encoder pass(es), plan of the first block, and a device-side `while` node
      // whose body is one iteration and whose condition the accept/commit kernel clears; no host round trip between them.
      // (a driver that does not know such a node: one body; no `while` node either: one replay per iteration)
      const LoopBodies one = {1, {h->pass[PK_VERIFY].M_cap}}, bodies = loop_bodies(h, !loop_drafts(*opts) && block_source(*opts, ovr) == SRC_POLICY);
      for (const LoopBodies* b : {&bodies, &one}) {
        if (!h->sw.devloop || (b == &one && bodies.n == 1)) break;
        if (build_whole_graph(h, *opts, ovr, capped, *b, &entry)) break;
        entry = ad_handle::GraphEntry{};
        cudaGetLastError();
      }
      if (!entry.exec) {
        const int before = h->launches;
        cudaGraph_t g = nullptr;
        AD_CUDA(h, cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
        const int rc = loop_iteration(h, *opts, ovr);
        cudaError_t e = cudaStreamEndCapture(h->stream, &g);
        entry.launches = h->launches - before;
        h->launches = before;
        if (rc != AD_OK) { if (g) cudaGraphDestroy(g); return rc; }
        if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("graph capture: ") + cudaGetErrorString(e));
        e = cudaGraphInstantiate(&entry.exec, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return fail(h, AD_ERR_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
      }
      entry.last_use = kept->last_use;
      *kept = entry;
    }
    exec = kept->exec;
    per_iter_launches = kept->launches;
    device_loop = kept->device_loop;
    if (device_loop) h->launches += kept->once;
  }

  if (device_loop) {
    AD_CUDA(h, cudaGraphLaunch(exec, h->stream));
  } else {
    char key[48];
    snprintf(key, sizeof(key), "encode B%d c%d", B, capped ? 1 : 0);
    AD_TRY(run_captured(h, being_captured(h), key, [&]() -> int { return encode_stage(h, capped); }));
    AD_CUDA(h, cudaEventRecord(h->ev1, h->stream));
    if (loop_plans_ahead(h)) AD_TRY(plan_first_pass(h, *opts, ovr));
  }
  h->encoded = true;
  h->last_vocab_which = -1;
  const int sync_every = opts->sync_every > 0 ? opts->sync_every : 1;
  int iters = 0;
  volatile int* flag = h->host_flag;
  flag[0] = 0;
  while (!device_loop && iters < max_iters + sync_every) {
    for (int s = 0; s < sync_every; ++s, ++iters) {
      if (exec) {
        AD_CUDA(h, cudaGraphLaunch(exec, h->stream));
        h->launches += per_iter_launches;
      } else {
        AD_TRY(loop_iteration(h, *opts, ovr));
      }
    }
    AD_CUDA(h, cudaMemcpyAsync(h->host_flag, h->st.all_fin, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    AD_CUDA(h, cudaStreamSynchronize(h->stream));
    if (flag[0]) break;
  }
  AD_CUDA(h, cudaEventRecord(h->ev2, h->stream));
  // Results, statistics and the status word in one block of mapped host memory, written by one kernel: the call ends
  // with a single synchronisation (device-resident result arrays are written directly by the same kernel).
  note_launch(h, "ad_generate");
  AD_CUDA(h, launch_k(finalize_generate_kernel, dim3(B), dim3(128), 0, h->stream, h->st, h->dims, on_host ? nullptr : out, out_stride,
                      on_host ? nullptr : out_len, h->down_dev));
  AD_CUDA(h, cudaStreamSynchronize(h->stream));
  const int* blk = h->down;
  if (device_loop) h->launches += blk[3];
  if (on_host) {
    const int w = out_stride < c.max_tgt ? out_stride : c.max_tgt;
    for (int b = 0; b < B; ++b) {
      memcpy(out + (size_t)b * out_stride, blk + 4 + 4 * B + (size_t)b * c.max_tgt, sizeof(int) * w);
      out_len[b] = blk[4 + 4 * b + 3];
    }
  }
  if (stats) {
    memset(stats, 0, sizeof(*stats));
    for (int b = 0; b < B; ++b) {
      stats->row_iterations += blk[4 + 4 * b];
      stats->accepted += blk[4 + 4 * b + 1];
      stats->offered += blk[4 + 4 * b + 2];
    }
    stats->iterations = blk[2];
    cudaEventElapsedTime(&stats->encode_ms, h->ev0, h->ev1);
    cudaEventElapsedTime(&stats->device_ms, h->ev1, h->ev2);
    stats->kernel_launches = h->launches;
  }
  const int dev_status = blk[1];      // already cleared on the device by the kernel that read it
  if (dev_status != 0)
    return fail(h, dev_status, dev_status == AD_ERR_TIMEOUT ? "a bounded device-side wait ran out" : "device-side argument check failed");
  return AD_OK;
}

extern "C" int ad_debug_logits(ad_handle* h, int32_t which, float* logits, size_t capacity_elems) {
  if (!h || !logits) return AD_ERR_ARG;
  if (h->last_vocab_which != which) return fail(h, AD_ERR_STATE, "no matching projection has just run");
  PassCfg& pc = h->pass[PK_VERIFY];
  int M = 0;
  AD_CUDA(h, cudaMemcpyAsync(&M, pc.plan.M, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  AD_CUDA(h, cudaStreamSynchronize(h->stream));
  if ((size_t)M * h->cfg.vocab > capacity_elems) return fail(h, AD_ERR_CAPACITY, "logits buffer too small");
  Model& m = which == 1 ? h->nar : h->ar;
  GemmParams p = {};
  p.out_f32 = logits;
  AD_TRY(gemm(h, EPI_F32, m.emb, which == 1 ? h->xg : h->yb, PK_VERIFY, pc.plan.M, pc.M_cap, p));
  return AD_OK;
}

extern "C" int ad_debug_encoder_memory(ad_handle* h, int32_t b, float* mem, size_t capacity_elems) {
  if (!h || !mem) return AD_ERR_ARG;
  if (!h->encoded || b < 0 || b >= h->B) return fail(h, AD_ERR_STATE, "no encoded row b");
  PassPlan& pl = h->pass[PK_ENCODE].plan;
  int off = 0, len = 0;
  AD_CUDA(h, cudaMemcpyAsync(&off, pl.seg_off + b, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  AD_CUDA(h, cudaMemcpyAsync(&len, pl.seg_len + b, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  AD_CUDA(h, cudaStreamSynchronize(h->stream));
  const size_t n = (size_t)len * h->cfg.d_model;
  if (n > capacity_elems) return fail(h, AD_ERR_CAPACITY, "memory buffer too small");
  const size_t start = (size_t)off * h->cfg.d_model;
  if (h->bf16) to_f32_kernel<bf16><<<64, 256, 0, h->stream>>>((const bf16*)h->encmem.ptr + start, mem, n);
  else to_f32_kernel<float><<<64, 256, 0, h->stream>>>((const float*)h->encmem.ptr + start, mem, n);
  AD_CUDA(h, cudaGetLastError());
  return AD_OK;
}


extern "C" int ad_debug_profile_verify(ad_handle* h, const int32_t* drafts, const int32_t* k, char* names, float* us,
                                       int32_t capacity, int32_t* n_launches) {
  if (!h || !drafts || !k || !names || !us || !n_launches || capacity < 1) return AD_ERR_ARG;
  if (!h->encoded) return fail(h, AD_ERR_STATE, "ad_debug_profile_verify before ad_encode");
  t_serialise_launches = true;     // serialised launches: an event between two kernels then brackets exactly one of them
  h->profiling = true;
  h->prof.clear();
  const int rc = ad_verify_block(h, drafts, k, nullptr, nullptr, 1);
  h->profiling = false;
  t_serialise_launches = false;
  cudaEvent_t last = nullptr;
  if (cudaEventCreate(&last) == cudaSuccess) { cudaEventRecord(last, h->stream); h->prof.emplace_back("end", last); }
  cudaStreamSynchronize(h->stream);
  int n = 0;
  for (size_t i = 0; i + 1 < h->prof.size() && n < capacity; ++i, ++n) {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, h->prof[i].second, h->prof[i + 1].second);
    us[n] = ms * 1e3f;
    snprintf(names + (size_t)n * 64, 64, "%s", h->prof[i].first.c_str());
  }
  for (auto& pr : h->prof) cudaEventDestroy(pr.second);
  h->prof.clear();
  *n_launches = n;
  return rc;
}

extern "C" int ad_debug_stage_timeline(ad_handle* h, uint64_t* stamps, int32_t capacity, int32_t* n_stages) {
  if (!h || !stamps || !n_stages) return AD_ERR_ARG;
  const int n = mega::ST_PER_LAYER * h->cfg.n_dec + 1;
  if (capacity < 2 * n) return fail(h, AD_ERR_CAPACITY, "timeline buffer too small");
  AD_CUDA(h, cudaStreamSynchronize(h->stream));
  AD_CUDA(h, cudaMemcpy(stamps, h->mega_timeline, sizeof(uint64_t) * 2 * (size_t)n, cudaMemcpyDeviceToHost));
  *n_stages = n;
  return AD_OK;
}

extern "C" int ad_debug_graph_count(const ad_handle* h, int32_t* n) {
  if (!h || !n) return AD_ERR_ARG;
  *n = 0;
  for (const auto& kv : h->graphs) *n += kv.second.exec != nullptr;
  return AD_OK;
}

extern "C" int ad_debug_projection_shapes(const ad_model_cfg* cfg, int32_t* rows, int32_t capacity, int32_t* n_rows) {
  std::string why;
  if (!rows || !n_rows || capacity < 1) return fail(nullptr, AD_ERR_ARG, "null output pointer");
  if (check_cfg(cfg, &why) != AD_OK) return fail(nullptr, AD_ERR_ARG, why);
  ad_handle h;
  h.cfg = *cfg;
  h.bf16 = cfg->dtype == AD_DTYPE_BF16;
  h.esz = h.bf16 ? 2 : 4;
  layout(&h, nullptr);
  *n_rows = 0;
  if (!h.bf16) return AD_OK;
  const int d = cfg->d_model, F = cfg->d_ffn;
  // the projections of a decoder pass in launch order; the query projection in both of its forms
  struct { int epi, N, K; bool split, bias; } list[] = {
      {EPI_SCATTER, 3 * d, d, false, true}, {EPI_F32, d, d, true, false}, {EPI_ACT, d, d, false, true}, {EPI_F32, d, d, true, false},
      {EPI_ACT, F, d, false, true},         {EPI_F32, d, F, true, false}, {EPI_ARGMAX, cfg->vocab, d, false, false}, {EPI_F32, cfg->vocab, d, false, false}};
  const PassCfg& pc = h.pass[PK_VERIFY];
  for (const auto& q : list) {
    const GeoRule r = geo_rule(pc, q.epi, q.N, q.K, q.split, q.bias);
    if (always_few(pc, r) || (q.epi == EPI_ARGMAX && pc.ntile == 256 && vocab_goes_persistent(q.K, q.N, pc.M_cap, nullptr))) continue;
    const TcShape& sh = cached_shape(&h, r, pc.M_cap);
    int ctas = 0, smem = 0;
    for (int M = 0; M <= pc.M_cap; ++M) {
      ctas = std::max(ctas, tc::geometry_ctas(r, M));
      smem = std::max(smem, tc_smem_need(r, M, sh.budget));
    }
    if (*n_rows >= capacity) return fail(nullptr, AD_ERR_CAPACITY, "ad_debug_projection_shapes: more projections than rows");
    const int32_t row[7] = {q.epi, q.N, q.K, sh.ctas, ctas, sh.smem, smem};
    memcpy(rows + 7 * (size_t)(*n_rows)++, row, sizeof(row));
  }
  return AD_OK;
}

// ---- bounded-wait self-test ---------------------------------------------------------------------------

namespace {
// One thread waits, with the given time budget, on an mbarrier phase that nothing ever completes.
__global__ void wait_probe_kernel(int* status, unsigned int budget_us, int* waited_us) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    tc::mbar_init(tc::smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    const unsigned long long t0 = tc::global_ns();
    tc::mbar_wait_budget(tc::smem_u32(&bar), 0, status, (unsigned long long)budget_us * 1000ull);
    if (waited_us) *waited_us = (int)((tc::global_ns() - t0) / 1000ull);
  }
}
}  // namespace

extern "C" int ad_debug_wait_probe(int32_t* status, int32_t budget_us, int32_t* waited_us, void* stream) {
  if (!status || budget_us < 1 || budget_us > (1 << 16)) return AD_ERR_ARG;
  wait_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(status, (unsigned int)budget_us, waited_us);
  return cudaGetLastError() == cudaSuccess ? AD_OK : AD_ERR_CUDA;
}

// ---- grid-barrier self-test and timing ------------------------------------------------------------------

namespace {
// Every CTA: per round, publish a word, pass the grid barrier, read the next CTA's word (bypassing L1) and check
// it.  CTA `absent` (if any) leaves at once without ever arriving, so everybody else's first wait runs out.
// result[0] = nanoseconds per barrier seen by CTA 0, result[1] = rounds CTA 0 completed, result[2] = payload
// mismatches seen by any CTA (must be 0).
__global__ void __launch_bounds__(256, 1)
grid_barrier_probe_kernel(unsigned int* ctr, unsigned int* payload, int rounds, int absent, unsigned long long budget_ns,
                          int* status, float* result, int variant) {
  extern __shared__ uint8_t probe_smem[];    // only there to hold the SM: one CTA per SM, as in the persistent kernels
  __shared__ int flag;
  const unsigned int n = gridDim.x;
  if ((int)blockIdx.x == absent) return;
  unsigned int gen = 0;
  int bad = 0, done = 0;
  if (threadIdx.x == 0) probe_smem[0] = 0;
  const unsigned long long t0 = gs::now_ns();
  for (int r = 0; r < rounds; ++r) {
    // variant bit 0: relaxed polls + one acquire fence instead of an acquire load per poll; bit 1: no payload (barrier alone)
    unsigned int* slot = payload + (size_t)(r & 1) * n;
    if (threadIdx.x == 0 && !(variant & 2)) slot[blockIdx.x] = (unsigned int)r * 4096u + blockIdx.x;
    if (!gs::grid_barrier(ctr, gen, n, budget_ns, &flag, (variant & 1) != 0)) {
      if (threadIdx.x == 0) latch_error(status, AD_ERR_TIMEOUT);
      break;
    }
    const unsigned int nb = (blockIdx.x + 1) % n;
    if (threadIdx.x == 0 && !(variant & 2) && __ldcg(slot + nb) != (unsigned int)r * 4096u + nb) bad++;
    ++done;
  }
  const unsigned long long t1 = gs::now_ns();
  if (threadIdx.x == 0) {
    if (bad) atomicAdd(reinterpret_cast<int*>(result + 2), bad);
    if (blockIdx.x == (absent == 0 ? 1 : 0)) {
      result[0] = done > 0 ? (float)(t1 - t0) / (float)done : 0.f;
      result[1] = (float)done;
    }
  }
}
constexpr int kProbeSmem = 160 * 1024;
}  // namespace

extern "C" int ad_debug_grid_barrier_probe(int32_t n_ctas, int32_t rounds, int32_t absent_cta, int32_t budget_us,
                                           void* scratch, size_t scratch_bytes, int32_t* status, float* result,
                                           void* stream) {
  int variant = 0;
  if (rounds < 0) { variant = (-rounds) & 3; rounds = (-rounds) >> 2; }   // timing variants of the probe (see the kernel)
  if (!scratch || !status || !result || rounds < 1 || rounds > (1 << 20) || budget_us < 1 || budget_us > (1 << 16))
    return fail(nullptr, AD_ERR_ARG, "ad_debug_grid_barrier_probe: bad argument");
  if (n_ctas <= 0) n_ctas = num_sms();
  if (absent_cta >= n_ctas) return fail(nullptr, AD_ERR_ARG, "ad_debug_grid_barrier_probe: absent_cta outside the grid");
  if (scratch_bytes < 256 + sizeof(unsigned int) * 2 * (size_t)n_ctas || reinterpret_cast<uintptr_t>(scratch) % 256)
    return fail(nullptr, AD_ERR_CAPACITY, "ad_debug_grid_barrier_probe: scratch too small or not 256-byte aligned");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (cudaFuncSetAttribute(grid_barrier_probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kProbeSmem) != cudaSuccess)
    return fail(nullptr, AD_ERR_CUDA, "ad_debug_grid_barrier_probe: cudaFuncSetAttribute failed");
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, grid_barrier_probe_kernel, 256, kProbeSmem) != cudaSuccess)
    return fail(nullptr, AD_ERR_CUDA, "ad_debug_grid_barrier_probe: occupancy query failed");
  if (n_ctas > per_sm * num_sms()) return fail(nullptr, AD_ERR_CAPACITY, "ad_debug_grid_barrier_probe: more CTAs than the device holds at once");
  unsigned int* ctr = static_cast<unsigned int*>(scratch);
  unsigned int* payload = ctr + 64;
  if (cudaMemsetAsync(scratch, 0, 256, st) != cudaSuccess || cudaMemsetAsync(result, 0, sizeof(float) * 4, st) != cudaSuccess)
    return fail(nullptr, AD_ERR_CUDA, "ad_debug_grid_barrier_probe: memset failed");
  unsigned long long budget_ns = (unsigned long long)budget_us * 1000ull;
  int absent = absent_cta;
  void* args[] = {&ctr, &payload, &rounds, &absent, &budget_ns, &status, &result, &variant};
  // cooperative launch: the runtime refuses the launch unless all CTAs can be resident at once
  cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<void*>(grid_barrier_probe_kernel), dim3(n_ctas), dim3(256), args,
                                              kProbeSmem, st);
  if (e != cudaSuccess) return fail(nullptr, AD_ERR_CUDA, std::string("ad_debug_grid_barrier_probe: ") + cudaGetErrorString(e));
  return AD_OK;
}

// ---- single-kernel entry points -----------------------------------------------------------------

namespace {
constexpr int kMaxOpTokens = 65536;   // operator-level entries: token rows per call (256-token tiles along grid.y)
}

extern "C" size_t ad_vocab_argmax_scratch_bytes(int32_t vocab, int32_t M) {
  const size_t tiles = (size_t)(vocab + 127) / 128;
  return align_up(tiles * (size_t)M * sizeof(float), 256) + align_up(tiles * (size_t)M * sizeof(int), 256);
}

namespace {

// Arg-max over tiles for M rows without any decoding state: four rows per CTA, a warp each (few rows: one row per CTA, whose
// warps share its tiles), up to eight tiles per lane in flight.  grid = ceil(M / rows), block = 128.
__global__ void __launch_bounds__(128)
argmax_rows_kernel(const float* __restrict__ part_val, const int* __restrict__ part_idx, int n_tiles, int M, int rows, int vocab, int* __restrict__ out) {
  __shared__ float s_v[4];
  __shared__ int s_i[4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = rows == 1 ? blockIdx.x : blockIdx.x * 4 + warp;
  const int first = rows == 1 ? threadIdx.x : lane, step = rows == 1 ? 128 : 32;
  float v = -INFINITY;
  int idx = 0x7fffffff;
  pdl_launch();
  pdl_wait();   // the partials come from the kernel before this one
  if (m < M) {
    for (int t0 = 0; t0 < n_tiles; t0 += 8 * step) {
      float pv[8];
      int pi[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = t0 + u * step + first;
        pv[u] = t < n_tiles ? part_val[(size_t)m * n_tiles + t] : -INFINITY;
        pi[u] = t < n_tiles ? part_idx[(size_t)m * n_tiles + t] : 0x7fffffff;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (pv[u] > v || (pv[u] == v && pi[u] < idx)) { v = pv[u]; idx = pi[u]; }
    }
    tc::warp_argmax(v, idx);
    if (rows > 1 && lane == 0) out[m] = idx < vocab ? idx : 0;       // (no ordered score, NaN: still an id that exists)
  }
  if (rows == 1) {
    if (lane == 0) { s_v[warp] = v; s_i[warp] = idx; }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 4; ++w)
        if (s_v[w] > v || (s_v[w] == v && s_i[w] < idx)) { v = s_v[w]; idx = s_i[w]; }
      out[m] = idx < vocab ? idx : 0;
    }
  }
}

}  // namespace

namespace {
// Geometry of an operator-level call over M tokens (by the passes' rule), and the token operand's map for its tile.
bool op_maps(GemmParams* p, tc::TileMaps* mx, const void* x, int M, int K) {
  p->rule = GeoRule{p->N, K, clampi(pow2ceil(M), 16, 256), 1, num_sms(), 0, 0, 0};
  int tile = geometry(p->rule, M).tile;
  // No K split here: tiles of half the tokens while they leave SMs without work (1800 x 2048 x 512, 60 CTAs with the passes' 128-token
  // tiles: a call 25.5 us, 23.6 with 64; 1100 tokens 24.8, 22.7 with 64, 22.1 with 32; 100 x 4096 x 1024 26.1, 24.8 with 32).
  const int nf = (p->N + tc::BLOCK_N_FEAT - 1) / tc::BLOCK_N_FEAT;
  while (tile > 32 && 2 * nf * ((M + tile - 1) / tile) <= num_sms()) tile /= 2;
  p->rule.fixed_tile = tile;
  int i = 0;
  while ((16 << i) < tile) ++i;
  memset(mx, 0, sizeof(*mx));
  return make_map(&mx->m[i], x, M, K, tile);
}
}  // namespace

extern "C" int ad_vocab_argmax(const void* x, const void* emb, int32_t dtype, int32_t M, int32_t d, int32_t vocab,
                               int32_t* argmax, void* scratch, size_t scratch_bytes, int32_t* status, void* stream) {
  if (!x || !emb || !scratch || M < 1 || d < 1 || vocab < 1) return AD_ERR_ARG;
  if (scratch_bytes < ad_vocab_argmax_scratch_bytes(vocab, M)) return AD_ERR_CAPACITY;
  if (reinterpret_cast<uintptr_t>(scratch) % 256) return AD_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int tiles = (vocab + 127) / 128;
  float* pv = static_cast<float*>(scratch);
  int* pi = reinterpret_cast<int*>(static_cast<char*>(scratch) + align_up((size_t)tiles * M * sizeof(float), 256));
  GemmParams p = {};
  p.K = d; p.N = vocab; p.M_ptr = nullptr; p.M_host = M; p.M_cap = M; p.part_val = pv; p.part_idx = pi; p.status = status;
  cudaError_t e;
  if (dtype == AD_DTYPE_BF16) {
    if (d % 64 || M > kMaxOpTokens) return AD_ERR_ARG;
    CUtensorMap mw;
    const bool persistent = vocab_goes_persistent(d, vocab, M, nullptr);
    if (!make_map(&mw, emb, vocab, d, persistent ? tc::P_BOX : tc::BLOCK_N_FEAT)) return AD_ERR_CUDA;
    if (persistent) {
      CUtensorMap mx128;
      if (!make_map(&mx128, x, M, d, tc::P_TOK)) return AD_ERR_CUDA;
      e = launch_vocab_persistent(st, mw, mx128, p, M);
    } else {
      tc::TileMaps mx;
      if (!op_maps(&p, &mx, x, M, d)) return AD_ERR_CUDA;
      e = launch_tc<EPI_ARGMAX>(st, mw, mx, p, tc_shape(p.rule, M, true));
    }
  } else if (dtype == AD_DTYPE_FP32) {
    e = launch_simt<EPI_ARGMAX>(st, emb, x, p, M);
  } else {
    return AD_ERR_ARG;
  }
  if (e != cudaSuccess) return AD_ERR_CUDA;
  if (!argmax) return AD_OK;   // projection kernel alone: partials stay in scratch
  const int rows = M <= num_sms() ? 1 : 4;
  e = launch_k(argmax_rows_kernel, dim3((M + rows - 1) / rows), dim3(128), 0, st, (const float*)pv, (const int*)pi, tiles, M, rows, vocab, argmax);
  return e == cudaSuccess ? AD_OK : AD_ERR_CUDA;
}

extern "C" int ad_linear(const void* x, const void* W, const float* bias, int32_t dtype, int32_t M, int32_t K,
                         int32_t N, float* y, int32_t* status, void* stream) {
  if (!x || !W || !y || M < 1 || K < 1 || N < 1) return AD_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  GemmParams p = {};
  p.K = K; p.N = N; p.M_ptr = nullptr; p.M_host = M; p.M_cap = M; p.bias = bias; p.out_f32 = y; p.status = status;
  cudaError_t e;
  if (dtype == AD_DTYPE_BF16) {
    if (K % 64 || M > kMaxOpTokens) return AD_ERR_ARG;
    CUtensorMap mw;
    tc::TileMaps mx;
    if (!make_map(&mw, W, N, K, tc::BLOCK_N_FEAT) || !op_maps(&p, &mx, x, M, K)) return AD_ERR_CUDA;
    e = launch_tc<EPI_F32>(st, mw, mx, p, tc_shape(p.rule, M, true));
  } else if (dtype == AD_DTYPE_FP32) {
    e = launch_simt<EPI_F32>(st, W, x, p, M);
  } else {
    return AD_ERR_ARG;
  }
  return e == cudaSuccess ? AD_OK : AD_ERR_CUDA;
}

// ---- projection + arg-max for callers that cannot allocate -------------------------------------------
// The scratch that ad_vocab_argmax takes from its caller is, here, a fixed array inside the library image.
// In host code the array's name is only a handle for the runtime, not a device address: the address is asked
// for once per device (cudaGetSymbolAddress with that device current) and then passed to the kernels.
static __device__ __align__(256) unsigned char g_static_scratch[AD_STATIC_SCRATCH_BYTES];

namespace {
void* g_static_scratch_addr[kMaxDevices] = {};
}  // namespace

extern "C" int ad_vocab_argmax_static(const void* x, const void* emb, int32_t dtype, int32_t M, int32_t d,
                                      int32_t vocab, int32_t* argmax, int32_t* status, void* stream) {
  if (!x || !emb || !argmax || M < 1 || d < 1 || vocab < 1) return fail(nullptr, AD_ERR_ARG, "ad_vocab_argmax_static: bad argument");
  const size_t need = ad_vocab_argmax_scratch_bytes(vocab, M);
  if (need > AD_STATIC_SCRATCH_BYTES)
    return fail(nullptr, AD_ERR_CAPACITY, "ad_vocab_argmax_static: problem needs " + std::to_string(need) +
                " bytes of scratch, the built-in array holds " + std::to_string((size_t)AD_STATIC_SCRATCH_BYTES));
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return fail(nullptr, AD_ERR_CUDA, "ad_vocab_argmax_static: no current CUDA device");
  if (!g_static_scratch_addr[dev]) {   // first call on this device: resolve the array's device address
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess || !p)
      return fail(nullptr, AD_ERR_CUDA, std::string("ad_vocab_argmax_static: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    g_static_scratch_addr[dev] = p;
  }
  const int rc = ad_vocab_argmax(x, emb, dtype, M, d, vocab, argmax, g_static_scratch_addr[dev], AD_STATIC_SCRATCH_BYTES, status, stream);
  if (rc != AD_OK)
    return fail(nullptr, rc, rc == AD_ERR_ARG ? "ad_vocab_argmax_static: unsupported shape or dtype (BF16 needs d % 64 == 0 and M <= 65536)"
                                              : "ad_vocab_argmax_static: encoding a TMA descriptor or launching a kernel failed");
  return AD_OK;
}

#ifdef AD_TRACE
// Timeline dump of a tracing build: copies up to cap stamps to the host and optionally clears the buffer.
extern "C" int ad_debug_trace(unsigned long long* host_buf, int cap, int reset) {
  unsigned int n = 0;
  if (cudaDeviceSynchronize() != cudaSuccess) return -1;
  if (cudaMemcpyFromSymbol(&n, g_trace_n, sizeof(n)) != cudaSuccess) return -1;
  if (n > (1u << 15)) n = 1u << 15;
  if ((int)n > cap) n = cap;
  if (n && cudaMemcpyFromSymbol(host_buf, g_trace_buf, sizeof(unsigned long long) * n) != cudaSuccess) return -1;
  if (reset) { unsigned int z = 0; cudaMemcpyToSymbol(g_trace_n, &z, sizeof(z)); }
  return (int)n;
}
#endif
