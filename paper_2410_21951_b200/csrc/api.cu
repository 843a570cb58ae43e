// libvadusa: host engine and C ABI.  Every step of the draft-and-verify path runs in
// the kernels included below; this file only validates, lays out memory and launches.
#include <cuda_runtime.h>
#include <stdarg.h>

#include <type_traits>

#include <algorithm>
#include <map>
#include <new>
#include <string>
#include <tuple>

#include "accept.cuh"
#include "attention_simt.cuh"
#include "attention_tc.cuh"
#include "attention_prefill_tc.cuh"
#include "attention_stream_tc.cuh"
#include "elementwise.cuh"
#include "fit.cuh"
#include "fwd_fused.cuh"
#include "gemm_simt.cuh"
#include "gemm_tc.cuh"
#include "gemm_tc2.cuh"
#include "layout.h"
#include "select.cuh"

using namespace vadusa;

struct LayerW {
  const float *ln1_g, *ln1_b, *bqkv, *bo, *ln2_g, *ln2_b, *b1, *b2;
  const void *wqkv, *wo, *w1, *w2;
};

struct vadusa_ctx {
  vadusa_config cfg;
  std::vector<LayerW> layers;
  const void *emb_audio = nullptr, *emb_phon = nullptr, *pos = nullptr, *lm = nullptr, *dw = nullptr, *du = nullptr;
  const float *lnf_g = nullptr, *lnf_b = nullptr, *db = nullptr;
  long long dw_stride = 0, du_stride = 0;     // bytes between draft heads
  WorkspaceLayout ws;
  std::vector<TensorDesc> wl;
  const char* blob = nullptr;
  char* wsp = nullptr;
  cudaStream_t stream = nullptr;
  int batch = 0;
  const float* logit_bias = nullptr;   // caller's [batch][logit_bias_ld] fp32 added to the base head's logits (sampler hook)
  int logit_bias_ld = 0;
  int n_nodes = 0;            // current tree size (0: none set)
  int tree_per_seq = 0;
  int tree_copies = 1;        // trees in the workspace's tree area (packed: see vadusa_set_tree)
  int tree_max_depth = 0;
  int tree_inner = 0;         // most nodes with children of any of the trees
  // draft-head fitting (vadusa_fit_*): the caller's state buffer and the schedule
  char* fit = nullptr;
  int fit_tokens = 0, fit_step = 0, fit_warmup = 0;
  float fit_lambda = 0.f, fit_lr = 0.f;
  void* pf_tap = nullptr;     // where prefill also leaves the final hidden state of every prefix token ([batch][stride][d])
  int pf_tap_stride = 0;
  int pf_tiles = 0;           // > 0 while a prefill pass runs: attention CTAs of the pass (pairs of chunks), listed in pf_pairs
  const int2* pf_pairs = nullptr;
  bool in_prefill = false;    // a prefill pass: the context of its later chunks is written by the pass itself
  int att_stream = 0;         // batches: attention as one persistent kernel over the stream of K/V pages (0: one CTA per head and sequence)
  int fused_enabled = 0;      // single-sequence passes run as one persistent kernel (0: no, 1: yes, 6 / 8: with that cluster size)
  int fused_clusters = -1;    // clusters of that kernel that can be resident at once on this device (-1: not asked yet)
  int fused_cs = -1;          // CTAs per cluster chosen for it (8 or 6; 0: the device cannot hold one cluster per head)
  int fused_n8 = 0, fused_n6 = 0;
  long long ctx_bound = 0;    // host-side upper bound of the longest context (grows by the longest path per commit)
  long long ctx_lo = 0;       // host-side lower estimate of it (one token per iteration); exact after begin, prefill, get_lengths
  const int32_t* block_table = nullptr;
  bool have_draft = false, have_verify = false;
  int64_t launches = 0;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  // Host-visible words: the generation loop's progress (see run_generate), then the sequences' token counts and error word
  int32_t* h_pinned = nullptr;
  // Pinned staging of host arrays on their way to the device: two halves, each with an event behind its last copy, so
  // that a call returns as soon as its arrays are staged instead of waiting for the stream
  char* up = nullptr;
  size_t up_at = 0;
  int up_half = 0;
  bool up_used[2] = {false, false};
  cudaEvent_t ev_up[2] = {nullptr, nullptr};
  // context lengths as the host knows them (exact after begin, prefill, get_lengths and generate)
  std::vector<int32_t> h_ctx;
  bool h_ctx_exact = false;
  char err[512] = {0};
  // TMA descriptors of the operands of the tensor-core products, made on first use
  typedef std::tuple<const void*, int, int, int, int, long long> MapKey;   // ptr, rows, K, box rows, batches, batch stride
  std::map<MapKey, CUtensorMap> maps;
  void* encode_fn = nullptr;       // cuTensorMapEncodeTiled, resolved through the runtime
  // CUDA graphs of the launch sequences of the hot calls, keyed by their baked-in arguments
  struct GraphRec { cudaGraphExec_t exec = nullptr; int seen = 0; int64_t launches = 0, used = 0; };
  int64_t graph_clock = 0;
  std::map<std::string, GraphRec> graphs;
  // per-kernel timing (vadusa_profile_begin/end): one event pair per launch
  struct ProfRec { cudaEvent_t a, b; int cls; };
  bool prof_on = false, prof_pending = false;
  std::vector<ProfRec> prof;
};

enum KClass { K_EMBED, K_LAYERNORM, K_GEMM_QKV, K_ATTENTION, K_GEMM_OUT, K_GEMM_FFN1, K_GEMM_FFN2, K_GEMM_LM,
              K_DRAFT_HIDDEN, K_DRAFT_LOGITS, K_DRAFT_SELECT, K_ACCEPT, K_COMMIT, K_MISC, K_FUSED, K_NCLASS };
static const char* const kClassName[K_NCLASS] = {
    "tree_embed", "layernorm", "gemm_qkv", "tree_attention", "gemm_out", "gemm_ffn1", "gemm_ffn2", "gemm_lm",
    "draft_hidden", "draft_logits", "draft_select", "accept", "commit", "misc", "fused_forward"};

namespace {

vadusa_status fail(vadusa_ctx* c, vadusa_status s, const char* fmt, ...) {
  if (c) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(c->err, sizeof(c->err), fmt, ap);
    va_end(ap);
  }
  return s;
}

#define CU(call)                                                                                   \
  do {                                                                                             \
    cudaError_t e_ = (call);                                                                       \
    if (e_ != cudaSuccess) return fail(ctx, VADUSA_ECUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

#define LAUNCH_CHECK()                                                                             \
  do {                                                                                             \
    cudaError_t e_ = cudaGetLastError();                                                           \
    if (e_ != cudaSuccess) return fail(ctx, VADUSA_ECUDA, "kernel launch: %s", cudaGetErrorString(e_)); \
    ctx->launches++;                                                                               \
    if (ctx->prof_pending) { cudaEventRecord(ctx->prof.back().b, ctx->stream); ctx->prof_pending = false; } \
  } while (0)

// Call right before a kernel launch: when profiling is on, brackets the launch with events.
void PROF(vadusa_ctx* c, int cls) {
  if (!c->prof_on) return;
  vadusa_ctx::ProfRec r;
  r.cls = cls;
  if (cudaEventCreate(&r.a) != cudaSuccess || cudaEventCreate(&r.b) != cudaSuccess) return;
  cudaEventRecord(r.a, c->stream);
  c->prof.push_back(r);
  c->prof_pending = true;
}

template <typename P> P* wsptr(vadusa_ctx* c, int64_t off) { return reinterpret_cast<P*>(c->wsp + off); }

const TensorDesc* find(const vadusa_ctx* c, const std::string& name) {
  for (const auto& t : c->wl)
    if (t.name == name) return &t;
  return nullptr;
}
const void* wraw(const vadusa_ctx* c, const std::string& name) {
  const TensorDesc* t = find(c, name);
  return t ? c->blob + t->offset : nullptr;
}

void resolve_weights(vadusa_ctx* c) {
  auto f = [&](const std::string& n) { return reinterpret_cast<const float*>(wraw(c, n)); };
  c->layers.resize(c->cfg.n_layers);
  for (int l = 0; l < c->cfg.n_layers; ++l) {
    const std::string p = "l" + std::to_string(l) + ".";
    LayerW& w = c->layers[l];
    w.ln1_g = f(p + "ln1_g"); w.ln1_b = f(p + "ln1_b"); w.bqkv = f(p + "bqkv"); w.bo = f(p + "bo");
    w.ln2_g = f(p + "ln2_g"); w.ln2_b = f(p + "ln2_b"); w.b1 = f(p + "b1"); w.b2 = f(p + "b2");
    w.wqkv = wraw(c, p + "wqkv"); w.wo = wraw(c, p + "wo"); w.w1 = wraw(c, p + "w1"); w.w2 = wraw(c, p + "w2");
  }
  c->emb_audio = wraw(c, "emb_audio"); c->emb_phon = wraw(c, "emb_phon"); c->pos = wraw(c, "pos");
  c->lnf_g = f("lnf_g"); c->lnf_b = f("lnf_b"); c->lm = wraw(c, "lm");
  c->dw = wraw(c, "draft0.w"); c->db = f("draft0.b"); c->du = wraw(c, "draft0.u");
  if (c->cfg.n_draft_heads > 1) {
    c->dw_stride = find(c, "draft1.w")->offset - find(c, "draft0.w")->offset;
    c->du_stride = find(c, "draft1.u")->offset - find(c, "draft0.u")->offset;
  }
}
template <typename T> const T* as(const void* p) { return reinterpret_cast<const T*>(p); }

uint32_t* err_word(vadusa_ctx* c) { return wsptr<uint32_t>(c, c->ws.scalars); }
int32_t* done_word(vadusa_ctx* c) { return wsptr<int32_t>(c, c->ws.scalars) + 1; }

KvGeom geom_of(const vadusa_ctx* c) {
  KvGeom g;
  g.n_heads = c->cfg.n_heads;
  g.head_dim = c->cfg.d_model / c->cfg.n_heads;
  g.max_blocks_per_seq = c->cfg.max_blocks_per_seq;
  g.num_blocks = c->cfg.kv_num_blocks;
  g.layer_stride = (long long)c->cfg.kv_num_blocks * 2 * c->cfg.d_model * kKvBlock;
  return g;
}

TreeView tree_of(vadusa_ctx* c, bool chain) {
  TreeView t;
  if (chain) {
    t.parent = wsptr<int32_t>(c, c->ws.chain_parent);
    t.depth = wsptr<int32_t>(c, c->ws.chain_depth);
    t.rank = wsptr<int32_t>(c, c->ws.chain_rank);
    t.anc = wsptr<unsigned long long>(c, c->ws.chain_anc);
    t.n_nodes = c->cfg.max_tree_nodes;
    t.per_seq = 0;
  } else {
    const size_t nn = (size_t)c->tree_copies * c->n_nodes;
    t.parent = wsptr<int32_t>(c, c->ws.tree);
    t.depth = t.parent + nn;
    t.rank = t.depth + nn;
    t.anc = reinterpret_cast<const unsigned long long*>(
        c->wsp + c->ws.tree + ((nn * 12 + (size_t)c->tree_copies * VADUSA_MAX_TREE_NODES * 4 + 15) & ~(size_t)15));
    t.n_nodes = c->n_nodes;
    t.per_seq = c->tree_per_seq;
  }
  return t;
}

SeqState state_of(vadusa_ctx* c, int32_t* out_tokens, int out_cap, int target) {
  SeqState s;
  s.ctx_len = wsptr<int32_t>(c, c->ws.ctx_len);
  s.nvalid = wsptr<int32_t>(c, c->ws.nvalid);
  s.gen_count = wsptr<int32_t>(c, c->ws.gen_count);
  s.commit_base = wsptr<int32_t>(c, c->ws.commit_base);
  s.commit_nv = wsptr<int32_t>(c, c->ws.commit_nv);
  s.node_ok = wsptr<int32_t>(c, c->ws.node_ok);
  s.node_top = wsptr<int32_t>(c, c->ws.node_top);
  s.out_tokens = out_tokens;
  s.done_count = done_word(c);
  s.out_cap = out_cap;
  s.target = target;
  s.stats = wsptr<unsigned long long>(c, c->ws.acc_stats);
  return s;
}
static_assert(kStatDepth == VADUSA_MAX_DEPTH && kStatTopk == VADUSA_MAX_DRAFT_TOPK, "statistics table follows the C ABI's maxima");

vadusa_status sampling_dev(vadusa_ctx* ctx, const vadusa_sampling* s, SamplingDev* o) {
  if (!s) return fail(ctx, VADUSA_EINVAL, "sampling is NULL");
  if (s->tau < 1) return fail(ctx, VADUSA_EINVAL, "tau must be >= 1");
  if (!(s->temperature >= 0.f)) return fail(ctx, VADUSA_EINVAL, "temperature must be >= 0");
  if (!(s->top_p > 0.f)) return fail(ctx, VADUSA_EINVAL, "top_p must be > 0");
  if (s->accept_rule != 0 && s->accept_rule != 1) return fail(ctx, VADUSA_EINVAL, "accept_rule must be 0 or 1");
  memset(o, 0, sizeof(*o));            // the bytes of this struct key the graph cache: no stray padding
  o->tau = s->tau;
  o->temperature = s->temperature;
  o->inv_temperature = s->temperature > 0.f ? (float)(1.0 / (double)s->temperature) : 1.f;
  o->top_p = s->top_p;
  o->eos_masked = s->eos_masked ? 1 : 0;
  o->accept_rule = s->accept_rule;
  o->eos_id = ctx->cfg.vocab - 1;
  o->seed = s->seed;
  o->bias = ctx->logit_bias;
  o->bias_ld = ctx->logit_bias_ld;
  return VADUSA_OK;
}

constexpr size_t kUpHalf = 1 << 20;
constexpr int kHostWords = 4;       // h_pinned: iterations finished, sequences done, error word, unused; then [batch] token counts

// Copies `bytes` from host memory (the caller's, free again on return) to dst in stream order.
vadusa_status upload(vadusa_ctx* ctx, void* dst, const void* src, size_t bytes) {
  if (bytes > kUpHalf) {
    CU(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, ctx->stream));
    CU(cudaStreamSynchronize(ctx->stream));
    return VADUSA_OK;
  }
  if (ctx->up_at + bytes > kUpHalf) {
    CU(cudaEventRecord(ctx->ev_up[ctx->up_half], ctx->stream));
    ctx->up_used[ctx->up_half] = true;
    ctx->up_half ^= 1;
    ctx->up_at = 0;
    if (ctx->up_used[ctx->up_half]) CU(cudaEventSynchronize(ctx->ev_up[ctx->up_half]));
  }
  char* at = ctx->up + ctx->up_half * kUpHalf + ctx->up_at;
  memcpy(at, src, bytes);
  ctx->up_at += (bytes + 15) & ~(size_t)15;
  CU(cudaMemcpyAsync(dst, at, bytes, cudaMemcpyHostToDevice, ctx->stream));
  return VADUSA_OK;
}

// Launch of a kernel that begins with griddepcontrol.wait: it may be set up while its predecessor is still running.
template <typename K, typename... A>
cudaError_t launch_dependent(vadusa_ctx* ctx, K kernel, dim3 grid, int threads, size_t smem, A... args) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = dim3(threads);
  lc.dynamicSmemBytes = smem;
  lc.stream = ctx->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at; lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, kernel, args...);
}

// ---- typed engine ------------------------------------------------------------------

// Plain FMA product; rn: LayerNorm of the operand rows on the way (few tokens only).
template <typename T, typename Epi>
vadusa_status gemm(vadusa_ctx* ctx, int cls, const T* A, const T* W, int M, int N, int K, int batches, long long a_z,
                   long long w_z, const Epi& epi, const RowNorm* rn = nullptr) {
  PROF(ctx, cls);
  if (M <= kFewTokens) {
    const int mw = M <= 4 ? 1 : M <= 8 ? 2 : 4, nw = 4 / mw;         // warps of a block along tokens / features
    const dim3 grid((N + 4 * nw - 1) / (4 * nw), (M + 4 * mw - 1) / (4 * mw), batches);
    if (rn) CU(launch_dependent(ctx, gemm_few_kernel<T, Epi, true>, grid, 128, 0, A, W, M, N, K, a_z, w_z, mw, epi, *rn));
    else CU(launch_dependent(ctx, gemm_few_kernel<T, Epi, false>, grid, 128, 0, A, W, M, N, K, a_z, w_z, mw, epi, RowNorm{}));
  } else {
    CU(launch_dependent(ctx, gemm_simt_kernel<T, Epi>, dim3((N + 63) / 64, (M + 63) / 64, batches), 256, 0, A, W, M, N, K, a_z,
                        w_z, epi));
  }
  LAUNCH_CHECK();
  return VADUSA_OK;
}

// ---- tensor-core products (bf16 models) ------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Descriptor of a row-major bf16 matrix [batches][rows][K] read in boxes of box_rows x 64
// elements with the 128-byte swizzle; rows outside the matrix read as zero.
vadusa_status tensor_map(vadusa_ctx* ctx, const void* ptr, int rows, int K, int box_rows, int batches,
                         long long batch_stride_elems, const CUtensorMap** out) {
  vadusa_ctx::MapKey key(ptr, rows, K, box_rows, batches, batch_stride_elems);
  auto it = ctx->maps.find(key);
  if (it == ctx->maps.end()) {
    if (!ctx->encode_fn) return fail(ctx, VADUSA_ECUDA, "cuTensorMapEncodeTiled is not available");
    CUtensorMap m;
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)batches};
    cuuint64_t strides[2] = {(cuuint64_t)K * 2, (cuuint64_t)(batches > 1 ? batch_stride_elems : (long long)rows * K) * 2};
    cuuint32_t box[3] = {(cuuint32_t)kGemmBK, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = reinterpret_cast<EncodeTiledFn>(ctx->encode_fn)(
        &m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(ctx, VADUSA_ECUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
    it = ctx->maps.emplace(key, m).first;
  }
  *out = &it->second;
  return VADUSA_OK;
}

// X == nullptr with ln != nullptr: the LayerNorm-fused variant (the operand is made in the kernel).
template <int TN, typename Epi, bool LN = false>
vadusa_status launch_gemm_tc(vadusa_ctx* ctx, int cls, const void* X, const void* W, int w_rows, int M, int N, int K,
                             int batches, long long x_z, long long w_z, int ksplit, const Epi& epi,
                             const LnFuse* ln = nullptr) {
  using Cfg = GemmTcCfg<TN>;
  static unsigned long long attr_done = 0ull;              // per device: function attributes belong to a device's context
  const unsigned long long dev_bit = 1ull << (ctx->cfg.device & 63);
  if (!(attr_done & dev_bit)) {
    CU(cudaFuncSetAttribute(gemm_tc_kernel<TN, Epi, LN>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmemMax));
    CU(cudaFuncSetAttribute(gemm_tc_kernel<TN, Epi, LN>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    CU(cudaFuncSetAttribute(gemm_tc_kernel<TN, Epi, LN>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    attr_done |= dev_bit;
  }
  const int chunks = K / kGemmBK / ksplit;
  const int smem = Cfg::smem_for(chunks, ksplit);
  const CUtensorMap *mw, *mx;
  if (vadusa_status s = tensor_map(ctx, W, w_rows, K, kGemmRowsW, batches, w_z, &mw)) return s;
  if (LN) mx = mw;                                       // unused by the kernel
  else if (vadusa_status s = tensor_map(ctx, X, M, K, TN, batches, x_z, &mx)) return s;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((N + kGemmRowsW - 1) / kGemmRowsW, (M + TN - 1) / TN, batches * ksplit);
  lc.blockDim = dim3(128);
  lc.dynamicSmemBytes = smem;
  lc.stream = ctx->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = ksplit;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel calls griddepcontrol.wait
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at; lc.numAttrs = 2;
  PROF(ctx, cls);
  CU(cudaLaunchKernelEx(&lc, gemm_tc_kernel<TN, Epi, LN>, *mw, *mx, M, N, chunks, ksplit, Cfg::stages_for(chunks),
                        Cfg::ring_for(chunks, ksplit), epi, wsptr<float>(ctx, ctx->ws.gemm_part), err_word(ctx),
                        ln ? *ln : LnFuse{}));
  LAUNCH_CHECK();
  return VADUSA_OK;
}

// Many-token product on CTA pairs (256 features x TN tokens per pair, no K split).
template <int TN, int ST, int KB, typename Epi>
vadusa_status launch_gemm_tc2(vadusa_ctx* ctx, int cls, const void* X, const void* W, int w_rows, int M, int N, int K,
                              int slices, const Epi& epi) {
  using Cfg = GemmTc2Cfg<TN, ST, KB>;
  // whole stages; and all CTAs that fit on an SM have room in its tensor memory, so that no pair ever waits for another's
  constexpr int kPerSm = 227 * 1024 / (Cfg::kSmem + 1024), kAccCols = 512 / kPerSm < 256 ? 512 / kPerSm : 256;
  while (slices > 1 && (slices * TN > kAccCols || K / (kGemmBK * KB) % slices)) slices /= 2;
  static unsigned long long attr_done = 0ull;              // per device, like launch_gemm_tc
  const unsigned long long dev_bit = 1ull << (ctx->cfg.device & 63);
  if (!(attr_done & dev_bit)) {
    CU(cudaFuncSetAttribute(gemm_tc2_kernel<TN, ST, KB, false, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmem));
    CU(cudaFuncSetAttribute(gemm_tc2_kernel<TN, ST, KB, true, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmem));
    CU(cudaFuncSetAttribute(gemm_tc2_kernel<TN, ST, KB, false, Epi>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    CU(cudaFuncSetAttribute(gemm_tc2_kernel<TN, ST, KB, true, Epi>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    attr_done |= dev_bit;
  }
  const CUtensorMap *mw, *mx;
  if (vadusa_status s = tensor_map(ctx, W, w_rows, K, kGemmRowsW, 1, 0, &mw)) return s;
  if (vadusa_status s = tensor_map(ctx, X, M, K, TN / 2, 1, 0, &mx)) return s;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(N / kGemmRowsW, (M + TN - 1) / TN, 1);           // N is a multiple of 256: whole pairs
  lc.blockDim = dim3(128);
  lc.dynamicSmemBytes = Cfg::kSmem;
  lc.stream = ctx->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // the kernel calls griddepcontrol.wait
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at; lc.numAttrs = 2;
  PROF(ctx, cls);
  CU(cudaLaunchKernelEx(&lc, slices > 1 ? gemm_tc2_kernel<TN, ST, KB, true, Epi> : gemm_tc2_kernel<TN, ST, KB, false, Epi>, *mw, *mx, M, N, K / (kGemmBK * KB), slices, epi, err_word(ctx)));
  LAUNCH_CHECK();
  return VADUSA_OK;
}

// Persistent CTA pairs: tiles of 256 features x 256 tokens dealt round-robin to as many pairs as balance the rounds.
template <typename Epi>
vadusa_status launch_gemm_tc2p(vadusa_ctx* ctx, int cls, const void* X, const void* W, int w_rows, int M, int N, int K,
                               const Epi& epi) {
  static unsigned long long attr_done = 0ull;
  const unsigned long long dev_bit = 1ull << (ctx->cfg.device & 63);
  if (!(attr_done & dev_bit)) {
    CU(cudaFuncSetAttribute(gemm_tc2p_kernel<Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemmP2Smem));
    CU(cudaFuncSetAttribute(gemm_tc2p_kernel<Epi>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    attr_done |= dev_bit;
  }
  const CUtensorMap *mw, *mx;
  if (vadusa_status s = tensor_map(ctx, W, w_rows, K, kGemmRowsW, 1, 0, &mw)) return s;
  if (vadusa_status s = tensor_map(ctx, X, M, K, kGemmP2TN / 2, 1, 0, &mx)) return s;
  const int tiles = (N / (2 * kGemmRowsW)) * ((M + kGemmP2TN - 1) / kGemmP2TN);
  const int rounds = (tiles + 73) / 74, npairs = (tiles + rounds - 1) / rounds;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(2 * npairs, 1, 1);
  lc.blockDim = dim3(kGemmP2Threads);
  lc.dynamicSmemBytes = kGemmP2Smem;
  lc.stream = ctx->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at; lc.numAttrs = 2;
  PROF(ctx, cls);
  CU(cudaLaunchKernelEx(&lc, gemm_tc2p_kernel<Epi>, *mw, *mx, M, N, K / kGemmBK, tiles, epi, err_word(ctx)));
  LAUNCH_CHECK();
  return VADUSA_OK;
}

// K split of a product with `tiles` output tiles of tn tokens: about one CTA per SM streams weights.
static int gemm_ksplit(int tiles, int chunks, int tn) {
  int ksplit = 1;
  while (ksplit < kGemmMaxSplit && tiles * ksplit < 148 && chunks % (ksplit * 2) == 0 && ksplit * 2 <= tn &&
         (long long)tiles * ksplit * 2 * tn * kGemmRowsW * 4 <= kGemmPartBytes)
    ksplit *= 2;
  return ksplit;
}

// Does a residual product of N = d_model features over K inputs leave LayerNorm statistics for M
// tokens?  (Its split-K epilogue does; the fused consumer handles at most 64 tokens and 8 groups.)
static bool residual_leaves_stats(int M, int d, int K) {
  if (M > 64 || d % 128 || d / 128 > 8 || K % kGemmBK) return false;
  const int tn = M <= 16 ? 16 : M <= 32 ? 32 : 64;
  return gemm_ksplit(d / kGemmRowsW, K / kGemmBK, tn) >= 2;
}

// LayerNorm(x) * W^T with the normalisation done inside the product kernel from the statistics the
// producer of x left; applies when the tokens fit one tile of at most 64 and the K slices of the
// cluster are 128 columns.  Returns false (nothing launched) when the shape does not qualify.
template <typename Epi>
bool gemm_tc_ln(vadusa_ctx* ctx, int cls, const float* x, const float* g, const float* b, const void* W, int w_rows,
                int M, int N, int K, const Epi& epi, vadusa_status* st, bf16* y = nullptr) {
  if (M > 64 || K % 128 || K / 128 > 8) return false;
  const int tn = M <= 16 ? 16 : M <= 32 ? 32 : 64;
  const int tiles = (N + kGemmRowsW - 1) / kGemmRowsW;
  const int ksplit = K / 128;                            // one CTA of the cluster per group of 128 columns
  if (ksplit < 2 || ksplit > tn || (long long)tiles * ksplit * tn * kGemmRowsW * 4 > kGemmPartBytes) return false;
  const LnFuse ln{x, g, b, wsptr<float2>(ctx, ctx->ws.ln_stats), y, K, ctx->cfg.ln_eps};
  switch (tn) {
    case 16: *st = launch_gemm_tc<16, Epi, true>(ctx, cls, nullptr, W, w_rows, M, N, K, 1, 0, 0, ksplit, epi, &ln); break;
    case 32: *st = launch_gemm_tc<32, Epi, true>(ctx, cls, nullptr, W, w_rows, M, N, K, 1, 0, 0, ksplit, epi, &ln); break;
    default: *st = launch_gemm_tc<64, Epi, true>(ctx, cls, nullptr, W, w_rows, M, N, K, 1, 0, 0, ksplit, epi, &ln); break;
  }
  return true;
}

// Tile width by token count; K split so that about one CTA per SM streams weights.
template <typename Epi>
vadusa_status gemm_tc(vadusa_ctx* ctx, int cls, const void* X, const void* W, int w_rows, int M, int N, int K,
                      int batches, long long x_z, long long w_z, const Epi& epi) {
  const int ntiles_n = (N + kGemmRowsW - 1) / kGemmRowsW;
  // More than 64 tokens and features in whole pairs of tiles: CTA pairs.  While a tile width gives at most one CTA per SM, the
  // narrowest such tile with the deepest ring of two-chunk stages (every CTA streams operands, latency decides); then
  // 128-token tiles with two or three CTAs per SM, whose epilogues hide behind one another's main loops; beyond three
  // full SMs' worth, resident pairs that walk 256 x 256 tiles.  32-token tiles read every weight M / 32 times: up to 72 CTAs, and
  // up to a full device where the weights are not the wider operand (N <= K).  Measured with weights from DRAM, us:
  //   512 tokens: q/k/v 13.8 -> 8.0, out 8.7 -> 4.9, FFN1 13.9 -> 8.6, FFN2 11.4 -> 11.1 (before: one CTA per tile, K split)
  //   2048 tokens: FFN1 17.8 -> 15.9, FFN2 21.4 -> 16.1; 1344 tokens: out 17.2 -> 8.0, FFN2 25.8 -> 15.4
  // Few tokens against a long K (second feed-forward matrix) stay with the K split below: 7.9 us at 128 tokens, 10.5 as pairs.
  if (M > 64 && batches == 1 && N % (2 * kGemmRowsW) == 0 && !(M <= 128 && K > 2 * N)) {
    auto ctas = [&](int tn) { return ntiles_n * ((M + tn - 1) / tn); };
    // Accumulators: one; for a prefix, whose rows every later token reads, one per K slice that a single-CTA product of 128-token
    // tiles would be split into (shorter chains of truncating additions: the rows are the split form's to the bit).  One prefix
    // of 325 tokens 668 -> 713 us a call; the same in a batch-8 step would be 3.00 -> 3.19 ms.
    const int slices = !ctx->in_prefill || (M > 512 && ctas(128) >= 128) ? 1 : gemm_ksplit(ctas(128), K / kGemmBK, 128);
    const bool two = K % (2 * kGemmBK) == 0;             // stages of two chunks
    if (two && ctas(32) <= (N <= K ? 148 : 72)) {
      if (ctas(32) <= 72 || K > 1024) return launch_gemm_tc2<32, 5, 2>(ctx, cls, X, W, w_rows, M, N, K, slices, epi);
      return launch_gemm_tc2<32, 3, 2>(ctx, cls, X, W, w_rows, M, N, K, slices, epi);
    }
    if (two && ctas(64) <= 148) return launch_gemm_tc2<64, 4, 2>(ctx, cls, X, W, w_rows, M, N, K, slices, epi);
    if (two && ctas(128) <= 148) return launch_gemm_tc2<128, 4, 2>(ctx, cls, X, W, w_rows, M, N, K, slices, epi);
    if (!two && ctas(64) <= 296) return launch_gemm_tc2<64, 5, 1>(ctx, cls, X, W, w_rows, M, N, K, slices, epi);
    if (ctas(128) <= 296) return launch_gemm_tc2<128, 4, 1>(ctx, cls, X, W, w_rows, M, N, K, slices, epi);
    if (ctas(128) <= 444) return launch_gemm_tc2<128, 3, 1>(ctx, cls, X, W, w_rows, M, N, K, slices, epi);
    return launch_gemm_tc2p(ctx, cls, X, W, w_rows, M, N, K, epi);
  }
  // token tile: as narrow as the token count allows for weight streaming; 256 where that still gives every SM a CTA pair
  int tn = M <= 16 ? 16 : M <= 32 ? 32 : M <= 64 ? 64 : M <= 1024 ? 128 : 256;
  if (tn == 256 && ntiles_n * ((M + 255) / 256) * batches < 200) tn = 128;
  const int tiles = ((N + kGemmRowsW - 1) / kGemmRowsW) * ((M + tn - 1) / tn) * batches;
  const int ksplit = gemm_ksplit(tiles, K / kGemmBK, tn);
  switch (tn) {
    case 16: return launch_gemm_tc<16>(ctx, cls, X, W, w_rows, M, N, K, batches, x_z, w_z, ksplit, epi);
    case 32: return launch_gemm_tc<32>(ctx, cls, X, W, w_rows, M, N, K, batches, x_z, w_z, ksplit, epi);
    case 64: return launch_gemm_tc<64>(ctx, cls, X, W, w_rows, M, N, K, batches, x_z, w_z, ksplit, epi);
    case 128: return launch_gemm_tc<128>(ctx, cls, X, W, w_rows, M, N, K, batches, x_z, w_z, ksplit, epi);
    default: return launch_gemm_tc<256>(ctx, cls, X, W, w_rows, M, N, K, batches, x_z, w_z, ksplit, epi);
  }
}

// Product dispatch by model type: fp32 models use plain FMA arithmetic, bf16 models the
// tensor cores (K must be a multiple of 64 there, else the FMA kernel serves).
template <typename T, typename Epi>
vadusa_status product(vadusa_ctx* ctx, int cls, const T* X, const T* W, int w_rows, int M, int N, int K, int batches,
                      long long x_z, long long w_z, const Epi& epi) {
  if constexpr (std::is_same<T, bf16>::value) {
    if (K % kGemmBK == 0) return gemm_tc(ctx, cls, X, W, w_rows, M, N, K, batches, x_z, w_z, epi);
  }
  return gemm<T>(ctx, cls, X, W, M, N, K, batches, x_z, w_z, epi);
}

// LayerNorm followed by a product, in one kernel where the shape allows (few tokens; bf16: from the statistics that the
// producer of x left).
template <typename T, typename Epi>
bool ln_product(vadusa_ctx* ctx, int cls, const float* x, const float* g, const float* b, const T* W, int w_rows, int M,
                int N, int K, const Epi& epi, vadusa_status* st, T* y = nullptr) {
  if constexpr (std::is_same<T, bf16>::value) return gemm_tc_ln(ctx, cls, x, g, b, W, w_rows, M, N, K, epi, st, y);
  if constexpr (std::is_same<T, float>::value) {
    if (M > kFewTokens || K > kFewNormK) return false;
    const RowNorm rn{g, b, y, ctx->cfg.ln_eps};
    *st = gemm<float>(ctx, cls, x, W, M, N, K, 1, 0, 0, epi, &rn);
    return true;
  }
  return false;
}

// KV splits of the tensor-core attention: enough CTAs for about two per SM even at batch 1, but no more than four
// per (head, sequence) while the contexts are short (a 16-head pass over 400-1100 tokens: 64 CTAs of two to five
// pages leave SMs to the next kernel's early CTAs and their weight loads, 128 CTAs of one or two pages do not;
// 0.538 -> 0.528 ms per step).  The estimate of the context is the host's lower one: never behind by more than
// the tokens accepted beyond one per iteration since the last exact value.
// (Ragged batches are balanced by visiting the sequences longest first, see tree_embed_kernel.)
constexpr long long kAttLongContext = 1536;
int attention_splits(const vadusa_ctx* ctx, int n_nodes) {
  int splits = 1;
  const int ntile = (n_nodes + 63) / 64;                 // CTAs per (head, sequence): one per 64 nodes
  const int cap = ctx->ctx_lo + n_nodes > kAttLongContext ? 8 : 4;
  while (splits < cap && ctx->cfg.n_heads * ctx->batch * ntile * splits * 2 <= 296) splits *= 2;
  return splits;
}

// Batches whose (head, sequence) items alone fill the device go through the persistent page-stream kernel.
bool attention_streams(const vadusa_ctx* ctx, int n_nodes) {
  const vadusa_config& c = ctx->cfg;
  return ctx->att_stream && c.dtype == 1 && c.d_model / c.n_heads == 64 && n_nodes <= 64 && ctx->batch <= kAsMaxBatch &&
         attention_splits(ctx, n_nodes) == 1 && (long long)c.max_blocks_per_seq * kKvBlock < (1ll << 24);
}

template <typename T>
vadusa_status attention(vadusa_ctx* ctx, const T* q, const T* pool, const TreeView& tv, T* out) {
  const vadusa_config& c = ctx->cfg;
  const int dh = c.d_model / c.n_heads;
  const KvGeom g = geom_of(ctx);
  const float scale = (float)(1.0 / sqrt((double)dh));
  const int ntile = (tv.n_nodes + 63) / 64;
  // four nodes per block while that makes at most four blocks per SM, else eight
  const int ng = c.n_heads * ctx->batch * ((tv.n_nodes + 3) / 4) <= 4 * 148 ? 4 : 8;
  auto go = [&](auto kern) -> vadusa_status {
    PROF(ctx, K_ATTENTION);
    CU(launch_dependent(ctx, kern, dim3(c.n_heads, ctx->batch, (tv.n_nodes + ng - 1) / ng), 256, att_simt_smem(dh), q, pool, ctx->block_table,
                        (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.ctx_len), (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.nvalid),
                        tv, g, c.d_model, scale, ctx->in_prefill ? 0 : 1, out, err_word(ctx)));
    LAUNCH_CHECK();
    return VADUSA_OK;
  };
  if constexpr (std::is_same<T, bf16>::value) {
    if (dh == 64) {
      if (ctx->pf_tiles > 0 && tv.n_nodes == 64) {
        // prefill pass: two consecutive chunks of a sequence per CTA (128 query rows per K/V page fetched)
        const CUtensorMap *mq, *mkv;
        const int M = ctx->batch * tv.n_nodes;
        if (vadusa_status s = tensor_map(ctx, q, M, c.d_model, 64, 1, 0, &mq)) return s;
        const long long rows = (long long)c.kv_num_blocks * 2 * c.n_heads * kKvBlock;
        if (rows > 0x7fffffffLL) return fail(ctx, VADUSA_EINVAL, "KV pool too large for one tensor map");
        if (vadusa_status s = tensor_map(ctx, c.kv_pool, (int)rows, 64, 64, c.n_layers, g.layer_stride, &mkv)) return s;
        const int layer = (int)((reinterpret_cast<const char*>(pool) - reinterpret_cast<const char*>(c.kv_pool)) /
                                (g.layer_stride * (long long)sizeof(bf16)));
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3(c.n_heads, ctx->pf_tiles, 1);
        lc.blockDim = dim3(kPfThreads);
        lc.dynamicSmemBytes = kAttSmemBytes;
        lc.stream = ctx->stream;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        lc.attrs = at; lc.numAttrs = 1;
        PROF(ctx, K_ATTENTION);
        CU(cudaLaunchKernelEx(&lc, prefill_attention_tc_kernel, *mq, *mkv, layer, ctx->block_table,
                              (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.ctx_len),
                              (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.nvalid),
                              ctx->pf_pairs, g, c.d_model,
                              scale * 1.4426950408889634f, reinterpret_cast<bf16*>(out), err_word(ctx)));
        LAUNCH_CHECK();
        return VADUSA_OK;
      }
      // tensor-core kernel; KV splits so that about two CTAs per SM exist even at batch 1
      const int splits = attention_splits(ctx, tv.n_nodes);
      const CUtensorMap *mq, *mkv;
      const int M = ctx->batch * tv.n_nodes;
      if (vadusa_status s = tensor_map(ctx, q, M, c.d_model, 64, 1, 0, &mq)) return s;
      const long long rows = (long long)c.kv_num_blocks * 2 * c.n_heads * kKvBlock;
      if (rows > 0x7fffffffLL) return fail(ctx, VADUSA_EINVAL, "KV pool too large for one tensor map");
      if (vadusa_status s = tensor_map(ctx, c.kv_pool, (int)rows, 64, 64, c.n_layers, g.layer_stride, &mkv)) return s;
      const int layer = (int)((reinterpret_cast<const char*>(pool) - reinterpret_cast<const char*>(c.kv_pool)) /
                              (g.layer_stride * (long long)sizeof(bf16)));
      if (attention_streams(ctx, tv.n_nodes)) {
        // batches: every CTA takes an equal share of the stream of K/V pages of all (sequence, head) items
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3(kAsGrid);
        lc.blockDim = dim3(kAsThreads);
        lc.dynamicSmemBytes = kAsSmemBytes;
        lc.stream = ctx->stream;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        lc.attrs = at; lc.numAttrs = 1;
        PROF(ctx, K_ATTENTION);
        CU(cudaLaunchKernelEx(&lc, tree_attention_stream_kernel, *mq, *mkv, layer, ctx->block_table,
                              (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.ctx_len),
                              (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.nvalid), tv, g, ctx->batch, c.d_model,
                              scale * 1.4426950408889634f, reinterpret_cast<bf16*>(out),
                              wsptr<float>(ctx, ctx->ws.att_xch), wsptr<uint32_t>(ctx, ctx->ws.att_cnt), err_word(ctx)));
        LAUNCH_CHECK();
        return VADUSA_OK;
      }
      cudaLaunchConfig_t lc = {};
      lc.gridDim = dim3(c.n_heads, ctx->batch * ntile, splits);
      lc.blockDim = dim3(kAttThreads);
      lc.dynamicSmemBytes = kAttSmemBytes;
      lc.stream = ctx->stream;
      cudaLaunchAttribute at[2];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = 1; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = splits;
      at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      at[1].val.programmaticStreamSerializationAllowed = 1;
      lc.attrs = at; lc.numAttrs = 2;
      PROF(ctx, K_ATTENTION);
      CU(cudaLaunchKernelEx(&lc, tree_attention_tc_kernel, *mq, *mkv, layer, ctx->block_table,
                            (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.ctx_len),
                            (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.nvalid),
                            (const int32_t*)(ctx->batch > 1 ? wsptr<int32_t>(ctx, ctx->ws.seq_order) : nullptr), tv, g, c.d_model,
                            scale * 1.4426950408889634f, splits, ctx->in_prefill ? 0 : 1, reinterpret_cast<bf16*>(out),
                            wsptr<float>(ctx, ctx->ws.att_xch), err_word(ctx)));
      LAUNCH_CHECK();
      return VADUSA_OK;
    }
  }
  if constexpr (!std::is_same<T, bf16>::value) {
    if (dh == 64) return ng == 4 ? go(tree_attention_simt_kernel<T, 64, 4>) : go(tree_attention_simt_kernel<T, 64, 8>);
  }
  return ng == 4 ? go(tree_attention_simt_kernel<T, 32, 4>) : go(tree_attention_simt_kernel<T, 32, 8>);
}

template <typename T>
vadusa_status layernorm(vadusa_ctx* ctx, const float* x, const float* g, const float* b, T* y, int rows) {
  const int d = ctx->cfg.d_model;
  const bool by_warp = rows >= 64 && d % 128 == 0 && d <= 2048;   // many rows: one warp per row
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(by_warp ? (rows + 3) / 4 : rows);
  lc.blockDim = dim3(by_warp ? 128 : 256);
  lc.stream = ctx->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;       // the kernel calls griddepcontrol.wait
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at; lc.numAttrs = 1;
  PROF(ctx, K_LAYERNORM);
  if (by_warp) CU(cudaLaunchKernelEx(&lc, layernorm_rows_kernel<T>, x, g, b, y, rows, d, ctx->cfg.ln_eps));
  else CU(cudaLaunchKernelEx(&lc, layernorm_kernel<T>, x, g, b, y, rows, d, ctx->cfg.ln_eps));
  LAUNCH_CHECK();
  return VADUSA_OK;
}

// Can this pass run as the single persistent kernel?  One sequence of at most 64 nodes, bf16, head_dim 64,
// 8 or 16 heads (one cluster per head), feed-forward width in whole 128-row blocks per cluster (at most two),
// and a device that holds all clusters at once (asked when the kernel is first wanted).
bool fused_shape_ok(const vadusa_ctx* ctx, const TreeView& tv) {
  const vadusa_config& c = ctx->cfg;
  if (!ctx->fused_enabled || c.dtype != 1 || ctx->batch != 1 || tv.n_nodes > 64) return false;
  const int H = c.n_heads, d = c.d_model, F = c.d_ffn;
  if (d != 64 * H || (H != 8 && H != 16)) return false;
  if (F % (128 * H) || F / H > 256) return false;
  if ((ctx->ctx_bound + 64) / kKvBlock / 6 + 1 > kFfMaxPages) return false;
  if (c.n_layers > 1) {
    // the per-layer tensors must repeat at a constant stride (they do in the blob this library lays out)
    const long long st = find(ctx, "l1.wqkv")->offset - find(ctx, "l0.wqkv")->offset;
    if (st % 16) return false;
  }
  return true;
}

template <int CS>
vadusa_status fused_launch(vadusa_ctx* ctx, bool query_only, int* clusters, const CUtensorMap* const* maps, const FusedArgs* a) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(CS * ctx->cfg.n_heads);
  lc.blockDim = dim3(kFfThreads);
  lc.dynamicSmemBytes = FfCfg<CS>::kSmemBytes;
  lc.stream = ctx->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  if (query_only) {
    lc.numAttrs = 1;
    CU(cudaFuncSetAttribute(fused_forward_kernel<CS>, cudaFuncAttributeMaxDynamicSharedMemorySize, FfCfg<CS>::kSmemBytes));
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fused_forward_kernel<CS>, &lc) != cudaSuccess) { cudaGetLastError(); n = 0; }
    *clusters = n;
    return VADUSA_OK;
  }
  lc.numAttrs = 2;
  PROF(ctx, K_FUSED);
  CU(cudaLaunchKernelEx(&lc, fused_forward_kernel<CS>, *maps[0], *maps[1], *maps[2], *maps[3], *maps[4], *maps[5], *maps[6], *maps[7], *a));
  LAUNCH_CHECK();
  return VADUSA_OK;
}

vadusa_status fused_forward(vadusa_ctx* ctx, const TreeView& tv, const int32_t* override_tokens, bf16* attn_tap, bool* launched) {
  *launched = false;
  const vadusa_config& c = ctx->cfg;
  const int H = c.n_heads, d = c.d_model, F = c.d_ffn, L = c.n_layers, M = tv.n_nodes, vp = vpad(&c);
  if (ctx->fused_cs < 0) {
    // clusters of 8 where the device holds one per head at once, else clusters of 6
    int n8 = 0, n6 = 0;
    if (vadusa_status s = fused_launch<8>(ctx, true, &n8, nullptr, nullptr)) return s;
    if (vadusa_status s = fused_launch<6>(ctx, true, &n6, nullptr, nullptr)) return s;
    ctx->fused_cs = n8 >= H ? 8 : n6 >= H ? 6 : 0;
    ctx->fused_clusters = ctx->fused_cs == 8 ? n8 : n6;
    ctx->fused_n8 = n8; ctx->fused_n6 = n6;
  }
  int cs = ctx->fused_cs;
  if (ctx->fused_enabled == 8 && ctx->fused_n8 >= H) cs = 8;
  if (ctx->fused_enabled == 6 && ctx->fused_n6 >= H) cs = 6;
  if (cs == 0) return VADUSA_OK;                            // not all clusters fit at once: the caller takes the other path
  const long long lstride = L > 1 ? find(ctx, "l1.wqkv")->offset - find(ctx, "l0.wqkv")->offset : 0;
  const LayerW& w0 = ctx->layers[0];
  const KvGeom g = geom_of(ctx);
  const CUtensorMap* maps[8];
  if (vadusa_status s = tensor_map(ctx, w0.wqkv, 3 * d, d, 64, L, lstride / 2, &maps[0])) return s;
  if (vadusa_status s = tensor_map(ctx, w0.wo, d, d, 64, L, lstride / 2, &maps[1])) return s;
  if (vadusa_status s = tensor_map(ctx, w0.w1, F, d, 128, L, lstride / 2, &maps[2])) return s;
  if (vadusa_status s = tensor_map(ctx, w0.w2, d, F, 64, L, lstride / 2, &maps[3])) return s;
  if (vadusa_status s = tensor_map(ctx, ctx->lm, vp, d, 128, 1, 0, &maps[4])) return s;
  if (vadusa_status s = tensor_map(ctx, ctx->wsp + ctx->ws.o, M, d, 64, 1, 0, &maps[5])) return s;
  if (vadusa_status s = tensor_map(ctx, ctx->wsp + ctx->ws.mid, M, F, 64, 1, 0, &maps[6])) return s;
  const long long rows = (long long)c.kv_num_blocks * 2 * c.n_heads * kKvBlock;
  if (rows > 0x7fffffffLL) return fail(ctx, VADUSA_EINVAL, "KV pool too large for one tensor map");
  if (vadusa_status s = tensor_map(ctx, c.kv_pool, (int)rows, 64, 64, c.n_layers, g.layer_stride, &maps[7])) return s;
  FusedArgs a;
  memset(&a, 0, sizeof(a));
  a.L = L; a.d = d; a.H = H; a.F = F; a.vocab = c.vocab; a.vpad = vp; a.n_phonemes = c.n_phonemes; a.max_pos = c.max_pos; a.M = M;
  a.eps = c.ln_eps;
  a.scale_log2e = (float)(1.0 / sqrt(64.0)) * 1.4426950408889634f;
  a.ln1_g = w0.ln1_g; a.ln1_b = w0.ln1_b; a.bqkv = w0.bqkv; a.bo = w0.bo; a.ln2_g = w0.ln2_g; a.ln2_b = w0.ln2_b;
  a.b1 = w0.b1; a.b2 = w0.b2;
  a.layer_stride = lstride;
  a.lnf_g = ctx->lnf_g; a.lnf_b = ctx->lnf_b;
  a.emb_audio = as<bf16>(ctx->emb_audio); a.emb_phon = as<bf16>(ctx->emb_phon); a.pos = as<bf16>(ctx->pos);
  a.xa = wsptr<float>(ctx, ctx->ws.x); a.xb = wsptr<float>(ctx, ctx->ws.f_xb);
  a.stats_a = wsptr<float2>(ctx, ctx->ws.f_stats_a); a.stats_b = wsptr<float2>(ctx, ctx->ws.f_stats_b);
  a.o = wsptr<bf16>(ctx, ctx->ws.o); a.mid = wsptr<bf16>(ctx, ctx->ws.mid); a.hfinal = wsptr<bf16>(ctx, ctx->ws.hfinal);
  a.logits = wsptr<float>(ctx, ctx->ws.logits);
  a.attn_tap = attn_tap;
  a.tokens = wsptr<int32_t>(ctx, ctx->ws.tokens);
  a.kv_row = wsptr<long long>(ctx, ctx->ws.kv_row);
  a.override_tokens = override_tokens;
  a.root = wsptr<int32_t>(ctx, ctx->ws.root); a.topk = wsptr<int32_t>(ctx, ctx->ws.topk);
  a.n_draft_heads = c.n_draft_heads; a.draft_topk = c.draft_topk;
  a.ctx_len = wsptr<int32_t>(ctx, ctx->ws.ctx_len); a.nvalid = wsptr<int32_t>(ctx, ctx->ws.nvalid);
  a.block_table = ctx->block_table;
  a.tree = tv; a.geom = g;
  a.kv_pool = reinterpret_cast<bf16*>(c.kv_pool);
  a.sync = wsptr<uint32_t>(ctx, ctx->ws.f_sync);
  a.err = err_word(ctx);
  vadusa_status s = cs == 8 ? fused_launch<8>(ctx, false, nullptr, maps, &a) : fused_launch<6>(ctx, false, nullptr, maps, &a);
  if (s) return s;
  *launched = true;
  return VADUSA_OK;
}

// Tokens and embeddings of all tree nodes, and the order in which attention visits the sequences.
template <typename T>
vadusa_status embed(vadusa_ctx* ctx, const TreeView& tv, const int32_t* override_tokens, long long* kv_row, float2* stats) {
  const vadusa_config& c = ctx->cfg;
  const int M = ctx->batch * tv.n_nodes;
  const bool ordered = ctx->batch > 1;
  PROF(ctx, K_EMBED);
  CU(launch_dependent(ctx, tree_embed_kernel<T>, dim3(M + (ordered ? 1 : 0)), 128, 0, tv, override_tokens,
                      (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.root), (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.topk),
                      c.n_draft_heads, c.draft_topk, (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.ctx_len),
                      (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.nvalid), as<T>(ctx->emb_audio), as<T>(ctx->emb_phon),
                      as<T>(ctx->pos), c.vocab, c.n_phonemes, c.max_pos, c.d_model, wsptr<int32_t>(ctx, ctx->ws.tokens),
                      wsptr<float>(ctx, ctx->ws.x), ctx->block_table, geom_of(ctx), kv_row, stats, M,
                      ordered ? wsptr<int32_t>(ctx, ctx->ws.seq_order) : (int32_t*)nullptr, err_word(ctx)));
  LAUNCH_CHECK();
  return VADUSA_OK;
}

// The rows of a prefill pass that the last layer is needed for: the last token of every prefix that ends in the pass.
struct PrefillTail {
  int rows;                  // 0: no prefix ends here
  int tiles;                 // attention tiles that hold these rows
  const int2* pairs;
  const int32_t* m;          // device [rows]: row of the pass
};

// Everything behind the last layer's q/k/v product for those rows alone: the other rows of that layer only leave K/V behind.
// (One layer of twelve and the vocabulary head for a few rows: a tenth of a long prefill's work.)
template <typename T>
vadusa_status prefill_tail(vadusa_ctx* ctx, const TreeView& tv, const PrefillTail& t, const T* pool) {
  const vadusa_config& c = ctx->cfg;
  const int d = c.d_model, f = c.d_ffn, vp = vpad(&c), n = t.rows;
  if (n == 0) return VADUSA_OK;
  const LayerW& w = ctx->layers[c.n_layers - 1];
  float* xg = wsptr<float>(ctx, ctx->ws.q);               // (q is free once attention has run)
  T *a = wsptr<T>(ctx, ctx->ws.a), *o = wsptr<T>(ctx, ctx->ws.o), *mid = wsptr<T>(ctx, ctx->ws.mid), *hf = wsptr<T>(ctx, ctx->ws.hfinal);
  if (ctx->pf_tiles > 0) { ctx->pf_tiles = t.tiles; ctx->pf_pairs = t.pairs; }
  if (vadusa_status s = attention<T>(ctx, wsptr<T>(ctx, ctx->ws.q), pool, tv, o)) return s;
  CU(launch_dependent(ctx, prefill_pick_kernel<T>, dim3(n), 128, 0, t.m, (const T*)o, (const float*)wsptr<float>(ctx, ctx->ws.x), d, a, xg));
  LAUNCH_CHECK();
  vadusa_status s = product<T>(ctx, K_GEMM_OUT, a, as<T>(w.wo), d, n, d, d, 1, 0, 0, EpiResidual{w.bo, xg, d});
  if (s) return s;
  const EpiRelu<T> e1{w.b1, mid, f};
  bool fused = std::is_same<T, float>::value && ln_product<T>(ctx, K_GEMM_FFN1, xg, w.ln2_g, w.ln2_b, as<T>(w.w1), f, n, f, d, e1, &s);
  if (!fused) {
    if ((s = layernorm<T>(ctx, xg, w.ln2_g, w.ln2_b, o, n))) return s;
    s = product<T>(ctx, K_GEMM_FFN1, o, as<T>(w.w1), f, n, f, d, 1, 0, 0, e1);
  }
  if (s) return s;
  if ((s = product<T>(ctx, K_GEMM_FFN2, mid, as<T>(w.w2), d, n, d, f, 1, 0, 0, EpiResidual{w.b2, xg, d}))) return s;
  if ((s = layernorm<T>(ctx, xg, ctx->lnf_g, ctx->lnf_b, hf, n))) return s;
  return product<T>(ctx, K_GEMM_LM, hf, as<T>(ctx->lm), vp, n, vp, d, 1, 0, 0, EpiLogits{wsptr<float>(ctx, ctx->ws.logits), vp, 0});
}

// One forward pass of the base model over batch * tv.n_nodes rows (verify step; with `tail` a prefill pass).
template <typename T>
vadusa_status forward(vadusa_ctx* ctx, const TreeView& tv, const int32_t* override_tokens, T* attn_tap,
                      const PrefillTail* tail = nullptr) {
  const vadusa_config& c = ctx->cfg;
  const int B = ctx->batch, N = tv.n_nodes, M = B * N, d = c.d_model, f = c.d_ffn, vp = vpad(&c);
  const KvGeom g = geom_of(ctx);
  if constexpr (std::is_same<T, bf16>::value) {
    if (fused_shape_ok(ctx, tv)) {
      bool launched = false;
      if (vadusa_status s = fused_forward(ctx, tv, override_tokens, attn_tap, &launched)) return s;
      if (launched) return VADUSA_OK;
    }
  }
  float* x = wsptr<float>(ctx, ctx->ws.x);
  T* a = wsptr<T>(ctx, ctx->ws.a);
  T* q = wsptr<T>(ctx, ctx->ws.q);
  T* o = wsptr<T>(ctx, ctx->ws.o);
  T* mid = wsptr<T>(ctx, ctx->ws.mid);
  T* hfinal = wsptr<T>(ctx, ctx->ws.hfinal);
  float* logits = wsptr<float>(ctx, ctx->ws.logits);

  // LayerNorm statistics for the products that normalise their own operand (bf16 models, few tokens): left by
  // the embedding kernel and by the residual products
  const bool tc = std::is_same<T, bf16>::value;
  const bool embed_stats = tc && M <= 64 && d % 128 == 0 && d / 128 <= 8;
  const bool stats_out = tc && residual_leaves_stats(M, d, d), stats_ffn = tc && residual_leaves_stats(M, d, f);
  float2* stats = wsptr<float2>(ctx, ctx->ws.ln_stats);
  if (vadusa_status s = embed<T>(ctx, tv, override_tokens, wsptr<long long>(ctx, ctx->ws.kv_row), embed_stats ? stats : nullptr)) return s;
  bool have_stats = embed_stats || !tc;                    // (fp32 models need none)
  for (int l = 0; l < c.n_layers; ++l) {
    const LayerW& w = ctx->layers[l];
    T* pool = reinterpret_cast<T*>(c.kv_pool) + (long long)l * g.layer_stride;
    vadusa_status s = VADUSA_OK;
    EpiQKV<T> eq{w.bqkv, q, pool, wsptr<long long>(ctx, ctx->ws.kv_row), (long long)c.n_heads * kKvBlock * g.head_dim,
                 kKvBlock * g.head_dim, g.head_dim, d};
    if (!(have_stats && ln_product<T>(ctx, K_GEMM_QKV, x, w.ln1_g, w.ln1_b, as<T>(w.wqkv), 3 * d, M, 3 * d, d, eq, &s))) {
      s = layernorm<T>(ctx, x, w.ln1_g, w.ln1_b, a, M);
      if (s) return s;
      s = product<T>(ctx, K_GEMM_QKV, a, as<T>(w.wqkv), 3 * d, M, 3 * d, d, 1, 0, 0, eq);
    }
    if (s) return s;
    if (tail && l == c.n_layers - 1) return prefill_tail<T>(ctx, tv, *tail, pool);
    s = attention<T>(ctx, q, pool, tv, o);
    if (s) return s;
    if (attn_tap)
      CU(cudaMemcpyAsync(attn_tap + (long long)l * M * d, o, (size_t)M * d * sizeof(T), cudaMemcpyDeviceToDevice, ctx->stream));
    if (stats_out) {
      EpiResidualStats eo{w.bo, x, d, stats};
      s = product<T>(ctx, K_GEMM_OUT, o, as<T>(w.wo), d, M, d, d, 1, 0, 0, eo);
      have_stats = true;
    } else {
      EpiResidual eo{w.bo, x, d};
      s = product<T>(ctx, K_GEMM_OUT, o, as<T>(w.wo), d, M, d, d, 1, 0, 0, eo);
    }
    if (s) return s;
    EpiRelu<T> e1{w.b1, mid, f};
    if (!(have_stats && ln_product<T>(ctx, K_GEMM_FFN1, x, w.ln2_g, w.ln2_b, as<T>(w.w1), f, M, f, d, e1, &s))) {
      s = layernorm<T>(ctx, x, w.ln2_g, w.ln2_b, a, M);
      if (s) return s;
      s = product<T>(ctx, K_GEMM_FFN1, a, as<T>(w.w1), f, M, f, d, 1, 0, 0, e1);
    }
    if (s) return s;
    if (stats_ffn) {
      EpiResidualStats e2{w.b2, x, d, stats};
      s = product<T>(ctx, K_GEMM_FFN2, mid, as<T>(w.w2), d, M, d, f, 1, 0, 0, e2);
    } else {
      EpiResidual e2{w.b2, x, d};
      s = product<T>(ctx, K_GEMM_FFN2, mid, as<T>(w.w2), d, M, d, f, 1, 0, 0, e2);
    }
    have_stats = stats_ffn || !tc;
    if (s) return s;
  }
  EpiLogits el{logits, vp, 0};
  vadusa_status s = VADUSA_OK;
  // the final LayerNorm folds into the vocabulary head, which also stores the normalised rows (the draft heads
  // and the carried state read them)
  if (have_stats && ln_product<T>(ctx, K_GEMM_LM, x, ctx->lnf_g, ctx->lnf_b, as<T>(ctx->lm), vp, M, vp, d, el, &s, hfinal))
    return s;
  if ((s = layernorm<T>(ctx, x, ctx->lnf_g, ctx->lnf_b, hfinal, M))) return s;
  return product<T>(ctx, K_GEMM_LM, hfinal, as<T>(ctx->lm), vp, M, vp, d, 1, 0, 0, el);
}

template <typename T>
vadusa_status draft(vadusa_ctx* ctx, const SamplingDev& sp) {
  const vadusa_config& c = ctx->cfg;
  const int B = ctx->batch, d = c.d_model, vp = vpad(&c), hd = c.n_draft_heads;
  const T* hstar = wsptr<T>(ctx, ctx->ws.hstar);
  T* z = wsptr<T>(ctx, ctx->ws.z);
  float* dl = wsptr<float>(ctx, ctx->ws.dlogits);
  const long long w_stride = ctx->dw_stride / (long long)sizeof(T), u_stride = ctx->du_stride / (long long)sizeof(T);
  if (hd > 1 && w_stride != (long long)d * d) return fail(ctx, VADUSA_EINVAL, "draft matrices are not contiguous");
  EpiDraftHiddenFlat<T> eh{ctx->db, hstar, z, d, B};
  vadusa_status s = product<T>(ctx, K_DRAFT_HIDDEN, hstar, as<T>(ctx->dw), hd * d, B, hd * d, d, 1, 0, 0, eh);
  if (s) return s;
  EpiLogits el{dl, vp, (long long)B * vp};
  s = product<T>(ctx, K_DRAFT_LOGITS, z, as<T>(ctx->du), vp, B, vp, d, hd, (long long)B * d, u_stride, el);
  if (s) return s;
  dim3 grid(hd + 1, B);
  PROF(ctx, K_DRAFT_SELECT);
  CU(launch_dependent(ctx, draft_select_kernel, grid, select_threads(c.vocab), row_keys_smem(vp, sp), (const float*)dl,
                      (const float*)wsptr<float>(ctx, ctx->ws.logits_star), vp, c.vocab, B, hd, c.draft_topk,
                      (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.ctx_len), (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.nvalid),
                      sp, wsptr<int32_t>(ctx, ctx->ws.topk), wsptr<int32_t>(ctx, ctx->ws.root)));
  LAUNCH_CHECK();
  return VADUSA_OK;
}

// tokens = tree built from the draft (no model pass): used when the caller wants them.
template <typename T>
vadusa_status accept_commit(vadusa_ctx* ctx, const SamplingDev& sp, const int32_t* forced, const AcceptOut& out,
                            int32_t* out_tokens, int out_cap, int target, int32_t* progress = nullptr) {
  const vadusa_config& c = ctx->cfg;
  const int B = ctx->batch, vp = vpad(&c);
  const KvGeom g = geom_of(ctx);
  const TreeView tv = tree_of(ctx, false);
  SeqState st = state_of(ctx, out_tokens, out_cap, target);
  st.progress = progress;
  PROF(ctx, K_ACCEPT);
  // the next root is wanted and the device holds a block per node at once: every node's first draw along with the rest
  const bool tops = out.next_root && sp.accept_rule == 0 && tv.n_nodes * B <= 2 * 148;
  const int draw_smem = out.next_root && !tops ? (int)row_keys_smem(vp, sp) : 0;
  CU(launch_dependent(ctx, accept_kernel, dim3(tops ? tv.n_nodes : ctx->tree_inner, B), accept_threads(c.vocab, tv.n_nodes * B), row_keys_smem(vp, sp),
                      (const float*)wsptr<float>(ctx, ctx->ws.logits), vp, c.vocab,
                      (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.tokens), tv,
                      (const int32_t*)(tops ? nullptr : wsptr<int32_t>(ctx, ctx->ws.tree) + 3ll * ctx->tree_copies * tv.n_nodes), sp, st));
  LAUNCH_CHECK();
  PROF(ctx, K_COMMIT);
  CU(launch_dependent(ctx, commit_kernel<T>, dim3(c.n_layers + (vp + kCommitLogits - 1) / kCommitLogits + 1, B),
                      draw_smem ? select_threads(c.vocab) : 256, draw_smem, reinterpret_cast<T*>(c.kv_pool), g, ctx->block_table, st,
                      c.n_layers, tv, (const int32_t*)wsptr<int32_t>(ctx, ctx->ws.tokens), sp, forced, tops ? 1 : 0, out,
                      (const T*)wsptr<T>(ctx, ctx->ws.hfinal), c.d_model, (const float*)wsptr<float>(ctx, ctx->ws.logits), vp,
                      c.vocab, wsptr<T>(ctx, ctx->ws.hstar), wsptr<float>(ctx, ctx->ws.logits_star), err_word(ctx)));
  LAUNCH_CHECK();
  return VADUSA_OK;
}

// While alive, the model's passes see `rows` rows described by the given arrays instead of the batch.
struct RowsView {
  vadusa_ctx* c;
  int batch; const int32_t* table; int64_t ctx_len, nvalid;
  RowsView(vadusa_ctx* ctx, int rows, const int32_t* block_table, int64_t ctx_len_off, int64_t nvalid_off)
      : c(ctx), batch(ctx->batch), table(ctx->block_table), ctx_len(ctx->ws.ctx_len), nvalid(ctx->ws.nvalid) {
    ctx->batch = rows; ctx->block_table = block_table; ctx->ws.ctx_len = ctx_len_off; ctx->ws.nvalid = nvalid_off;
  }
  ~RowsView() { c->batch = batch; c->block_table = table; c->ws.ctx_len = ctx_len; c->ws.nvalid = nvalid; }
};

// A prefill pass's arrays in ws.pf_stage, packed behind one another so that one copy brings them.
struct PassArrays {
  int rows, n_nodes;
  size_t pairs() const { return 0; }                            // int2: rows that share an attention CTA (y < 0: a single chunk)
  size_t tail_pairs() const { return (size_t)rows * 8; }        // int2: those of them that hold the end of a prefix
  size_t word(int i) const { return (size_t)rows * (16 + 4 * i); }
  size_t ctx() const { return word(0); }                        // int32: tokens before the chunk
  size_t nvalid() const { return word(1); }                     // its length
  size_t seq() const { return word(2); }                        // its sequence
  size_t tail_m() const { return word(3); }                     // [tail]: row of a prefix's last token,
  size_t tail_seq() const { return word(4); }                   //         its sequence,
  size_t tail_len() const { return word(5); }                   //         and the sequence's new length
  size_t tokens() const { return word(6); }                     // int32 [rows][n_nodes]
  size_t total() const { return tokens() + (size_t)rows * n_nodes * 4; }
};

template <typename T>
vadusa_status prefill(vadusa_ctx* ctx, const int32_t* h_tokens, const int32_t* h_len, int stride) {
  const vadusa_config& c = ctx->cfg;
  const int B = ctx->batch, N = c.max_tree_nodes, vp = vpad(&c), R = pass_rows(&c);
  int longest = 0;
  for (int b = 0; b < B; ++b) {
    if (h_len[b] < 1 || h_len[b] > stride) return fail(ctx, VADUSA_EINVAL, "prefix length of sequence %d out of range", b);
    if (ctx->pf_tap && h_len[b] > ctx->pf_tap_stride) return fail(ctx, VADUSA_EINVAL, "prefill tap: row stride shorter than the prefix");
    longest = h_len[b] > longest ? h_len[b] : longest;
  }
  // what the cache holds already
  if (!ctx->h_ctx_exact) {
    ctx->h_ctx.resize(B);
    CU(cudaMemcpyAsync(ctx->h_ctx.data(), ctx->wsp + ctx->ws.ctx_len, B * sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
    CU(cudaStreamSynchronize(ctx->stream));
    ctx->h_ctx_exact = true;
  }
  // chunks in sequence order, so that a chunk never precedes an earlier chunk of its sequence
  struct Chunk { int b, s0, n, last; };
  std::vector<Chunk> chunks;
  for (int b = 0; b < B; ++b)
    for (int s0 = 0; s0 < h_len[b]; s0 += N) {
      const int n = h_len[b] - s0 < N ? h_len[b] - s0 : N;
      chunks.push_back({b, s0, n, s0 + n == h_len[b] ? b : -1});
    }
  int32_t* d_table = wsptr<int32_t>(ctx, ctx->ws.pf_block_table);
  int32_t* real_ctx_len = wsptr<int32_t>(ctx, ctx->ws.ctx_len);
  const int32_t* real_table = ctx->block_table;
  std::vector<char> pack;
  const TreeView tv = tree_of(ctx, true);
  for (size_t c0 = 0; c0 < chunks.size(); c0 += R) {
    const int rows = (int)(chunks.size() - c0 < (size_t)R ? chunks.size() - c0 : R);
    const PassArrays pa{rows, N};
    pack.assign(pa.total(), 0);
    auto at = [&](size_t off) { return reinterpret_cast<int32_t*>(pack.data() + off); };
    int ends = 0;
    for (int r = 0; r < rows; ++r) {
      const Chunk& ch = chunks[c0 + r];
      at(pa.ctx())[r] = ctx->h_ctx[ch.b] + ch.s0; at(pa.nvalid())[r] = ch.n; at(pa.seq())[r] = ch.b;
      if (ch.last >= 0) {
        at(pa.tail_m())[ends] = r * N + ch.n - 1; at(pa.tail_seq())[ends] = ch.b;
        at(pa.tail_len())[ends] = ctx->h_ctx[ch.b] + ch.s0 + ch.n;
        ++ends;
      }
      memcpy(at(pa.tokens()) + (size_t)r * N, h_tokens + (size_t)ch.b * stride + ch.s0, ch.n * sizeof(int32_t));
    }
    // attention tiles of the pass: a full chunk and the chunk behind it in the same sequence share a CTA
    int tiles = 0, tail_tiles = 0;
    for (int r = 0; r < rows;) {
      const Chunk& ch = chunks[c0 + r];
      const bool pair = r + 1 < rows && chunks[c0 + r + 1].b == ch.b && ch.n == N;
      at(pa.pairs())[2 * tiles] = r; at(pa.pairs())[2 * tiles + 1] = pair ? r + 1 : -1;
      ++tiles;
      if (ch.last >= 0 || (pair && chunks[c0 + r + 1].last >= 0)) {
        at(pa.tail_pairs())[2 * tail_tiles] = r; at(pa.tail_pairs())[2 * tail_tiles + 1] = pair ? r + 1 : -1;
        ++tail_tiles;
      }
      r += pair ? 2 : 1;
    }
    // Longest contexts first: their CTAs would otherwise be the last to start (80 000 tokens in ragged prefixes: 39.6 -> 37.0 ms).
    // Not where all CTAs run at once: the first few share SMs that the projection left free, and these should be the short
    // ones (one prefix of 325 tokens: 11.8 us a launch in order of position, 15.5 sorted)
    auto longest_first = [&](int32_t* pairs, int n) {
      if (ctx->cfg.n_heads * n <= 2 * 148) return;
      struct Pair { int32_t x, y; };
      Pair* q = reinterpret_cast<Pair*>(pairs);
      const int32_t* cl = at(pa.ctx());
      std::stable_sort(q, q + n, [&](const Pair& u, const Pair& v) { return cl[u.x] > cl[v.x]; });
    };
    longest_first(at(pa.pairs()), tiles);
    longest_first(at(pa.tail_pairs()), tail_tiles);
    char* dev = ctx->wsp + ctx->ws.pf_stage;
    if (vadusa_status s = upload(ctx, dev, pack.data(), pack.size())) return s;
    auto dp = [&](size_t off) { return reinterpret_cast<int32_t*>(dev + off); };
    CU(launch_dependent(ctx, prefill_gather_kernel, dim3(rows), 128, 0, real_table, (const int32_t*)dp(pa.seq()), c.max_blocks_per_seq, d_table));
    LAUNCH_CHECK();
    // (the persistent pass has no tail of its own; the gathered residual rows take the place of q)
    const bool whole = ctx->pf_tap != nullptr || ctx->fused_enabled || (size_t)ends * 4 > (size_t)rows * N * sizeof(T);
    {
      RowsView view(ctx, rows, d_table, ctx->ws.pf_stage + (int64_t)pa.ctx(), ctx->ws.pf_stage + (int64_t)pa.nvalid());
      const PrefillTail tail{ends, tail_tiles, reinterpret_cast<const int2*>(dev + pa.tail_pairs()), dp(pa.tail_m())};
      ctx->pf_tiles = tiles;
      ctx->in_prefill = true;
      ctx->pf_pairs = reinterpret_cast<const int2*>(dev + pa.pairs());
      const vadusa_status s = forward<T>(ctx, tv, dp(pa.tokens()), nullptr, whole ? nullptr : &tail);
      ctx->pf_tiles = 0;
      ctx->in_prefill = false;
      if (s) return s;
    }
    if (ends > 0) {
      CU(launch_dependent(ctx, prefill_finish_kernel<T>, dim3(ends), 256, 0, (const int32_t*)dp(pa.tail_m()), (const int32_t*)dp(pa.tail_seq()),
                          (const int32_t*)dp(pa.tail_len()), whole ? 1 : 0, (const T*)wsptr<T>(ctx, ctx->ws.hfinal), c.d_model,
                          (const float*)wsptr<float>(ctx, ctx->ws.logits), vp, wsptr<T>(ctx, ctx->ws.hstar),
                          wsptr<float>(ctx, ctx->ws.logits_star), real_ctx_len));
      LAUNCH_CHECK();
    }
    if (ctx->pf_tap)
      for (int r = 0; r < rows; ++r) {
        const Chunk& ch = chunks[c0 + r];
        CU(cudaMemcpyAsync(reinterpret_cast<T*>(ctx->pf_tap) + ((long long)ch.b * ctx->pf_tap_stride + ch.s0) * c.d_model,
                           wsptr<T>(ctx, ctx->ws.hfinal) + (long long)r * N * c.d_model, (size_t)ch.n * c.d_model * sizeof(T),
                           cudaMemcpyDeviceToDevice, ctx->stream));
      }
  }
  for (int b = 0; b < B; ++b) ctx->h_ctx[b] += h_len[b];
  ctx->ctx_bound += longest;
  ctx->ctx_lo += longest;
  return VADUSA_OK;
}

// ---- draft-head fitting -------------------------------------------------------------------
struct FitLayout {
  int64_t W, U, b;                         // fp32 masters: [heads][d][d], [heads][vpad][d], [heads][d]
  int64_t mW, vW, mU, vU, mb, vb;          // Adam moments, same shapes
  int64_t Wp, Up;                          // parts of the masters, bf16 [3] of the same shapes
  int64_t hf, hp, pre, zp, dl, dp, logits, ce, count, total;
};
FitLayout fit_layout(const vadusa_config* c, int max_tokens) {
  FitLayout f;
  const int64_t hd = c->n_draft_heads, d = c->d_model, vp = vpad(c), T = max_tokens;
  int64_t off = 0;
  auto take = [&](int64_t bytes) { int64_t o = off; off = align_up(off + bytes, 256); return o; };
  const int64_t nW = hd * d * d, nU = hd * vp * d, nb = hd * d;
  f.W = take(nW * 4); f.U = take(nU * 4); f.b = take(nb * 4);
  f.mW = take(nW * 4); f.vW = take(nW * 4); f.mU = take(nU * 4); f.vU = take(nU * 4); f.mb = take(nb * 4); f.vb = take(nb * 4);
  f.Wp = take(nW * 6); f.Up = take(nU * 6);
  f.hf = take(T * d * 4); f.hp = take(T * d * 6); f.pre = take(hd * T * d * 4); f.zp = take(hd * T * d * 6);
  f.dl = take(hd * T * vp * 6); f.dp = take(hd * T * d * 6); f.logits = take(hd * T * vp * 4);
  f.ce = take(hd * T * 4); f.count = take(hd * 4);
  f.total = off;
  return f;
}

template <typename T>
vadusa_status fit_begin(vadusa_ctx* ctx, const FitLayout& f) {
  const vadusa_config& c = ctx->cfg;
  const long long hd = c.n_draft_heads, d = c.d_model, vp = vpad(&c);
  auto up = [&](const T* src, int64_t off, int64_t parts, long long n) -> vadusa_status {
    fit_masters_kernel<T><<<(unsigned)((n / 8 + 255) / 256), 256, 0, ctx->stream>>>(src, reinterpret_cast<float*>(ctx->fit + off),
                                                                                   reinterpret_cast<bf16*>(ctx->fit + parts), n);
    LAUNCH_CHECK();
    return VADUSA_OK;
  };
  if (vadusa_status s = up(as<T>(ctx->dw), f.W, f.Wp, hd * d * d)) return s;
  if (vadusa_status s = up(as<T>(ctx->du), f.U, f.Up, hd * vp * d)) return s;
  CU(cudaMemcpyAsync(ctx->fit + f.b, ctx->db, (size_t)(hd * d * 4), cudaMemcpyDeviceToDevice, ctx->stream));
  CU(cudaMemsetAsync(ctx->fit + f.mW, 0, (size_t)(f.Wp - f.mW), ctx->stream));
  return VADUSA_OK;
}

// One product of a fitting step: C[r][c] = sum_k A(r, k) B(c, k) per head (fit_tc_kernel).
struct FitOperand { const void* parts; int rows, cols, heads; };   // the array as it lies: [part][heads][rows][cols]
template <int NA, int NB, bool AMN, bool BMN, typename Epi>
vadusa_status fit_product(vadusa_ctx* ctx, const FitOperand& A, const FitOperand& B, int R, int C, int K, const Epi& epi) {
  static unsigned long long attr_done = 0ull;              // per device, like launch_gemm_tc
  const unsigned long long dev_bit = 1ull << (ctx->cfg.device & 63);
  if (!(attr_done & dev_bit)) {
    CU(cudaFuncSetAttribute(fit_tc_kernel<NA, NB, AMN, BMN, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, FitCfg<NA, NB>::kSmem));
    attr_done |= dev_bit;
  }
  const CUtensorMap *ma, *mb;
  if (vadusa_status s = tensor_map(ctx, A.parts, A.rows, A.cols, AMN ? 64 : kFitTile, NA * A.heads, (long long)A.rows * A.cols, &ma)) return s;
  if (vadusa_status s = tensor_map(ctx, B.parts, B.rows, B.cols, BMN ? 64 : kFitTile, NB * B.heads, (long long)B.rows * B.cols, &mb)) return s;
  CU(launch_dependent(ctx, fit_tc_kernel<NA, NB, AMN, BMN, Epi>,
                      dim3((C + kFitTile - 1) / kFitTile, (R + kFitTile - 1) / kFitTile, ctx->cfg.n_draft_heads), kFitThreads,
                      FitCfg<NA, NB>::kSmem, *ma, *mb, R, C, K, A.heads, B.heads, epi, err_word(ctx)));
  LAUNCH_CHECK();
  return VADUSA_OK;
}

template <typename T>
vadusa_status fit_step(vadusa_ctx* ctx, const FitLayout& f, const T* hidden, const int32_t* targets, int Tn, float* loss_out) {
  constexpr int NH = sizeof(T) == 2 ? 1 : 3;               // parts of the hidden states
  const vadusa_config& c = ctx->cfg;
  const int hd = c.n_draft_heads, d = c.d_model, vp = vpad(&c), V = c.vocab;
  auto P = [&](int64_t off) { return reinterpret_cast<float*>(ctx->fit + off); };
  auto H = [&](int64_t off) { return reinterpret_cast<bf16*>(ctx->fit + off); };
  int32_t* count = reinterpret_cast<int32_t*>(ctx->fit + f.count);
  const FitOperand h{H(f.hp), Tn, d, 1}, z{H(f.zp), Tn, d, hd}, dl{H(f.dl), Tn, vp, hd}, dpre{H(f.dp), Tn, d, hd}, W{H(f.Wp), d, d, hd},
      U{H(f.Up), vp, d, hd};
  ctx->fit_step++;
  const float lr = ctx->fit_lr * fminf(1.0f, (float)ctx->fit_step / (float)(ctx->fit_warmup > 0 ? ctx->fit_warmup : 1));
  const float c1 = (float)(1.0 - pow(0.9, (double)ctx->fit_step)), c2 = (float)(1.0 - pow(0.999, (double)ctx->fit_step));
  const long long n = (long long)Tn * d;
  CU(launch_dependent(ctx, fit_inputs_kernel<T>, dim3((unsigned)((n / 8 + 255) / 256) + 1), 256, 0, hidden, P(f.hf), H(f.hp), n, targets,
                      Tn, hd, count));
  LAUNCH_CHECK();
  // forward: pre = h W^T + b, z = h + SiLU(pre), logits = z U^T
  const FitHidden eh{P(f.b), P(f.hf), P(f.pre), H(f.zp), Tn, d, hd};
  if (vadusa_status s = fit_product<NH, 3, false, false>(ctx, h, W, Tn, d, d, eh)) return s;
  if (vadusa_status s = fit_product<3, 3, false, false>(ctx, z, U, Tn, vp, d, FitStore{P(f.logits), Tn, vp})) return s;
  // loss and d loss / d logits
  CU(launch_dependent(ctx, fit_softmax_ce_kernel, dim3(Tn, hd), 256, 0, (const float*)P(f.logits), targets, (const int32_t*)count, Tn, hd, V,
                      vp, ctx->fit_lambda, H(f.dl), P(f.ce)));
  LAUNCH_CHECK();
  // backward and update: dz = dl U, dpre = dz SiLU'(pre); then dU = dl^T z and dW = dpre^T h with Adam behind the sums
  // (linear warm-up; masters, their parts, and the heads in the weight blob)
  if (vadusa_status s = fit_product<3, 3, false, true>(ctx, dl, U, Tn, d, vp, FitDpre{P(f.pre), H(f.dp), Tn, d, hd})) return s;
  const FitAdam<T> aU{P(f.U), P(f.mU), P(f.vU), const_cast<T*>(as<T>(ctx->du)), H(f.Up), vp, d, hd, lr, c1, c2};
  if (vadusa_status s = fit_product<3, 3, true, true>(ctx, dl, z, vp, d, Tn, aU)) return s;
  const FitAdam<T> aW{P(f.W), P(f.mW), P(f.vW), const_cast<T*>(as<T>(ctx->dw)), H(f.Wp), d, d, hd, lr, c1, c2};
  if (vadusa_status s = fit_product<3, NH, true, true>(ctx, dpre, h, d, d, Tn, aW)) return s;
  CU(launch_dependent(ctx, fit_bias_kernel, dim3((d + 31) / 32 + 1, hd), 1024, 0, (const bf16*)H(f.dp), Tn, d, hd, P(f.b), P(f.mb), P(f.vb),
                      const_cast<float*>(ctx->db), lr, c1, c2, (const float*)P(f.ce), (const int32_t*)count, ctx->fit_lambda, loss_out));
  LAUNCH_CHECK();
  return VADUSA_OK;
}

vadusa_status set_kernel_attributes(vadusa_ctx* ctx) {
  const auto smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
  CU(cudaFuncSetAttribute(tree_attention_simt_kernel<float, 64, 4>, smem, att_simt_smem(64)));
  CU(cudaFuncSetAttribute(tree_attention_simt_kernel<float, 64, 8>, smem, att_simt_smem(64)));
  CU(cudaFuncSetAttribute(tree_attention_simt_kernel<float, 32, 4>, smem, att_simt_smem(32)));
  CU(cudaFuncSetAttribute(tree_attention_simt_kernel<float, 32, 8>, smem, att_simt_smem(32)));
  CU(cudaFuncSetAttribute(tree_attention_simt_kernel<bf16, 32, 4>, smem, att_simt_smem(32)));
  CU(cudaFuncSetAttribute(tree_attention_simt_kernel<bf16, 32, 8>, smem, att_simt_smem(32)));
  CU(cudaFuncSetAttribute(tree_attention_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttSmemBytes));
  CU(cudaFuncSetAttribute(prefill_attention_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttSmemBytes));
  CU(cudaFuncSetAttribute(tree_attention_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAsSmemBytes));
  CU(cudaFuncSetAttribute(prefill_attention_tc_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  // the kernels that draw keep one row of keys and one of logits in shared memory.  The limit is an attribute of
  // the function on this device, shared by every context: always the library's largest vocabulary
  CU(cudaFuncSetAttribute(accept_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 24576 * (int)sizeof(float)));
  CU(cudaFuncSetAttribute(accept_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  CU(cudaFuncSetAttribute(commit_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 24576 * (int)sizeof(float)));
  CU(cudaFuncSetAttribute(commit_kernel<bf16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 24576 * (int)sizeof(float)));
  CU(cudaFuncSetAttribute(draft_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 24576 * (int)sizeof(float)));
  // the small kernels between the products too: an SM that keeps its carve-out takes the next kernel's CTAs beside them
  const auto carve = cudaFuncAttributePreferredSharedMemoryCarveout;
  CU(cudaFuncSetAttribute(layernorm_rows_kernel<float>, carve, cudaSharedmemCarveoutMaxShared));
  CU(cudaFuncSetAttribute(layernorm_rows_kernel<bf16>, carve, cudaSharedmemCarveoutMaxShared));
  CU(cudaFuncSetAttribute(layernorm_kernel<bf16>, carve, cudaSharedmemCarveoutMaxShared));
  CU(cudaFuncSetAttribute(tree_embed_kernel<bf16>, carve, cudaSharedmemCarveoutMaxShared));
  CU(cudaFuncSetAttribute(commit_kernel<bf16>, carve, cudaSharedmemCarveoutMaxShared));
  CU(cudaFuncSetAttribute(draft_select_kernel, carve, cudaSharedmemCarveoutMaxShared));
  // ask for the largest shared-memory carve-out so that several CTAs fit on an SM
  CU(cudaFuncSetAttribute(tree_attention_tc_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  CU(cudaFuncSetAttribute(tree_attention_stream_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  return VADUSA_OK;
}

__global__ void begin_kernel(uint32_t* scalars /*[64]*/, uint32_t* f_sync /*[64]*/, uint32_t* att_cnt, int n_cnt, int32_t* gen_count,
                             int32_t* ctx_len /*or null*/, int32_t* nvalid, int batch, int n_nodes) {
  const int t = threadIdx.x;
  if (t < 64) { scalars[t] = 0u; f_sync[t] = 0u; }
  for (int i = t; i < n_cnt; i += blockDim.x) att_cnt[i] = 0u;
  for (int b = t; b < batch; b += blockDim.x) {
    gen_count[b] = 0; nvalid[b] = n_nodes;
    if (ctx_len) ctx_len[b] = 0;
  }
}

__global__ void generate_begin_kernel(int32_t* gen_count, int32_t* nvalid, int batch, int n_nodes, int32_t* done /*[3]: done, iterations, arrived*/) {
  if (threadIdx.x < 3) done[threadIdx.x] = 0;
  for (int b = threadIdx.x; b < batch; b += blockDim.x) { gen_count[b] = 0; nvalid[b] = n_nodes; }
}

__global__ void fill_i32_kernel(int32_t* p, int n, int32_t v) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

vadusa_status set_active(vadusa_ctx* ctx, int value) {
  fill_i32_kernel<<<(ctx->batch + 255) / 256, 256, 0, ctx->stream>>>(wsptr<int32_t>(ctx, ctx->ws.nvalid), ctx->batch,
                                                                     value);
  LAUNCH_CHECK();
  return VADUSA_OK;
}

vadusa_status error_of(vadusa_ctx* ctx, uint32_t e) {
  if (e & kErrTimeout) return fail(ctx, VADUSA_ETIMEOUT, "a bounded device-side wait expired (error word 0x%x)", e);
  if (e & kErrCapacity)
    return fail(ctx, VADUSA_ECAPACITY, "a sequence ran past its KV blocks, the position table or the token range (error word 0x%x)", e);
  return VADUSA_OK;
}

vadusa_status device_errors(vadusa_ctx* ctx) {
  uint32_t e = 0;
  CU(cudaMemcpyAsync(&e, err_word(ctx), sizeof(e), cudaMemcpyDeviceToHost, ctx->stream));
  CU(cudaStreamSynchronize(ctx->stream));
  return error_of(ctx, e);
}

// Key of a launch sequence: a tag plus the raw bytes of everything baked into its kernels' arguments.
struct KeyBuilder {
  std::string k;
  explicit KeyBuilder(const char* tag) : k(tag) {}
  template <typename V> KeyBuilder& add(const V& v) { k.append(reinterpret_cast<const char*>(&v), sizeof(V)); return *this; }
};

// Runs `body` (which only enqueues work on ctx->stream) eagerly the first time a key is seen,
// captures it into a CUDA graph the second time, and replays the graph afterwards.  The legacy
// default stream cannot be captured, and profiling wants separate launches: both run eagerly.
template <typename F>
vadusa_status run_graphed(vadusa_ctx* ctx, const std::string& key, F&& body) {
  if (ctx->stream == nullptr || ctx->prof_on) return body();
  if (ctx->graphs.size() > 64 && ctx->graphs.find(key) == ctx->graphs.end()) {
    // the sequence that was asked for longest ago makes room
    auto old = ctx->graphs.begin();
    for (auto it = ctx->graphs.begin(); it != ctx->graphs.end(); ++it)
      if (it->second.used < old->second.used) old = it;
    if (old->second.exec) cudaGraphExecDestroy(old->second.exec);
    ctx->graphs.erase(old);
  }
  vadusa_ctx::GraphRec& r = ctx->graphs[key];
  r.used = ++ctx->graph_clock;
  if (r.exec) {
    CU(cudaGraphLaunch(r.exec, ctx->stream));
    ctx->launches += r.launches;
    return VADUSA_OK;
  }
  if (r.seen++ == 0) return body();
  const int64_t l0 = ctx->launches;
  CU(cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal));
  vadusa_status s = body();
  cudaGraph_t graph = nullptr;
  cudaError_t ce = cudaStreamEndCapture(ctx->stream, &graph);
  if (s != VADUSA_OK || ce != cudaSuccess || !graph) {
    if (graph) cudaGraphDestroy(graph);
    cudaGetLastError();
    if (s != VADUSA_OK) return s;
    return fail(ctx, VADUSA_ECUDA, "stream capture failed: %s", cudaGetErrorString(ce));
  }
  ce = cudaGraphInstantiate(&r.exec, graph, 0);
  cudaGraphDestroy(graph);
  if (ce != cudaSuccess) { r.exec = nullptr; return fail(ctx, VADUSA_ECUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(ce)); }
  r.launches = ctx->launches - l0;
  ctx->launches = l0;
  CU(cudaGraphLaunch(r.exec, ctx->stream));
  ctx->launches += r.launches;
  return VADUSA_OK;
}

#define DISPATCH(expr_f32, expr_bf16) (ctx->cfg.dtype == 1 ? (expr_bf16) : (expr_f32))

vadusa_status need_batch(vadusa_ctx* ctx) {
  if (!ctx) return VADUSA_EINVAL;
  if (ctx->batch == 0) return fail(ctx, VADUSA_ESTATE, "vadusa_begin has not been called");
  return VADUSA_OK;
}

// The words in h_pinned, written by the device while the host looks on.
struct HostWords { volatile int32_t iters, done; volatile uint32_t err; int32_t unused; volatile int32_t gen[1]; };

// out_len[b] = min(gen_count[b], cap); token counts and the error word to the host.  One block.
__global__ void generate_end_kernel(const int32_t* gen_count, const uint32_t* err, int batch, int cap, int32_t* out_len /*or null*/,
                                    HostWords* host) {
  for (int b = threadIdx.x; b < batch; b += blockDim.x) {
    const int g = gen_count[b];
    host->gen[b] = g;
    if (out_len) out_len[b] = g < cap ? g : cap;
  }
  if (threadIdx.x == 0) host->err = *err;
}

// The decoding loop.  The host stays one iteration ahead of the device: the commit of an iteration leaves (iterations
// finished, sequences done) in pinned host memory, and iteration k is enqueued once k - 2 has been reported, so that the
// device always has one queued and the loop ends with at most one iteration that finds nothing to do (with a copy and an
// event every eighth iteration up to sixteen ran behind the end: a quarter of a short request).
// h_out_tokens / h_out_len: host destinations, or null (then out_len, a device pointer, or null).
vadusa_status run_generate(vadusa_ctx* ctx, const vadusa_sampling* sampling, int32_t max_new_tokens, int32_t max_iters,
                           int32_t* out_tokens, int32_t* out_len, int32_t* h_out_tokens, int32_t* h_out_len, vadusa_stats* h_stats) {
  if (vadusa_status s = need_batch(ctx)) return s;
  if (ctx->n_nodes == 0 || ctx->tree_per_seq) return fail(ctx, VADUSA_ESTATE, "generate needs a shared tree template");
  if (max_new_tokens < 1) return fail(ctx, VADUSA_EINVAL, "max_new_tokens must be positive");
  SamplingDev sp;
  if (vadusa_status s = sampling_dev(ctx, sampling, &sp)) return s;
  const int64_t launches0 = ctx->launches;
  const int limit = max_iters > 0 ? max_iters : max_new_tokens;
  const TreeView tv = tree_of(ctx, false);
  AcceptOut none{nullptr, nullptr, nullptr, nullptr, nullptr, 1, nullptr};
  HostWords* host = reinterpret_cast<HostWords*>(ctx->h_pinned);
  // (nothing of an earlier generate is in flight: each ends with a synchronisation)
  host->iters = 0; host->done = 0; host->err = 0u;
  generate_begin_kernel<<<1, 256, 0, ctx->stream>>>(wsptr<int32_t>(ctx, ctx->ws.gen_count), wsptr<int32_t>(ctx, ctx->ws.nvalid),
                                                    ctx->batch, ctx->n_nodes, done_word(ctx));
  LAUNCH_CHECK();
  int iters = 0;
  CU(cudaEventRecord(ctx->ev0, ctx->stream));
  for (; iters < limit; ++iters) {
    for (int spins = 1; host->iters < iters - 1; ++spins) {
      if ((spins & 0xfff) == 0) {
        // the device has gone idle without a report: it failed
        const cudaError_t q = cudaStreamQuery(ctx->stream);
        if (q != cudaErrorNotReady && host->iters < iters - 1)
          return fail(ctx, VADUSA_ECUDA, "generate: %s", q == cudaSuccess ? "an iteration was not reported" : cudaGetErrorString(q));
      }
    }
    if (host->done >= ctx->batch) break;
    const std::string iter_key = KeyBuilder("iteration").add(sp).add(out_tokens).add(max_new_tokens).add(ctx->batch)
                                     .add(ctx->n_nodes).add(ctx->block_table).add(attention_splits(ctx, ctx->n_nodes)).add(ctx->fused_enabled).add(ctx->att_stream).k;
    vadusa_status s = run_graphed(ctx, iter_key, [&]() -> vadusa_status {
      vadusa_status s = DISPATCH(draft<float>(ctx, sp), draft<bf16>(ctx, sp));
      if (s) return s;
      s = DISPATCH(forward<float>(ctx, tv, nullptr, nullptr), forward<bf16>(ctx, tv, nullptr, nullptr));
      if (s) return s;
      return DISPATCH(accept_commit<float>(ctx, sp, nullptr, none, out_tokens, max_new_tokens, max_new_tokens, ctx->h_pinned),
                      accept_commit<bf16>(ctx, sp, nullptr, none, out_tokens, max_new_tokens, max_new_tokens, ctx->h_pinned));
    });
    if (s) return s;
    ctx->ctx_bound += ctx->tree_max_depth + 1;
    ctx->ctx_lo += 1;
  }
  CU(cudaEventRecord(ctx->ev1, ctx->stream));
  generate_end_kernel<<<1, 256, 0, ctx->stream>>>(wsptr<int32_t>(ctx, ctx->ws.gen_count), err_word(ctx), ctx->batch, max_new_tokens,
                                                  out_len, host);
  LAUNCH_CHECK();
  if (h_out_tokens)
    CU(cudaMemcpyAsync(h_out_tokens, out_tokens, (size_t)ctx->batch * max_new_tokens * 4, cudaMemcpyDeviceToHost, ctx->stream));
  CU(cudaStreamSynchronize(ctx->stream));
  int64_t total = 0;
  for (int b = 0; b < ctx->batch; ++b) {
    const int32_t g = host->gen[b];
    total += g;
    if (h_out_len) h_out_len[b] = g > max_new_tokens ? max_new_tokens : g;
    if (ctx->h_ctx_exact) ctx->h_ctx[b] += g;               // (every committed token is counted in both)
  }
  if (h_stats) {
    float ms = 0.f;
    CU(cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1));
    h_stats->iterations = iters;
    h_stats->tokens_generated = total;
    h_stats->elapsed_ms = ms;
    h_stats->kernel_launches = ctx->launches - launches0;
  }
  ctx->have_draft = ctx->have_verify = false;
  return error_of(ctx, host->err);
}

}  // namespace

// ---- C ABI -------------------------------------------------------------------------

extern "C" {

int64_t vadusa_workspace_bytes(const vadusa_config* cfg) {
  if (check_config(cfg)) return -1;
  return workspace_layout(cfg).total;
}

int64_t vadusa_weights_bytes(const vadusa_config* cfg) {
  if (check_config(cfg)) return -1;
  int64_t total = 0;
  weight_layout(cfg, &total);
  return total;
}

int64_t vadusa_kv_pool_bytes(const vadusa_config* cfg) {
  if (check_config(cfg)) return -1;
  return kv_pool_bytes(cfg);
}

int32_t vadusa_weight_count(const vadusa_config* cfg) {
  if (check_config(cfg)) return -1;
  return (int32_t)weight_layout(cfg, nullptr).size();
}

vadusa_status vadusa_weight_info(const vadusa_config* cfg, int32_t index, vadusa_tensor_info* h_out) {
  if (check_config(cfg) || !h_out) return VADUSA_EINVAL;
  auto v = weight_layout(cfg, nullptr);
  if (index < 0 || index >= (int32_t)v.size()) return VADUSA_EINVAL;
  const TensorDesc& t = v[index];
  memset(h_out, 0, sizeof(*h_out));
  snprintf(h_out->name, sizeof(h_out->name), "%s", t.name.c_str());
  h_out->offset = t.offset; h_out->nbytes = t.nbytes;
  h_out->rows = t.rows; h_out->cols = t.cols; h_out->rows_padded = t.rows_padded; h_out->is_matrix = t.is_matrix;
  return VADUSA_OK;
}

vadusa_status vadusa_init(const vadusa_weights* weights, const vadusa_config* cfg, vadusa_ctx** h_out) {
  if (!h_out) return VADUSA_EINVAL;
  *h_out = nullptr;
  vadusa_ctx* ctx = new (std::nothrow) vadusa_ctx();
  if (!ctx) return VADUSA_ENOMEM;
  *h_out = ctx;     // returned even on failure so that vadusa_last_error can be read; destroy it either way
  if (const char* why = check_config(cfg)) return fail(ctx, VADUSA_EINVAL, "%s", why);
  ctx->cfg = *cfg;
  if (!weights || !weights->blob) return fail(ctx, VADUSA_EINVAL, "weights are NULL");
  int64_t wbytes = 0;
  ctx->wl = weight_layout(cfg, &wbytes);
  if (weights->nbytes < wbytes) return fail(ctx, VADUSA_ENOMEM, "weight blob has %lld bytes, %lld needed", (long long)weights->nbytes, (long long)wbytes);
  ctx->ws = workspace_layout(cfg);
  if (!cfg->workspace || cfg->workspace_bytes < ctx->ws.total)
    return fail(ctx, VADUSA_ENOMEM, "workspace has %lld bytes, %lld needed", (long long)cfg->workspace_bytes, (long long)ctx->ws.total);
  if (((uintptr_t)cfg->workspace & 255) || ((uintptr_t)weights->blob & 255) || ((uintptr_t)cfg->kv_pool & 255))
    return fail(ctx, VADUSA_EINVAL, "workspace, weight blob and KV pool must be 256-byte aligned");
  if (!cfg->kv_pool || cfg->kv_pool_bytes < kv_pool_bytes(cfg))
    return fail(ctx, VADUSA_ENOMEM, "KV pool has %lld bytes, %lld needed", (long long)cfg->kv_pool_bytes, (long long)kv_pool_bytes(cfg));
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
    cudaGetLastError();
    return fail(ctx, VADUSA_ECUDA, "no CUDA device: this library has no CPU path");
  }
  if (cfg->device < 0 || cfg->device >= ndev) return fail(ctx, VADUSA_EINVAL, "device ordinal out of range");
  CU(cudaSetDevice(cfg->device));
  cudaDeviceProp prop;
  CU(cudaGetDeviceProperties(&prop, cfg->device));
  if (prop.major != 10) return fail(ctx, VADUSA_ECUDA, "device is sm_%d%d; this library is built for sm_100a only", prop.major, prop.minor);
  ctx->blob = reinterpret_cast<const char*>(weights->blob);
  ctx->wsp = reinterpret_cast<char*>(cfg->workspace);
  ctx->stream = reinterpret_cast<cudaStream_t>(cfg->stream);
  resolve_weights(ctx);
  {
    cudaDriverEntryPointQueryResult qres;
    void* fn = nullptr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      ctx->encode_fn = fn;
    else
      cudaGetLastError();
  }
  if (vadusa_status s = set_kernel_attributes(ctx)) return s;
  CU(cudaEventCreate(&ctx->ev0));
  CU(cudaEventCreate(&ctx->ev1));
  for (int i = 0; i < 2; ++i) CU(cudaEventCreateWithFlags(&ctx->ev_up[i], cudaEventDisableTiming));
  CU(cudaMallocHost(&ctx->h_pinned, (kHostWords + cfg->max_batch) * sizeof(int32_t)));
  CU(cudaMallocHost(&ctx->up, 2 * kUpHalf));
  CU(cudaMemsetAsync(ctx->wsp, 0, ctx->ws.tokens, ctx->stream));     // scalars, per-sequence state, trees
  CU(cudaMemsetAsync(ctx->wsp + ctx->ws.acc_stats, 0, 2ull * kStatDepth * kStatTopk * 8, ctx->stream));
  CU(cudaMemsetAsync(ctx->wsp + ctx->ws.f_sync, 0, 256, ctx->stream));
  CU(cudaMemsetAsync(ctx->wsp + ctx->ws.att_cnt, 0, 2 * kAsGrid * 4, ctx->stream));
  // chain-shaped tree used by prefill: node i is the child of node i-1
  constexpr int T = VADUSA_MAX_TREE_NODES;
  static_assert(T == kMaxNodes, "node limit of the kernels");
  int32_t par[T], dep[T], rnk[T];
  unsigned long long anc[2 * T];
  auto low_bits = [](int n) { return n <= 0 ? 0ull : n >= 64 ? ~0ull : ((1ull << n) - 1); };   // n lowest bits set
  for (int i = 0; i < T; ++i) { par[i] = i - 1; dep[i] = i; rnk[i] = 0; anc[2 * i] = low_bits(i + 1); anc[2 * i + 1] = low_bits(i + 1 - 64); }
  CU(cudaMemcpyAsync(ctx->wsp + ctx->ws.chain_parent, par, sizeof(par), cudaMemcpyHostToDevice, ctx->stream));
  CU(cudaMemcpyAsync(ctx->wsp + ctx->ws.chain_depth, dep, sizeof(dep), cudaMemcpyHostToDevice, ctx->stream));
  CU(cudaMemcpyAsync(ctx->wsp + ctx->ws.chain_rank, rnk, sizeof(rnk), cudaMemcpyHostToDevice, ctx->stream));
  CU(cudaMemcpyAsync(ctx->wsp + ctx->ws.chain_anc, anc, sizeof(anc), cudaMemcpyHostToDevice, ctx->stream));
  CU(cudaStreamSynchronize(ctx->stream));
  return VADUSA_OK;
}

vadusa_status vadusa_destroy(vadusa_ctx* ctx) {
  if (!ctx) return VADUSA_EINVAL;
  if (ctx->ev0) cudaEventDestroy(ctx->ev0);
  if (ctx->ev1) cudaEventDestroy(ctx->ev1);
  for (int i = 0; i < 2; ++i) if (ctx->ev_up[i]) cudaEventDestroy(ctx->ev_up[i]);
  if (ctx->h_pinned) cudaFreeHost(ctx->h_pinned);
  if (ctx->up) cudaFreeHost(ctx->up);
  for (auto& r : ctx->prof) { cudaEventDestroy(r.a); cudaEventDestroy(r.b); }
  for (auto& kv : ctx->graphs) if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
  delete ctx;
  return VADUSA_OK;
}

const char* vadusa_last_error(const vadusa_ctx* ctx) { return ctx ? ctx->err : "context is NULL"; }

vadusa_status vadusa_set_tree(vadusa_ctx* ctx, int32_t n_nodes, const int32_t* h_parent, const int32_t* h_rank,
                              int32_t per_sequence) {
  if (!ctx) return VADUSA_EINVAL;
  if (!ctx->wsp) return fail(ctx, VADUSA_ESTATE, "context is not initialised");
  if (!h_parent || !h_rank) return fail(ctx, VADUSA_EINVAL, "tree arrays are NULL");
  if (n_nodes < 1 || n_nodes > ctx->cfg.max_tree_nodes) return fail(ctx, VADUSA_EINVAL, "n_nodes must be in 1..max_tree_nodes");
  int copies = 1;
  if (per_sequence) {
    if (ctx->batch == 0) return fail(ctx, VADUSA_ESTATE, "per-sequence trees need vadusa_begin first");
    copies = ctx->batch;
  }
  std::vector<int32_t> depth((size_t)copies * n_nodes);
  std::vector<unsigned long long> anc((size_t)copies * n_nodes * 2);
  std::vector<int32_t> inner((size_t)copies * VADUSA_MAX_TREE_NODES, -1);
  int max_depth = 0, max_inner = 0;
  for (int s = 0; s < copies; ++s) {
    const int32_t* par = h_parent + (size_t)s * n_nodes;
    const int32_t* rnk = h_rank + (size_t)s * n_nodes;
    int32_t* dep = depth.data() + (size_t)s * n_nodes;
    unsigned long long* an = anc.data() + (size_t)s * n_nodes * 2;       // two words per node
    if (par[0] != -1) return fail(ctx, VADUSA_EINVAL, "node 0 must be the root (parent -1)");
    dep[0] = 0; an[0] = 1ull; an[1] = 0ull;
    for (int n = 1; n < n_nodes; ++n) {
      if (par[n] < 0 || par[n] >= n) return fail(ctx, VADUSA_EINVAL, "node %d: parent %d must precede it", n, par[n]);
      dep[n] = dep[par[n]] + 1;
      an[2 * n] = an[2 * par[n]] | (n < 64 ? 1ull << n : 0ull);
      an[2 * n + 1] = an[2 * par[n] + 1] | (n >= 64 ? 1ull << (n - 64) : 0ull);
      if (dep[n] > VADUSA_MAX_DEPTH) return fail(ctx, VADUSA_EINVAL, "node %d: deeper than %d", n, VADUSA_MAX_DEPTH);
      if (!per_sequence) {
        if (dep[n] > ctx->cfg.n_draft_heads) return fail(ctx, VADUSA_EINVAL, "node %d: depth %d exceeds the number of draft heads", n, dep[n]);
        if (rnk[n] < 0 || rnk[n] >= ctx->cfg.draft_topk) return fail(ctx, VADUSA_EINVAL, "node %d: rank %d outside the draft top-k", n, rnk[n]);
      } else if (rnk[n] < 0) {
        return fail(ctx, VADUSA_EINVAL, "node %d: negative rank", n);
      }
      if (dep[n] < dep[n - 1]) return fail(ctx, VADUSA_EINVAL, "node %d: nodes must be ordered by depth", n);
      // (depth, rank path) order: within a depth, parents ascend, and siblings ascend by rank
      if (n > 1 && dep[n] == dep[n - 1]) {
        if (par[n] < par[n - 1] || (par[n] == par[n - 1] && rnk[n] <= rnk[n - 1]))
          return fail(ctx, VADUSA_EINVAL, "node %d: nodes of one depth must be in rank-path order", n);
      }
      max_depth = dep[n] > max_depth ? dep[n] : max_depth;
    }
    bool has[VADUSA_MAX_TREE_NODES] = {false};
    for (int n = 1; n < n_nodes; ++n) has[par[n]] = true;
    int k = 0;
    for (int n = 0; n < n_nodes; ++n)
      if (has[n]) inner[(size_t)s * VADUSA_MAX_TREE_NODES + k++] = n;
    max_inner = k > max_inner ? k : max_inner;
  }
  // one staged copy: parent, depth, rank [copies][n_nodes], the lists of inner nodes, the ancestor words
  const size_t nn = (size_t)copies * n_nodes;
  std::vector<char> pack(nn * 12 + inner.size() * 4 + 16 + nn * 16);
  const size_t at_anc = (nn * 12 + inner.size() * 4 + 15) & ~(size_t)15;
  memcpy(pack.data(), h_parent, nn * 4);
  memcpy(pack.data() + nn * 4, depth.data(), nn * 4);
  memcpy(pack.data() + nn * 8, h_rank, nn * 4);
  memcpy(pack.data() + nn * 12, inner.data(), inner.size() * 4);
  memcpy(pack.data() + at_anc, anc.data(), nn * 16);
  if (vadusa_status s = upload(ctx, ctx->wsp + ctx->ws.tree, pack.data(), at_anc + nn * 16)) return s;
  ctx->tree_copies = copies;
  ctx->n_nodes = n_nodes;
  ctx->tree_per_seq = per_sequence ? 1 : 0;
  ctx->tree_max_depth = max_depth;
  ctx->tree_inner = max_inner > 0 ? max_inner : 1;
  ctx->have_draft = ctx->have_verify = false;
  if (ctx->batch > 0) return set_active(ctx, ctx->n_nodes);
  return VADUSA_OK;
}

vadusa_status vadusa_begin(vadusa_ctx* ctx, int32_t batch, const int32_t* block_table, const int32_t* h_ctx_len) {
  if (!ctx) return VADUSA_EINVAL;
  if (!ctx->wsp) return fail(ctx, VADUSA_ESTATE, "context is not initialised");
  if (batch < 1 || batch > ctx->cfg.max_batch) return fail(ctx, VADUSA_EINVAL, "batch must be in 1..max_batch");
  if (!block_table) return fail(ctx, VADUSA_EINVAL, "block_table is NULL");
  if (ctx->tree_per_seq) { ctx->n_nodes = 0; ctx->tree_per_seq = 0; }
  ctx->batch = batch;
  ctx->block_table = block_table;
  ctx->have_draft = ctx->have_verify = false;
  ctx->ctx_bound = 0;
  ctx->h_ctx.assign(batch, 0);
  ctx->h_ctx_exact = true;
  if (h_ctx_len) {
    for (int b = 0; b < batch; ++b) {
      if (h_ctx_len[b] < 0 || h_ctx_len[b] > (int64_t)ctx->cfg.max_blocks_per_seq * 64)
        return fail(ctx, VADUSA_EINVAL, "context length of sequence %d out of range", b);
      if (h_ctx_len[b] > ctx->ctx_bound) ctx->ctx_bound = h_ctx_len[b];
      ctx->h_ctx[b] = h_ctx_len[b];
    }
    if (vadusa_status s = upload(ctx, ctx->wsp + ctx->ws.ctx_len, h_ctx_len, batch * 4)) return s;
  }
  ctx->ctx_lo = ctx->ctx_bound;
  // one launch for everything a new batch clears
  begin_kernel<<<1, 256, 0, ctx->stream>>>(wsptr<uint32_t>(ctx, ctx->ws.scalars), wsptr<uint32_t>(ctx, ctx->ws.f_sync),
                                           wsptr<uint32_t>(ctx, ctx->ws.att_cnt), 2 * kAsGrid, wsptr<int32_t>(ctx, ctx->ws.gen_count),
                                           h_ctx_len ? nullptr : wsptr<int32_t>(ctx, ctx->ws.ctx_len),
                                           wsptr<int32_t>(ctx, ctx->ws.nvalid), batch, ctx->n_nodes);
  LAUNCH_CHECK();
  return VADUSA_OK;
}

vadusa_status vadusa_prefill(vadusa_ctx* ctx, const int32_t* h_tokens, const int32_t* h_len, int32_t stride) {
  if (vadusa_status s = need_batch(ctx)) return s;
  if (!h_tokens || !h_len || stride < 1) return fail(ctx, VADUSA_EINVAL, "prefill arguments are NULL or empty");
  vadusa_status s = DISPATCH(prefill<float>(ctx, h_tokens, h_len, stride), prefill<bf16>(ctx, h_tokens, h_len, stride));
  if (s) return s;

  ctx->have_draft = ctx->have_verify = false;
  return set_active(ctx, ctx->n_nodes);
}

vadusa_status vadusa_load_state(vadusa_ctx* ctx, const void* hstar, const float* logits_star) {
  if (vadusa_status s = need_batch(ctx)) return s;
  if (!hstar || !logits_star) return fail(ctx, VADUSA_EINVAL, "state pointers are NULL");
  const vadusa_config& c = ctx->cfg;
  CU(cudaMemcpyAsync(ctx->wsp + ctx->ws.hstar, hstar, (size_t)ctx->batch * c.d_model * esize(&c), cudaMemcpyDeviceToDevice, ctx->stream));
  CU(cudaMemcpy2DAsync(ctx->wsp + ctx->ws.logits_star, (size_t)vpad(&c) * 4, logits_star, (size_t)c.vocab * 4,
                       (size_t)c.vocab * 4, ctx->batch, cudaMemcpyDeviceToDevice, ctx->stream));
  return VADUSA_OK;
}

vadusa_status vadusa_draft(vadusa_ctx* ctx, const vadusa_sampling* sampling, int32_t* tree_tokens,
                           int32_t* draft_topk_out) {
  if (vadusa_status s = need_batch(ctx)) return s;
  if (ctx->n_nodes == 0) return fail(ctx, VADUSA_ESTATE, "no tree set");
  if (ctx->tree_per_seq && tree_tokens) return fail(ctx, VADUSA_EINVAL, "per-sequence topologies take their tokens from the override");
  SamplingDev sp;
  if (vadusa_status s = sampling_dev(ctx, sampling, &sp)) return s;
  const vadusa_config& c = ctx->cfg;
  const std::string key = KeyBuilder("draft").add(sp).add(tree_tokens).add(draft_topk_out).add(ctx->batch)
                              .add(ctx->n_nodes).add(ctx->tree_per_seq).add(ctx->block_table).k;
  vadusa_status s = run_graphed(ctx, key, [&]() -> vadusa_status {
    vadusa_status s = DISPATCH(draft<float>(ctx, sp), draft<bf16>(ctx, sp));
    if (s) return s;
    if (draft_topk_out)
      CU(cudaMemcpyAsync(draft_topk_out, ctx->wsp + ctx->ws.topk, (size_t)ctx->batch * c.n_draft_heads * c.draft_topk * 4,
                         cudaMemcpyDeviceToDevice, ctx->stream));
    if (tree_tokens) {
      // tokens of the tree without a model pass: the embed kernel computes them; run it alone
      const TreeView tv = tree_of(ctx, false);
      const int M = ctx->batch * tv.n_nodes;
      if (vadusa_status s = DISPATCH(embed<float>(ctx, tv, nullptr, nullptr, nullptr), embed<bf16>(ctx, tv, nullptr, nullptr, nullptr))) return s;
      CU(cudaMemcpyAsync(tree_tokens, ctx->wsp + ctx->ws.tokens, (size_t)M * 4, cudaMemcpyDeviceToDevice, ctx->stream));
    }
    return VADUSA_OK;
  });
  if (s) return s;
  ctx->have_draft = true;
  return VADUSA_OK;
}

vadusa_status vadusa_verify_step(vadusa_ctx* ctx, const int32_t* tree_tokens_override, float* logits_out,
                                 void* attn_tap, void* hidden_out) {
  if (vadusa_status s = need_batch(ctx)) return s;
  if (ctx->n_nodes == 0) return fail(ctx, VADUSA_ESTATE, "no tree set");
  if (!tree_tokens_override && !ctx->have_draft) return fail(ctx, VADUSA_ESTATE, "verify without a draft or an override");
  if (!tree_tokens_override && ctx->tree_per_seq) return fail(ctx, VADUSA_ESTATE, "per-sequence topologies need a token override");
  const TreeView tv = tree_of(ctx, false);
  const vadusa_config& c = ctx->cfg;
  const int M = ctx->batch * tv.n_nodes;
  const std::string key = KeyBuilder("verify").add(tree_tokens_override).add(logits_out).add(attn_tap).add(hidden_out)
                              .add(ctx->batch).add(ctx->n_nodes).add(ctx->tree_per_seq).add(ctx->block_table)
                              .add(attention_splits(ctx, ctx->n_nodes)).add(ctx->fused_enabled).add(ctx->att_stream).k;
  vadusa_status s = run_graphed(ctx, key, [&]() -> vadusa_status {
    vadusa_status s = DISPATCH(forward<float>(ctx, tv, tree_tokens_override, reinterpret_cast<float*>(attn_tap)),
                               forward<bf16>(ctx, tv, tree_tokens_override, reinterpret_cast<bf16*>(attn_tap)));
    if (s) return s;
    if (logits_out)
      CU(cudaMemcpy2DAsync(logits_out, (size_t)c.vocab * 4, ctx->wsp + ctx->ws.logits, (size_t)vpad(&c) * 4,
                           (size_t)c.vocab * 4, M, cudaMemcpyDeviceToDevice, ctx->stream));
    if (hidden_out)
      CU(cudaMemcpyAsync(hidden_out, ctx->wsp + ctx->ws.hfinal, (size_t)M * c.d_model * esize(&c), cudaMemcpyDeviceToDevice, ctx->stream));
    return VADUSA_OK;
  });
  if (s) return s;
  ctx->have_verify = true;
  return VADUSA_OK;
}

vadusa_status vadusa_accept_and_commit(vadusa_ctx* ctx, const vadusa_sampling* sampling, const int32_t* forced_best_node,
                                       int32_t* accept_len, int32_t* path_nodes, int32_t* path_tokens,
                                       int64_t* kv_slots, uint64_t* edge_bits, int32_t* next_root) {
  if (vadusa_status s = need_batch(ctx)) return s;
  if (!ctx->have_verify) return fail(ctx, VADUSA_ESTATE, "accept without a verify step");
  SamplingDev sp;
  if (vadusa_status s = sampling_dev(ctx, sampling, &sp)) return s;
  AcceptOut out{accept_len, path_nodes, path_tokens, reinterpret_cast<long long*>(kv_slots),
                reinterpret_cast<unsigned long long*>(edge_bits), ctx->cfg.max_tree_nodes > 64 ? 2 : 1, next_root};
  const std::string key = KeyBuilder("accept").add(sp).add(forced_best_node).add(out).add(ctx->batch).add(ctx->n_nodes)
                              .add(ctx->tree_per_seq).add(ctx->block_table).k;
  vadusa_status s = run_graphed(ctx, key, [&]() -> vadusa_status {
    return DISPATCH(accept_commit<float>(ctx, sp, forced_best_node, out, nullptr, 0, 0),
                    accept_commit<bf16>(ctx, sp, forced_best_node, out, nullptr, 0, 0));
  });
  if (s) return s;
  ctx->ctx_bound += ctx->tree_max_depth + 1;
  ctx->ctx_lo += 1;
  ctx->h_ctx_exact = false;
  ctx->have_verify = ctx->have_draft = false;
  return VADUSA_OK;
}

vadusa_status vadusa_generate(vadusa_ctx* ctx, const vadusa_sampling* sampling, int32_t max_new_tokens,
                              int32_t max_iters, int32_t* out_tokens, int32_t* out_len, vadusa_stats* h_stats) {
  return run_generate(ctx, sampling, max_new_tokens, max_iters, out_tokens, out_len, nullptr, nullptr, h_stats);
}

vadusa_status vadusa_generate_host(vadusa_ctx* ctx, const vadusa_sampling* sampling, int32_t batch,
                                   const int32_t* block_table, const int32_t* h_tokens, const int32_t* h_len,
                                   int32_t stride, int32_t max_new_tokens, int32_t* h_out_tokens,
                                   int32_t* h_out_len, vadusa_stats* h_stats) {
  if (!ctx) return VADUSA_EINVAL;
  if (!h_out_tokens || !h_out_len) return fail(ctx, VADUSA_EINVAL, "output pointers are NULL");
  if (max_new_tokens < 1 || max_new_tokens > kGenHostCap)
    return fail(ctx, VADUSA_EINVAL, "vadusa_generate_host: max_new_tokens must be in 1..%d", kGenHostCap);
  vadusa_status s = vadusa_begin(ctx, batch, block_table, nullptr);
  if (s) return s;
  s = vadusa_prefill(ctx, h_tokens, h_len, stride);
  if (s) return s;
  return run_generate(ctx, sampling, max_new_tokens, 0, wsptr<int32_t>(ctx, ctx->ws.gen_out), nullptr, h_out_tokens, h_out_len, h_stats);
}

vadusa_status vadusa_get_lengths(vadusa_ctx* ctx, int32_t* h_ctx_len) {
  if (vadusa_status s = need_batch(ctx)) return s;
  if (!h_ctx_len) return fail(ctx, VADUSA_EINVAL, "h_ctx_len is NULL");
  CU(cudaMemcpyAsync(h_ctx_len, ctx->wsp + ctx->ws.ctx_len, ctx->batch * 4, cudaMemcpyDeviceToHost, ctx->stream));
  if (vadusa_status s = device_errors(ctx)) return s;       // (synchronises)
  long long longest = 0;
  for (int b = 0; b < ctx->batch; ++b) longest = h_ctx_len[b] > longest ? h_ctx_len[b] : longest;
  ctx->ctx_lo = ctx->ctx_bound = longest;                   // both estimates are exact again
  ctx->h_ctx.assign(h_ctx_len, h_ctx_len + ctx->batch);
  ctx->h_ctx_exact = true;
  return VADUSA_OK;
}

vadusa_status vadusa_check(vadusa_ctx* ctx) {
  if (!ctx || !ctx->wsp) return VADUSA_EINVAL;
  return device_errors(ctx);
}

vadusa_status vadusa_set_logit_bias(vadusa_ctx* ctx, const float* bias, int32_t ld) {
  if (!ctx) return VADUSA_EINVAL;
  if (!ctx->wsp) return fail(ctx, VADUSA_ESTATE, "context is not initialised");
  if (bias && ld < ctx->cfg.vocab) return fail(ctx, VADUSA_EINVAL, "bias rows must hold at least vocab entries");
  ctx->logit_bias = bias;
  ctx->logit_bias_ld = bias ? ld : 0;
  return VADUSA_OK;
}

vadusa_status vadusa_accept_stats(vadusa_ctx* ctx, int64_t* h_tested, int64_t* h_accepted, int32_t reset) {
  if (!ctx) return VADUSA_EINVAL;
  if (!ctx->wsp) return fail(ctx, VADUSA_ESTATE, "context is not initialised");
  if (!h_tested || !h_accepted) return fail(ctx, VADUSA_EINVAL, "statistics arrays are NULL");
  const size_t n = (size_t)kStatDepth * kStatTopk;
  static_assert(sizeof(int64_t) == sizeof(unsigned long long), "counter width");
  CU(cudaMemcpyAsync(h_tested, ctx->wsp + ctx->ws.acc_stats, n * 8, cudaMemcpyDeviceToHost, ctx->stream));
  CU(cudaMemcpyAsync(h_accepted, ctx->wsp + ctx->ws.acc_stats + n * 8, n * 8, cudaMemcpyDeviceToHost, ctx->stream));
  if (reset) CU(cudaMemsetAsync(ctx->wsp + ctx->ws.acc_stats, 0, 2 * n * 8, ctx->stream));
  CU(cudaStreamSynchronize(ctx->stream));
  return VADUSA_OK;
}

vadusa_status vadusa_build_sparse_tree(const double* h_prob, int32_t depth, int32_t topk, int32_t n_nodes,
                                       int32_t* h_parent, int32_t* h_rank, double* h_expected_len) {
  if (!h_prob || !h_parent || !h_rank) return VADUSA_EINVAL;
  if (depth < 1 || depth > VADUSA_MAX_DEPTH || topk < 1 || topk > VADUSA_MAX_DRAFT_TOPK) return VADUSA_EINVAL;
  if (n_nodes < 1 || n_nodes > VADUSA_MAX_TREE_NODES) return VADUSA_EINVAL;
  struct Node { std::vector<int> path; double p; };
  auto before = [](const Node& a, const Node& b) {       // higher probability, then shallower, then smaller path
    if (a.p != b.p) return a.p > b.p;
    if (a.path.size() != b.path.size()) return a.path.size() < b.path.size();
    return a.path < b.path;
  };
  std::vector<Node> tree(1, Node{{}, 1.0}), frontier;
  auto grow = [&](const Node& parent) {
    if ((int)parent.path.size() == depth) return;
    for (int r = 0; r < topk; ++r) {
      Node c{parent.path, parent.p * h_prob[(size_t)parent.path.size() * topk + r]};
      c.path.push_back(r);
      frontier.push_back(c);
    }
  };
  grow(tree[0]);
  double expected = 1.0;
  while ((int)tree.size() < n_nodes) {
    if (frontier.empty()) return VADUSA_EINVAL;
    size_t best = 0;
    for (size_t i = 1; i < frontier.size(); ++i)
      if (before(frontier[i], frontier[best])) best = i;
    const Node pick = frontier[best];
    frontier.erase(frontier.begin() + (long)best);
    expected += pick.p;
    tree.push_back(pick);
    grow(pick);
  }
  std::sort(tree.begin(), tree.end(), [](const Node& a, const Node& b) {
    return a.path.size() != b.path.size() ? a.path.size() < b.path.size() : a.path < b.path;
  });
  std::map<std::vector<int>, int> index;
  for (int i = 0; i < n_nodes; ++i) index[tree[i].path] = i;
  for (int i = 0; i < n_nodes; ++i) {
    if (tree[i].path.empty()) { h_parent[i] = -1; h_rank[i] = 0; continue; }
    std::vector<int> up(tree[i].path.begin(), tree[i].path.end() - 1);
    h_parent[i] = index[up];
    h_rank[i] = tree[i].path.back();
  }
  if (h_expected_len) *h_expected_len = expected;
  return VADUSA_OK;
}

int64_t vadusa_fit_state_bytes(const vadusa_config* cfg, int32_t max_tokens) {
  if (check_config(cfg) || max_tokens < 1) return -1;
  return fit_layout(cfg, max_tokens).total;
}

vadusa_status vadusa_fit_begin(vadusa_ctx* ctx, void* state, int64_t state_bytes, int32_t max_tokens, float lambda,
                               float learning_rate, int32_t warmup_steps) {
  if (!ctx) return VADUSA_EINVAL;
  if (!ctx->wsp) return fail(ctx, VADUSA_ESTATE, "context is not initialised");
  if (!state || max_tokens < 1 || ((uintptr_t)state & 255)) return fail(ctx, VADUSA_EINVAL, "fit state is NULL, unaligned or sized for no token");
  if (!(lambda > 0.f && lambda <= 1.f) || !(learning_rate > 0.f) || warmup_steps < 0) return fail(ctx, VADUSA_EINVAL, "lambda must be in (0, 1], the learning rate positive");
  const FitLayout f = fit_layout(&ctx->cfg, max_tokens);
  if (state_bytes < f.total) return fail(ctx, VADUSA_ENOMEM, "fit state has %lld bytes, %lld needed", (long long)state_bytes, (long long)f.total);
  if (ctx->cfg.n_draft_heads > 1 && ctx->dw_stride != (long long)ctx->cfg.d_model * ctx->cfg.d_model * esize(&ctx->cfg))
    return fail(ctx, VADUSA_EINVAL, "draft matrices are not contiguous");
  ctx->fit = reinterpret_cast<char*>(state);
  ctx->fit_tokens = max_tokens; ctx->fit_step = 0; ctx->fit_warmup = warmup_steps;
  ctx->fit_lambda = lambda; ctx->fit_lr = learning_rate;
  return DISPATCH(fit_begin<float>(ctx, f), fit_begin<bf16>(ctx, f));
}

vadusa_status vadusa_fit_step(vadusa_ctx* ctx, const void* hidden, const int32_t* targets, int32_t n_tokens, float* loss_out) {
  if (!ctx) return VADUSA_EINVAL;
  if (!ctx->fit) return fail(ctx, VADUSA_ESTATE, "vadusa_fit_begin has not been called");
  if (!hidden || !targets || n_tokens < 1 || n_tokens > ctx->fit_tokens) return fail(ctx, VADUSA_EINVAL, "fit step: NULL input or token count out of range");
  const FitLayout f = fit_layout(&ctx->cfg, ctx->fit_tokens);
  ctx->have_draft = false;
  return DISPATCH(fit_step<float>(ctx, f, reinterpret_cast<const float*>(hidden), targets, n_tokens, loss_out),
                  fit_step<bf16>(ctx, f, reinterpret_cast<const bf16*>(hidden), targets, n_tokens, loss_out));
}

vadusa_status vadusa_fit_end(vadusa_ctx* ctx) {
  if (!ctx) return VADUSA_EINVAL;
  ctx->fit = nullptr;
  return VADUSA_OK;
}

vadusa_status vadusa_set_prefill_tap(vadusa_ctx* ctx, void* hidden_out, int32_t stride) {
  if (!ctx) return VADUSA_EINVAL;
  if (hidden_out && stride < 1) return fail(ctx, VADUSA_EINVAL, "prefill tap: stride must be positive");
  ctx->pf_tap = hidden_out;
  ctx->pf_tap_stride = hidden_out ? stride : 0;
  return VADUSA_OK;
}

int64_t vadusa_kernel_launches(const vadusa_ctx* ctx) { return ctx ? ctx->launches : 0; }

int32_t vadusa_fused_pass_clusters(const vadusa_ctx* ctx) { return ctx ? ctx->fused_clusters : -1; }

vadusa_status vadusa_set_attention_stream(vadusa_ctx* ctx, int32_t enable) {
  if (!ctx) return VADUSA_EINVAL;
  if (enable != 0 && enable != 1) return fail(ctx, VADUSA_EINVAL, "enable must be 0 or 1");
  ctx->att_stream = enable;
  return VADUSA_OK;
}

vadusa_status vadusa_set_fused_pass(vadusa_ctx* ctx, int32_t enable) {
  if (!ctx) return VADUSA_EINVAL;
  if (enable != 0 && enable != 1 && enable != 6 && enable != 8) return fail(ctx, VADUSA_EINVAL, "enable must be 0, 1, 6 or 8");
  ctx->fused_enabled = enable;
  return VADUSA_OK;
}

vadusa_status vadusa_profile_begin(vadusa_ctx* ctx) {
  if (!ctx || !ctx->wsp) return VADUSA_EINVAL;
  for (auto& r : ctx->prof) { cudaEventDestroy(r.a); cudaEventDestroy(r.b); }
  ctx->prof.clear();
  ctx->prof_on = true;
  ctx->prof_pending = false;
  return VADUSA_OK;
}

vadusa_status vadusa_profile_end(vadusa_ctx* ctx, vadusa_kernel_time* h_out, int32_t capacity, int32_t* h_count) {
  if (!ctx || !ctx->wsp) return VADUSA_EINVAL;
  if (!h_out || !h_count || capacity < K_NCLASS) return fail(ctx, VADUSA_EINVAL, "profile output needs room for %d entries", (int)K_NCLASS);
  ctx->prof_on = false;
  CU(cudaStreamSynchronize(ctx->stream));
  double total[K_NCLASS] = {0};
  int64_t count[K_NCLASS] = {0};
  for (auto& r : ctx->prof) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, r.a, r.b) == cudaSuccess) { total[r.cls] += ms; count[r.cls]++; }
    cudaEventDestroy(r.a); cudaEventDestroy(r.b);
  }
  ctx->prof.clear();
  int n = 0;
  for (int k = 0; k < K_NCLASS; ++k) {
    if (!count[k]) continue;
    memset(&h_out[n], 0, sizeof(h_out[n]));
    snprintf(h_out[n].name, sizeof(h_out[n].name), "%s", kClassName[k]);
    h_out[n].launches = count[k];
    h_out[n].total_ms = total[k];
    ++n;
  }
  *h_count = n;
  return VADUSA_OK;
}

}  // extern "C"
