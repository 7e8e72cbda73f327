// C-ABI layer of the d2Cache step: argument validation, the carve-up of the caller's workspace and
// the launch sequence of one step.  No device memory is allocated here.
#include <cuda.h>
#include <math.h>
#include <stdarg.h>
#include <string.h>

#include <new>
#include <vector>

#include "common.cuh"

namespace d2c {

static thread_local char g_err[512] = "";
void set_global_error(const char* fmt, ...) {
  va_list ap; va_start(ap, fmt); vsnprintf(g_err, sizeof(g_err), fmt, ap); va_end(ap);
}
const char* global_error() { return g_err; }

int sm_count_current() {
  static int count[kMaxDevices] = {};
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  if (dev >= 0 && dev < kMaxDevices && count[dev] > 0) return count[dev];
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
  if (dev >= 0 && dev < kMaxDevices) count[dev] = n;
  return n;
}

static thread_local long long g_launches = 0;
void count_launch(int n) { g_launches += n; }

static const char* const kPhaseNames[D2C_N_PHASES] = {
    "select", "gather_norm", "rmsnorm", "gemm_qkv", "rope_scatter", "attention", "gemm_o",
    "gemm_gate_up", "gemm_down", "lm_head", "rollout", "copy_out", "attn_abar"};
enum Phase { PH_SELECT = 0, PH_GATHER, PH_NORM, PH_QKV, PH_ROPE, PH_ATTN, PH_O, PH_GATEUP, PH_DOWN, PH_LM, PH_ROLLOUT, PH_OUT, PH_ABAR };

// Hands out 256-byte aligned pieces of a buffer; with base == null it only measures.
struct Carver {
  char* base; size_t off = 0;
  explicit Carver(void* b) : base(static_cast<char*>(b)) {}
  template <typename T> T* take(size_t count) {
    off = align_up(off, 256);
    T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
    off += count * sizeof(T);
    return p;
  }
};

struct Buffers {
  bf16 *kcache, *vcache; float *conf, *c, *key; int32_t *pred, *status;
  int32_t *sel_idx, *row_seq, *row_off, *lm_rows, *lm_off, *slot_of_pos, *rank_s, *rank_lm, *n_b, *nm_b;
  uint32_t* phi; float2* rope;
  bf16 *x, *xn, *qkv, *o, *hmid, *xm; float *lse, *abar, *ssq;
  float *st_max, *st_sum; int32_t* st_arg;
  float *u0, *u1, *partial;
  float* sk_partials; int32_t* sk_counters; long long* gemm_clocks; char* records;
  bf16* h0_stage; uint8_t* mask_stage; int32_t *forced_stage, *forced_off_stage; float *okey_stage, *oc_stage;
  int32_t* committed_stage;
};

static int rollout_depth(const d2c_config& c) {
  return (c.rollout_layers > 0 && c.rollout_layers < c.n_layers) ? c.rollout_layers : c.n_layers;
}
static const int kCounters = 2 * kSkMaxTiles + 2 * kPairCounters;
static int lm_tiles(int vocab) { return ceil_div(vocab, 128); }

// The fused QKV projection leaves only Q and, after attention, the log-sum-exp in activation buffers.  Each layer uses the
// next of up to six of them, so that the probabilities pass of a layer, on a stream of its own, may take longer than the layer
// without holding up the projections of the next ones.  The last layer uses the first.  As many are carved as the rows of one
// whole QKV buffer and of the buffers that share a place (see carve) leave room for, so that they cost no memory of their own:
// six for as many KV heads as query heads, five for 28 and 4.
static int q_buffers(const d2c_config& c) {
  const size_t d = c.d_model, hq_dh = (size_t)c.n_q_heads * c.head_dim, qkv_out = (size_t)(c.n_q_heads + 2 * c.n_kv_heads) * c.head_dim;
  const size_t stats = 6 * (size_t)lm_tiles(c.vocab), shared = stats < (size_t)c.d_ffn ? stats : (size_t)c.d_ffn;      // in elements of bf16
  const size_t n = (qkv_out + 2 * (d < hq_dh ? d : hq_dh) + shared) / hq_dh;
  return n < 6 ? (int)n : 6;
}
// Slots for parked parts: four for every cluster that the pair kernel can have at these sizes, and what the one-SM kernel may use.
static int sk_tiles(const d2c_config& c) {
  const int shapes[5][2] = {{(c.n_q_heads + 2 * c.n_kv_heads) * c.head_dim, c.d_model}, {c.d_model, c.n_q_heads * c.head_dim},
                            {2 * c.d_ffn, c.d_model}, {c.d_model, c.d_ffn}, {c.vocab, c.d_model}};      // {weight rows, K}
  const long long rows = (long long)c.max_batch * c.max_seq;
  long long most = 0;
  for (const auto& s : shapes) {
    const long long n = rows >= kPairRows ? gemm_tc2_clusters(ceil_div(s[0], 256), rows, s[1]) : 0;
    most = n > most ? n : most;
  }
  const long long n = 4 * most < kSkMaxTiles ? 4 * most : kSkMaxTiles;
  return n > 160 ? (int)n : 160;
}
// Pieces that are never live at the same time share a place: the attention output of the layers, the LM head's rows and the
// staged h0 (read by the first kernel behind selection); the FFN's middle and the LM head's statistics.
static size_t carve(const d2c_config& c, void* base, Buffers* out) {
  Carver w(base);
  Buffers b;
  const size_t B = c.max_batch, L = c.max_seq, R = B * L, d = c.d_model, n_q = q_buffers(c);
  const size_t hq_dh = (size_t)c.n_q_heads * c.head_dim, kv = (size_t)c.n_kv_heads * c.head_dim, qkv_out = (size_t)(c.n_q_heads + 2 * c.n_kv_heads) * c.head_dim;
  b.kcache = w.take<bf16>((size_t)c.n_layers * R * kv);
  b.vcache = w.take<bf16>((size_t)c.n_layers * R * kv);
  b.conf = w.take<float>(R); b.c = w.take<float>(R); b.key = w.take<float>(R);
  b.pred = w.take<int32_t>(R); b.status = w.take<int32_t>(64);                 // (four status words; counters of the one-launch step from the 32nd on)
  b.sel_idx = w.take<int32_t>(R); b.row_seq = w.take<int32_t>(R); b.row_off = w.take<int32_t>(B + 1);
  b.lm_rows = w.take<int32_t>(R); b.lm_off = w.take<int32_t>(B + 1); b.slot_of_pos = w.take<int32_t>(R);
  b.rank_s = w.take<int32_t>(R); b.rank_lm = w.take<int32_t>(R); b.n_b = w.take<int32_t>(B); b.nm_b = w.take<int32_t>(B);
  b.phi = w.take<uint32_t>(L); b.rope = w.take<float2>(L * (c.head_dim / 2));
  b.x = w.take<bf16>(R * d); b.xn = w.take<bf16>(R * d); b.qkv = w.take<bf16>(R * (qkv_out > n_q * hq_dh ? qkv_out : n_q * hq_dh));
  b.o = b.xm = b.h0_stage = w.take<bf16>(R * (d > hq_dh ? d : hq_dh));
  const size_t stat = align_up(R * lm_tiles(c.vocab) * sizeof(float), 256), mid = R * (size_t)c.d_ffn * sizeof(bf16);
  char* shared = w.take<char>(3 * stat > mid ? 3 * stat : mid);
  b.hmid = reinterpret_cast<bf16*>(shared);
  b.st_max = reinterpret_cast<float*>(shared); b.st_sum = reinterpret_cast<float*>(shared + stat); b.st_arg = reinterpret_cast<int32_t*>(shared + 2 * stat);
  b.lse = w.take<float>(n_q * R * (size_t)c.n_q_heads);
  b.ssq = w.take<float>(R * (d / 32));                      // per (row, 32 columns): sum of squares of the residual stream
  b.abar = w.take<float>((size_t)rollout_depth(c) * R * L);
  b.u0 = w.take<float>(R); b.u1 = w.take<float>(R);
  b.partial = w.take<float>((size_t)kRolloutSplit * R + (R + 3) / 4);     // partial sums + selected-flag bytes
  b.sk_partials = w.take<float>((size_t)sk_tiles(c) * 128 * 256); b.sk_counters = w.take<int32_t>(kCounters);     // the one-SM kernel's arrival and done counters, two sets of the pair kernel's
  b.gemm_clocks = w.take<long long>(4);
  b.records = R >= kPairRows ? w.take<char>((size_t)kWorkPlans * kWorkClusters * kWorkRecordBytes) : nullptr;
  b.mask_stage = w.take<uint8_t>(R);
  b.forced_stage = w.take<int32_t>(R); b.forced_off_stage = w.take<int32_t>(B + 1);
  b.okey_stage = w.take<float>(R); b.oc_stage = w.take<float>(R); b.committed_stage = w.take<int32_t>(B);
  if (out) *out = b;
  return align_up(w.off, 256);
}

static const char* check_config(const d2c_config* c) {
  if (!c) return "config is null";
  if (c->n_layers < 1 || c->d_model < 64 || c->n_q_heads < 1 || c->n_kv_heads < 1 || c->d_ffn < 64 || c->vocab < 2)
    return "non-positive model dimension";
  if (c->head_dim != 64 && c->head_dim != 128) return "head_dim must be 64 or 128";
  if (c->d_model % 64 || c->d_ffn % 64 || (c->n_q_heads * c->head_dim) % 64) return "d_model, d_ffn and n_q_heads*head_dim must be multiples of 64";
  if (c->n_q_heads % c->n_kv_heads) return "n_q_heads must be a multiple of n_kv_heads";
  if (c->vocab & 1) return "vocab must be even";
  if (c->max_batch < 1 || c->max_seq < 1 || c->max_seq > 8192) return "max_batch >= 1 and 1 <= max_seq <= 8192 required";
  if (!(c->rope_base > 1.f) || !(c->rms_eps >= 0.f) || !(c->sigma > 0.f)) return "rope_base > 1, rms_eps >= 0, sigma > 0 required";
  if (c->stage2_candidates != 0 && c->stage2_candidates != 1) return "stage2_candidates must be 0 or 1";
  if (c->rollout_layers < 0 || (c->flags & ~(D2C_FLAG_PORTABLE_GEMM | D2C_FLAG_PORTABLE_ATTENTION | D2C_FLAG_ONE_SM_GEMM | D2C_FLAG_SERIAL | D2C_FLAG_FOLDED_NORMS))) return "rollout_layers >= 0 and no unknown flag bits required";
  return nullptr;
}

}  // namespace d2c

using namespace d2c;

struct d2c_ctx {
  d2c_config cfg;
  std::vector<const bf16*> wqkv, bqkv, wo, w_gate, w_up, w_down, g_attn, g_ffn;
  const bf16 *g_final, *w_lm;
  cudaStream_t stream;
  Buffers buf;
  int phi_len, q_bufs, sk_tiles;
  // Selected-row count of the previous step, which chooses between the GEMM kernels (both are correct for any
  // count, but they add fp32 partial sums in different orders).  The selection kernel writes the count into one
  // of two words of mapped host memory; the next step waits for the event recorded behind that kernel before it
  // reads the word, so the choice depends on the step sequence only, never on how far the host runs ahead.
  int32_t* hint_host[2] = {nullptr, nullptr};
  int32_t* hint_dev[2] = {nullptr, nullptr};
  cudaEvent_t ev_hint[2] = {nullptr, nullptr};
  long long hint_step[2] = {-1, -1};     // step number whose count the word holds
  bool hint_tagged[2] = {false, false};  // it was a step in one launch: it writes its number and the count as one 64-bit word
  long long step_no = 0;
  int asked_k = 0; float asked_p = 0.f;  // rows of stage 1 at most, and mass of stage 2, that the step before asked for
  bool few_rows = false;                 // this step's regime: at most 128 rows expected
  std::vector<MapCache> maps;            // six launches of each layer (QKV, forward, probabilities, output, gate/up, down), LM head
  int max_pairs = 0;                     // SM pairs the projections of this step may use (0: all)
  int narrow_pairs = 0;                  // those 64-token tiles may spread over (0: all)
  int lm_pairs = 0;                      // those the LM head may use (0: all)
  int small_clusters = 0;                // clusters of the kernel that does the whole step (0: the model is not one for it)
  bool host_call = false, h0_far = false;      // in d2c_step_host; its h0 lies in host memory
  WorkPlan plan{};                       // the pair kernel's launches of the current step
  int pair_launches = 0;                 // how many of them are enqueued
  int used_batch = 0, used_seq = 0;      // the (batch, seq_len) of the first step: the per-position state is laid out for it
  // d2c_step_host: the device-to-host copy of the hidden rows runs on its own stream, ordered after the
  // last layer by an event, so that it overlaps the LM head and the rollout
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t layers_done = nullptr;
  void* early_hidden_host = nullptr;     // set by d2c_step_host for the duration of one step
  void* early_hidden_dev = nullptr;      // the same buffer as the device sees it: only the live rows are written (null: copy all)
  // The head-averaged probabilities and the rollout feed only the next step's selection.  They run on a
  // low-priority stream beside the projections, the FFN and the LM head, filling the SMs those leave idle
  // (partial last waves); the rest of the step runs on a high-priority stream so that it wins every SM it
  // can use.  Both are forked from and joined to the caller's stream by events inside d2c_step.
  cudaStream_t work_stream = nullptr, side_stream = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr, ev_fwd = nullptr, ev_side = nullptr, ev_begun = nullptr, ev_abar[4] = {};      // ev_abar: layers l, l + 4, ... share one
  cudaStream_t run = nullptr;            // where the current step's critical path is enqueued
  char err[512];
  // optional per-phase timing: one event at every phase boundary, resolved by d2c_profile_read
  bool prof = false;
  std::vector<cudaEvent_t> ev;
  std::vector<int> ev_phase;      // phase that starts at event i, -1 = end of a step
  size_t ev_used = 0;
  double phase_ms[D2C_N_PHASES] = {0};
  long long phase_launches[D2C_N_PHASES] = {0};
  long long launch_mark = 0;
  int prof_phase = -1;
};

static void destroy_overlap(d2c_ctx* ctx) {
  if (ctx->work_stream) cudaStreamDestroy(ctx->work_stream);
  if (ctx->side_stream) cudaStreamDestroy(ctx->side_stream);
  for (cudaEvent_t* ev : {&ctx->ev_in, &ctx->ev_out, &ctx->ev_fwd, &ctx->ev_side, &ctx->ev_begun, &ctx->ev_abar[0], &ctx->ev_abar[1], &ctx->ev_abar[2], &ctx->ev_abar[3]}) {
    if (*ev) cudaEventDestroy(*ev);
    *ev = nullptr;
  }
  ctx->work_stream = ctx->side_stream = nullptr;
}

// Marks the start of `phase` (or the end of the step with phase < 0) on the context's stream.
static int mark(d2c_ctx* ctx, int phase) {
  if (!ctx->prof) return D2C_OK;
  if (ctx->prof_phase >= 0) ctx->phase_launches[ctx->prof_phase] += g_launches - ctx->launch_mark;
  ctx->launch_mark = g_launches; ctx->prof_phase = phase;
  if (ctx->ev_used == ctx->ev.size()) {
    cudaEvent_t e;
    D2C_CUDA_OK(cudaEventCreate(&e));
    ctx->ev.push_back(e); ctx->ev_phase.push_back(-1);
  }
  ctx->ev_phase[ctx->ev_used] = phase;
  D2C_CUDA_OK(cudaEventRecord(ctx->ev[ctx->ev_used], ctx->stream));
  ctx->ev_used++;
  return D2C_OK;
}

static int fail(d2c_ctx* ctx, int code, const char* fmt, ...) {
  char tmp[512];
  va_list ap; va_start(ap, fmt); vsnprintf(tmp, sizeof(tmp), fmt, ap); va_end(ap);
  if (ctx) { strncpy(ctx->err, tmp, sizeof(ctx->err) - 1); ctx->err[sizeof(ctx->err) - 1] = 0; }
  set_global_error("%s", tmp);
  return code;
}
// Propagates an error raised by a launcher (its text is in the thread-local slot).
static int pass(d2c_ctx* ctx, int rc) {
  if (rc != D2C_OK && ctx) { strncpy(ctx->err, global_error(), sizeof(ctx->err) - 1); ctx->err[sizeof(ctx->err) - 1] = 0; }
  return rc;
}
// A product with what the pair kernel needs from the context.
static GemmArgs pair_args(const d2c_ctx* ctx, const GemmArgs& g, GemmEpilogue epi) {
  GemmArgs g2 = g;
  g2.narrow_pairs = ctx->narrow_pairs;
  g2.max_pairs = epi == EPI_LMSTATS ? ctx->lm_pairs : ctx->max_pairs;
  g2.sk_partials = ctx->buf.sk_partials; g2.sk_counters = ctx->buf.sk_counters; g2.sk_max_tiles = ctx->sk_tiles;
  return g2;
}
// Notes that the step has such a product, for the kernel that writes the records of its launches.
static void plan_pair(d2c_ctx* ctx, const GemmArgs& g, GemmEpilogue epi) {
  WorkPlan& p = ctx->plan;
  if ((ctx->cfg.flags & (D2C_FLAG_PORTABLE_GEMM | D2C_FLAG_ONE_SM_GEMM)) || !ctx->buf.records || !gemm_tc2_supported(g) || p.n == kWorkPlans) return;
  const WorkShape s = gemm_tc2_shape(pair_args(ctx, g, epi), epi);
  if (s.clusters > kWorkClusters) return;
  p.lm[p.n] = epi == EPI_LMSTATS;
  p.shape[p.n++] = s;
}
// The step's GEMMs: tcgen05 kernel unless the context was created with D2C_FLAG_PORTABLE_GEMM.  use_records: the kernel that
// writes them is complete when this launch starts.
static int gemm(d2c_ctx* ctx, const GemmArgs& g, GemmEpilogue epi, bool use_records = true) {
  if (ctx->cfg.flags & D2C_FLAG_PORTABLE_GEMM) return launch_gemm_mma(g, epi, ctx->run);
  if (!(ctx->cfg.flags & D2C_FLAG_ONE_SM_GEMM) && gemm_tc2_supported(g))
  {
    GemmArgs g2 = pair_args(ctx, g, epi);
    const WorkShape s = gemm_tc2_shape(g2, epi);
    for (int i = 0; i < ctx->plan.n && use_records; ++i) {
      const WorkShape& t = ctx->plan.shape[i];
      if (t.blocks == s.blocks && t.K == s.K && t.clusters == s.clusters && t.slots == s.slots && ctx->plan.lm[i] == (epi == EPI_LMSTATS))
        g2.records = ctx->plan.records + (size_t)i * kWorkClusters * kWorkRecordBytes;
    }
    int32_t* sets = ctx->buf.sk_counters + 2 * kSkMaxTiles;                // (see the kernel: launches take turns)
    const int turn = ctx->pair_launches++ & 1;
    g2.sk_counters = sets + turn * kPairCounters; g2.sk_clear = sets + (turn ^ 1) * kPairCounters;
    return launch_gemm_tc2(g2, epi, ctx->run, ctx->buf.status);
  }
  GemmArgs gs = g;
  gs.sk_partials = ctx->buf.sk_partials; gs.sk_counters = ctx->buf.sk_counters; gs.sk_max_tiles = ctx->sk_tiles;
  return launch_gemm_tc(gs, epi, ctx->run, ctx->buf.status);
}
// A CUDA runtime call inside the step: its error text goes where launcher errors go.
static int cu(cudaError_t e) {
  if (e == cudaSuccess) return D2C_OK;
  set_global_error("d2c_step: %s", cudaGetErrorString(e));
  return D2C_ECUDA;
}
// The device's address of a host buffer that kernels may use in place: all of its bytes lie in one pinned allocation or
// registration (the first byte's attributes are not enough: a registered range may end inside the buffer, and a kernel that
// runs past it faults where a copy returns an error), and it starts at a word.  Null for every other buffer, which is copied.
static void* mapped(const void* p, size_t bytes) {
  typedef CUresult (*GetAttributes)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
  static GetAttributes get = []() -> GetAttributes {                       // (the library does not link libcuda)
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    const bool ok = cudaGetDriverEntryPoint("cuPointerGetAttributes", &fn, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess;
    if (!ok) (void)cudaGetLastError();
    return ok ? reinterpret_cast<GetAttributes>(fn) : nullptr;
  }();
  cudaPointerAttributes at;
  if (!p || bytes == 0 || !get) return nullptr;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) { (void)cudaGetLastError(); return nullptr; }
  if (at.type != cudaMemoryTypeHost || !at.devicePointer || reinterpret_cast<uintptr_t>(at.devicePointer) % 4) return nullptr;
  CUdeviceptr start = 0;
  size_t size = 0;
  CUpointer_attribute what[2] = {CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
  void* to[2] = {&start, &size};
  const CUdeviceptr first = reinterpret_cast<CUdeviceptr>(at.devicePointer);
  if (get(2, what, to, first) != CUDA_SUCCESS) return nullptr;
  return first >= start && first - start <= size && bytes <= size - (first - start) ? at.devicePointer : nullptr;
}
#define D2C_TRY(ctx, expr) do { int rc__ = (expr); if (rc__ != D2C_OK) return pass((ctx), rc__); } while (0)

// The arguments of a step in one launch, but for those of the call.
static SmallArgs small_args(const d2c_ctx* ctx, int batch, int seq_len) {
  const d2c_config& c = ctx->cfg;
  const Buffers& b = ctx->buf;
  SmallArgs a{};
  a.sel.batch = batch; a.sel.seq_len = seq_len;
  for (int l = 0; l < c.n_layers; ++l)
    a.layer[l] = SmallLayer{ctx->wqkv[l], ctx->bqkv[l], ctx->wo[l], ctx->w_gate[l], ctx->w_up[l], ctx->w_down[l], ctx->g_attn[l], ctx->g_ffn[l]};
  a.g_final = ctx->g_final; a.w_lm = ctx->w_lm;
  a.n_layers = c.n_layers; a.d = c.d_model; a.hq = c.n_q_heads; a.hkv = c.n_kv_heads; a.ffn = c.d_ffn; a.vocab = c.vocab;
  a.cache_seq = c.max_seq; a.depth = rollout_depth(c); a.eps = c.rms_eps;
  a.rope = b.rope; a.kc = b.kcache; a.vc = b.vcache; a.cache_layer = (size_t)c.max_batch * c.max_seq * c.n_kv_heads * c.head_dim;
  a.q = b.qkv; a.o = b.o; a.hmid = b.hmid; a.lse = b.lse; a.abar = b.abar; a.abar_layer = (size_t)c.max_batch * c.max_seq * c.max_seq;
  a.c = b.c; a.conf = b.conf; a.pred = b.pred;
  a.clear = b.sk_counters; a.n_clear = kCounters;
  a.sync = reinterpret_cast<uint32_t*>(b.status) + 32; a.status = b.status;
  return a;
}
// Clusters of the kernel that does a whole step, 0 where the model is not one for it.
static int small_clusters(const d2c_ctx* ctx) {
  const d2c_config& c = ctx->cfg;
  const int hq_dh = c.n_q_heads * c.head_dim, qkv_out = (c.n_q_heads + 2 * c.n_kv_heads) * c.head_dim;
  if ((c.flags & ~D2C_FLAG_SERIAL) || c.head_dim != 64 || c.n_layers > kSmallMaxLayers || c.max_batch > kSmallMaxBatch) return 0;
  if (c.d_model < 256 || c.d_model > 512 || hq_dh > 512 || c.d_ffn > 1024 || c.max_seq > 8192) return 0;
  // (every CTA has columns of the products of the layers; the LM head may leave some without)
  if (c.d_ffn < 8 * kSmallCluster || qkv_out < 16 * kSmallCluster || (long long)c.vocab * c.d_model > (1 << 20)) return 0;
  uintptr_t low = reinterpret_cast<uintptr_t>(ctx->g_final) | reinterpret_cast<uintptr_t>(ctx->w_lm);      // (the layers' are checked; a bias may lie anywhere)
  for (const bf16* p : ctx->bqkv) low |= reinterpret_cast<uintptr_t>(p);
  if (low % 16) return 0;
  const SmallArgs a = small_args(ctx, c.max_batch, c.max_seq);
  const int most = small_step_clusters(), tiles = c.max_batch * ceil_div(c.max_seq, 16), n = most < tiles ? most : tiles;
  if (n == 0 || n > kSmallMaxClusters || ceil_div(tiles, n) > kSmallMaxTiles || n * kSmallCluster < c.max_batch) return 0;
  return small_step_scratch(a, n, nullptr, nullptr) <= (size_t)ctx->sk_tiles * 128 * 256 ? n : 0;
}

extern "C" {

size_t d2c_workspace_bytes(const d2c_config* cfg) {
  if (check_config(cfg)) return 0;
  return carve(*cfg, nullptr, nullptr);
}

int d2c_create(const d2c_config* cfg, const d2c_weights* w, void* workspace, size_t workspace_bytes,
               void* cuda_stream, d2c_ctx** out) {
  if (!out) return fail(nullptr, D2C_EINVAL, "d2c_create: out is null");
  *out = nullptr;
  if (const char* why = check_config(cfg)) return fail(nullptr, cfg ? D2C_ESHAPE : D2C_EINVAL, "d2c_create: %s", why);
  if (!w || !workspace) return fail(nullptr, D2C_EINVAL, "d2c_create: weights or workspace is null");
  if (reinterpret_cast<uintptr_t>(workspace) % 256) return fail(nullptr, D2C_EINVAL, "d2c_create: workspace must be 256-byte aligned");
  const size_t need = carve(*cfg, nullptr, nullptr);
  if (workspace_bytes < need) return fail(nullptr, D2C_ECAPACITY, "d2c_create: workspace %zu bytes < %zu needed", workspace_bytes, need);
  if (!w->wqkv || !w->wo || !w->w_gate || !w->w_up || !w->w_down || !w->g_attn || !w->g_ffn || !w->g_final || !w->w_lm ||
      (cfg->qkv_bias && !w->bqkv))
    return fail(nullptr, D2C_EINVAL, "d2c_create: a weight pointer is null");
  d2c_ctx* ctx = new (std::nothrow) d2c_ctx();
  if (!ctx) return fail(nullptr, D2C_EINVAL, "d2c_create: out of host memory");
  ctx->cfg = *cfg; ctx->err[0] = 0;
  ctx->stream = static_cast<cudaStream_t>(cuda_stream);
  for (int l = 0; l < cfg->n_layers; ++l) {
    const void* ptrs[] = {w->wqkv[l], w->wo[l], w->w_gate[l], w->w_up[l], w->w_down[l], w->g_attn[l], w->g_ffn[l]};
    for (const void* p : ptrs)
      if (!p || reinterpret_cast<uintptr_t>(p) % 16) { delete ctx; return fail(nullptr, D2C_EINVAL, "d2c_create: layer %d weight pointer null or not 16-byte aligned", l); }
    ctx->wqkv.push_back((const bf16*)w->wqkv[l]); ctx->wo.push_back((const bf16*)w->wo[l]);
    ctx->w_gate.push_back((const bf16*)w->w_gate[l]); ctx->w_up.push_back((const bf16*)w->w_up[l]);
    ctx->w_down.push_back((const bf16*)w->w_down[l]); ctx->g_attn.push_back((const bf16*)w->g_attn[l]);
    ctx->g_ffn.push_back((const bf16*)w->g_ffn[l]);
    ctx->bqkv.push_back(cfg->qkv_bias ? (const bf16*)w->bqkv[l] : nullptr);
    if (cfg->qkv_bias && !w->bqkv[l]) { delete ctx; return fail(nullptr, D2C_EINVAL, "d2c_create: layer %d bias is null", l); }
  }
  ctx->maps.resize(6 * (size_t)cfg->n_layers + 1);
  ctx->g_final = (const bf16*)w->g_final; ctx->w_lm = (const bf16*)w->w_lm;
  carve(*cfg, workspace, &ctx->buf);
  ctx->q_bufs = q_buffers(*cfg); ctx->sk_tiles = sk_tiles(*cfg);
  ctx->small_clusters = small_clusters(ctx);
  {
    bool ok = cudaHostAlloc(reinterpret_cast<void**>(&ctx->hint_host[0]), 4 * sizeof(int32_t), cudaHostAllocMapped) == cudaSuccess;
    if (ok) {
      ctx->hint_host[1] = ctx->hint_host[0] + 2;
      ctx->hint_host[0][0] = ctx->hint_host[1][0] = 1 << 30; ctx->hint_host[0][1] = ctx->hint_host[1][1] = -1;
      ok = cudaHostGetDevicePointer(reinterpret_cast<void**>(&ctx->hint_dev[0]), ctx->hint_host[0], 0) == cudaSuccess;
      ctx->hint_dev[1] = ctx->hint_dev[0] + 2;
      for (int i = 0; i < 2 && ok; ++i) ok = cudaEventCreateWithFlags(&ctx->ev_hint[i], cudaEventDisableTiming) == cudaSuccess;
    }
    if (!ok) {                                               // the step then always takes the many-row kernels
      for (int i = 0; i < 2; ++i) if (ctx->ev_hint[i]) { cudaEventDestroy(ctx->ev_hint[i]); ctx->ev_hint[i] = nullptr; }
      if (ctx->hint_host[0]) cudaFreeHost(ctx->hint_host[0]);
      ctx->hint_host[0] = ctx->hint_host[1] = nullptr; (void)cudaGetLastError();
    }
  }
  if (cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&ctx->layers_done, cudaEventDisableTiming) != cudaSuccess) {
    if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
    ctx->copy_stream = nullptr; ctx->layers_done = nullptr; (void)cudaGetLastError();
  }
  ctx->run = ctx->stream;
  if (!(cfg->flags & D2C_FLAG_SERIAL)) {
    int least = 0, greatest = 0;
    bool ok = cudaDeviceGetStreamPriorityRange(&least, &greatest) == cudaSuccess && greatest < least &&
              cudaStreamCreateWithPriority(&ctx->work_stream, cudaStreamNonBlocking, greatest) == cudaSuccess &&
              cudaStreamCreateWithPriority(&ctx->side_stream, cudaStreamNonBlocking, least) == cudaSuccess;
    for (cudaEvent_t* ev : {&ctx->ev_in, &ctx->ev_out, &ctx->ev_fwd, &ctx->ev_side, &ctx->ev_begun, &ctx->ev_abar[0], &ctx->ev_abar[1], &ctx->ev_abar[2], &ctx->ev_abar[3]})
      ok = ok && cudaEventCreateWithFlags(ev, cudaEventDisableTiming) == cudaSuccess;
    if (!ok) { destroy_overlap(ctx); (void)cudaGetLastError(); }      // the step then runs on the caller's stream alone
  }
  cudaError_t e = cudaMemsetAsync(workspace, 0, need, ctx->stream);
  if (e == cudaSuccess) {
    std::vector<uint32_t> tab(cfg->max_seq);
    ctx->phi_len = build_phi_table(cfg->sigma, tab.data(), cfg->max_seq);
    e = cudaMemcpyAsync(ctx->buf.phi, tab.data(), tab.size() * sizeof(uint32_t), cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) {
      int rc = launch_rope_table(ctx->buf.rope, cfg->max_seq, cfg->head_dim, cfg->rope_base, ctx->stream);
      if (rc != D2C_OK) { delete ctx; return rc; }
      e = cudaStreamSynchronize(ctx->stream);      // the host table above must outlive the copy
    }
  }
  if (e != cudaSuccess) { delete ctx; return fail(nullptr, D2C_ECUDA, "d2c_create: %s", cudaGetErrorString(e)); }
  *out = ctx;
  return D2C_OK;
}

int d2c_destroy(d2c_ctx* ctx) {
  if (!ctx) return D2C_EINVAL;
  for (cudaEvent_t e : ctx->ev) cudaEventDestroy(e);
  for (int i = 0; i < 2; ++i) if (ctx->ev_hint[i]) cudaEventDestroy(ctx->ev_hint[i]);
  if (ctx->hint_host[0]) cudaFreeHost(ctx->hint_host[0]);
  if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
  if (ctx->layers_done) cudaEventDestroy(ctx->layers_done);
  destroy_overlap(ctx);
  delete ctx;
  return D2C_OK;
}

const char* d2c_last_error(const d2c_ctx* ctx) { return ctx ? ctx->err : global_error(); }

int d2c_state_ptrs(d2c_ctx* ctx, d2c_state* out) {
  if (!ctx || !out) return D2C_EINVAL;
  const Buffers& b = ctx->buf;
  out->kcache = b.kcache; out->vcache = b.vcache; out->conf = b.conf; out->pred = b.pred; out->c = b.c; out->key = b.key;
  out->sel_idx = b.sel_idx; out->row_off = b.row_off; out->lm_rows = b.lm_rows; out->lm_off = b.lm_off;
  out->abar = b.abar; out->lse = b.lse; out->status = b.status; out->gemm_clocks = reinterpret_cast<int64_t*>(b.gemm_clocks);
  return D2C_OK;
}

int d2c_sync_status(d2c_ctx* ctx) {
  if (!ctx) return D2C_EINVAL;
  cudaError_t e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) return fail(ctx, D2C_ECUDA, "d2c_sync_status: %s", cudaGetErrorString(e));
  int32_t st[4];
  e = cudaMemcpy(st, ctx->buf.status, sizeof(st), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return fail(ctx, D2C_ECUDA, "d2c_sync_status: %s", cudaGetErrorString(e));
  if (st[0] != 0) return fail(ctx, st[0], "device status %d raised at site %d", st[0], st[1]);
  return D2C_OK;
}

static int check_step_args(d2c_ctx* ctx, const d2c_step_args* a) {
  if (!ctx) return D2C_EINVAL;
  if (!a) return fail(ctx, D2C_EINVAL, "d2c_step: args is null");
  if (a->batch < 1 || a->seq_len < 1) return fail(ctx, D2C_EINVAL, "d2c_step: batch %d / seq_len %d must be positive", a->batch, a->seq_len);
  if (a->batch > ctx->cfg.max_batch || a->seq_len > ctx->cfg.max_seq)
    return fail(ctx, D2C_ECAPACITY, "d2c_step: batch %d x seq_len %d exceeds the context's %d x %d", a->batch, a->seq_len, ctx->cfg.max_batch, ctx->cfg.max_seq);
  if (!a->h0 || !a->mask) return fail(ctx, D2C_EINVAL, "d2c_step: h0 or mask is null");
  if (a->k < 0) return fail(ctx, D2C_EINVAL, "d2c_step: k = %d is negative", a->k);
  if (isnan(a->p)) return fail(ctx, D2C_EINVAL, "d2c_step: p is NaN");
  if ((a->forced == nullptr) != (a->forced_off == nullptr)) return fail(ctx, D2C_EINVAL, "d2c_step: forced and forced_off must be given together");
  if (ctx->used_batch == 0) { ctx->used_batch = a->batch; ctx->used_seq = a->seq_len; }
  if (a->batch != ctx->used_batch || a->seq_len != ctx->used_seq)
    return fail(ctx, D2C_EINVAL, "d2c_step: batch %d x seq_len %d differs from the %d x %d this context was first used with",
                a->batch, a->seq_len, ctx->used_batch, ctx->used_seq);
  return D2C_OK;
}

static bool stream_captures(const d2c_ctx* ctx) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(ctx->stream, &cs) != cudaSuccess) { (void)cudaGetLastError(); return true; }
  return cs != cudaStreamCaptureStatusNone;
}
// The row count of the step before, read behind that step's selection kernel, which the next one goes by; left alone if there is none.
static int previous_rows(d2c_ctx* ctx, bool capturing, int* rows) {
  const int prev = (int)(ctx->step_no & 1) ^ 1;
  if (!ctx->hint_host[0] || capturing || ctx->hint_step[prev] != ctx->step_no - 1) return D2C_OK;
  if (ctx->hint_tagged[prev]) {
    // (an event behind a step in one launch would come with its end, and cost the GPU 8 of 50 us between two of them)
    const volatile uint64_t* word = reinterpret_cast<const volatile uint64_t*>(ctx->hint_host[prev]);
    for (bool ended = false;;) {
      for (int i = 0; i < 20000; ++i) {
        const uint64_t v = *word;
        if ((uint32_t)(v >> 32) == (uint32_t)ctx->hint_step[prev]) { *rows = (int)(uint32_t)v; return D2C_OK; }
        if (ended) return D2C_OK;                              // it said nothing: like a step that was not watched
      }
      const cudaError_t e = cudaStreamQuery(ctx->stream);
      if (e == cudaErrorNotReady) (void)cudaGetLastError();
      else if (e != cudaSuccess) return cu(e);
      else ended = true;
    }
  }
  const int rc = cu(cudaEventSynchronize(ctx->ev_hint[prev]));
  if (rc == D2C_OK) *rows = *reinterpret_cast<volatile int32_t*>(ctx->hint_host[prev]);
  return rc;
}

static SelectArgs select_args(const d2c_ctx* ctx, const d2c_step_args* a, bool track) {
  const Buffers& b = ctx->buf;
  const int L = a->seq_len;
  SelectArgs s{};
  s.mask = a->mask; s.conf = b.conf; s.c = a->override_c ? a->override_c : b.c; s.override_key = a->override_key;
  s.forced = a->forced; s.forced_off = a->forced_off; s.batch = a->batch; s.seq_len = L; s.k = a->k; s.p = a->p;
  s.stage2_candidates = ctx->cfg.stage2_candidates; s.block_lo = a->block_lo; s.block_hi = a->block_hi; s.phi_q30 = b.phi; s.phi_len = ctx->phi_len < L ? ctx->phi_len : L;
  s.key = b.key; s.sel_idx = b.sel_idx; s.row_seq = b.row_seq; s.row_off = b.row_off; s.lm_rows = b.lm_rows;
  s.lm_off = b.lm_off; s.slot_of_pos = b.slot_of_pos; s.rank_s = b.rank_s; s.rank_lm = b.rank_lm; s.n_b = b.n_b; s.nm_b = b.nm_b;
  s.n_host = track ? ctx->hint_dev[ctx->step_no & 1] : nullptr;
  return s;
}
// The index outputs of a step, copied by one of its kernels.
static CopyOut index_outputs(const d2c_ctx* ctx, const d2c_step_out* out, int rows, int batch) {
  CopyOut copies{};
  if (out && out->sel_idx) { copies.src[0] = ctx->buf.sel_idx; copies.dst[0] = out->sel_idx; copies.n[0] = rows; }
  if (out && out->row_off) { copies.src[1] = ctx->buf.row_off; copies.dst[1] = out->row_off; copies.n[1] = batch + 1; }
  return copies;
}
// Whether a small model's step goes in one launch: while each cluster has one tile of 16 rows, and of a narrow model two, or three where
// the rows are a part of the room only and so mostly known ones, without work for the LM head.  (us, one launch / separate kernels, one layer
// of d 256: 61 rows of 256 positions 40 / 60, 216 of 600 56 / 71, 224 of 16 x 300 60 / 75, all of 112 rows 41 / 86, all of 224 in four
// sequences, three tiles, 56 / 55, with 4096 columns of the LM head 71 / 58; two of d 384: 109 of 256 73 / 90, all of 112 70 / 181, 125 rows, two
// tiles, 93 / 88; three of d 512: 106 of 600 128 / 151, 125 rows 135 / 124.  One layer of d 256 with 1500 columns, 110 rows, 51 / 66, with 2048
// 52 / 67, all 221 masked in part 61 / 70; of four and eight layers, d 256 to 512, 59 to 328 rows of 256 to 3000 positions, one to four
// sequences, the one launch is ahead by 4 % (four of d 512, 59 rows, 153 / 160) to 35 % (eight of d 256, 110 rows, 250 / 337).)
static bool few_for_one_launch(const d2c_ctx* ctx, int batch, int room, int rows) {
  const d2c_config& c = ctx->cfg;
  const int most = c.d_model > 256 || (long long)c.vocab * c.d_model > 1 << 18 ? 1 : 2 * rows <= room ? 3 : 2;
  return batch * ceil_div(rows, 16 * batch) <= ctx->small_clusters * most;
}
// Rows that stage 1 of a call selects at most.
static int most_of_stage1(const d2c_step_args* a) {
  const int lo = a->block_lo > 0 ? a->block_lo : 0, hi = a->block_hi < a->seq_len ? a->block_hi : a->seq_len;
  const int width = a->block_hi > a->block_lo ? (hi > lo ? hi - lo : 0) : a->seq_len;
  return a->k < width ? a->k : width;
}
static void note_asked(d2c_ctx* ctx, const d2c_step_args* a) { ctx->asked_k = most_of_stage1(a); ctx->asked_p = a->p; }
// It is on the caller's stream.  Where the GPU has no room for it, as in a part of one that has fewer SMs than were counted, the context goes
// on with the separate kernels.
static int step_in_one_launch(d2c_ctx* ctx, const d2c_step_args* a, const d2c_step_out* out, bool track, bool* refused) {
  const d2c_config& c = ctx->cfg;
  const Buffers& b = ctx->buf;
  const int B = a->batch, L = a->seq_len, R = B * L, slot = (int)(ctx->step_no & 1);
  SmallArgs s = small_args(ctx, B, L);
  s.sel = select_args(ctx, a, false);
  s.h0 = static_cast<const bf16*>(a->h0); s.h0_far = ctx->h0_far;
  s.x = (out && out->hidden_out) ? static_cast<bf16*>(out->hidden_out) : b.x;
  s.layer_in = out ? static_cast<bf16*>(out->layer_in) : nullptr; s.rows_cap = R;
  s.logits = out ? out->logits : nullptr;
  s.copies = index_outputs(ctx, out, R, B);
  if (track) { s.n_word = reinterpret_cast<uint64_t*>(ctx->hint_dev[slot]); s.n_tag = (int)ctx->step_no; }
  small_step_scratch(s, ctx->small_clusters, b.sk_partials, &s);
  D2C_TRY(ctx, launch_small_step(s, ctx->small_clusters, ctx->stream, refused));
  if (*refused) { ctx->small_clusters = 0; return D2C_OK; }
  if (track) { ctx->hint_step[slot] = ctx->step_no; ctx->hint_tagged[slot] = true; }
  ctx->step_no++; note_asked(ctx, a);
  if (ctx->early_hidden_host && ctx->copy_stream) {           // d2c_step_host's rows
    if (ctx->early_hidden_dev) { D2C_TRY(ctx, launch_rows_to_host(s.x, b.row_off + B, c.d_model, ctx->early_hidden_dev, ctx->stream)); }
    else D2C_TRY(ctx, cu(cudaMemcpyAsync(ctx->early_hidden_host, s.x, (size_t)R * c.d_model * sizeof(bf16), cudaMemcpyDeviceToHost, ctx->stream)));
  }
  return D2C_OK;
}

int d2c_step(d2c_ctx* ctx, const d2c_step_args* a, const d2c_step_out* out) {
  D2C_TRY(ctx, check_step_args(ctx, a));
  const d2c_config& c = ctx->cfg;
  const Buffers& b = ctx->buf;
  {
    const void* x = (out && out->hidden_out) ? out->hidden_out : b.x;
    if (reinterpret_cast<uintptr_t>(x) % 16 || reinterpret_cast<uintptr_t>(a->h0) % 16)
      return fail(ctx, D2C_EINVAL, "d2c_step: h0 and hidden_out must be 16-byte aligned");
  }
  // the row count of the previous step, read behind that step's selection, once (a call for an event or the stream takes 0.5 us)
  const bool capturing = stream_captures(ctx);
  int expect_rows = 1 << 30;
  bool read = false;
  if (ctx->small_clusters > 0 && !ctx->prof && !(out && reinterpret_cast<uintptr_t>(out->layer_in) % 16)) {
    // One launch where few rows are expected, going by the step before like everything here, or where there is room for no more.  Not where
    // the call asks for more than that one did, so that its count says nothing: many rows behind few cost the separate kernels hardly
    // more than behind many, and the one launch several passes a cluster.  Behind 16 + 2 % of the rows, us, separate / one launch, all rows of
    // one layer of d 256: 600 positions 79 / 105, 2048 155 / 376, 4096 390 / 1011; three layers, four of 700 248 / 746; three of d 512, 2048 528 / 1516;
    // 16 + 90 %: 143 / 250 at 2048, 343 / 703 at 4096.
    const int rows = a->batch * a->seq_len;
    const bool any = few_for_one_launch(ctx, a->batch, rows, rows);
    const bool track = ctx->hint_host[0] != nullptr && !capturing && (!any || ctx->host_call);
    const bool asks_more = most_of_stage1(a) > ctx->asked_k || a->p > ctx->asked_p;
    if (!any) { D2C_TRY(ctx, previous_rows(ctx, capturing, &expect_rows)); read = true; }
    if (few_for_one_launch(ctx, a->batch, rows, any || asks_more || expect_rows > rows ? rows : expect_rows)) {
      bool refused = false;
      const int rc = step_in_one_launch(ctx, a, out, track, &refused);
      if (!refused) return rc;
    }
  }
  // critical path on `st`, probabilities + rollout on `side` (the same stream while profiling or when serial)
  const int B = a->batch, L = a->seq_len, R = B * L, d = c.d_model;
  // Whether a product's weights alone give all SMs work, with one tile of tokens and whichever kernel takes it.  (By the tiles of all
  // tokens that there is room for the smallest models' products would, at lengths where most of those CTAs find no rows; called
  // large, they lose: one layer of d 256, us, 1200 positions 106 / 120, all rows 93 / 112, 2048 positions 149 / 176; two of d 512 at
  // 2 x 2048 303 / 310, all rows 319 / 332, 103 rows of 2048 positions 131 / 150.  The other way: two of d 512, all of 1200 rows, 180 / 174.)
  auto takes_all = [&](int n, int k, GemmEpilogue epi) {
    GemmArgs t{};
    t.max_rows = R < 256 ? R : 256; t.N = n; t.K = k;
    return gemm_tc2_ctas(t, epi, false) >= sm_count_current() - 1;
  };
  const bool lm_takes_all = takes_all(c.vocab, d, EPI_LMSTATS), layers_take_all = takes_all(c.d_ffn, d, EPI_SWIGLU);
  bool fills = false;                                  // the LM head takes all SMs, and can be told to leave some
  {
    GemmArgs t{};
    t.A = b.xm; t.W = ctx->w_lm; t.max_rows = R; t.N = c.vocab; t.K = t.lda = d;
    fills = lm_takes_all && !(c.flags & (D2C_FLAG_PORTABLE_GEMM | D2C_FLAG_ONE_SM_GEMM)) && gemm_tc2_supported(t);
  }
  // Models whose products leave SMs free need no priority over the passes beside them: their chain stays on the caller's stream,
  // without the two events between streams (one layer of d 256 at 94 rows 56.4 -> 53.4 us, two of d 512 at 299 rows 121.1 -> 119.6).
  const bool overlap = ctx->work_stream != nullptr && !ctx->prof, hop = overlap && (lm_takes_all || layers_take_all);
  cudaStream_t st = hop ? ctx->work_stream : ctx->stream;
  cudaStream_t side = overlap ? ctx->side_stream : st;
  ctx->run = st;
  if (hop) {
    D2C_TRY(ctx, cu(cudaEventRecord(ctx->ev_in, ctx->stream)));
    D2C_TRY(ctx, cu(cudaStreamWaitEvent(st, ctx->ev_in, 0)));
  }
  // The probabilities pass of a layer goes to the side stream when its CTAs cannot hold up the projections that follow:
  // with few rows or in small models, for a single layer whose products leave SMs free (it then overlaps the LM head), and on SM
  // pairs that the projections leave alone.  Otherwise a statically scheduled GEMM whose CTAs start late behind side-stream CTAs
  // loses more than the overlap gains (measured at 488 rows x 32 layers: +5 %).
  // regime of this step: the row count of the previous step
  const bool track = ctx->hint_host[0] != nullptr && !capturing;
  const int slot = (int)(ctx->step_no & 1);
  if (!read) D2C_TRY(ctx, previous_rows(ctx, capturing, &expect_rows));
  ctx->few_rows = expect_rows <= 128;
  const bool few_rows = ctx->few_rows;
  // With few rows the projections stream weights and 96 of the 148 SMs take all the HBM gives (32 layers at 81 rows: 64
  // pairs 4.60 ms, 48 pairs 4.77), while a projection whose share of SMs is held by the probabilities pass waits for it
  // (74 pairs: 5.21 ms; with that pass spread over all SMs and short: 4.93).  So they leave it the SMs it needs.
  ctx->max_pairs = 0;
  if (few_rows) {
    const int free_pairs = sm_count_current() / 2 - ceil_div(a->seq_len, 256) * a->batch;
    ctx->max_pairs = free_pairs >= 64 ? 64 : (free_pairs >= 56 ? 56 : 48);
  }
  // Eq. 6-9 for the next step's stage 2: enqueued right after the last probabilities pass it needs
  RolloutArgs r{};
  r.abar = b.abar; r.layer_stride = (size_t)c.max_batch * c.max_seq * c.max_seq; r.n_layers = rollout_depth(c); r.sel_idx = b.sel_idx;
  r.expect_rows = expect_rows < a->batch * a->seq_len ? expect_rows : 0;
  r.row_off = b.row_off; r.batch = a->batch; r.seq_len = a->seq_len; r.c = b.c; r.u0 = b.u0; r.u1 = b.u1; r.partial = b.partial; r.n_split = kRolloutSplit;
  int abar_last = -1;                                  // last layer whose probabilities run on the side stream
  bool rollout_done = false;
  // With eight layers or more the rollout goes beside the LM head, which leaves it the SMs it needs: that product is bound by
  // the weights it reads and 60 of the 74 SM pairs take all the HBM gives.  Beside the last layers' projections, where it could
  // begin, its CTAs hold up statically scheduled ones (32 layers: 4262 us, 4080 this way at 81 rows; 8500 and 8330 at 489).
  // A shorter one goes in launches of many CTAs, also beside the LM head if it reads no more than the eight SMs left to it get
  // through meanwhile (about 0.1 TB/s each), else over the whole GPU where it can begin.  Models whose products do not fill the
  // GPU have no such conflict.
  const bool rollout_late = fills && !capturing && r.n_layers >= 8 && sm_count_current() - B * kRolloutCluster >= 120 && rollout_single(r);
  r.spread = fills && !rollout_late;
  // With few rows (192 are a tile of tokens that the weights still bound) the LM head leaves eight SMs to that and to the rows that
  // a host call gets from a kernel.  (Where it took all SMs, those left behind it, and the kernels after it, whose start waits for
  // every write under way to the host, came 17 us later: one layer called with host buffers 382 -> 370 us.)  One layer without / with
  // the room, us: 32 rows in the LM head 523 / 515, 64 337 / 335 and 546 / 535, 128 364 / 359 and (in four sequences) 469 / 461, 192
  // 490 / 504 and 1419 / 1389, 384 680 / 698, 512 803 / 819.  The rollout beside it or where it could begin: no difference up to 12 MB
  // but for 1530 rows of 2048 positions, 823 / 880; four layers, 69 MB 3219 / 3115, 94 MB 7221 / 7116.
  const bool lm_room = fills && c.stage2_candidates == 0 && (long long)B * a->k <= 192;
  const float rollout_mb = 4e-6f * r.n_layers * (float)(expect_rows < R ? expect_rows : R) * (float)L;
  const bool spread_late = r.spread && lm_room && rollout_mb <= 32.f;
  ctx->lm_pairs = rollout_late ? (sm_count_current() - B * kRolloutCluster) / 2 - (lm_room ? 2 : 0) : (lm_room ? sm_count_current() / 2 - 4 : 0);
  const int hq = c.n_q_heads, hkv = c.n_kv_heads, dh = c.head_dim;
  const int qkv_out = (hq + 2 * hkv) * dh;
  const size_t cache_layer = (size_t)c.max_batch * c.max_seq * hkv * dh;
  bf16* x = (out && out->hidden_out) ? static_cast<bf16*>(out->hidden_out) : b.x;

  D2C_TRY(ctx, mark(ctx, PH_SELECT));
  D2C_TRY(ctx, launch_select(select_args(ctx, a, track), st));
  if (track) {
    D2C_TRY(ctx, cu(cudaEventRecord(ctx->ev_hint[slot], st)));
    ctx->hint_step[slot] = ctx->step_no; ctx->hint_tagged[slot] = false;
  }
  ctx->step_no++; note_asked(ctx, a);
  const int32_t* n_rows = b.row_off + B;
  const int32_t* n_lm = b.lm_off + B;

  const int depth = rollout_depth(c);
  // The RMSNorms inside the layers ride in the tcgen05 GEMMs' epilogues (all four projections must run on those kernels)
  // with few rows, where two launches a layer count (32 layers at 81 rows 4.50 -> 4.38 ms), or on request.  Otherwise the
  // longer epilogues and the row scaling cost the GEMMs more than the two small kernels per layer take (8.6 -> 8.85 ms at
  // 489 rows x 32 layers, 46.0 -> 48.0 ms at 3907 rows x 28).
  bool fold = (few_rows || (c.flags & D2C_FLAG_FOLDED_NORMS)) && !(c.flags & D2C_FLAG_PORTABLE_GEMM);
  {
    const int shapes[4][2] = {{qkv_out, d}, {d, hq * dh}, {c.d_ffn, d}, {d, c.d_ffn}};       // {N, K}
    const bf16* as[4] = {b.xn, b.o, b.xn, b.hmid};
    for (int i = 0; i < 4 && fold; ++i) {
      GemmArgs t{};
      t.A = as[i]; t.lda = shapes[i][1]; t.W = ctx->wqkv[0]; t.max_rows = R; t.N = shapes[i][0]; t.K = shapes[i][1];
      fold = gemm_tc_supported(t) && (d & 7) == 0;
    }
  }
  bool fused_qkv = !(c.flags & D2C_FLAG_PORTABLE_GEMM);
  {
    GemmArgs t{};
    t.A = b.xn; t.lda = d; t.W = ctx->wqkv[0]; t.max_rows = R; t.N = qkv_out; t.K = d;
    fused_qkv = fused_qkv && gemm_tc_supported(t);
  }
  // Small models: the probabilities pass also goes to the side stream when its CTAs and those of any projection fit the
  // GPU together (two layers of d 512, 277 rows: 12 us a layer off the chain).
  bool small = false;
  // Grids grow for 64-token tiles only with up to 1024 positions: with more, kernels around them (attention, whose time goes
  // with the positions, and the probabilities beside the chain) want the SMs, whatever the rows.  Without / with, us: three
  // layers of d 256 at 2000 positions 58 rows 242 / 242, 259 rows 263 / 275, 929 rows 320 / 404, 1668 rows 400 / 445; two of d 512
  // 134 / 137, 156 / 156, 191 / 195, 234 / 238.  At 1100 it can go either way (497 rows 230 / 224, two layers 158 / 159), at 768
  // with wins (299 rows in two layers of d 512: 155 / 143).
  ctx->narrow_pairs = c.n_layers > 1 && R > 1024 ? 1 : 0;
  if (!few_rows && fused_qkv) {
    AttnArgs t{};
    t.q = b.qkv; t.ldq = hq * dh; t.kc = b.kcache; t.vc = b.vcache; t.batch = B; t.seq_len = L; t.cache_seq = c.max_seq;
    t.hq = hq; t.hkv = hkv; t.dh = dh; t.max_rows_per_seq = L; t.q_rows = R; t.portable = (c.flags & D2C_FLAG_PORTABLE_ATTENTION) ? 1 : 0;
    t.expect_rows = expect_rows < R ? expect_rows : 0;
    const int shapes[4][2] = {{qkv_out, d}, {d, hq * dh}, {c.d_ffn, d}, {d, c.d_ffn}};       // {N, K}
    const GemmEpilogue epis[4] = {EPI_QKV_ROPE, EPI_RESIDUAL, EPI_SWIGLU, EPI_RESIDUAL};
    int most = 0;
    for (int i = 0; i < 4; ++i) {
      GemmArgs s{};
      s.A = b.xn; s.W = ctx->wqkv[0]; s.max_rows = R; s.N = shapes[i][0]; s.K = s.lda = shapes[i][1]; s.q_dh = dh;
      const int n = !(c.flags & D2C_FLAG_ONE_SM_GEMM) && gemm_tc2_supported(s) ? gemm_tc2_ctas(s, epis[i], false) : gemm_tc_ctas(s, epis[i]);
      most = n > most ? n : most;
    }
    const int free_pairs = (sm_count_current() - attention_abar_sms(t)) / 2;
    small = c.n_layers > 1 && most <= 2 * free_pairs;
    if (small) ctx->max_pairs = free_pairs;
    // The pass of a single layer whose products leave SMs free runs beside them in any case: 64-token tiles only spread over the SMs
    // it leaves (one layer of d 256, 1200 rows: 93 us, over all SMs 113, which then wait for the pass).
    if (c.n_layers == 1 && !layers_take_all) ctx->narrow_pairs = free_pairs > 1 ? free_pairs : 1;
  }
  // Large models, more rows: the pass is short (489 rows x 768 keys: 17 us) but takes that on the whole GPU, mostly latency.  A
  // few SM pairs do it in the time of a layer, and the layer's other kernels lose less by those than the pass took between
  // them (489 rows x 32 layers: 8500 -> 8370 us; 8 layers, 190 rows, 2179 keys: 1670 -> 1530).
  int abar_pairs = 0;
  if (c.n_layers > 1 && !few_rows && !small && fused_qkv && !(c.flags & (D2C_FLAG_PORTABLE_ATTENTION | D2C_FLAG_ONE_SM_GEMM))) {
    AttnArgs t{};
    t.q = b.qkv; t.ldq = hq * dh; t.kc = b.kcache; t.vc = b.vcache; t.batch = B; t.seq_len = L; t.cache_seq = c.max_seq;
    t.hq = hq; t.hkv = hkv; t.dh = dh; t.max_rows_per_seq = L; t.q_rows = R; t.expect_rows = expect_rows < R ? expect_rows : 0;
    const float rows = (float)(expect_rows < R ? expect_rows : R);
    const float flops = 2.f * rows * ((float)d * (qkv_out + hq * dh) + 3.f * d * c.d_ffn) + 4.f * rows * L * hq * dh;
    if (attention_tc_supported(t)) abar_pairs = attention_abar_pairs(t, 40.f + flops / 1.1e9f);      // 1.1 PFLOP/s and 40 us of small kernels
    if (abar_pairs > 0) ctx->max_pairs = sm_count_current() / 2 - abar_pairs;
  }
  // A single layer's pass stays on the chain where the layer's products take all SMs: beside them it gets SMs in the gaps between launches,
  // where it holds up the statically scheduled CTAs behind it, and ends after the LM head.  One layer beside / on the chain, us: d 4096,
  // 831 rows x 1024 positions 561 / 553, 797 x 797 567 / 552, 588 rows of four sequences x 1187 613 / 587, 1499 of five x 3071 1230 / 1140.
  // An LM head of that size alone is no reason: d 768 and 16000 words, 2000 rows of four sequences 167 / 176, 301 rows 87 / 96; d 1536 and
  // 50000, 2048 positions 180 / 207; all of 2048 rows at d 768 256 / 245.
  const bool abar_aside = overlap && ((c.n_layers == 1 && !layers_take_all) || few_rows || small || abar_pairs > 0);
  // The launches of the pair kernel: with the SM pairs that the layers leave to the passes beside them and, where the passes end
  // before the layers do, with all.
  ctx->plan.n = 0;
  ctx->pair_launches = 0;
  ctx->plan.n_rows[0] = n_rows; ctx->plan.n_rows[1] = n_lm; ctx->plan.records = b.records;
  {
    const int shapes[5][3] = {{qkv_out, d, hq * dh}, {d, hq * dh, d}, {c.d_ffn, d, c.d_ffn}, {d, c.d_ffn, d}, {c.vocab, d, 0}};       // {N, K, ldc}
    const GemmEpilogue epis[5] = {fused_qkv ? EPI_QKV_ROPE : EPI_STORE, EPI_RESIDUAL, EPI_SWIGLU, EPI_RESIDUAL, EPI_LMSTATS};
    const int pairs = ctx->max_pairs;
    for (int all = 0; all < (abar_pairs > 0 && depth + 1 < c.n_layers ? 2 : 1); ++all) {
      ctx->max_pairs = all ? 0 : pairs;
      for (int i = 0; i < (all ? 4 : 5); ++i) {
        GemmArgs t{};
        t.A = b.xn; t.W = ctx->wqkv[0]; t.max_rows = R; t.N = shapes[i][0]; t.K = t.lda = shapes[i][1]; t.ldc = shapes[i][2];
        plan_pair(ctx, t, epis[i]);
      }
    }
    ctx->max_pairs = pairs;
  }
  D2C_TRY(ctx, mark(ctx, PH_GATHER));
  // Every step starts with cleared meeting counters, whatever the one before left in them: the one-SM kernel puts its own back at each
  // meeting, unless a wait gave up, and the pair kernel's are cleared by the launch after (the last one's by lm_reduce).  What was left
  // would let a launch add parts of another.  In this kernel, which no GEMM overlaps that has come past its wait (in the selection
  // kernel it took 0.3 us of the smallest step).
  D2C_TRY(ctx, launch_gather_norm((const bf16*)a->h0, b.sel_idx, b.row_seq, n_rows, R, L, d, ctx->g_attn[0], c.rms_eps, x, b.xn,
                                  b.sk_counters, kCounters, ctx->plan, st));
  auto rollout = [&]() {
    int rc = launch_rollout(r, side);
    if (rc == D2C_OK && overlap) rc = cu(cudaEventRecord(ctx->ev_side, side));
    rollout_done = true;
    return rc;
  };
  AttnArgs last_pass{};                                // the last layer's pass, if it is enqueued behind the LM head
  bool pass_left = false;
  for (int l = 0; l < c.n_layers; ++l) {
    if (out && out->layer_in) {
      cudaError_t e = cudaMemcpyAsync(static_cast<bf16*>(out->layer_in) + (size_t)l * R * d, x, (size_t)R * d * sizeof(bf16),
                                      cudaMemcpyDeviceToDevice, st);
      if (e != cudaSuccess) return fail(ctx, D2C_ECUDA, "d2c_step: %s", cudaGetErrorString(e));
    }
    // RMSNorm folded into the projections (tcgen05 GEMMs): the residual epilogue before a norm leaves x * gain in xn
    // and the row's sums of squares in ssq, the projection after it scales its accumulator rows by rsqrt(mean + eps)
    if (l > 0 && !fold) {
      D2C_TRY(ctx, mark(ctx, PH_NORM));
      D2C_TRY(ctx, launch_rmsnorm(x, nullptr, n_rows, R, d, ctx->g_attn[l], c.rms_eps, b.xn, st));
    }
    D2C_TRY(ctx, mark(ctx, PH_QKV));
    const int qbuf = (c.n_layers - 1 - l) % ctx->q_bufs;
    // Probabilities passes on the side stream still read their layers' Q and LSE.  Every fourth layer waits for those whose
    // buffers it and the next three write: with six buffers for the pass three layers back, and with it for those before, as
    // layers l to l + 3 write the buffers of l - 6 to l - 3.  (With fewer than four buffers every layer waits for its own.)
    const bool by_four = fused_qkv && ctx->q_bufs >= 4;
    const int need = by_four ? l + 3 - ctx->q_bufs : l - (fused_qkv ? ctx->q_bufs : 1);
    if (abar_last >= 0 && need >= 0 && (!by_four || (l & 3) == 0))
      D2C_TRY(ctx, cu(cudaStreamWaitEvent(st, ctx->ev_abar[(need < abar_last ? need : abar_last) & 3], 0)));
    GemmArgs g{};
    g.A = b.xn; g.lda = d; g.W = ctx->wqkv[l]; g.bias = ctx->bqkv[l]; g.C = b.qkv; g.ldc = qkv_out;
    g.n_rows = n_rows; g.max_rows = R; g.N = qkv_out; g.K = d;
    MapCache* maps = &ctx->maps[6 * (size_t)l];
    g.cache = maps;
    if (fold && l > 0) { g.in_ssq = b.ssq; g.in_eps = c.rms_eps; }
    bf16* kc = b.kcache + (size_t)l * cache_layer; bf16* vc = b.vcache + (size_t)l * cache_layer;
    if (fused_qkv) {
      g.C = b.qkv + (size_t)qbuf * R * hq * dh; g.ldc = hq * dh;
      // QKV projection with bias, rotary embedding and the K/V scatter in its epilogue
      g.q_sel_idx = b.sel_idx; g.q_row_seq = b.row_seq; g.q_rope = b.rope; g.q_kc = kc; g.q_vc = vc;
      g.q_cache_seq = c.max_seq; g.q_hq = hq; g.q_hkv = hkv; g.q_dh = dh;
      D2C_TRY(ctx, gemm(ctx, g, EPI_QKV_ROPE, l > 0));
    } else {
      D2C_TRY(ctx, gemm(ctx, g, EPI_STORE, l > 0));
      D2C_TRY(ctx, mark(ctx, PH_ROPE));
      D2C_TRY(ctx, launch_rope_scatter(b.qkv, b.sel_idx, b.row_seq, n_rows, R, hq, hkv, dh, b.rope, kc, vc, c.max_seq, st));
    }
    AttnArgs at{};
    at.q = fused_qkv ? g.C : b.qkv; at.ldq = fused_qkv ? hq * dh : qkv_out; at.kc = kc; at.vc = vc; at.row_off = b.row_off; at.batch = B; at.seq_len = L;
    at.cache_seq = c.max_seq; at.hq = hq; at.hkv = hkv; at.dh = dh; at.max_rows_per_seq = L;
    at.q_rows = R; at.portable = (c.flags & D2C_FLAG_PORTABLE_ATTENTION) ? 1 : 0; at.status = b.status;
    at.expect_rows = expect_rows < R ? expect_rows : 0; 
    at.cache[0] = maps + 1; at.cache[1] = maps + 2;
    at.o = b.o; at.lse = b.lse + (size_t)qbuf * R * hq; at.abar = l < depth ? b.abar + (size_t)l * c.max_batch * c.max_seq * c.max_seq : nullptr;
    D2C_TRY(ctx, mark(ctx, PH_ATTN));
    at.which = 1;
    D2C_TRY(ctx, launch_attention(at, st));
    // (with shared SMs the last layer's pass takes the whole GPU: the rollout waits for it)
    const bool aside = at.abar && abar_aside && !(abar_pairs > 0 && l == c.n_layers - 1);
    const bool rollout_here = at.abar && l == depth - 1 && !rollout_late && !spread_late;
    at.which = 2;
    at.pairs = aside ? abar_pairs : 0;
    at.beside = few_rows || (abar_pairs > 0 && l < c.n_layers - 1);          // (cut alike on one stream: the same sums)
    if (aside) {
      D2C_TRY(ctx, cu(cudaEventRecord(ctx->ev_fwd, st)));                      // launched below, behind the chain's next kernels
    } else if (at.abar) {
      D2C_TRY(ctx, mark(ctx, PH_ABAR));
      D2C_TRY(ctx, launch_attention(at, st));
      if (rollout_here) {
        D2C_TRY(ctx, mark(ctx, PH_ROLLOUT));
        if (overlap) {                                                         // the side stream must follow this layer's pass
          D2C_TRY(ctx, cu(cudaEventRecord(ctx->ev_fwd, st)));
          D2C_TRY(ctx, cu(cudaStreamWaitEvent(side, ctx->ev_fwd, 0)));
        }
        D2C_TRY(ctx, rollout());
      }
    }
    D2C_TRY(ctx, mark(ctx, PH_O));
    GemmArgs go{};
    go.A = b.o; go.lda = hq * dh; go.W = ctx->wo[l]; go.C = x; go.ldc = d; go.n_rows = n_rows; go.max_rows = R; go.N = d; go.K = hq * dh;
    go.cache = maps + 3;
    if (fold) { go.nx_out = b.xn; go.nx_gain = ctx->g_ffn[l]; go.nx_ssq = b.ssq; }
    D2C_TRY(ctx, gemm(ctx, go, EPI_RESIDUAL));
    if (!fold) {
      D2C_TRY(ctx, mark(ctx, PH_NORM));
      D2C_TRY(ctx, launch_rmsnorm(x, nullptr, n_rows, R, d, ctx->g_ffn[l], c.rms_eps, b.xn, st));
    }
    D2C_TRY(ctx, mark(ctx, PH_GATEUP));
    GemmArgs gf{};
    gf.A = b.xn; gf.lda = d; gf.W = ctx->w_gate[l]; gf.W2 = ctx->w_up[l]; gf.C = b.hmid; gf.ldc = c.d_ffn;
    gf.n_rows = n_rows; gf.max_rows = R; gf.N = c.d_ffn; gf.K = d; gf.cache = maps + 4;
    gf.clock_probe = ctx->prof ? b.gemm_clocks : nullptr;
    if (fold) { gf.in_ssq = b.ssq; gf.in_eps = c.rms_eps; }
    D2C_TRY(ctx, gemm(ctx, gf, EPI_SWIGLU));
    if (abar_pairs > 0 && l > depth) ctx->max_pairs = 0;                     // no pass runs any more
    GemmArgs gd{};
    gd.A = b.hmid; gd.lda = c.d_ffn; gd.W = ctx->w_down[l]; gd.C = x; gd.ldc = d; gd.n_rows = n_rows; gd.max_rows = R; gd.N = d; gd.K = c.d_ffn;
    gd.cache = maps + 5;
    if (fold && l + 1 < c.n_layers) { gd.nx_out = b.xn; gd.nx_gain = ctx->g_attn[l + 1]; gd.nx_ssq = b.ssq; }
    D2C_TRY(ctx, mark(ctx, PH_DOWN));
    D2C_TRY(ctx, gemm(ctx, gd, EPI_RESIDUAL));
    if (aside) {
      // The host needs longer for these calls than small kernels run, so the chain's came first: those of this layer, behind the
      // last one also the LM head's, unless that takes all SMs (the smallest step 51.5 -> 51.1 us; the others do not wait for the host).
      if (l == c.n_layers - 1 && !lm_takes_all) { last_pass = at; pass_left = true; continue; }
      D2C_TRY(ctx, cu(cudaStreamWaitEvent(side, ctx->ev_fwd, 0)));
      D2C_TRY(ctx, launch_attention(at, side));
      D2C_TRY(ctx, cu(cudaEventRecord(ctx->ev_abar[l & 3], side)));
      abar_last = l;
      if (rollout_here) D2C_TRY(ctx, rollout());
    }
  }
  if (ctx->early_hidden_host && ctx->copy_stream) {
    // the residual stream is final here: ship it to the host while the LM head and the rollout run
    // (the row count is not known on the host yet, so the worst case is copied)
    cudaError_t e = cudaEventRecord(ctx->layers_done, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(ctx->copy_stream, ctx->layers_done, 0);
    if (e == cudaSuccess && ctx->early_hidden_dev) D2C_TRY(ctx, launch_rows_to_host(x, n_rows, d, ctx->early_hidden_dev, ctx->copy_stream));
    else if (e == cudaSuccess) e = cudaMemcpyAsync(ctx->early_hidden_host, x, (size_t)R * d * sizeof(bf16), cudaMemcpyDeviceToHost, ctx->copy_stream);
    if (e != cudaSuccess) return fail(ctx, D2C_ECUDA, "d2c_step: %s", cudaGetErrorString(e));
  }
  if (rollout_late) {
    D2C_TRY(ctx, mark(ctx, PH_ROLLOUT));
    if (overlap) {
      D2C_TRY(ctx, cu(cudaEventRecord(ctx->ev_fwd, st)));
      D2C_TRY(ctx, cu(cudaStreamWaitEvent(side, ctx->ev_fwd, 0)));
      r.begun = ctx->ev_begun;
    }
    D2C_TRY(ctx, launch_rollout(r, side));
    if (overlap) {
      D2C_TRY(ctx, cu(cudaEventRecord(ctx->ev_side, side)));
      D2C_TRY(ctx, cu(cudaStreamWaitEvent(st, ctx->ev_begun, 0)));     // it has its SMs: a cluster needs neighbouring ones
    }
    rollout_done = true;
  }
  if (spread_late) {
    D2C_TRY(ctx, mark(ctx, PH_ROLLOUT));
    if (overlap) {
      D2C_TRY(ctx, cu(cudaEventRecord(ctx->ev_fwd, st)));
      D2C_TRY(ctx, cu(cudaStreamWaitEvent(side, ctx->ev_fwd, 0)));
    }
    D2C_TRY(ctx, rollout());
  }
  // Eq. 1 on the selected rows that are still masked
  D2C_TRY(ctx, mark(ctx, PH_LM));
  D2C_TRY(ctx, launch_rmsnorm(x, b.lm_rows, n_lm, R, d, ctx->g_final, c.rms_eps, b.xm, st));
  GemmArgs gl{};
  gl.A = b.xm; gl.lda = d; gl.W = ctx->w_lm; gl.n_rows = n_lm; gl.max_rows = R; gl.N = c.vocab; gl.K = d; gl.cache = &ctx->maps.back();
  gl.st_max = b.st_max; gl.st_sum = b.st_sum; gl.st_arg = b.st_arg; gl.n_tiles = lm_tiles(c.vocab);
  gl.logits = out ? out->logits : nullptr;
  D2C_TRY(ctx, gemm(ctx, gl, EPI_LMSTATS));
  const CopyOut copies = index_outputs(ctx, out, R, B);      // they leave with the last kernel of the chain
  D2C_TRY(ctx, launch_lm_reduce(b.st_max, b.st_sum, b.st_arg, gl.n_tiles, n_lm, R, b.lm_rows, b.sel_idx, b.row_seq, L, b.conf, b.pred, copies, b.sk_counters + 2 * kSkMaxTiles, 2 * kPairCounters, st));
  if (pass_left) {
    D2C_TRY(ctx, cu(cudaStreamWaitEvent(side, ctx->ev_fwd, 0)));
    D2C_TRY(ctx, launch_attention(last_pass, side));
    D2C_TRY(ctx, rollout());                           // (it is put off itself only where the LM head takes all SMs)
  }
  if (!rollout_done) return fail(ctx, D2C_EINVAL, "d2c_step: no layer produced attention probabilities");
  if (overlap) D2C_TRY(ctx, cu(cudaStreamWaitEvent(st, ctx->ev_side, 0)));

  D2C_TRY(ctx, mark(ctx, PH_OUT));
  D2C_TRY(ctx, mark(ctx, -1));
  if (hop) {
    D2C_TRY(ctx, cu(cudaEventRecord(ctx->ev_out, st)));
    D2C_TRY(ctx, cu(cudaStreamWaitEvent(ctx->stream, ctx->ev_out, 0)));
  }
  ctx->run = ctx->stream;
  return D2C_OK;
}

int d2c_profile(d2c_ctx* ctx, int32_t enable) {
  if (!ctx) return D2C_EINVAL;
  ctx->prof = enable != 0;
  ctx->prof_phase = -1;
  return D2C_OK;
}

int d2c_profile_read(d2c_ctx* ctx, float* phase_ms, int64_t* phase_launches, int32_t reset) {
  if (!ctx) return D2C_EINVAL;
  cudaError_t e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) return fail(ctx, D2C_ECUDA, "d2c_profile_read: %s", cudaGetErrorString(e));
  for (size_t i = 0; i + 1 < ctx->ev_used; ++i) {
    if (ctx->ev_phase[i] < 0) continue;
    float ms = 0.f;
    e = cudaEventElapsedTime(&ms, ctx->ev[i], ctx->ev[i + 1]);
    if (e != cudaSuccess) return fail(ctx, D2C_ECUDA, "d2c_profile_read: %s", cudaGetErrorString(e));
    ctx->phase_ms[ctx->ev_phase[i]] += ms;
  }
  ctx->ev_used = 0;
  for (int i = 0; i < D2C_N_PHASES; ++i) {
    if (phase_ms) phase_ms[i] = (float)ctx->phase_ms[i];
    if (phase_launches) phase_launches[i] = ctx->phase_launches[i];
    if (reset) { ctx->phase_ms[i] = 0; ctx->phase_launches[i] = 0; }
  }
  return D2C_OK;
}

const char* d2c_phase_name(int32_t i) { return (i >= 0 && i < D2C_N_PHASES) ? kPhaseNames[i] : ""; }

// Enqueues the copies and the step of a host call.
static int enqueue_step_host(d2c_ctx* ctx, const d2c_step_args* h, const d2c_host_out* out) {
  const d2c_config& c = ctx->cfg;
  const Buffers& b = ctx->buf;
  cudaStream_t st = ctx->stream;
  const size_t B = h->batch, L = h->seq_len, R = B * L;
#define D2C_CP(dst, src, bytes, kind)                                                         \
  do { cudaError_t e__ = cudaMemcpyAsync((dst), (src), (bytes), (kind), st);                  \
       if (e__ != cudaSuccess) return fail(ctx, D2C_ECUDA, "d2c_step_host: %s", cudaGetErrorString(e__)); } while (0)
  // Pinned buffers are read and written in place by the step's kernels: the selection reads the masks and scores over
  // the link, the gather only the selected rows of h0 and the copy at the end only those rows.  A copy engine moves whole
  // arrays faster, so h0 and the hidden rows go that way when most rows are expected, going by the step before as d2c_step
  // does (one layer, 1024 rows of 8 KB, 116 selected: 150 us of copies saved on each side; a transfer of all rows by kernels
  // is no faster than the engine's).
  d2c_step_args a = *h;
  int expect_rows = 1 << 30;
  D2C_TRY(ctx, previous_rows(ctx, stream_captures(ctx), &expect_rows));
  const bool few_expected = (size_t)expect_rows <= R / 2;
  const void* h0_dev = few_expected ? mapped(h->h0, R * c.d_model * sizeof(bf16)) : nullptr;
  if (h0_dev && reinterpret_cast<uintptr_t>(h0_dev) % 16 == 0) a.h0 = h0_dev;
  else { D2C_CP(b.h0_stage, h->h0, R * c.d_model * sizeof(bf16), cudaMemcpyHostToDevice); a.h0 = b.h0_stage; }
  auto input = [&](const void* src, void* stage, size_t bytes) -> const void* {
    if (const void* p = bytes <= 64 * 1024 ? mapped(src, bytes) : nullptr) return p;
    const cudaError_t e = cudaMemcpyAsync(stage, src, bytes, cudaMemcpyHostToDevice, st);
    return e == cudaSuccess ? stage : nullptr;
  };
#define D2C_IN(field, stage, bytes)                                                                                  \
  do { a.field = static_cast<decltype(a.field)>(input(h->field, (stage), (bytes)));                                  \
       if (!a.field) return fail(ctx, D2C_ECUDA, "d2c_step_host: copying %s failed: %s", #field, cudaGetErrorString(cudaGetLastError())); } while (0)
  D2C_IN(mask, b.mask_stage, R);
  if (h->forced) {
    const int32_t n_forced = h->forced_off[B];
    D2C_IN(forced_off, b.forced_off_stage, (B + 1) * sizeof(int32_t));
    if (n_forced) D2C_IN(forced, b.forced_stage, (size_t)n_forced * sizeof(int32_t));
    else a.forced = b.forced_stage;
  }
  if (h->override_key) D2C_IN(override_key, b.okey_stage, R * sizeof(float));
  if (h->override_c) D2C_IN(override_c, b.oc_stage, R * sizeof(float));
#undef D2C_IN
  d2c_step_out dev_out{};
  const bool early = out && out->hidden_out_host && ctx->copy_stream;
  ctx->early_hidden_host = early ? out->hidden_out_host : nullptr;
  ctx->early_hidden_dev = early && few_expected ? mapped(out->hidden_out_host, R * c.d_model * sizeof(bf16)) : nullptr;
  if (reinterpret_cast<uintptr_t>(ctx->early_hidden_dev) % 16) ctx->early_hidden_dev = nullptr;
  ctx->host_call = true; ctx->h0_far = a.h0 != b.h0_stage;
  const int step_rc = d2c_step(ctx, &a, &dev_out);
  ctx->early_hidden_host = ctx->early_hidden_dev = nullptr; ctx->host_call = ctx->h0_far = false;
  if (step_rc != D2C_OK) return step_rc;
  // every other result is copied without knowing the row count (worst-case sizes), then one synchronisation
  if (out) {
    const void* src[4] = {b.row_off, b.sel_idx, b.conf, b.pred};
    void* dst[4] = {out->row_off_host, out->sel_idx_host, out->conf_host, out->pred_host};
    const size_t n[4] = {B + 1, R, R, R};
    HostResults hr{};
    bool any = false;
    for (int k = 0; k < 4; ++k) {
      if (!dst[k]) continue;
      if (void* p = n[k] * 4 <= 64 * 1024 ? mapped(dst[k], n[k] * 4) : nullptr) {
        hr.src[k] = static_cast<const uint32_t*>(src[k]); hr.dst[k] = static_cast<uint32_t*>(p); hr.n[k] = (int)n[k]; any = true;
      } else {
        D2C_CP(dst[k], src[k], n[k] * 4, cudaMemcpyDeviceToHost);
      }
    }
    if (any) D2C_TRY(ctx, launch_results_to_host(hr, st));
    if (out->hidden_out_host && !early) D2C_CP(out->hidden_out_host, b.x, R * c.d_model * sizeof(bf16), cudaMemcpyDeviceToHost);
  }
#undef D2C_CP
  return D2C_OK;
}

int d2c_step_host(d2c_ctx* ctx, const d2c_step_args* h, const d2c_host_out* out) {
  D2C_TRY(ctx, check_step_args(ctx, h));
  if (h->forced && (h->forced_off[h->batch] < 0 || (size_t)h->forced_off[h->batch] > (size_t)h->batch * h->seq_len))
    return fail(ctx, D2C_EINVAL, "d2c_step_host: %d forced rows", h->forced_off[h->batch]);
  const int rc = enqueue_step_host(ctx, h, out);
  // The caller may free its buffers once it has the answer, also when that is an error: nothing enqueued so far may use them
  // any longer.  (Behind an error the step's own streams need not have been joined.)
  cudaError_t e = cudaStreamSynchronize(ctx->stream);
  if (ctx->copy_stream && out && out->hidden_out_host) { const cudaError_t e2 = cudaStreamSynchronize(ctx->copy_stream); if (e == cudaSuccess) e = e2; }
  if (rc == D2C_OK) return e == cudaSuccess ? D2C_OK : fail(ctx, D2C_ECUDA, "d2c_step_host: %s", cudaGetErrorString(e));
  if (ctx->work_stream) { cudaStreamSynchronize(ctx->work_stream); cudaStreamSynchronize(ctx->side_stream); }
  (void)cudaGetLastError();                                  // reported by this call, not to whoever asks next
  return rc;
}

int d2c_commit(d2c_ctx* ctx, int32_t batch, int32_t seq_len, const void* embed_table, void* h0,
               uint8_t* mask, int32_t* tokens, int32_t* committed, int32_t rule, float threshold) {
  if (!ctx) return D2C_EINVAL;
  if (!embed_table || !h0 || !mask || !tokens || !committed) return fail(ctx, D2C_EINVAL, "d2c_commit: null pointer");
  if (batch < 1 || batch > ctx->cfg.max_batch || seq_len < 1 || seq_len > ctx->cfg.max_seq)
    return fail(ctx, D2C_ECAPACITY, "d2c_commit: batch %d x seq_len %d out of range", batch, seq_len);
  if (rule < 0 || rule > 2 || isnan(threshold)) return fail(ctx, D2C_EINVAL, "d2c_commit: rule %d / threshold", rule);
  if (ctx->used_batch != 0 && (batch != ctx->used_batch || seq_len != ctx->used_seq))
    return fail(ctx, D2C_EINVAL, "d2c_commit: batch %d x seq_len %d differs from the %d x %d of this context's steps", batch, seq_len, ctx->used_batch, ctx->used_seq);
  const Buffers& b = ctx->buf;
  D2C_TRY(ctx, launch_commit(batch, seq_len, ctx->cfg.d_model, ctx->cfg.vocab, rule, threshold, b.slot_of_pos, b.conf, b.pred, b.phi,
                             ctx->phi_len < seq_len ? ctx->phi_len : seq_len, (const bf16*)embed_table, (bf16*)h0, mask,
                             tokens, committed, ctx->stream));
  return D2C_OK;
}

}  // extern "C"
