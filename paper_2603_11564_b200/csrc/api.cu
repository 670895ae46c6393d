// C ABI of libdapq: context, argument checking, workspace, and the launch sequences.
// See include/dapq.h for the contract of every entry point.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <new>
#include <vector>

#include "dapq_internal.cuh"

using namespace dapq;

struct dapq_ctx {
  int device = 0;
  dapq_shape shape{};
  Dims dims{};
  int elem_bytes = 2;
  int n_sm = 148;
  int64_t max_chunks = 0;
  int64_t q_rows_max = 0;        // max_batch * H_q * N
  // device workspace
  void* owned[24] = {};          // its allocations
  int n_owned = 0;
  double* inv_freq = nullptr;    // [d/2]
  int* status = nullptr;         // device status word
  void* q_rot = nullptr;         // [max_batch, H_q, N, d]
  float2* part = nullptr;        // [max_chunks, H_q, N]
  // (of these, room for flow_layers layers)
  float* lse2 = nullptr;         // [max_batch, H_q, N]
  float* scores = nullptr;       // [H_kv, max_total_rows]
  float* pooled = nullptr;       // [H_kv, max_total_rows] (pooling only)
  float* slots = nullptr;        // [query groups, H_kv, max_total_rows] (sized for groups of 256 query rows; used when sweep 2 has more than one group)
  long long wait_limit = 0;      // cycles a device-side wait may take (0: the default, about a second)
  int32_t* idx = nullptr;        // [H_kv, max_total_rows]
  int flow_layers = 1;           // layers of the full size that one launch may cover
  int score_slots = 2;           // layers of the full size that `scores` has room for, that of `idx` included
  int64_t flow_chunks = 0;       // rows of `part` in the layout of score_flow.cu
  uint32_t* sync[2] = {};        // tickets and counters of its launches, used in turn
  int64_t sync_words = 0;
  int sync_turn = 0;
  PruneBuffers prune = {};       // the pruned selection (sums == nullptr: not available)
  // staging for the host-buffer entry points (allocated on first use): two sets, so that the copies of one
  // layer run beside the kernels of the layer before
  struct HostStage {
    void *q = nullptr, *k = nullptr, *v = nullptr, *ko = nullptr, *vo = nullptr;
    int32_t* idx = nullptr;
    cudaEvent_t in_done = nullptr;    // the layer's inputs have arrived (recorded on the copy stream)
    cudaEvent_t out_done = nullptr;   // the layer's results have left (recorded on the caller's stream)
  } hs[2];
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t fork = nullptr;         // orders the copy stream behind what the caller's stream already holds
  LaunchLog log;
  char err[512] = "";
};

// ---- launch accounting and per-kernel event timing ----------------------------------------
namespace dapq {
struct ProfImpl {
  std::vector<cudaEvent_t> pool;      // event pairs, reused after every drain
  std::vector<int> kinds;             // kind of each pending pair
  double ms[kKindCount] = {};
  int64_t count[kKindCount] = {};
  ~ProfImpl() { for (cudaEvent_t e : pool) cudaEventDestroy(e); }
};

void LaunchLog::begin(int kind, cudaStream_t s) {
  ++n_launch;
  if (!profiling) return;
  ProfImpl* p = static_cast<ProfImpl*>(impl);
  const size_t n = p->kinds.size();
  while (p->pool.size() < 2 * (n + 1)) {
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) { profiling = false; return; }
    p->pool.push_back(e);
  }
  p->kinds.push_back(kind);
  cudaEventRecord(p->pool[2 * n], s);
}

void LaunchLog::end(cudaStream_t s) {
  if (!profiling) return;
  ProfImpl* p = static_cast<ProfImpl*>(impl);
  cudaEventRecord(p->pool[2 * (p->kinds.size() - 1) + 1], s);
}
}  // namespace dapq

namespace {

// Message of the last failed dapq_create on this thread (there is no context to hold it).
thread_local char g_create_err[256] = "";

struct DeviceGuard {
  int prev = -1;
  bool ok = true;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; return; }
    if (prev != dev && cudaSetDevice(dev) != cudaSuccess) ok = false;
  }
  ~DeviceGuard() { if (prev >= 0) cudaSetDevice(prev); }
};

dapq_status fail(dapq_ctx* ctx, dapq_status st, const char* fmt, ...) {
  if (ctx) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(ctx->err, sizeof(ctx->err), fmt, ap);
    va_end(ap);
  }
  return st;
}

dapq_status cuda_fail(dapq_ctx* ctx, cudaError_t e, const char* what) {
  return fail(ctx, DAPQ_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define DAPQ_CUDA(ctx, call)                                        \
  do {                                                              \
    cudaError_t e_ = (call);                                        \
    if (e_ != cudaSuccess) return cuda_fail((ctx), e_, #call);      \
  } while (0)

constexpr double kFlowPairs = 6e8;             // query-key pairs of a launch of score_flow.cu that make its start and end small
constexpr int kMaxGridY = 65535;
constexpr double kAlonePairs = 3.3e8;          // query-key pairs of one prompt from which a layer goes by itself
constexpr size_t kFlowLeastPairs = 16;         // key pairs of a unit for which its partial row sums have room in any call

// Device buffers allocated together: as one block, cut up at 256-byte boundaries, where a block of its own for each
// would cost up to a millisecond apiece (large ones), or each by itself, where the driver has small blocks at hand.
struct Arena {
  struct Part { void** p; size_t bytes; };
  Part parts[16];
  int n = 0;
  size_t size = 0;
  template <typename T> void add(T** p, size_t bytes) {
    parts[n++] = {reinterpret_cast<void**>(p), (bytes + 255) & ~(size_t)255};
    size += parts[n - 1].bytes;
  }
  bool allocate(dapq_ctx* ctx) {
    const bool together = size >= (4u << 20);
    char* at = nullptr;
    if (together) {
      if (cudaMalloc(&at, size) != cudaSuccess) return false;
      ctx->owned[ctx->n_owned++] = at;
    }
    for (int i = 0; i < n; ++i) {
      if (together) {
        *parts[i].p = at;
        at += parts[i].bytes;
      } else {
        if (cudaMalloc(parts[i].p, parts[i].bytes) != cudaSuccess) return false;
        ctx->owned[ctx->n_owned++] = *parts[i].p;
      }
    }
    return true;
  }
};

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Fill the sequence table from the caller's host arrays and check it against the context.
// Any of cu_rows / prompt_len may come from a cache view; k_keep and pos_start are optional.
dapq_status build_table(dapq_ctx* ctx, int32_t batch, const int32_t* cu_rows, const int32_t* prompt_len,
                        const int32_t* cu_prompt, const int32_t* k_keep, const int32_t* pos_start,
                        SeqTable* t) {
  const dapq_shape& sh = ctx->shape;
  if (batch < 1) return fail(ctx, DAPQ_ERR_INVALID_ARG, "batch must be >= 1 (got %d)", batch);
  if (batch > sh.max_batch)
    return fail(ctx, DAPQ_ERR_WORKSPACE, "batch %d exceeds max_batch %d", batch, sh.max_batch);
  memset(t, 0, sizeof(*t));
  t->batch = batch;
  int64_t rows = 0, prompt = 0, keep = 0, chunks = 0;
  for (int b = 0; b < batch; ++b) {
    int64_t L;
    if (prompt_len) {
      L = prompt_len[b];
    } else if (cu_prompt) {
      L = (int64_t)cu_prompt[b + 1] - cu_prompt[b];
    } else {
      L = 1;  // rope-only tables carry no lengths
    }
    if (L < 1) return fail(ctx, DAPQ_ERR_INVALID_ARG, "prompt length of sequence %d is %lld (must be >= 1)", b, (long long)L);
    if (cu_prompt && cu_prompt[b] != prompt)
      return fail(ctx, DAPQ_ERR_INVALID_ARG, "cu_prompt[%d] = %d, expected %lld", b, cu_prompt[b], (long long)prompt);
    if (cu_rows) {
      if (b == 0 && cu_rows[0] < 0) return fail(ctx, DAPQ_ERR_INVALID_ARG, "cu_rows[0] is negative");
      if ((int64_t)cu_rows[b + 1] - cu_rows[b] != L + sh.n_pseudo)
        return fail(ctx, DAPQ_ERR_INVALID_ARG,
                    "sequence %d owns %lld cache rows, expected L_b + N = %lld", b,
                    (long long)((int64_t)cu_rows[b + 1] - cu_rows[b]), (long long)(L + sh.n_pseudo));
      t->cu_rows[b] = cu_rows[b];
      t->cu_rows[b + 1] = cu_rows[b + 1];
    } else {
      t->cu_rows[b] = (int32_t)rows;
      t->cu_rows[b + 1] = (int32_t)(rows + L + sh.n_pseudo);
    }
    int64_t kb = L;
    if (k_keep) {
      if (k_keep[b] < 1) return fail(ctx, DAPQ_ERR_INVALID_ARG, "k_keep[%d] = %d (must be >= 1)", b, k_keep[b]);
      kb = k_keep[b] < L ? k_keep[b] : L;
    }
    t->prompt_len[b] = (int32_t)L;
    t->pos_start[b] = pos_start ? pos_start[b] : (int32_t)L;
    if (pos_start && pos_start[b] < 0) return fail(ctx, DAPQ_ERR_INVALID_ARG, "pos_start[%d] is negative", b);
    t->cu_prompt[b] = (int32_t)prompt;
    t->cu_keep[b] = (int32_t)keep;
    rows += L + sh.n_pseudo;
    prompt += L;
    keep += kb;
    chunks += (L + kChunkKeys - 1) / kChunkKeys + 1;
  }
  t->cu_prompt[batch] = (int32_t)prompt;
  t->cu_keep[batch] = (int32_t)keep;
  const int64_t last_row = cu_rows ? cu_rows[batch] : rows;
  if ((prompt_len || cu_prompt) && last_row > sh.max_total_rows)
    return fail(ctx, DAPQ_ERR_WORKSPACE, "%lld cache rows exceed max_total_rows %lld",
                (long long)last_row, (long long)sh.max_total_rows);
  if ((prompt_len || cu_prompt) && chunks > ctx->max_chunks)
    return fail(ctx, DAPQ_ERR_WORKSPACE, "%lld work chunks of %d keys exceed the %lld the workspace was sized for "
                "(more or longer sequences than max_batch / max_total_rows allow)",
                (long long)chunks, kChunkKeys, (long long)ctx->max_chunks);
  return DAPQ_OK;
}

dapq_status check_view(dapq_ctx* ctx, const dapq_cache_view* cv, bool need_v, bool host, CacheDev* out) {
  if (!cv) return fail(ctx, DAPQ_ERR_INVALID_ARG, "cache view is NULL");
  if (!cv->k || (need_v && !cv->v)) return fail(ctx, DAPQ_ERR_INVALID_ARG, "cache view has a NULL K or V pointer");
  if (!cv->cu_rows_host || !cv->prompt_len_host)
    return fail(ctx, DAPQ_ERR_INVALID_ARG, "cache view needs cu_rows_host and prompt_len_host");
  if (cv->reserved != 0) return fail(ctx, DAPQ_ERR_INVALID_ARG, "cache view reserved field must be 0");
  const int per16 = 16 / ctx->elem_bytes;
  const bool use_v = cv->v != nullptr;
  if (cv->k_row_stride < kHeadDim || cv->k_head_stride < 0 || (use_v && (cv->v_row_stride < kHeadDim || cv->v_head_stride < 0)))
    return fail(ctx, DAPQ_ERR_INVALID_ARG, "row strides must be >= head_dim and head strides >= 0");
  if (!host) {
    if (cv->k_row_stride % per16 || cv->k_head_stride % per16 || !aligned16(cv->k) ||
        (use_v && (cv->v_row_stride % per16 || cv->v_head_stride % per16 || !aligned16(cv->v))))
      return fail(ctx, DAPQ_ERR_UNSUPPORTED, "K/V base pointers and strides must be multiples of 16 bytes");
  }
  out->k = cv->k;
  out->v = cv->v;
  out->k_head_stride = cv->k_head_stride;
  out->k_row_stride = cv->k_row_stride;
  out->v_head_stride = cv->v_head_stride;
  out->v_row_stride = cv->v_row_stride;
  return DAPQ_OK;
}

// The fp16 tensor-core scorer takes bf16 caches whose query block is at least half an MMA tile high; fp32 storage
// and smaller query blocks go to the one that splits its operands (run_score); views TMA cannot describe and
// syn_mass requests to the CUDA-core scorer.
bool wants_umma(const dapq_ctx* ctx) {
  return ctx->shape.dtype == DAPQ_BF16 && !(ctx->shape.flags & DAPQ_FLAG_CUDA_CORE_SCORER) &&
         ctx->dims.group * ctx->dims.n_pseudo >= 64;
}

// ... and the one with split operands what the other does not take, unless the context asks for the CUDA cores.
bool wants_split(const dapq_ctx* ctx) { return !(ctx->shape.flags & DAPQ_FLAG_CUDA_CORE_SCORER) && !wants_umma(ctx); }

dapq_status run_score_umma(dapq_ctx* ctx, const UmmaPlan& plan, const SeqTable& t, const float* lse_in,
                           float* scores, int64_t score_stride, float* lse_out, cudaStream_t s) {
  cudaError_t e = launch_score_umma(plan, t, ctx->dims, lse_in, ctx->part, scores, score_stride,
                                    lse_out, ctx->status, ctx->wait_limit, s, &ctx->log);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "tensor-core score kernels (two-part bf16 queries)");
  return DAPQ_OK;
}

dapq_status run_score_qg(dapq_ctx* ctx, const QgPlan& plan, const SeqTable& t, const float* lse_in,
                         float* scores, int64_t score_stride, float* lse_out, bool after_rope, cudaStream_t s) {
  cudaError_t e = launch_score_qg(plan, t, ctx->dims, lse_in, ctx->part, ctx->slots, scores, score_stride, lse_out,
                                  ctx->lse2, ctx->status, ctx->wait_limit, after_rope, s, &ctx->log);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "tensor-core score kernels");
  return DAPQ_OK;
}

// The scorer over several layers a launch: the eviction path's own fp16 queries (more than 256 query rows a KV head: in groups, each
// with its own score slot).
bool wants_flow(const dapq_ctx* ctx) {
  return wants_umma(ctx) && !(ctx->shape.flags & (DAPQ_FLAG_Q_BF16 | DAPQ_FLAG_Q_LO_SWEEP1 | DAPQ_FLAG_Q_LO_SWEEP2));
}

// The older tensor-core kernels (a second MMA pass with the low-order bf16 part of the queries) serve
// the contexts that ask for that part in either sweep.
bool wants_lo(const dapq_ctx* ctx) { return (ctx->shape.flags & (DAPQ_FLAG_Q_LO_SWEEP1 | DAPQ_FLAG_Q_LO_SWEEP2)) != 0; }

// fp32 arithmetic on unrounded queries: on the tensor cores with split operands, or on the CUDA cores where the
// context asks for them, the attention mass of the synthetic keys is wanted, or TMA cannot describe the view.
dapq_status run_score(dapq_ctx* ctx, int q_dtype, const void* q_rot, const CacheDev& cd, const SeqTable& t,
                      const float* lse_in, float* scores, int64_t score_stride, float* lse_out,
                      float* syn_mass, bool after_rope, cudaStream_t s) {
  cudaError_t e;
  SplitPlan plan;
  if (wants_split(ctx) && !syn_mass && split_plan(ctx->shape.dtype, cd, t, ctx->dims, ctx->n_sm, &plan))
    e = launch_score_split(plan, q_dtype, q_rot, t, ctx->dims, lse_in, ctx->part, ctx->slots, scores, score_stride, lse_out,
                           ctx->status, ctx->wait_limit, after_rope, s, &ctx->log);
  else
    e = launch_score_fma(ctx->shape.dtype, q_dtype, q_rot, cd, t, ctx->dims, lse_in, ctx->part, ctx->max_chunks, ctx->n_sm,
                         ctx->lse2, scores, score_stride, lse_out, syn_mass, s, &ctx->log);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "score kernels");
  return DAPQ_OK;
}

IndexOut one_index(const dapq_ctx* ctx, int32_t* idx) {
  IndexOut out = {};
  out.p[0] = idx;
  out.heads_per_layer = ctx->dims.n_kv_heads;
  return out;
}

RopeBatch one_rope(const dapq_ctx* ctx, const void* q_pre) {
  RopeBatch rb = {};
  rb.q[0] = q_pre;
  rb.n_layers = 1;
  rb.group = ctx->dims.group;
  return rb;
}

// Eq. 5 on the scores ([n_layers][H_kv][score_stride]), or on their pooled image if the context asks for pooling.
dapq_status run_select(dapq_ctx* ctx, int n_layers, const float* scores, int64_t score_stride, const IndexOut& idx, int64_t idx_stride,
                       const SeqTable& t, cudaStream_t s) {
  cudaError_t e;
  if (ctx->shape.pool_mode != DAPQ_POOL_NONE) {
    e = launch_pool(scores, ctx->pooled, score_stride, t, n_layers * ctx->dims.n_kv_heads, ctx->shape.pool_kernel,
                    ctx->shape.pool_mode, s, &ctx->log);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "pooling kernel");
    scores = ctx->pooled;
  }
  e = launch_topk(scores, score_stride, idx, idx_stride, t, n_layers * ctx->dims.n_kv_heads, s, &ctx->log);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "top-k kernel");
  return DAPQ_OK;
}

}  // namespace

extern "C" {

dapq_status dapq_create(dapq_ctx** out, const dapq_shape* sh, int device) {
  if (!out || !sh) return DAPQ_ERR_INVALID_ARG;
  *out = nullptr;
  dapq_ctx* ctx = new (std::nothrow) dapq_ctx();
  if (!ctx) return DAPQ_ERR_CUDA;
  // Errors before the context exists are reported through a context that is then freed:
  // keep the message reachable by returning the status only.
  auto bail = [&](dapq_status st, const char* why) {
    snprintf(g_create_err, sizeof(g_create_err), "dapq_create: %s", why);
    dapq_destroy(ctx);
    return st;
  };
  if (sh->head_dim != kHeadDim) return bail(DAPQ_ERR_UNSUPPORTED, "head_dim must be 128");
  if (sh->n_pseudo < 1 || sh->n_pseudo > kMaxPseudo) return bail(DAPQ_ERR_UNSUPPORTED, "n_pseudo must be in 1..128");
  if (sh->n_q_heads < 1 || sh->n_kv_heads < 1 || sh->n_q_heads % sh->n_kv_heads)
    return bail(DAPQ_ERR_INVALID_ARG, "n_kv_heads must divide n_q_heads");
  if (sh->max_batch < 1 || sh->max_total_rows < 1) return bail(DAPQ_ERR_INVALID_ARG, "max_batch and max_total_rows must be >= 1");
  if (sh->max_batch > kMaxBatch || sh->max_total_rows > 0x7fffffffLL)
    return bail(DAPQ_ERR_UNSUPPORTED, "max_batch > 128 or max_total_rows >= 2^31");
  if (sh->dtype != DAPQ_BF16 && sh->dtype != DAPQ_F32) return bail(DAPQ_ERR_INVALID_ARG, "unknown dtype");
  if (sh->flags & ~(DAPQ_FLAG_CUDA_CORE_SCORER | DAPQ_FLAG_ROPE_INTERLEAVED | DAPQ_FLAG_Q_BF16 | DAPQ_FLAG_Q_LO_SWEEP1 |
                    DAPQ_FLAG_Q_LO_SWEEP2))
    return bail(DAPQ_ERR_INVALID_ARG, "unknown flag");
  if (sh->pool_mode != DAPQ_POOL_NONE && sh->pool_mode != DAPQ_POOL_MAX && sh->pool_mode != DAPQ_POOL_AVG)
    return bail(DAPQ_ERR_INVALID_ARG, "unknown pool_mode");
  if (sh->pool_mode != DAPQ_POOL_NONE && (sh->pool_kernel < 3 || sh->pool_kernel > DAPQ_MAX_POOL_KERNEL || sh->pool_kernel % 2 == 0))
    return bail(DAPQ_ERR_UNSUPPORTED, "pool_kernel must be odd, 3 .. 127");
  if (!sh->inv_freq_host && !(sh->rope_base > 0.0)) return bail(DAPQ_ERR_INVALID_ARG, "rope_base must be > 0");
  if (!(sh->softmax_scale >= 0.f)) return bail(DAPQ_ERR_INVALID_ARG, "softmax_scale must be >= 0");

  ctx->device = device;
  ctx->shape = *sh;
  ctx->shape.inv_freq_host = nullptr;
  ctx->elem_bytes = sh->dtype == DAPQ_BF16 ? 2 : 4;
  ctx->dims.n_q_heads = sh->n_q_heads;
  ctx->dims.n_kv_heads = sh->n_kv_heads;
  ctx->dims.group = sh->n_q_heads / sh->n_kv_heads;
  ctx->dims.n_pseudo = sh->n_pseudo;
  ctx->dims.rope_interleaved = (sh->flags & DAPQ_FLAG_ROPE_INTERLEAVED) ? 1 : 0;
  const double scale = sh->softmax_scale > 0.f ? (double)sh->softmax_scale : 1.0 / sqrt((double)kHeadDim);
  ctx->dims.scale_log2e = (float)(scale * 1.4426950408889634074);

  DeviceGuard guard(device);
  if (!guard.ok) return bail(DAPQ_ERR_CUDA, "cannot make the device current");
  double freq[kHeadDim / 2];
  for (int c = 0; c < kHeadDim / 2; ++c)
    freq[c] = sh->inv_freq_host ? sh->inv_freq_host[c] : pow(sh->rope_base, -2.0 * c / (double)kHeadDim);
  if (cudaDeviceGetAttribute(&ctx->n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || ctx->n_sm < 1)
    return bail(DAPQ_ERR_CUDA, "cannot query the device");
  // partials of the CUDA-core sweeps: the chunks at 512 keys each, plus room to cut small inputs
  // finer (down to 64 keys) until every SM has two CTAs
  ctx->max_chunks = (sh->max_total_rows + kChunkKeys - 1) / kChunkKeys + 2LL * sh->max_batch +
                    (2LL * ctx->n_sm + sh->n_kv_heads - 1) / sh->n_kv_heads;
  const size_t hq_n = (size_t)sh->n_q_heads * sh->n_pseudo;
  ctx->q_rows_max = (int64_t)sh->max_batch * hq_n;
  const size_t part_umma = (size_t)umma_part_elems(sh->max_batch, sh->n_q_heads, sh->n_kv_heads, sh->n_pseudo);
  const size_t rows = (size_t)sh->max_total_rows;
  const bool flow = wants_flow(ctx);
  if (flow) {
    // enough layers a launch for some 6e8 query-key pairs; small calls of a large context may take more
    const double layers = kFlowPairs / ((double)hq_n * rows);
    ctx->flow_layers = layers >= kFlowLayers ? kFlowLayers : (int)layers + 1;
  }
  const int n_slots = wants_umma(ctx) ? qg_groups(ctx->dims) : (wants_split(ctx) ? split_groups(ctx->dims) : 1);
  const size_t score_bytes = (size_t)sh->n_kv_heads * rows * sizeof(float);
  auto allocate = [&] {
    const size_t nl = (size_t)ctx->flow_layers, part_fma = (size_t)ctx->max_chunks * hq_n;
    size_t part_elems = part_umma > part_fma ? part_umma : part_fma;
    if (flow) {
      const size_t chunk_elems = (size_t)sh->n_kv_heads * flow_rows_pad(ctx->dims);
      const size_t runs = nl * (rows / (256 * kFlowLeastPairs) + 1), few = 4 * (size_t)ctx->n_sm / ((size_t)sh->n_kv_heads * qg_groups(ctx->dims)) + 1;
      const size_t want = nl * sh->max_batch + (runs > few ? runs : few);
      const size_t need = want * chunk_elems * 3 / 2;                // (a float2 and a float each)
      if (need > part_elems) part_elems = need;
      ctx->flow_chunks = (int64_t)(part_elems * 2 / 3 / chunk_elems);
      ctx->sync_words = (int64_t)nl * sh->max_batch * sh->n_kv_heads * qg_groups(ctx->dims) + 1;
    }
    Arena ar;
    ar.add(&ctx->inv_freq, sizeof(freq));
    ar.add(&ctx->status, sizeof(int));
    ar.add(&ctx->q_rot, (size_t)sh->max_batch * hq_n * kHeadDim * (nl > 1 ? nl * sizeof(__half) : sizeof(float)));
    ar.add(&ctx->part, part_elems * sizeof(float2));
    ar.add(&ctx->lse2, (nl * sh->max_batch * hq_n + 32) * sizeof(float));
    // (the indices have the last of the score slots, which launches whose caller takes the indices fill with scores too)
    ctx->score_slots = nl > 2 ? (int)nl : 2;
    ar.add(&ctx->scores, ctx->score_slots * score_bytes);
    if (sh->pool_mode != DAPQ_POOL_NONE) ar.add(&ctx->pooled, nl * score_bytes);
    if (n_slots > 1) ar.add(&ctx->slots, nl * n_slots * score_bytes);
    if (flow)
      for (auto& w : ctx->sync) ar.add(&w, ctx->sync_words * sizeof(uint32_t));
    return ar.allocate(ctx);
  };
  bool ok = allocate();
  if (!ok && ctx->flow_layers > 1) {
    // no room for several layers of the full size: what one takes will do (64 prompts of 130 tokens on 64 heads: 290 of 696 MB)
    cudaGetLastError();
    while (ctx->n_owned > 0) cudaFree(ctx->owned[--ctx->n_owned]);
    ctx->flow_layers = 1;
    ok = allocate();
  }
  if (ok) ctx->idx = reinterpret_cast<int32_t*>(ctx->scores + (size_t)(ctx->score_slots - 1) * sh->n_kv_heads * rows);
  ok = ok && cudaMemcpy(ctx->inv_freq, freq, sizeof(freq), cudaMemcpyHostToDevice) == cudaSuccess;
  ok = ok && cudaMemset(ctx->status, 0, sizeof(int)) == cudaSuccess;
  if (!ok) { cudaGetLastError(); return bail(DAPQ_ERR_CUDA, "workspace allocation failed"); }
  if (wants_umma(ctx) && !wants_lo(ctx) && !(sh->flags & DAPQ_FLAG_Q_BF16) && sh->pool_mode == DAPQ_POOL_NONE &&
      qg_groups(ctx->dims) <= kPruneSums && (double)hq_n * rows >= kPruneLeastPairs &&
      (int64_t)rows >= (int64_t)kPruneLeastLen * sh->max_batch && prune_available()) {
    // (some 20 bytes a row and KV head: not for contexts of many short prompts, whose calls never take the route.  No room:
    // the two full sweeps need none of these)
    PruneBuffers& pr = ctx->prune;
    Arena pa;
    pa.add(&pr.part_m, part_umma * sizeof(float2));
    pa.add(&pr.sums, kPruneSums * (score_bytes + 16));
    pa.add(&pr.cand, (size_t)sh->n_kv_heads * rows * sizeof(int32_t));
    pa.add(&pr.hist, (size_t)sh->max_batch * sh->n_kv_heads * kPruneHist * sizeof(uint32_t));
    pa.add(&pr.route, 2 * sizeof(float2));
    pa.add(&pr.est, (size_t)sh->max_batch * hq_n * sizeof(float));
    if (!pa.allocate(ctx)) {
      cudaGetLastError();
      pr.sums = nullptr;
    }
    pr.part_s = ctx->part;
    pr.ref = ctx->lse2;
  }
  *out = ctx;
  return DAPQ_OK;
}

void dapq_destroy(dapq_ctx* ctx) {
  if (!ctx) return;
  {
    DeviceGuard guard(ctx->device);
    for (int i = 0; i < ctx->n_owned; ++i) cudaFree(ctx->owned[i]);
    for (auto& st : ctx->hs) {
      void* sb[] = {st.q, st.k, st.v, st.ko, st.vo, st.idx};
      for (void* p : sb)
        if (p) cudaFree(p);
      if (st.in_done) cudaEventDestroy(st.in_done);
      if (st.out_done) cudaEventDestroy(st.out_done);
    }
    if (ctx->fork) cudaEventDestroy(ctx->fork);
    if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
  }
  delete static_cast<dapq::ProfImpl*>(ctx->log.impl);
  delete ctx;
}

const char* dapq_last_error(const dapq_ctx* ctx) { return ctx ? ctx->err : g_create_err; }

int64_t dapq_launch_count(const dapq_ctx* ctx) { return ctx ? ctx->log.n_launch : 0; }

dapq_status dapq_rope_inv_freq_llama3(double rope_base, double factor, double low_freq_factor, double high_freq_factor,
                                      int32_t original_context, double* inv_freq_out) {
  if (!inv_freq_out || !(rope_base > 0.0) || !(factor >= 1.0) || !(low_freq_factor > 0.0) ||
      !(high_freq_factor > low_freq_factor) || original_context < 1)
    return DAPQ_ERR_INVALID_ARG;
  const double two_pi = 6.283185307179586476925286766559;
  const double short_wave = original_context / high_freq_factor, long_wave = original_context / low_freq_factor;
  for (int c = 0; c < kHeadDim / 2; ++c) {
    const double f = pow(rope_base, -2.0 * c / (double)kHeadDim), wave = two_pi / f;
    double g = f;
    if (wave > long_wave) {
      g = f / factor;
    } else if (wave >= short_wave) {
      const double smooth = (original_context / wave - low_freq_factor) / (high_freq_factor - low_freq_factor);
      g = (1.0 - smooth) * f / factor + smooth * f;
    }
    inv_freq_out[c] = g;
  }
  return DAPQ_OK;
}

dapq_status dapq_set_wait_limit(dapq_ctx* ctx, int64_t cycles) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  if (cycles < 0) return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_set_wait_limit: negative limit");
  ctx->wait_limit = cycles;
  return DAPQ_OK;
}

dapq_status dapq_poll_status(dapq_ctx* ctx, void* stream) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  DeviceGuard guard(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  int word = 0;
  DAPQ_CUDA(ctx, cudaStreamSynchronize(s));
  DAPQ_CUDA(ctx, cudaMemcpy(&word, ctx->status, sizeof(int), cudaMemcpyDeviceToHost));
  if (word) DAPQ_CUDA(ctx, cudaMemset(ctx->status, 0, sizeof(int)));
  if (word & kStatusTimeout) return fail(ctx, DAPQ_ERR_TIMEOUT, "a kernel gave up on a bounded wait; its results are undefined");
  if (word & kStatusBadIndex) return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_compact_kv skipped indices outside [0, L_b)");
  if (word & kStatusSmemAlign)
    return fail(ctx, DAPQ_ERR_UNSUPPORTED, "the score kernels found their shared memory off a 1024-byte boundary and did nothing");
  return DAPQ_OK;
}

dapq_status dapq_profile(dapq_ctx* ctx, int32_t enable) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  if (!ctx->log.impl) {
    ctx->log.impl = new (std::nothrow) dapq::ProfImpl();
    if (!ctx->log.impl) return fail(ctx, DAPQ_ERR_CUDA, "out of host memory");
  }
  dapq::ProfImpl* p = static_cast<dapq::ProfImpl*>(ctx->log.impl);
  if (enable) {
    p->kinds.clear();
    for (int k = 0; k < kKindCount; ++k) { p->ms[k] = 0.0; p->count[k] = 0; }
  }
  ctx->log.profiling = enable != 0;
  return DAPQ_OK;
}

dapq_status dapq_profile_read(dapq_ctx* ctx, void* stream, double* ms_out, int64_t* count_out) {
  if (!ctx || !ms_out || !count_out) return DAPQ_ERR_INVALID_ARG;
  dapq::ProfImpl* p = static_cast<dapq::ProfImpl*>(ctx->log.impl);
  if (!p) return fail(ctx, DAPQ_ERR_INVALID_ARG, "profiling was never enabled");
  DeviceGuard guard(ctx->device);
  DAPQ_CUDA(ctx, cudaStreamSynchronize((cudaStream_t)stream));
  for (size_t i = 0; i < p->kinds.size(); ++i) {
    float ms = 0.f;
    DAPQ_CUDA(ctx, cudaEventElapsedTime(&ms, p->pool[2 * i], p->pool[2 * i + 1]));
    p->ms[p->kinds[i]] += ms;
    p->count[p->kinds[i]] += 1;
  }
  p->kinds.clear();
  for (int k = 0; k < kKindCount; ++k) { ms_out[k] = p->ms[k]; count_out[k] = p->count[k]; }
  return DAPQ_OK;
}

dapq_status dapq_rope_pseudo_q(dapq_ctx* ctx, const void* q_pre, const int32_t* pos_start_host,
                               int32_t batch, void* q_rot, void* stream) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  if (!q_pre || !q_rot || !pos_start_host) return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_rope_pseudo_q: NULL argument");
  SeqTable t;
  dapq_status st = build_table(ctx, batch, nullptr, nullptr, nullptr, nullptr, pos_start_host, &t);
  if (st != DAPQ_OK) return st;
  DeviceGuard guard(ctx->device);
  cudaError_t e = launch_rope(ctx->shape.dtype, ctx->shape.dtype, 0, one_rope(ctx, q_pre), q_rot, ctx->inv_freq, t, ctx->dims, false,
                              (cudaStream_t)stream, &ctx->log);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "rope kernel");
  return DAPQ_OK;
}

dapq_status dapq_score(dapq_ctx* ctx, const void* q_rot, const dapq_cache_view* cache,
                       const float* lse_in, float* scores, float* lse_out, float* syn_mass, void* stream) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  if (!q_rot || !scores) return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_score: NULL argument");
  if (!aligned16(q_rot)) return fail(ctx, DAPQ_ERR_UNSUPPORTED, "q_rot must be 16-byte aligned");
  CacheDev cd;
  dapq_status st = check_view(ctx, cache, false, false, &cd);
  if (st != DAPQ_OK) return st;
  SeqTable t;
  st = build_table(ctx, cache->batch, cache->cu_rows_host, cache->prompt_len_host, nullptr, nullptr, nullptr, &t);
  if (st != DAPQ_OK) return st;
  DeviceGuard guard(ctx->device);
  if (wants_umma(ctx) && !syn_mass) {
    // the caller's bf16 queries are exact in bf16: one bf16 x bf16 MMA pass, no conversion of K
    if (wants_lo(ctx)) {
      UmmaPlan plan;
      if (umma_plan(q_rot, 0, 0, cd, t, ctx->dims, ctx->n_sm, &plan))
        return run_score_umma(ctx, plan, t, lse_in, scores, t.cu_prompt[t.batch], lse_out, (cudaStream_t)stream);
    } else {
      QgPlan plan;
      if (qg_plan(q_rot, 0, cd, t, ctx->dims, ctx->n_sm, &plan))
        return run_score_qg(ctx, plan, t, lse_in, scores, t.cu_prompt[t.batch], lse_out, false, (cudaStream_t)stream);
    }
  }
  return run_score(ctx, ctx->shape.dtype, q_rot, cd, t, lse_in, scores, t.cu_prompt[t.batch], lse_out, syn_mass, false,
                   (cudaStream_t)stream);
}

dapq_status dapq_topk_select(dapq_ctx* ctx, const float* scores, const int32_t* cu_prompt_host,
                             const int32_t* k_keep_host, int32_t batch, int32_t* idx_out, void* stream) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  if (!scores || !cu_prompt_host || !k_keep_host || !idx_out)
    return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_topk_select: NULL argument");
  SeqTable t;
  dapq_status st = build_table(ctx, batch, nullptr, nullptr, cu_prompt_host, k_keep_host, nullptr, &t);
  if (st != DAPQ_OK) return st;
  DeviceGuard guard(ctx->device);
  return run_select(ctx, 1, scores, t.cu_prompt[batch], one_index(ctx, idx_out), t.cu_keep[batch], t, (cudaStream_t)stream);
}

dapq_status dapq_compact_kv(dapq_ctx* ctx, const dapq_cache_view* cache, const int32_t* idx,
                            const int32_t* k_keep_host, void* k_out, void* v_out, void* stream) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  if (!idx || !k_keep_host || !k_out || !v_out) return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_compact_kv: NULL argument");
  if (!aligned16(k_out) || !aligned16(v_out)) return fail(ctx, DAPQ_ERR_UNSUPPORTED, "k_out / v_out must be 16-byte aligned");
  CacheDev cd;
  dapq_status st = check_view(ctx, cache, true, false, &cd);
  if (st != DAPQ_OK) return st;
  SeqTable t;
  st = build_table(ctx, cache->batch, cache->cu_rows_host, cache->prompt_len_host, nullptr, k_keep_host, nullptr, &t);
  if (st != DAPQ_OK) return st;
  DeviceGuard guard(ctx->device);
  CompactBatch cb = {};
  cb.l[0] = {cd, idx, k_out, v_out};
  cudaError_t e = launch_compact(ctx->shape.dtype, cb, 1, t.cu_keep[t.batch], t, ctx->dims.n_kv_heads, ctx->status, (cudaStream_t)stream,
                                 &ctx->log);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "compaction kernel");
  return DAPQ_OK;
}

dapq_status dapq_recall(dapq_ctx* ctx, const int32_t* idx_gold, const int32_t* idx_pred,
                        const int32_t* prompt_len_host, const int32_t* k_keep_host, int32_t batch,
                        float* recall_out, void* stream) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  if (!idx_gold || !idx_pred || !prompt_len_host || !k_keep_host || !recall_out)
    return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_recall: NULL argument");
  SeqTable t;
  dapq_status st = build_table(ctx, batch, nullptr, prompt_len_host, nullptr, k_keep_host, nullptr, &t);
  if (st != DAPQ_OK) return st;
  DeviceGuard guard(ctx->device);
  cudaError_t e = launch_recall(idx_gold, idx_pred, t.cu_keep[batch], t, ctx->dims.n_kv_heads, recall_out,
                                (cudaStream_t)stream, &ctx->log);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "recall kernel");
  return DAPQ_OK;
}

namespace {

// The layers of a dapq_evict_layers call that took the pruned selection so far: the last one that did whatever the one
// before it had found, and which of the two route words holds what the next one is to do.
struct PruneRoute { int32_t last_try = -1, at = 0; };

// One layer's arguments, checked.
struct Layer {
  const void* q_pre;
  CacheDev cd;
  void *k_out, *v_out;
  int32_t* idx_out;
};
dapq_status check_layer(dapq_ctx* ctx, const void* q_pre, const dapq_cache_view* cache, const int32_t* k_keep_host, void* k_out, void* v_out,
                        int32_t* idx_out, Layer* y, SeqTable* t) {
  if (!q_pre || !k_keep_host || !k_out || !v_out) return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_evict: NULL argument");
  if (!aligned16(k_out) || !aligned16(v_out)) return fail(ctx, DAPQ_ERR_UNSUPPORTED, "k_out / v_out must be 16-byte aligned");
  *y = {q_pre, {}, k_out, v_out, idx_out};
  const dapq_status st = check_view(ctx, cache, true, false, &y->cd);
  if (st != DAPQ_OK) return st;
  return build_table(ctx, cache->batch, cache->cu_rows_host, cache->prompt_len_host, nullptr, k_keep_host, nullptr, t);
}

// What a layer's step reads and writes: [lo, hi) of its arrays.
struct Span {
  uintptr_t lo, hi;
  bool meets(const Span& o) const { return lo < o.hi && o.lo < hi; }
};
Span span_of(const void* p, size_t bytes) { return {(uintptr_t)p, p ? (uintptr_t)p + bytes : (uintptr_t)p}; }

// Layers may share launches if nothing that one of them writes is written or read by another, so that their order does
// not matter; and a rotation may begin beside the compaction of the layers before if none of its own layers reads what they write.
struct LayerSpans {
  Span out[3], in[3];
  LayerSpans() = default;
  LayerSpans(const dapq_ctx* ctx, const Layer& y, const SeqTable& t) {
    const size_t eb = (size_t)ctx->elem_bytes, H = (size_t)ctx->dims.n_kv_heads, kt = (size_t)t.cu_keep[t.batch];
    auto cache = [&](const void* p, int64_t head, int64_t row) {
      return span_of(p, ((H - 1) * (size_t)head + (size_t)(t.cu_rows[t.batch] - 1) * (size_t)row + kHeadDim) * eb);
    };
    out[0] = span_of(y.k_out, H * kt * kHeadDim * eb);
    out[1] = span_of(y.v_out, H * kt * kHeadDim * eb);
    out[2] = span_of(y.idx_out, H * kt * sizeof(int32_t));
    in[0] = cache(y.cd.k, y.cd.k_head_stride, y.cd.k_row_stride);
    in[1] = cache(y.cd.v, y.cd.v_head_stride, y.cd.v_row_stride);
    in[2] = span_of(y.q_pre, (size_t)t.batch * ctx->dims.n_q_heads * ctx->dims.n_pseudo * kHeadDim * eb);
  }
  bool apart(const LayerSpans& o) const {
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j)
        if (out[i].meets(o.out[j]) || out[i].meets(o.in[j]) || in[i].meets(o.out[j])) return false;
    return true;
  }
  bool reads(const LayerSpans& o) const {
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j)
        if (in[i].meets(o.out[j])) return true;
    return false;
  }
};

// Layers of this geometry that one launch may cover: their workspace fits the context's (own_idx: the indices take a part of
// it too).  Us a layer on 8 heads, a launch per sweep -> shared launches of 7 layers, in bursts of 10 ms | over seconds (power cap):
// 8 k tokens x 128 query rows 26.9 -> 10.3 | 26.8 -> 10.1, x 1024 68 -> 48 | 68 -> 50; 30 k x 512 97 -> 83 | 98 -> 93, x 1024 173 -> 163
// | 177 -> 176; 60 k x 128 80 -> 56 | 81 -> 64, x 256 108 -> 91 | 110 -> 99; 100 k x 128 115 -> 97 | 122 -> 109, x 256 168 -> 159 | 171 -> 168,
// x 512 279 -> 280 | 293 -> 303.  So layers of long prompts and the size from which the pruned selection pays go by themselves.
// From 3.3e8 pairs of one prompt on a sweep of its own is long enough whatever the length, and where it holds 512 query rows a CTA
// it fetches and converts keys half as often: 40 k x 1024 227 -> 225 | 231 -> 236, 48 k 263 -> 265 | 271 -> 278, 60 k 329 -> 327 | 335 -> 342
// (36 k, 3e8: 206 -> 195 | 210 -> 209).  A batch of as many pairs in short prompts gains (8 x 8 k x 1024 377 -> 329 | 402 -> 375).
int layers_that_fit(const dapq_ctx* ctx, const SeqTable& t, bool own_idx) {
  int longest = 0;
  for (int b = 0; b < t.batch; ++b) longest = t.prompt_len[b] > longest ? t.prompt_len[b] : longest;
  const double rows = (double)ctx->dims.n_q_heads * ctx->dims.n_pseudo;
  if ((longest >= kPruneLeastLen && t.cu_prompt[t.batch] * rows >= kPruneLeastPairs) || longest * rows >= kAlonePairs) return 1;
  const int64_t room = ctx->shape.max_total_rows, seqs = (int64_t)ctx->shape.max_batch * ctx->flow_layers / t.batch;
  const int slots = ctx->score_slots < ctx->flow_layers ? ctx->score_slots : ctx->flow_layers;
  int64_t n = room * (own_idx && slots == ctx->score_slots ? slots - 1 : slots) / t.cu_prompt[t.batch];
  if (own_idx && room / t.cu_keep[t.batch] < n) n = room / t.cu_keep[t.batch];
  if (seqs < n) n = seqs;
  if (kMaxGridY / ctx->dims.n_kv_heads < n) n = kMaxGridY / ctx->dims.n_kv_heads;   // (selection and pooling: a row of the grid per head)
  return n < 1 ? 1 : (n > kFlowLayers ? kFlowLayers : (int)n);
}

// n layers of one geometry and one row of budgets; *taken says how many of them were done (more than one only by score_flow.cu).
// after_own_compaction: the kernel before this call in `stream` is the compaction kernel of an
// earlier evict on the same context (the layers of dapq_evict_layers), which writes nothing that these layers read; the rotation
// then does not wait for it before it starts, and the first sweep's first keys are copied beside it too.
// route: the call's layers may take the pruned selection (NULL: they may not); layer: the first one's number.
dapq_status evict_impl(dapq_ctx* ctx, const Layer* y, int n, const SeqTable& t, float* scores_out, cudaStream_t s, bool after_own_compaction,
                       PruneRoute* route, int32_t layer, int* taken) {
  const CacheDev& cd = y[0].cd;
  float* scores = scores_out ? scores_out : ctx->scores;
  const int64_t score_stride = t.cu_prompt[t.batch], idx_stride = t.cu_keep[t.batch];
  UmmaPlan plan;
  QgPlan qplan;
  FlowPlan fplan;
  PrunePlan pplan;
  const int64_t lo_rows = ctx->q_rows_max;
  const int flags = ctx->shape.flags;
  cudaError_t e;
  dapq_status st = DAPQ_OK;
  CompactBatch cb = {};
  IndexOut idx = {};
  idx.heads_per_layer = ctx->dims.n_kv_heads;
  for (int l = 0; l < n; ++l) {
    idx.p[l] = y[l].idx_out ? y[l].idx_out : ctx->idx + (int64_t)l * ctx->dims.n_kv_heads * idx_stride;
    cb.l[l] = {y[l].cd, idx.p[l], y[l].k_out, y[l].v_out};
  }
  RopeBatch rb = one_rope(ctx, y[0].q_pre);
  auto with_references = [&](int layers) {
    // (with fp16 queries the rotation also leaves, in lse2, every query's logit against the first key of its
    // sequence: the reference that sweep 1 measures the row's other logits against)
    for (int l = 0; l < layers; ++l) {
      rb.q[l] = y[l].q_pre;
      rb.k[l] = (const __nv_bfloat16*)y[l].cd.k;
      rb.head_stride[l] = y[l].cd.k_head_stride;
      rb.row_stride[l] = y[l].cd.k_row_stride;
    }
    rb.n_layers = layers;
    rb.ref = ctx->lse2;
  };
  const bool qg = wants_umma(ctx) && !wants_lo(ctx) &&
                  qg_plan(ctx->q_rot, (flags & DAPQ_FLAG_Q_BF16) ? 0 : 1, cd, t, ctx->dims, ctx->n_sm, &qplan);
  const bool prune = qg && route && ctx->prune.sums && prune_plan(qplan, cd, t, ctx->dims, ctx->n_sm, &pplan);
  bool flow = false;
  *taken = 1;
  if (wants_flow(ctx) && !prune) {
    CacheDev cds[kFlowLayers];
    for (int l = 0; l < n; ++l) cds[l] = y[l].cd;
    while (n > 1 && !flow_plan(ctx->q_rot, cds, n, t, ctx->dims, ctx->n_sm, ctx->flow_chunks, &fplan)) --n;
    flow = n > 1;
  }
  if (flow) {
    // rotated queries rounded to fp16, K tiles converted to fp16 on their way to the MMAs; both sweeps of all n layers in one launch
    with_references(n);
    uint32_t* sync = ctx->sync[ctx->sync_turn ^= 1];
    rb.clear = sync;
    rb.n_clear = fplan.n_items + 1;
    e = launch_rope(ctx->shape.dtype, kRopeOutF16, 0, rb, ctx->q_rot, ctx->inv_freq, t, ctx->dims, after_own_compaction, s, &ctx->log);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "rope kernel");
    e = launch_score_flow(fplan, t, ctx->dims, ctx->part, ctx->flow_chunks, ctx->lse2, ctx->slots, scores, score_stride, sync, ctx->n_sm, ctx->status,
                          ctx->wait_limit, s, &ctx->log);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "tensor-core score kernel");
    *taken = n;
  } else if (qg) {
    // tensor-core scorer, a launch per sweep (DAPQ_FLAG_Q_BF16: queries rounded to bf16, no conversion)
    with_references(1);
    e = launch_rope(ctx->shape.dtype, qplan.q_is_f16 ? kRopeOutF16 : kRopeOutBf16, 0, rb, ctx->q_rot, ctx->inv_freq, t,
                    ctx->dims, after_own_compaction, s, &ctx->log);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "rope kernel");
    if (prune) {
      // nobody reads the scores: only those that can be among the K largest are computed
      const bool attempt = route->last_try < 0 || layer - route->last_try >= kPruneRetry;
      if (attempt) route->last_try = layer;
      e = launch_prune(pplan, cd, t, ctx->dims, ctx->prune, attempt ? -1 : route->at, route->at ^ 1, ctx->slots, scores, score_stride, ctx->status, ctx->wait_limit, s,
                       &ctx->log);
      if (e != cudaSuccess) return cuda_fail(ctx, e, "pruned score kernels");
      route->at ^= 1;
    } else {
      st = run_score_qg(ctx, qplan, t, nullptr, scores, score_stride, nullptr, true, s);
    }
  } else if (wants_umma(ctx) && wants_lo(ctx) && umma_plan(ctx->q_rot, 1, lo_rows, cd, t, ctx->dims, ctx->n_sm, &plan)) {
    // older tensor-core scorer: rotated queries as a bf16 pair hi + lo, the lo part added by a second MMA
    // pass in the sweeps that the flags name
    plan.lo_sweep1 = (flags & DAPQ_FLAG_Q_LO_SWEEP1) ? 1 : 0;
    plan.lo_sweep2 = (flags & DAPQ_FLAG_Q_LO_SWEEP2) ? 1 : 0;
    e = launch_rope(ctx->shape.dtype, kRopeOutSplitBf16, lo_rows * kHeadDim, rb, ctx->q_rot, ctx->inv_freq, t,
                    ctx->dims, after_own_compaction, s, &ctx->log);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "rope kernel");
    st = run_score_umma(ctx, plan, t, nullptr, scores, score_stride, nullptr, s);
  } else {
    // the rotated queries unrounded (fp32)
    e = launch_rope(ctx->shape.dtype, kRopeOutF32, 0, rb, ctx->q_rot, ctx->inv_freq, t, ctx->dims, after_own_compaction, s,
                    &ctx->log);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "rope kernel");
    st = run_score(ctx, DAPQ_F32, ctx->q_rot, cd, t, nullptr, scores, score_stride, nullptr, nullptr, true, s);
  }
  if (st != DAPQ_OK) return st;
  st = run_select(ctx, *taken, scores, score_stride, idx, idx_stride, t, s);
  if (st != DAPQ_OK) return st;
  e = launch_compact(ctx->shape.dtype, cb, *taken, idx_stride, t, ctx->dims.n_kv_heads, ctx->status, s, &ctx->log);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "compaction kernel");
  return DAPQ_OK;
}

}  // namespace

dapq_status dapq_evict(dapq_ctx* ctx, const void* q_pre, const dapq_cache_view* cache,
                       const int32_t* k_keep_host, void* k_out, void* v_out, int32_t* idx_out,
                       float* scores_out, void* stream) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  Layer y;
  SeqTable t;
  const dapq_status st = check_layer(ctx, q_pre, cache, k_keep_host, k_out, v_out, idx_out, &y, &t);
  if (st != DAPQ_OK) return st;
  DeviceGuard guard(ctx->device);
  int taken;
  return evict_impl(ctx, &y, 1, t, scores_out, (cudaStream_t)stream, false, nullptr, 0, &taken);
}

dapq_status dapq_evict_layers(dapq_ctx* ctx, int32_t n_layers, const void* const* q_pre,
                              const dapq_cache_view* caches, const int32_t* k_keep_host,
                              int64_t k_keep_layer_stride, void* const* k_out, void* const* v_out,
                              int32_t* const* idx_out, void* stream) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  if (n_layers < 0 || k_keep_layer_stride < 0) return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_evict_layers: negative count or stride");
  if (n_layers > 0 && (!q_pre || !caches || !k_keep_host || !k_out || !v_out))
    return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_evict_layers: NULL argument");
  DeviceGuard guard(ctx->device);
  PruneRoute route;
  auto check = [&](int32_t m, Layer* y, SeqTable* t) {
    return check_layer(ctx, q_pre[m], &caches[m], k_keep_host + (int64_t)m * k_keep_layer_stride, k_out[m], v_out[m], idx_out ? idx_out[m] : nullptr, y, t);
  };
  // what the launches before this one write: they have the layers before `l` and wait for the compaction before them, so nothing
  // older is still being written when this one's rotation begins
  LayerSpans before[kFlowLayers];
  int n_before = 0;
  for (int32_t l = 0; l < n_layers;) {
    Layer y[kFlowLayers];
    SeqTable t, other;
    dapq_status st = check(l, &y[0], &t);
    if (st != DAPQ_OK) return st;
    // The layers behind it that may share its launches: of the same geometry and budgets, as many as fit the workspace, none of them
    // touching another's outputs; in launches of equal size.  (A layer that is not in order says so when its own turn comes.)
    int n = 1;
    LayerSpans spans[kFlowLayers];
    spans[0] = LayerSpans(ctx, y[0], t);
    if (wants_flow(ctx)) {
      bool own_idx = false;
      for (int32_t m = l; m < n_layers && m < l + kFlowLayers; ++m) own_idx = own_idx || !idx_out || !idx_out[m];
      const int fit = layers_that_fit(ctx, t, own_idx), left = n_layers - l, launches = (left + fit - 1) / fit, most = (left + launches - 1) / launches;
      for (; n < most && check(l + n, &y[n], &other) == DAPQ_OK && memcmp(&other, &t, sizeof(t)) == 0; ++n) {
        spans[n] = LayerSpans(ctx, y[n], t);
        bool apart = true;
        for (int i = 0; i < n; ++i) apart = apart && spans[n].apart(spans[i]);
        if (!apart) break;
      }
    }
    bool beside = l > 0;
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n_before; ++j) beside = beside && !spans[i].reads(before[j]);
    int taken = 1;
    st = evict_impl(ctx, y, n, t, nullptr, (cudaStream_t)stream, beside, n_layers >= kPruneLeastLayers ? &route : nullptr, l, &taken);
    if (st != DAPQ_OK) return st;
    l += taken;
    n_before = taken;
    for (int i = 0; i < taken; ++i) before[i] = spans[i];
  }
  return DAPQ_OK;
}

namespace {

// First use of a staging set: its buffers (V only when some caller's V cannot be read in place) and events.
dapq_status ensure_stage(dapq_ctx* ctx, int set, bool need_v) {
  const dapq_shape& sh = ctx->shape;
  dapq_ctx::HostStage& hs = ctx->hs[set];
  const size_t row_bytes = (size_t)kHeadDim * ctx->elem_bytes;
  const size_t cache_bytes = (size_t)sh.n_kv_heads * (size_t)sh.max_total_rows * row_bytes;
  if (!ctx->copy_stream) {
    DAPQ_CUDA(ctx, cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking));
    DAPQ_CUDA(ctx, cudaEventCreateWithFlags(&ctx->fork, cudaEventDisableTiming));
  }
  if (!hs.k) {
    DAPQ_CUDA(ctx, cudaMalloc(&hs.q, (size_t)sh.max_batch * sh.n_q_heads * sh.n_pseudo * row_bytes));
    DAPQ_CUDA(ctx, cudaMalloc(&hs.k, cache_bytes));
    DAPQ_CUDA(ctx, cudaMalloc(&hs.ko, cache_bytes));
    DAPQ_CUDA(ctx, cudaMalloc(&hs.vo, cache_bytes));
    DAPQ_CUDA(ctx, cudaMalloc(&hs.idx, (size_t)sh.n_kv_heads * (size_t)sh.max_total_rows * sizeof(int32_t)));
    DAPQ_CUDA(ctx, cudaEventCreateWithFlags(&hs.in_done, cudaEventDisableTiming));
    DAPQ_CUDA(ctx, cudaEventCreateWithFlags(&hs.out_done, cudaEventDisableTiming));
  }
  if (need_v && !hs.v) DAPQ_CUDA(ctx, cudaMalloc(&hs.v, cache_bytes));
  return DAPQ_OK;
}

// Device address of the caller's V if the compaction kernel can read it in place (page-locked, addressable
// by the device, 16-byte geometry), else NULL.
const void* mapped_v(dapq_ctx* ctx, const CacheDev& hv) {
  cudaPointerAttributes pa;
  const int per16 = 16 / ctx->elem_bytes;
  if (hv.v_row_stride % per16 || hv.v_head_stride % per16) return nullptr;
  if (cudaPointerGetAttributes(&pa, hv.v) == cudaSuccess && pa.type == cudaMemoryTypeHost && pa.devicePointer &&
      aligned16(pa.devicePointer))
    return pa.devicePointer;
  cudaGetLastError();
  return nullptr;
}

}  // namespace

namespace {
dapq_status evict_layers_host_impl(dapq_ctx* ctx, int32_t n_layers, const void* const* q_pre_host,
                                   const dapq_cache_view* caches_host, const int32_t* k_keep_host,
                                   int64_t k_keep_layer_stride, void* const* k_out_host, void* const* v_out_host,
                                   int32_t* const* idx_out_host, void* stream);
}  // namespace

dapq_status dapq_evict_layers_host(dapq_ctx* ctx, int32_t n_layers, const void* const* q_pre_host,
                                   const dapq_cache_view* caches_host, const int32_t* k_keep_host,
                                   int64_t k_keep_layer_stride, void* const* k_out_host, void* const* v_out_host,
                                   int32_t* const* idx_out_host, void* stream) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  const dapq_status st = evict_layers_host_impl(ctx, n_layers, q_pre_host, caches_host, k_keep_host, k_keep_layer_stride,
                                                k_out_host, v_out_host, idx_out_host, stream);
  if (st != DAPQ_OK) {
    // a layer failed with copies of earlier layers possibly still in flight: the caller's buffers may be
    // reused as soon as this call returns, so wait for both streams first (their own errors do not matter now)
    DeviceGuard guard(ctx->device);
    if (ctx->copy_stream) cudaStreamSynchronize(ctx->copy_stream);
    cudaStreamSynchronize((cudaStream_t)stream);
    cudaGetLastError();
  }
  return st;
}

namespace {
dapq_status evict_layers_host_impl(dapq_ctx* ctx, int32_t n_layers, const void* const* q_pre_host,
                                   const dapq_cache_view* caches_host, const int32_t* k_keep_host,
                                   int64_t k_keep_layer_stride, void* const* k_out_host, void* const* v_out_host,
                                   int32_t* const* idx_out_host, void* stream) {
  if (n_layers < 0 || k_keep_layer_stride < 0) return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_evict_layers_host: negative count or stride");
  if (n_layers > 0 && (!q_pre_host || !caches_host || !k_keep_host || !k_out_host || !v_out_host))
    return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_evict_layers_host: NULL argument");
  DeviceGuard guard(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  const dapq_shape& sh = ctx->shape;
  const size_t eb = (size_t)ctx->elem_bytes, row_bytes = (size_t)kHeadDim * eb;
  bool forked = false;
  for (int32_t l = 0; l < n_layers; ++l) {
    const int32_t* keep = k_keep_host + (int64_t)l * k_keep_layer_stride;
    if (!q_pre_host[l] || !k_out_host[l] || !v_out_host[l]) return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_evict_layers_host: NULL layer pointer");
    CacheDev hv;
    dapq_status st = check_view(ctx, &caches_host[l], true, true, &hv);
    if (st != DAPQ_OK) return st;
    SeqTable t;
    st = build_table(ctx, caches_host[l].batch, caches_host[l].cu_rows_host, caches_host[l].prompt_len_host, nullptr, keep,
                     nullptr, &t);
    if (st != DAPQ_OK) return st;
    const void* v_in_place = mapped_v(ctx, hv);
    const int set = l & 1;
    st = ensure_stage(ctx, set, v_in_place == nullptr);
    if (st != DAPQ_OK) return st;
    dapq_ctx::HostStage& hs = ctx->hs[set];
    cudaStream_t cs = ctx->copy_stream;
    if (!forked) {                                       // the copies start behind the work already in `stream`
      DAPQ_CUDA(ctx, cudaEventRecord(ctx->fork, s));
      DAPQ_CUDA(ctx, cudaStreamWaitEvent(cs, ctx->fork, 0));
      forked = true;
    }
    if (l >= 2) DAPQ_CUDA(ctx, cudaStreamWaitEvent(cs, hs.out_done, 0));   // the set's last user is done with it
    // ---- inputs: q and the used row range [cu_rows[0], cu_rows[B]) of every head of K, packed from row 0
    const int64_t row0 = t.cu_rows[0], n_rows = t.cu_rows[t.batch] - row0;
    DAPQ_CUDA(ctx, cudaMemcpyAsync(hs.q, q_pre_host[l], (size_t)t.batch * sh.n_q_heads * sh.n_pseudo * row_bytes,
                                   cudaMemcpyHostToDevice, cs));
    for (int h = 0; h < sh.n_kv_heads; ++h) {
      const char* ks = (const char*)hv.k + ((size_t)h * hv.k_head_stride + (size_t)row0 * hv.k_row_stride) * eb;
      DAPQ_CUDA(ctx, cudaMemcpy2DAsync((char*)hs.k + (size_t)h * n_rows * row_bytes, row_bytes, ks,
                                       (size_t)hv.k_row_stride * eb, row_bytes, (size_t)n_rows, cudaMemcpyHostToDevice, cs));
      if (v_in_place) continue;
      const char* vs = (const char*)hv.v + ((size_t)h * hv.v_head_stride + (size_t)row0 * hv.v_row_stride) * eb;
      DAPQ_CUDA(ctx, cudaMemcpy2DAsync((char*)hs.v + (size_t)h * n_rows * row_bytes, row_bytes, vs,
                                       (size_t)hv.v_row_stride * eb, row_bytes, (size_t)n_rows, cudaMemcpyHostToDevice, cs));
    }
    DAPQ_CUDA(ctx, cudaEventRecord(hs.in_done, cs));
    // ---- the layer itself, on the caller's stream
    int32_t cu_local[kMaxBatch + 1];
    for (int b = 0; b <= t.batch; ++b) cu_local[b] = (int32_t)(t.cu_rows[b] - row0);
    dapq_cache_view dv;
    memset(&dv, 0, sizeof(dv));
    dv.k = hs.k;
    dv.k_head_stride = n_rows * kHeadDim;
    dv.k_row_stride = kHeadDim;
    if (v_in_place) {
      dv.v = (const char*)v_in_place + (size_t)row0 * hv.v_row_stride * eb;   // row 0 of the view = row cu_rows[0] of the caller's
      dv.v_head_stride = hv.v_head_stride;
      dv.v_row_stride = hv.v_row_stride;
    } else {
      dv.v = hs.v;
      dv.v_head_stride = n_rows * kHeadDim;
      dv.v_row_stride = kHeadDim;
    }
    dv.cu_rows_host = cu_local;
    dv.prompt_len_host = caches_host[l].prompt_len_host;
    dv.batch = t.batch;
    DAPQ_CUDA(ctx, cudaStreamWaitEvent(s, hs.in_done, 0));
    st = dapq_evict(ctx, hs.q, &dv, keep, hs.ko, hs.vo, hs.idx, nullptr, stream);
    if (st != DAPQ_OK) return st;
    // ---- results
    const size_t kt = (size_t)t.cu_keep[t.batch];
    DAPQ_CUDA(ctx, cudaMemcpyAsync(k_out_host[l], hs.ko, (size_t)sh.n_kv_heads * kt * row_bytes, cudaMemcpyDeviceToHost, s));
    DAPQ_CUDA(ctx, cudaMemcpyAsync(v_out_host[l], hs.vo, (size_t)sh.n_kv_heads * kt * row_bytes, cudaMemcpyDeviceToHost, s));
    if (idx_out_host && idx_out_host[l])
      DAPQ_CUDA(ctx, cudaMemcpyAsync(idx_out_host[l], hs.idx, (size_t)sh.n_kv_heads * kt * sizeof(int32_t),
                                     cudaMemcpyDeviceToHost, s));
    DAPQ_CUDA(ctx, cudaEventRecord(hs.out_done, s));
  }
  DAPQ_CUDA(ctx, cudaStreamSynchronize(s));
  return DAPQ_OK;
}
}  // namespace

dapq_status dapq_evict_host(dapq_ctx* ctx, const void* q_pre_host, const dapq_cache_view* cache_host,
                            const int32_t* k_keep_host, void* k_out_host, void* v_out_host,
                            int32_t* idx_out_host, void* stream) {
  if (!ctx) return DAPQ_ERR_INVALID_ARG;
  if (!q_pre_host || !cache_host || !k_keep_host || !k_out_host || !v_out_host)
    return fail(ctx, DAPQ_ERR_INVALID_ARG, "dapq_evict_host: NULL argument");
  return dapq_evict_layers_host(ctx, 1, &q_pre_host, cache_host, k_keep_host, 0, &k_out_host, &v_out_host, &idx_out_host, stream);
}

}  // extern "C"
