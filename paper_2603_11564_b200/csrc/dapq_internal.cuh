// Internal declarations shared by the translation units of libdapq (not installed).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "dapq.h"

namespace dapq {

constexpr int kHeadDim = DAPQ_HEAD_DIM;      // d
constexpr int kMaxBatch = DAPQ_MAX_BATCH;
constexpr int kMaxPseudo = DAPQ_MAX_PSEUDO;
constexpr int kChunkKeys = 512;              // most prompt keys per work chunk of the CUDA-core score sweeps

// Per-call sequence geometry, passed by value to the kernels (host arrays never have to
// be copied to the device, so a call adds no copy nodes to a stream).
struct SeqTable {
  int32_t batch;
  int32_t cu_rows[kMaxBatch + 1];   // first cache row of sequence b
  int32_t cu_prompt[kMaxBatch + 1]; // first score column of sequence b
  int32_t cu_keep[kMaxBatch + 1];   // first output row of sequence b (K_b clamped to L_b)
  int32_t prompt_len[kMaxBatch];    // L_b
  int32_t pos_start[kMaxBatch];     // position of pseudo query 0
};

// How the score sweeps cut the sequences into work chunks (one CTA per chunk and KV head).
//   CUDA-core path:   chunks of chunk_tiles prompt KEYS (64 .. kChunkKeys), then one chunk with the N
//                     synthetic rows;
//   tensor-core path: chunks of chunk_tiles whole K tiles (the tile size is the sweep's).
struct ChunkTable {
  int32_t chunk_tiles;
  int32_t n_chunks;
  int32_t cu_chunk[kMaxBatch + 1];  // first chunk of sequence b
};
constexpr int kUmmaMaxChunks = 256;  // the tensor-core planner never makes more chunks than max_batch + this

struct CacheDev {
  const void* k;
  const void* v;
  int64_t k_head_stride, k_row_stride, v_head_stride, v_row_stride;  // elements
};

struct Dims {
  int32_t n_q_heads, n_kv_heads, group, n_pseudo;
  float scale_log2e;                // softmax scale * log2(e): logits are kept in base 2
  int32_t rope_interleaved = 0;     // RoPE pairs are (2c, 2c + 1) instead of (c, c + d/2)
};

// Device status word bits (set by kernels, read by dapq_poll_status).
enum : int { kStatusTimeout = 1, kStatusBadIndex = 2, kStatusSmemAlign = 4 };

// Output formats of the rotation kernel.
enum : int { kRopeOutBf16 = DAPQ_BF16, kRopeOutF32 = DAPQ_F32, kRopeOutSplitBf16 = 2, kRopeOutF16 = 3 };

__device__ __forceinline__ int find_segment(const int32_t* cu, int n, int x) {
  // largest b in [0, n) with cu[b] <= x
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (cu[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Kernel kinds, for launch accounting and the optional per-kernel event timing.
enum KernelKind : int { kKindRope = 0, kKindSweep1, kKindLseMerge, kKindSweep2, kKindTopk, kKindCompact, kKindPool,
                        kKindRecall, kKindSlotSum, kKindCount };

// Counts launches and, while profiling is on, brackets every launch with CUDA events on
// the launching stream (implemented in api.cu; events come from a host-side pool).
struct LaunchLog {
  int64_t n_launch = 0;
  bool profiling = false;
  void* impl = nullptr;
  void begin(int kind, cudaStream_t s);
  void end(cudaStream_t s);
};

// ---- programmatic dependent launch --------------------------------------------------------
// Every kernel of the eviction path is launched with programmatic stream serialization and
// waits, before its first access to global memory, until the kernel before it has completed
// and its writes are visible (pdl_wait): its launch is then prepared, and its CTAs' set-up done,
// while the predecessor still runs.  The short kernels that precede a long one (rotation,
// behind its own wait, and selection) also signal early that the next kernel may be scheduled (pdl_trigger); the
// second sweeps do not: their successors' CTAs would only sit on the SMs the next sweep needs (measured:
// slower); the first sweeps do where a CTA's run is short (see there).  The compaction signals at its start too: in dapq_evict_layers the next layer's
// rotation, which touches nothing the compaction or the selection before it use, runs beside
// them and waits at its END, so that the kernels after it stay ordered behind the compaction.
// Both instructions are no-ops for a kernel launched the ordinary way.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch with programmatic stream serialization (and a cluster of cluster_x CTAs if > 1).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster_x,
                       Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[n].val.programmaticStreamSerializationAllowed = 1;
  ++n;
  if (cluster_x > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster_x;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ---- launchers (each returns the cudaError_t of its launch) -------------------------------
// Layers that one launch of the rotation, the scorer, the selection and the compaction may cover (dapq_evict_layers).
constexpr int kFlowLayers = 8;
// The rotation of the layers' queries q (element type `dtype`) to q_rot, [layers][B, H_q, N, d] as `out_mode` says: fp16 (times
// scale * log2 e, for the tensor-core scorer), bf16, fp32 (unrounded, for the CUDA-core scorer) or a bf16 pair hi + lo with
// lo = bf16(q - hi) stored `lo_offset` elements after hi.  Only the fp16 mode takes more than one layer.
// ref (fp16 mode only, may be NULL): where to write, per rotated query, its base-2 logit against the first key of its sequence in
// the layer's bf16 key cache (see rope.cu).  clear: words set to 0.
template <int kLayers>
struct RopeLayers {
  const void* q[kLayers];
  const __nv_bfloat16* k[kLayers];
  int64_t head_stride[kLayers], row_stride[kLayers];           // of k, elements
  int32_t n_layers, group;
  float* ref;                                                  // [layers][B, H_q, N]
  uint32_t* clear;
  int32_t n_clear;
};
using RopeBatch = RopeLayers<kFlowLayers>;
cudaError_t launch_rope(int dtype, int out_mode, int64_t lo_offset, const RopeBatch& rb, void* q_rot, const double* inv_freq_dev,
                        const SeqTable& t, const Dims& dm, bool late_wait, cudaStream_t s, LaunchLog* log);

// Generic CUDA-core scorer (any N <= 128, both dtypes).
//   part  : [n_chunks, H_q, N] float2 (running max, sum) in base-2 logits, room for max_chunks
//           chunks (at least the count at kChunkKeys keys per chunk; more lets small inputs
//           be cut finer so that they fill the n_sm SMs)
//   lse2  : [B, H_q, N] base-2 log-sum-exp
cudaError_t launch_score_fma(int dtype, int q_dtype, const void* q_rot, const CacheDev& cv, const SeqTable& t,
                             const Dims& dm, const float* lse_in, float2* part, int64_t max_chunks, int n_sm,
                             float* lse2, float* scores, int64_t score_stride, float* lse_out, float* syn_mass,
                             cudaStream_t s, LaunchLog* log);

// Makes the device code of every CUDA-core score kernel resident on the current device (no launch).
cudaError_t score_fma_preload();

// Tensor-core scorer (bf16 caches).  umma_plan encodes the TMA descriptors and cuts the work;
// it returns false when the view cannot be described to TMA (the caller then takes the
// CUDA-core path).  q_hi: [B*H_q*N, d] bf16; with has_lo the low-order parts follow
// lo_row_offset rows later in the same allocation.
struct UmmaPlan {
  CUtensorMap tm_k1, tm_k2, tm_q;   // K for sweep 1 / sweep 2 (different boxes), the query operand
  ChunkTable ct1, ct2;              // work cut of sweep 1 (192-key tiles over L_b + N) / sweep 2 (128-key tiles over L_b)
  int32_t has_lo;                   // the low-order parts exist in memory
  int32_t lo_sweep1, lo_sweep2;     // ... and which sweep adds them (a second MMA pass)
  int64_t lo_row_offset;
};
bool umma_plan(const void* q_hi, int has_lo, int64_t lo_row_offset, const CacheDev& cv, const SeqTable& t,
               const Dims& dm, int n_sm, UmmaPlan* plan);
int64_t umma_part_elems(int max_batch, int n_q_heads, int n_kv_heads, int n_pseudo);
cudaError_t launch_score_umma(const UmmaPlan& plan, const SeqTable& t, const Dims& dm, const float* lse_in,
                              float2* part, float* scores, int64_t score_stride, float* lse_out,
                              int* status, long long wait_limit, cudaStream_t s, LaunchLog* log);

// Pieces shared by the two tensor-core scorers (defined in score_qg.cu): the TMA descriptor of a
// 16-bit [.., rows, 128] tensor (boxes of 64 channels x box_rows rows, 128-byte swizzle), and the cut of
// the sequences' keys into chunks of whole tiles with ctas_per_chunk CTAs working on every chunk.
bool encode_tile_map(CUtensorMap* map, const void* base, bool f16, int rank, const uint64_t* dims,
                     const uint64_t* strides_bytes, int box_rows);
// fp32 tensor [H, rows, 128], boxes of box_cols (up to 32) channels x box_rows rows, 128-byte swizzle.
bool encode_rows_map_f32(CUtensorMap* map, const void* base, const uint64_t* dims, const uint64_t* strides_bytes, int box_cols,
                         int box_rows);
bool plan_chunks(const SeqTable& t, int extra_keys, int tile_keys, int ctas_per_chunk, int n_sm, ChunkTable* ct,
                 double cta_cost = 3.0);

// Tensor-core scorer with one query group per CTA (score_qg.cu).  q: [B*H_q*N, d], fp16 (the K tiles
// are then converted to fp16 in shared memory) or bf16.  qg_plan returns false when the view cannot be
// described to TMA.  With more than one query group per KV head the sweeps write one score slot per
// group into `slots` ([n_qgroups, H_kv, score_stride]) and a last kernel sums them into `scores`.
struct QgPlan {
  CUtensorMap tm_k1, tm_k2, tm_q;
  ChunkTable ct1, ct2;
  int32_t n_qgroups, rows_g, n_stages1, n_stages2, q_is_f16;
  int32_t n_qgroups2, rows_g2, wide2;     // sweep 2's own cut of the query rows (groups of up to 512 rows when wide2)
};
int qg_groups(const Dims& dm);
bool qg_plan(const void* q, int q_is_f16, const CacheDev& cv, const SeqTable& t, const Dims& dm, int n_sm, QgPlan* plan);
// ref: with fp16 queries, the [B, H_q, N] reference logits that the rotation kernel wrote beside them.
// after_own_kernel: the kernel before these in the stream is this library's rotation kernel (which waits for
// whatever precedes it), so the sweeps may copy the keys before their own wait for it.
cudaError_t launch_score_qg(const QgPlan& plan, const SeqTable& t, const Dims& dm, const float* lse_in, float2* part,
                            float* slots, float* scores, int64_t score_stride, float* lse_out, const float* ref, int* status,
                            long long wait_limit, bool after_own_kernel, cudaStream_t s, LaunchLog* log);

// The same scorer over several layers of the same geometry in one launch (score_flow.cu), for fp16 queries of the rotation
// ([layers][B, H_q, N, d]).  flow_plan returns false when a view cannot be described to TMA or the partials do not fit
// max_chunks rows of [H_kv][flow_rows_pad].  part: that many rows, and as many of floats behind them; ref: [layers][B, H_q, N];
// scores: [layers][H_kv][score_stride]; slots (more than one query group): n_qgroups arrays like scores; sync: 1 + n_items
// words, cleared.
struct FlowPlan {
  CUtensorMap tm_k[kFlowLayers], tm_q;
  ChunkTable ct;                          // runs of key pairs
  int32_t n_layers, n_qgroups, rows_g, rows_pad, two;
  int32_t n_units, n_items, block;
};
int flow_rows_pad(const Dims& dm);
bool flow_plan(const void* q, const CacheDev* cv, int n_layers, const SeqTable& t, const Dims& dm, int n_sm, int64_t max_chunks, FlowPlan* plan);
cudaError_t launch_score_flow(const FlowPlan& plan, const SeqTable& t, const Dims& dm, float2* part, int64_t max_chunks, const float* ref, float* slots,
                              float* scores, int64_t score_stride, uint32_t* sync, int n_sm, int* status, long long wait_limit, cudaStream_t s,
                              LaunchLog* log);

// Sum of n_slots score arrays of `count` values that lie one behind the other, in slot order.
cudaError_t launch_slots_sum(const float* slots, int n_slots, float* scores, int64_t count, cudaStream_t s, LaunchLog* log);

// Tensor-core scorer with unrounded operands (score_split.cu).  split_plan returns false when the view cannot be
// described to TMA; split_groups: score slots that sweep 2 needs (one per 128 query rows of a KV head).
struct SplitPlan {
  CUtensorMap tm_k;
  ChunkTable ct1, ct2;
  int32_t key_parts;                      // 3: fp32 keys, 1: bf16 keys
  int32_t R, n_qgroups;                   // query rows per sub-group (16 .. 64), sub-groups of a KV head
  int32_t n_sub2, n_qgroups2;             // sub-groups per CTA in sweep 2, CTAs per chunk there
  int32_t n_ring1, n_ring2, n_stage1, n_stage2, smem1, smem2;
};
int split_groups(const Dims& dm);
bool split_plan(int dtype, const CacheDev& cv, const SeqTable& t, const Dims& dm, int n_sm, SplitPlan* plan);
cudaError_t launch_score_split(const SplitPlan& plan, int q_dtype, const void* q, const SeqTable& t, const Dims& dm,
                               const float* lse_in, float2* part, float* slots, float* scores, int64_t score_stride, float* lse_out,
                               int* status, long long wait_limit, bool after_own_kernel, cudaStream_t s, LaunchLog* log);

// ---- the pruned selection: the layers of dapq_evict_layers (score_prune.cu) ----------------------------------
constexpr int kPruneSums = 4;              // partial sums per key
constexpr double kPruneLeastPairs = 2e8;   // query-key pairs of a layer below which the full sweeps are as fast (score_prune.cu)
constexpr int kPruneLeastLen = 65536;      // shortest prompt
constexpr int kPruneLeastLayers = 8;       // of a call: the first has to find out whether it pays, and loses a fifth if not
constexpr int kPruneRetry = 16;            // layers after which a call that went back to the full sweeps tries again
// histogram of a head's lower bounds, its candidate count, the largest magnitude of its rows' log-sum-exps (bits of a float)
constexpr int kPruneBins = 2048, kPruneHist = kPruneBins + 4;
struct PrunePlan {
  QgPlan qg;                               // the full scorer's plan; sweep 2's cut serves the candidates
  CUtensorMap tm_s;                        // every 16th key
  ChunkTable ct_s, ct_m, ct_g;             // chunks of the sample's sweep and of the one-pass sweep; CTAs per candidate list
  int32_t n_stages_m, per_cta;
  float most;                              // candidates of a head, as a share of its prompt, up to which a layer gains
};
struct PruneBuffers {                      // device workspace
  float2 *part_s, *part_m;                 // umma_part_elems each
  const float* ref;                        // [B, H_q, N] the rotation's reference logits
  float* est;                              // [B, H_q, N] the estimates
  float* sums;                             // kPruneSums * (H_kv * max_total_rows rounded up to 4)
  int32_t* cand;                           // [H_kv][max_total_rows]
  uint32_t* hist;                          // [max_batch, H_kv][kPruneHist]
  float2* route;                           // [2] what decides a layer's route, and the next one's
};
bool prune_available();
bool prune_plan(const QgPlan& qg, const CacheDev& cv, const SeqTable& t, const Dims& dm, int n_sm, PrunePlan* plan);
// route_at, route_next: which of buf.route holds this layer's route (-1: pruned, whatever the last one found) and which
// receives the next one's.
// scores: [H_kv][score_stride], those of keys that cannot be selected are negative; slots as for launch_score_qg.
cudaError_t launch_prune(const PrunePlan& plan, const CacheDev& cv, const SeqTable& t, const Dims& dm, const PruneBuffers& buf,
                         int route_at, int route_next, float* slots, float* scores, int64_t score_stride, int* status, long long wait_limit,
                         cudaStream_t s, LaunchLog* log);
// n_heads: heads of all layers, heads_per_layer of them to each of the index arrays.
struct IndexOut { int32_t* p[kFlowLayers]; int32_t heads_per_layer; };
cudaError_t launch_topk(const float* scores, int64_t score_stride, const IndexOut& idx, int64_t idx_stride,
                        const SeqTable& t, int n_heads, cudaStream_t s, LaunchLog* log);

// pooled[kvh, j] = max / mean of scores[kvh, j - kernel/2 .. j + kernel/2] within each sequence.
cudaError_t launch_pool(const float* scores, float* pooled, int64_t stride, const SeqTable& t, int n_kv_heads,
                        int kernel, int mode, cudaStream_t s, LaunchLog* log);

// recall[b, kvh] = |gold ∩ pred| / |gold| for two ascending index lists per (sequence, KV head).
cudaError_t launch_recall(const int32_t* gold, const int32_t* pred, int64_t idx_stride, const SeqTable& t,
                          int n_kv_heads, float* recall, cudaStream_t s, LaunchLog* log);

struct CompactLayer { CacheDev cv; const int32_t* idx; void *k_out, *v_out; };
struct CompactBatch { CompactLayer l[kFlowLayers]; };
cudaError_t launch_compact(int dtype, const CompactBatch& cb, int n_layers, int64_t idx_stride, const SeqTable& t, int n_kv_heads, int* status,
                           cudaStream_t s, LaunchLog* log);

}  // namespace dapq
