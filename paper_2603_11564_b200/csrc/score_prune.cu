// The retained set without the scores (Section 4.2, Eq. 5 needs the K largest S(j), not all of them): dapq_evict
// and its multi-layer and host forms, when no scores are asked for.  The same set as from the two full sweeps, for less
// than two thirds of their work on long prompts.
//
//   1. sample      sweep 1 over every 16th key: an estimate r_i of each query row's log-sum-exp;
//   2. one pass    over all keys with r_i in place of the log-sum-exp: e_ij = 2^(s_ij - r_i) is added to the sum of its
//                  row, Z_i, and to that of its key, E_g(j), in up to four sums g of some 64 to 256 rows each.  The row sums
//                  are what sweep 1 yields: log-sum-exp_i = r_i + log2 Z_i, in fp32 as there;
//   3. bounds      S(j) = sum_i e_ij / Z_i, so  sum_g E_g(j) / max_g Z  <=  S(j)  <=  sum_g E_g(j) / min_g Z.  With T the K-th
//                  largest lower bound (at least K keys score T or more), a key whose upper bound is below T is not
//                  among the K largest: what remains are the candidates;
//   4. candidates  sweep 2 over them, with the log-sum-exp from step 2: the scores that the full sweep 2 gives them
//                  (skipped, per KV head, when there are exactly K);
//   5. selection   as ever, on an array that holds -1 for all other keys.
// Nothing depends on how good the estimate is but the number of candidates.  A row sum that leaves the float range
// is done over again by itself (careful_row).
//
// Measured on B200, a layer with the two full sweeps -> here, on prompts whose relevant passages stand out (candidates = K):
// 128 k, 8 KV heads x 1024 query rows 690 -> 460 us; 128 k, 4 x 448 rows 182 -> 139; 32 k, 8 x 256 rows 64 -> 65 (four more
// launches, the sample and the bounds at their start-up times).  On N(0, 1) keys, which stand out by nothing, a fifth to a
// quarter of them are candidates at 128 k (704 -> 605 us with outlier channels, 188 -> 162), and a sample of 2 k keys is
// the least that bounds anything: 8 prompts of 32 k 270 -> 249 (logits of standard deviation 2: 296 -> 290; 3: 294 -> 341, the
// worst seen), 12 of 16 k 201 -> 237, 40 of 8 k 365 -> 446 (365 -> 290 where passages stand out), and 8 of 4 to 32 k that
// keep a tenth 206 -> 285.  Hence the conditions in prune_plan: prompts long enough for the sample, query-key pairs enough
// for the launches, and a budget of at most a sixteenth of a prompt (an eighth of a long one), so that the threshold lies
// in the tail of the scores.
#include "score_qg_sweep1.cuh"
#include "score_qg_sweep2.cuh"

namespace dapq {
namespace {

using namespace qg;

constexpr int kSampleStride = 16, kSamplePhase = 7;
constexpr float kLog2Sample = 4.f;

// ---- step 3: two kernels over tiles of kBoundTile keys of a head -------------------------------------------
constexpr int kBoundThreads = 512, kBoundKeys = 8, kBoundTile = kBoundThreads * kBoundKeys;

struct BoundArgs {
  const float2* part;                      // [chunks, H_kv, rows_pad] row sums of the one-pass sweep
  const float* ref;                        // [B, H_kv, rows_total] the estimates it worked with
  int32_t rows_total, rows_pad, rows_g;    // query rows per KV head, of a CTA of that sweep
  int32_t n_sums, per_cta;                 // partial sums per key in all, and of one CTA
  float* sums;                             // the sums, sum_stride (a multiple of 4) floats apart; the first is replaced by the upper bounds
  int64_t sum_stride, score_stride;
  uint32_t* hist;
  int32_t* cand;
  float* scores;                           // preset: n_slots arrays [H_kv][score_stride]
  int64_t slot_stride;
  int32_t n_slots;
};

// Bins of the lower bounds: 32 per octave from 2^-52 to 2^12, what lies outside goes to the end bins.
constexpr uint32_t kBinBase = (127u - 52u) << 5;
__device__ __forceinline__ int bound_bin(float lo) {
  const int x = (int)(__float_as_uint(lo) >> 18) - (int)kBinBase;
  return lo < 3e38f ? min(max(x, 0), kPruneBins - 1) : 0;       // (a sum beyond the float range bounds nothing from below)
}

// Scores between the 16-byte boundary before a head's first score and that score.
__device__ __forceinline__ int head_lead(const SeqTable& t, const BoundArgs& a, int b, int kvh) {
  return (int)(((int64_t)kvh * a.score_stride + t.cu_prompt[b]) & 3);
}

// The kBoundKeys positions of this thread begin at a 16-byte boundary of the head's arrays, whatever the head's offset.
struct BoundSpan {
  int base, v0, nv;
  int64_t at;                              // of position 0, in the arrays
  __device__ __forceinline__ BoundSpan(const SeqTable& t, const BoundArgs& a, int b, int kvh, int tile) {
    at = (int64_t)kvh * a.score_stride + t.cu_prompt[b];
    base = tile * kBoundTile + (int)threadIdx.x * kBoundKeys - head_lead(t, a, b, kvh);
    v0 = max(0, -base);
    nv = max(0, min(kBoundKeys, t.prompt_len[b] - base));
  }
  __device__ __forceinline__ bool whole() const { return v0 == 0 && nv == kBoundKeys; }
  __device__ __forceinline__ void load(const float* p, float (&v)[kBoundKeys]) const {
    p += at + base;
    if (whole()) {
      const float4 x = *reinterpret_cast<const float4*>(p), y = *reinterpret_cast<const float4*>(p + 4);
      v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
    } else {
#pragma unroll
      for (int e = 0; e < kBoundKeys; ++e) v[e] = (e >= v0 && e < nv) ? p[e] : 0.f;
    }
  }
  __device__ __forceinline__ void store(float* p, const float (&v)[kBoundKeys], bool vec) const {
    p += at + base;
    if (vec && whole()) {
      *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
    } else {
#pragma unroll
      for (int e = 0; e < kBoundKeys; ++e)
        if (e >= v0 && e < nv) p[e] = v[e];
    }
  }
};

// Upper bounds in place of the first sum, histogram of the lower bounds.
__global__ void __launch_bounds__(kBoundThreads)
bound_hist_kernel(const __grid_constant__ SeqTable t, const __grid_constant__ ChunkTable ct, const BoundArgs a) {
  __shared__ uint32_t hist[kPruneBins];
  __shared__ uint32_t f_min[kPruneSums], f_max[kPruneSums], lse_max;
  const int tid = threadIdx.x, kvh = blockIdx.y, b = blockIdx.z, H = gridDim.y;
  pdl_trigger();
  if ((int)blockIdx.x * kBoundTile - head_lead(t, a, b, kvh) >= t.prompt_len[b]) return;
  for (int x = tid; x < kPruneBins; x += kBoundThreads) hist[x] = 0u;
  if (tid < kPruneSums) { f_min[tid] = 0x7f800000u; f_max[tid] = 0u; }
  if (tid == 0) lse_max = 0u;
  __syncthreads();
  pdl_wait();
  const BoundSpan sp(t, a, b, kvh, blockIdx.x);
  float v[kPruneSums][kBoundKeys];
#pragma unroll
  for (int g = 0; g < kPruneSums; ++g)
    if (g < a.n_sums) sp.load(a.sums + g * a.sum_stride, v[g]);
  // factors 2^(estimate - log-sum-exp) of the query rows: their range over the rows behind each sum
  for (int row = tid; row < a.rows_total; row += kBoundThreads) {
    const int n = ct.cu_chunk[b + 1] - ct.cu_chunk[b];
    const float2* p = a.part + ((int64_t)ct.cu_chunk[b] * H + kvh) * a.rows_pad + row;
    float m = -CUDART_INF_F, z = 0.f;
    for (int c0 = 0; c0 < n; c0 += 8) {
      float2 q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = c0 + u < n ? __ldg(p + (int64_t)(c0 + u) * H * a.rows_pad) : make_float2(-CUDART_INF_F, 0.f);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float mm = fmaxf(m, q[u].x);
        if (c0 + u < n) z = z * exp2f(m - mm) + q[u].y * exp2f(q[u].x - mm);
        m = mm;
      }
    }
    const float lse = m + log2f(z), f = exp2f(a.ref[((int64_t)b * H + kvh) * a.rows_total + row] - lse);
    if (blockIdx.x == 0) atomicMax(&lse_max, __float_as_uint(fabsf(lse)));   // (NaN above infinity above all numbers)
    const int qg = row / a.rows_g, rr = row - qg * a.rows_g;
    const int nch = (min(a.rows_g, a.rows_total - qg * a.rows_g) + 15) >> 4;
    int eg = 3;
    while (eg > 0 && (rr >> 4) < (eg * nch) / 4) --eg;          // the epilogue group that held the row's column
    const int g = qg * a.per_cta + (a.per_cta == 4 ? eg : (a.per_cta == 2 ? eg >> 1 : 0));
    // (positive floats order like their bit patterns; a factor below the normal range keeps no bits that a bound could
    // rely on: at least 0 and at most the range's lower end)
    constexpr float kTiny = 0x1p-126f;
    atomicMin(&f_min[g], __float_as_uint(f < kTiny ? 0.f : f));
    atomicMax(&f_max[g], __float_as_uint(f < kTiny ? kTiny : f));
  }
  __syncthreads();
  float hi[kBoundKeys], lo[kBoundKeys];
#pragma unroll
  for (int e = 0; e < kBoundKeys; ++e) hi[e] = lo[e] = 0.f;
#pragma unroll
  for (int g = 0; g < kPruneSums; ++g) {
    if (g < a.n_sums) {
      const float mn = __uint_as_float(f_min[g]), mx = __uint_as_float(f_max[g]);
#pragma unroll
      for (int e = 0; e < kBoundKeys; ++e) {
        lo[e] = fmaf(v[g][e], mn, lo[e]);
        hi[e] = fmaf(v[g][e], mx, hi[e]);
      }
    }
  }
#pragma unroll
  for (int e = 0; e < kBoundKeys; ++e)
    if (e >= sp.v0 && e < sp.nv) atomicAdd(&hist[bound_bin(lo[e])], 1u);
  sp.store(a.sums, hi, true);
  __syncthreads();
  uint32_t* out = a.hist + (int64_t)(b * H + kvh) * kPruneHist;
  for (int x = tid; x < kPruneBins; x += kBoundThreads)
    if (hist[x]) atomicAdd(out + x, hist[x]);
  if (tid == 0 && blockIdx.x == 0) out[kPruneBins + 1] = lse_max;
}

// The candidates: keys whose upper bound reaches the lower edge of the bin that holds the K-th largest lower bound.
// Lists them and presets the scores (+1 for them, -1 for the others).
__global__ void __launch_bounds__(kBoundThreads)
bound_list_kernel(const __grid_constant__ SeqTable t, const BoundArgs a) {
  constexpr int kPer = kPruneBins / kBoundThreads;
  static_assert(kPer == 4, "a thread owns four bins");
  __shared__ uint32_t warp_sum[2][kBoundThreads / 32];
  __shared__ float edge;
  __shared__ uint32_t list_at;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, kvh = blockIdx.y, b = blockIdx.z, H = gridDim.y;
  pdl_trigger();
  if ((int)blockIdx.x * kBoundTile - head_lead(t, a, b, kvh) >= t.prompt_len[b]) return;
  pdl_wait();
  const BoundSpan sp(t, a, b, kvh, blockIdx.x);
  float hi[kBoundKeys];
  sp.load(a.sums, hi);
  uint32_t* hist = a.hist + (int64_t)(b * H + kvh) * kPruneHist;
  const int top = kPruneBins - 1 - kPer * tid;                   // this thread's highest bin
  const uint4 h4 = *reinterpret_cast<const uint4*>(hist + top - 3);
  const uint32_t h[4] = {h4.w, h4.z, h4.y, h4.x};
  const float lse_max = __uint_as_float(hist[kPruneBins + 1]);
  // inclusive prefix over the block, in thread order (every warp sums the totals of the warps before it by itself)
  auto prefix = [&](uint32_t mine, uint32_t* sums, uint32_t* total) {
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) sums[warp] = incl;
    __syncthreads();
    const uint32_t ws = lane < kBoundThreads / 32 ? sums[lane] : 0u;
    uint32_t before = lane < warp ? ws : 0u, all = ws;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      before += __shfl_xor_sync(0xffffffffu, before, o);
      all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    *total = all;
    return incl + before;
  };
  const uint32_t K = (uint32_t)(t.cu_keep[b + 1] - t.cu_keep[b]), mine = h[0] + h[1] + h[2] + h[3];
  uint32_t total;
  const uint32_t incl = prefix(mine, warp_sum[0], &total);
  if (incl >= K && incl - mine < K) {                            // exactly one thread
    uint32_t c = incl - mine;
    int bin = top;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      c += h[e];
      if (c >= K) break;
      --bin;
    }
    // with a margin for the roundings of either side: 2^-10 of the score, ten times what the polynomial exponentials and
    // the sums amount to, and 2^-20 of the largest log-sum-exp for what grows with the logits: an fp16 pair holds one
    // to 2^-23 of it (that of an estimate is the one the bounds use, that of the candidates' sweep is not known here), and the
    // MMA that subtracts it from a dot product of its size rounds to 2^-24 of that or, with fewer bits kept, 2^-23
    const float margin = 0x1p-10f + 0x1p-20f * lse_max;
    edge = bin > 0 ? __uint_as_float(((uint32_t)bin + kBinBase) << 18) * (1.f - margin) : 0.f;   // (NaN or negative: all keys)
  }
  __syncthreads();
  const float floor_ = edge;
  uint32_t take = 0u;
#pragma unroll
  for (int e = 0; e < kBoundKeys; ++e)
    if (e >= sp.v0 && e < sp.nv && !(hi[e] < floor_)) take |= 1u << e;   // (NaN: a candidate)
  const uint32_t n = __popc(take), upto = prefix(n, warp_sum[1], &total);
  if (tid == 0) list_at = total ? atomicAdd(hist + kPruneBins, total) : 0u;
  __syncthreads();
  int32_t* list = a.cand + sp.at + list_at + (upto - n);
  float preset[kBoundKeys];
#pragma unroll
  for (int e = 0; e < kBoundKeys; ++e) {
    preset[e] = (take >> e) & 1u ? 1.f : -1.f;
    if ((take >> e) & 1u) *list++ = sp.base + e;
  }
  for (int g = 0; g < a.n_slots; ++g) sp.store(a.scores + g * a.slot_stride, preset, a.slot_stride % 4 == 0 || g == 0);
}

}  // namespace

// The one-pass sweep's roles trade registers (setmaxnreg), and what the epilogue asks for has to be what a block was
// launched with: 80 per thread.
bool prune_available() {
  cudaFuncAttributes fa;
  return cudaFuncGetAttributes(&fa, colsum_kernel<true, false, kOnePass>) == cudaSuccess && fa.numRegs == 80;
}

bool prune_plan(const QgPlan& qg, const CacheDev& cv, const SeqTable& t, const Dims& dm, int n_sm, PrunePlan* plan) {
  if (!qg.q_is_f16 || qg.n_qgroups > kPruneSums) return false;
  const int rows = dm.group * dm.n_pseudo;
  double pairs = 0.0;
  for (int b = 0; b < t.batch; ++b) {
    const int L = t.prompt_len[b], K = t.cu_keep[b + 1] - t.cu_keep[b];
    if (L < 32768 || K > L / (L < 65536 ? 16 : 8)) return false;
    pairs += (double)rows * dm.n_kv_heads * L;
  }
  if (pairs < kPruneLeastPairs) return false;
  plan->qg = qg;
  plan->per_cta = kPruneSums / qg.n_qgroups;
  // ---- the sample: rows kSamplePhase, kSamplePhase + 16, ... of the cache, seen as a tensor of its own
  SeqTable& ts = plan->ts;
  memset(&ts, 0, sizeof(ts));
  ts.batch = t.batch;
  for (int b = 0; b < t.batch; ++b) {
    const int first = (t.cu_rows[b] + kSampleStride - 1 - kSamplePhase) / kSampleStride;      // first sampled row of the sequence
    const int end = (t.cu_rows[b] + t.prompt_len[b] - kSamplePhase + kSampleStride - 1) / kSampleStride;
    ts.cu_rows[b] = first;
    ts.prompt_len[b] = end - first;
  }
  const uint64_t rows_s = ((uint64_t)t.cu_rows[t.batch] - kSamplePhase + kSampleStride - 1) / kSampleStride;
  const uint64_t kd[3] = {(uint64_t)kHeadDim, rows_s, (uint64_t)dm.n_kv_heads};
  uint64_t ks[2] = {(uint64_t)cv.k_row_stride * 2 * kSampleStride, (uint64_t)cv.k_head_stride * 2};
  if (dm.n_kv_heads == 1 && ks[1] == 0) ks[1] = ks[0] * rows_s;
  if (ks[1] == 0 || ks[1] % 16) return false;
  const char* base = (const char*)cv.k + (size_t)kSamplePhase * cv.k_row_stride * 2;
  if (!encode_tile_map(&plan->tm_s, base, false, 3, kd, ks, kTile1)) return false;
  const int q_bytes = ((qg.rows_g + 127) / 128) * 2 * 128 * 128, s2 = (kRingEnd - kSlabBytes - q_bytes) / TileGeo<kTile2>::kStage;
  plan->n_stages_m = s2 < kMaxStages ? s2 : kMaxStages;
  if (plan->n_stages_m < 2) return false;
  if (!plan_chunks(ts, 0, kTile1, dm.n_kv_heads * qg.n_qgroups, n_sm, &plan->ct_s, 3.0)) return false;
  if (!plan_chunks(t, dm.n_pseudo, kTile2, dm.n_kv_heads * qg.n_qgroups, n_sm, &plan->ct_m, 6.0)) return false;
  // ---- the candidates: a wave of CTAs shared out by the prompts' lengths
  int64_t total = 0, upto = 0;
  for (int b = 0; b < t.batch; ++b) total += t.prompt_len[b];
  const int per_head = n_sm / (dm.n_kv_heads * qg.n_qgroups2);
  memset(&plan->ct_g, 0, sizeof(ChunkTable));
  for (int b = 0; b < t.batch; ++b) {
    upto += t.prompt_len[b];
    const int to = (int)(per_head * upto / total), least = plan->ct_g.cu_chunk[b] + 1;
    plan->ct_g.cu_chunk[b + 1] = to > least ? to : least;
  }
  plan->ct_g.n_chunks = plan->ct_g.cu_chunk[t.batch];
  return true;
}

cudaError_t launch_prune(const PrunePlan& plan, const CacheDev& cv, const SeqTable& t, const Dims& dm, const PruneBuffers& buf,
                         float* slots, float* scores, int64_t score_stride, int* status, long long wait_limit,
                         cudaStream_t s, LaunchLog* log) {
  Args a = {};
  a.n_pseudo = dm.n_pseudo;
  a.group = dm.group;
  a.n_q_heads = dm.n_q_heads;
  a.n_kv_heads = dm.n_kv_heads;
  a.rows_total = dm.group * dm.n_pseudo;
  a.n_qgroups = plan.qg.n_qgroups;
  a.rows_g = plan.qg.rows_g;
  a.rows_pad = (a.rows_total + 255) / 256 * 256;
  a.n_stages = plan.qg.n_stages1;
  a.early_loads = 1;                                            // (the kernel before these is the rotation)
  a.scale_log2e = 1.f;
  a.wait_limit = wait_limit > 0 ? wait_limit : kWaitLimit;
  a.status = status;
  a.score_stride = score_stride;
  a.k = cv.k;
  a.k_head_stride = cv.k_head_stride;
  a.k_row_stride = cv.k_row_stride;
  cudaError_t e;
  // 1: the sample
  a.sampled = 1;
  a.part = buf.part_s;
  a.ref = buf.ref;
  if ((e = cudaFuncSetAttribute(rowstat_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes)) != cudaSuccess) return e;
  log->begin(kKindLseMerge, s);
  e = launch_pdl(rowstat_kernel<true>, dim3(plan.ct_s.n_chunks * a.n_qgroups, dm.n_kv_heads), dim3(kThreads1), kSmemBytes, s, 1, plan.tm_s,
                 plan.qg.tm_q, plan.ts, plan.ct_s, a);
  log->end(s);
  if (e != cudaSuccess) return e;
  // 2: one pass over all keys
  a.sampled = 0;
  a.n_stages = plan.n_stages_m;
  a.log2_sample = kLog2Sample;
  a.sum_groups = plan.per_cta;
  a.scores = buf.sums;
  a.slot_stride = ((int64_t)dm.n_kv_heads * score_stride + 3) & ~(int64_t)3;
  a.part_out = buf.part_m;
  a.ref_out = buf.ref;
  a.hist = buf.hist;
  auto one = a.rows_g <= 128 ? colsum_kernel<true, false, kOnePass, true> : colsum_kernel<true, false, kOnePass, false>;
  if ((e = cudaFuncSetAttribute(one, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes)) != cudaSuccess) return e;
  log->begin(kKindSweep1, s);
  e = launch_pdl(one, dim3(plan.ct_m.n_chunks * a.n_qgroups, dm.n_kv_heads), dim3(kThreadsOne), kSmemBytes, s, 1, plan.qg.tm_k2, plan.qg.tm_q, t,
                 plan.ct_m, plan.ct_s, a);
  log->end(s);
  if (e != cudaSuccess) return e;
  // 3: bounds and candidates
  const int n_slots = plan.qg.n_qgroups2;
  float* out = n_slots > 1 ? slots : scores;
  const int64_t slot_stride = (int64_t)dm.n_kv_heads * score_stride;
  BoundArgs ba = {};
  ba.part = buf.part_m;
  ba.ref = buf.ref;
  ba.rows_total = a.rows_total;
  ba.rows_pad = a.rows_pad;
  ba.rows_g = a.rows_g;
  ba.n_sums = a.n_qgroups * plan.per_cta;
  ba.per_cta = plan.per_cta;
  ba.sums = buf.sums;
  ba.sum_stride = a.slot_stride;
  ba.score_stride = score_stride;
  ba.hist = buf.hist;
  ba.cand = buf.cand;
  ba.scores = out;
  ba.slot_stride = slot_stride;
  ba.n_slots = n_slots;
  int max_len = 1;
  for (int b = 0; b < t.batch; ++b) max_len = t.prompt_len[b] > max_len ? t.prompt_len[b] : max_len;
  const dim3 tiles((max_len + 3 + kBoundTile - 1) / kBoundTile, dm.n_kv_heads, t.batch);
  log->begin(kKindTopk, s);
  e = launch_pdl(bound_hist_kernel, tiles, dim3(kBoundThreads), 0, s, 1, t, plan.ct_m, ba);
  log->end(s);
  if (e != cudaSuccess) return e;
  log->begin(kKindTopk, s);
  e = launch_pdl(bound_list_kernel, tiles, dim3(kBoundThreads), 0, s, 1, t, ba);
  log->end(s);
  if (e != cudaSuccess) return e;
  // 4: the candidates' scores
  a.part = buf.part_m;
  a.cand = buf.cand;
  a.n_qgroups = plan.qg.n_qgroups2;
  a.rows_g = plan.qg.rows_g2;
  a.n_stages = plan.qg.n_stages2;
  a.scores = out;
  a.slot_stride = slot_stride;
  auto gather = [&](auto kernel, int smem) -> cudaError_t {
    cudaError_t e2 = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e2 != cudaSuccess) return e2;
    log->begin(kKindSweep2, s);
    e2 = launch_pdl(kernel, dim3(plan.ct_g.n_chunks * a.n_qgroups, dm.n_kv_heads), dim3(kThreads2), smem, s, 1, plan.qg.tm_k2, plan.qg.tm_q,
                    t, plan.ct_g, plan.ct_m, a);
    log->end(s);
    return e2;
  };
  e = plan.qg.wide2 ? gather(colsum_kernel<true, true, kGather>, SmemT<true>::total) : gather(colsum_kernel<true, false, kGather>, kSmemBytes);
  if (e != cudaSuccess) return e;
  if (n_slots > 1 && (e = launch_slots_sum(slots, n_slots, scores, slot_stride, s, log)) != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace dapq
