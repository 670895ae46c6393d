// The retained set without the scores (Section 4.2, Eq. 5 needs the K largest S(j), not all of them): layers of a
// dapq_evict_layers call, from kPruneLeastLayers layers on.  The set of the two full sweeps, up to keys whose scores agree
// with the K-th to rounding, for less than two thirds of their work where it pays.
//
//   1. sample      sweep 1 over every 16th key: with the first key an estimate r_i of each query row's log-sum-exp;
//   2. one pass    over all keys with r_i in place of the log-sum-exp: e_ij = 2^(s_ij - r_i) is added to the sum of its
//                  row, Z_i, and to that of its key, E_g(j), in up to four sums g of some 64 to 256 rows each.  The row sums
//                  are what sweep 1 yields: log-sum-exp_i = r_i + log2 Z_i, in fp32 as there;
//   3. bounds      S(j) = sum_i e_ij / Z_i, so  sum_g E_g(j) / max_g Z  <=  S(j)  <=  sum_g E_g(j) / min_g Z.  With T the K-th
//                  largest lower bound (at least K keys score T or more), a key whose upper bound is below T is not
//                  among the K largest: what remains are the candidates;
//   4. candidates  sweep 2 over them, with the log-sum-exp from step 2: the scores that the full sweep 2 gives them, up to
//                  the order in which that was summed (skipped, per KV head, when there are exactly K);
//   5. selection   as ever, on an array that holds -1 for all other keys.
// Nothing depends on how good the estimate is but the number of candidates.  A row sum that leaves the float range
// is done over again by itself (careful_row).
//
// Where it pays is a matter of the data: the bounds are as wide as the worst estimate among the rows behind a sum, and rows
// whose mass lies in few keys are estimated badly.  So the first layer of a call tries, and every layer that is pruned adds
// what its longest list of candidates gained or lost to a credit (Route); once that is used up, the next layers run the full
// sweeps, and one tries again after kPruneRetry layers.  The decision stays on the device: the launches are the same either
// way, the two sweeps do the one thing or the other, and the one pass and the bounds return at once.
//
// Measured on B200, us a layer of a 32-layer call, full sweeps -> here, 128 k keys:
//                                        8 heads x 1024 rows      4 x 448       8 x 256
//   N(0, 1) keys                             670 -> 573         177 -> 166    197 -> 184
//   the same times 2                         694 -> 715         175 -> 170    201 -> 190
//   times 3                                  713 -> 743         183 -> 193    209 -> 222
//   times 4                                  712 -> 739         176 -> 183    224 -> 236
//   four channels times 8                    683 -> 581         177 -> 165    215 -> 227
//   a first key 8 above the rest             670 -> 507         174 -> 156    200 -> 180
//   five keys that single rows attend to     679 -> 531         174 -> 166    214 -> 228
//   passages that stand out, K keys          662 -> 562         172 -> 152    192 -> 171
//   ... K/2 keys                             688 -> 621         180 -> 175    200 -> 206
// (every layer trying whatever the others found: times 3 691 -> 806, 181 -> 219, 198 -> 222.)  What the full route still loses is
// the three launches with nothing to do (some 2 us each) and the layers that tried: 12 layers, times 4, 671 -> 700, 184 -> 194,
// 196 -> 211; the shortest calls, 8 layers, 634 -> 702, 185 -> 196, 194 -> 207 (and 646 -> 535, 181 -> 159, 191 -> 173 with
// passages for K keys).  In a long call at the power cap (80 layers of 8 x 1024 rows, outlier channels and needles) 708 -> 603.
// Prompts of 32 k gained a tenth at best and lost a fifth (8 x 1024 rows: first key 190 -> 176, N(0, 1) 209 -> 238; 8
// prompts of 8 x 256: 434 -> 393, times 2 404 -> 479): a sample of 2 k keys says too little.  Fewer query-key pairs do
// not pay for the launches: 1.3e8 pairs 130 -> 129 to 108 -> 132 (8 x 128 rows of 128 k, 8 x 256 of 64 k).  Hence the
// conditions in prune_plan: prompts long enough for the sample, pairs enough for the launches, and a budget of at
// most an eighth of a prompt, so that the threshold lies in the tail of the scores.
#include "score_qg_sweep1.cuh"
#include "score_qg_sweep2.cuh"

namespace dapq {
namespace {

using namespace qg;

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
  const Route* route_in;                   // as in Args
  Route* route_out;
  float most;
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
  const bool pruned = route_of(a.route_in, a.most) >= 0.f;
  if (pruned && (int)blockIdx.x * kBoundTile - head_lead(t, a, b, kvh) >= t.prompt_len[b]) return;
  for (int x = tid; x < kPruneBins; x += kBoundThreads) hist[x] = 0u;
  if (tid < kPruneSums) { f_min[tid] = 0x7f800000u; f_max[tid] = 0u; }
  if (tid == 0) lse_max = 0u;
  if (!pruned) { wait_in_one_cta(); return; }
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
  if (!(route_of(a.route_in, a.most) >= 0.f)) { wait_in_one_cta(); return; }
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
  if (tid == 0) {
    list_at = total ? atomicAdd(hist + kPruneBins, total) : 0u;
    // (the count only grows: the block that comes last sees all of it; positive floats order like their bit patterns)
    atomicMax(reinterpret_cast<int*>(&a.route_out->worst), __float_as_int((float)(list_at + total) / (float)t.prompt_len[b]));
  }
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

// Sweep 1 of a layer on the full route, its sample on the pruned one, in one launch.
__global__ void __launch_bounds__(kThreads1, 1)
rowstat_route_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_s, const __grid_constant__ CUtensorMap tm_q,
                     const __grid_constant__ SeqTable t, const __grid_constant__ ChunkTable ct, const __grid_constant__ ChunkTable ct_s,
                     const Args a) {
  const bool sampled = route_of(a.route_in, a.most) >= 0.f;
  const ChunkTable& c = sampled ? ct_s : ct;
  // (the grid has room for either: the CTAs with work come first)
  const int nx = c.n_chunks * a.n_qgroups, id = blockIdx.y * gridDim.x + blockIdx.x, kvh = id / nx;
  if (kvh >= (int)gridDim.y) return;
  rowstat_cta<true>(sampled ? tm_s : tm_k, tm_q, t, c, a, id - kvh * nx, kvh, sampled, !sampled);
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
    if (L < kPruneLeastLen || K > L / 8) return false;
    pairs += (double)rows * dm.n_kv_heads * L;
  }
  if (pairs < kPruneLeastPairs) return false;
  plan->qg = qg;
  plan->per_cta = kPruneSums / qg.n_qgroups;
  // (the candidates' sweep takes the time of its longest list: with two jobs a tile about its share of a full sweep, with one
  // half as much again.  Break-even measured at 0.59 to 0.85 of a sweep's time for 8 x 1024 rows of 128 k, in bursts and at the
  // power cap, which the full sweeps reach; 0.50 for 4 x 448; 0.43 to 0.47 for 8 x 256)
  plan->most = (float)(qg.wide2 ? 0.78 - 6.8e7 / pairs : 0.45 - 4e7 / pairs);
  // ---- the sample: rows kSamplePhase, kSamplePhase + 16, ... of the cache, seen as a tensor of its own
  SeqTable ts;                                                  // (only what plan_chunks looks at)
  ts.batch = t.batch;
  for (int b = 0; b < t.batch; ++b) ts.prompt_len[b] = sample_first(t.cu_rows[b] + t.prompt_len[b]) - sample_first(t.cu_rows[b]);
  const uint64_t rows_s = (uint64_t)sample_first(t.cu_rows[t.batch]);
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
                         int route_at, int route_next, float* slots, float* scores, int64_t score_stride, int* status, long long wait_limit,
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
  a.route_in = route_at < 0 ? nullptr : reinterpret_cast<const Route*>(buf.route) + route_at;
  a.route_out = reinterpret_cast<Route*>(buf.route) + route_next;
  a.most = plan.most;
  // 1: the sample, or sweep 1
  a.part = buf.part_s;
  a.ref = buf.ref;
  if ((e = cudaFuncSetAttribute(rowstat_route_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes)) != cudaSuccess) return e;
  const int n_chunks = route_at >= 0 && plan.qg.ct1.n_chunks > plan.ct_s.n_chunks ? plan.qg.ct1.n_chunks : plan.ct_s.n_chunks;
  log->begin(kKindLseMerge, s);
  e = launch_pdl(rowstat_route_kernel, dim3(n_chunks * a.n_qgroups, dm.n_kv_heads), dim3(kThreads1), kSmemBytes, s, 1, plan.qg.tm_k1, plan.tm_s,
                 plan.qg.tm_q, t, plan.qg.ct1, plan.ct_s, a);
  log->end(s);
  if (e != cudaSuccess) return e;
  // 2: one pass over all keys
  a.n_stages = plan.n_stages_m;
  a.log2_sample = kLog2Sample;
  a.sum_groups = plan.per_cta;
  a.scores = buf.sums;
  a.slot_stride = ((int64_t)dm.n_kv_heads * score_stride + 3) & ~(int64_t)3;
  a.part_out = buf.part_m;
  a.ref_out = buf.est;
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
  ba.ref = buf.est;
  ba.rows_total = a.rows_total;
  ba.rows_pad = a.rows_pad;
  ba.rows_g = a.rows_g;
  ba.n_sums = a.n_qgroups * plan.per_cta;
  ba.per_cta = plan.per_cta;
  ba.sums = buf.sums;
  ba.sum_stride = a.slot_stride;
  ba.score_stride = score_stride;
  ba.hist = buf.hist;
  ba.route_in = a.route_in;
  ba.route_out = a.route_out;
  ba.most = plan.most;
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
  a.part_full = buf.part_s;
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
                    t, plan.ct_g, ChunkTables2{plan.ct_m, plan.qg.ct1}, a);
    log->end(s);
    return e2;
  };
  e = plan.qg.wide2 ? gather(colsum_kernel<true, true, kGather>, SmemT<true>::total) : gather(colsum_kernel<true, false, kGather>, kSmemBytes);
  if (e != cudaSuccess) return e;
  if (n_slots > 1 && (e = launch_slots_sum(slots, n_slots, scores, slot_stride, s, log)) != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace dapq
