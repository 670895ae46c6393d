// Host side of the scorer that runs both sweeps over several layers as one stream of units (score_flow.cuh).
#include "score_flow.cuh"

namespace dapq {

using namespace flow;

int flow_rows_pad(const Dims& dm) {
  const int rows = dm.group * dm.n_pseudo, groups = qg_groups(dm);
  return groups * ((((rows + groups - 1) / groups) + 15) & ~15);
}

bool flow_plan(const void* q, const CacheDev* cv, int n_layers, const SeqTable& t, const Dims& dm, int n_sm, int64_t max_chunks, FlowPlan* plan) {
  if (n_layers < 1 || n_layers > kMaxLayers) return false;
  const int rows_total = dm.group * dm.n_pseudo;
  plan->n_layers = n_layers;
  plan->n_qgroups = qg_groups(dm);
  plan->rows_g = (((rows_total + plan->n_qgroups - 1) / plan->n_qgroups) + 15) & ~15;
  plan->rows_pad = flow_rows_pad(dm);
  plan->two = plan->rows_g > 128 ? 1 : 0;
  const int per_chunk = dm.n_kv_heads * plan->n_qgroups;
  int64_t pairs = 0;
  for (int b = 0; b < t.batch; ++b) pairs += (t.prompt_len[b] + dm.n_pseudo + kPair - 1) / kPair;
  auto chunks = [&](int ct) {
    int64_t n = 0;
    for (int b = 0; b < t.batch; ++b) n += ((t.prompt_len[b] + dm.n_pseudo + kPair - 1) / kPair + ct - 1) / ct;
    return n;
  };
  // Pairs of a unit: units go to the CTAs one by one, so a sweep takes about as many rounds of them as units / CTAs, rounded up,
  // each of a unit's pairs and some half a pair of set-up.  Below four pairs the next unit's ticket, queries and
  // log-sum-exps no longer hide behind this one.
  int ct = 0;
  double best = 0.0;
  for (int c = 4; c <= 16; ++c) {
    const int64_t n = n_layers * chunks(c), units = n * per_chunk;
    if (n > max_chunks) continue;
    const double cost = (double)((2 * units + n_sm - 1) / n_sm) * ((double)n_layers * per_chunk * pairs / units + 0.4);
    if (ct == 0 || cost < best) { ct = c; best = cost; }
  }
  if (ct == 0) return false;
  plan->ct.chunk_tiles = ct;
  int32_t n = 0, most_chunks = 0;
  for (int b = 0; b < t.batch; ++b) {
    const int c = ((t.prompt_len[b] + dm.n_pseudo + kPair - 1) / kPair + ct - 1) / ct;
    plan->ct.cu_chunk[b] = n;
    n += c;
    most_chunks = c > most_chunks ? c : most_chunks;
  }
  plan->ct.cu_chunk[t.batch] = n;
  plan->ct.n_chunks = n;
  plan->n_units = n_layers * n * per_chunk;
  plan->n_items = n_layers * t.batch * per_chunk;
  // (a block holds at least the units of an item, so that a unit of sweep 2 depends on lower tickets only)
  const int item = most_chunks * plan->n_qgroups;
  plan->block = item > n_sm ? item : n_sm;
  // ---- tensor maps: K of every layer as [d, rows, H_kv], the queries of all layers as [d, rows]
  const uint64_t rows_k = (uint64_t)t.cu_rows[t.batch];
  const uint64_t kd[3] = {(uint64_t)kHeadDim, rows_k, (uint64_t)dm.n_kv_heads};
  for (int l = 0; l < n_layers; ++l) {
    uint64_t ks[2] = {(uint64_t)cv[l].k_row_stride * 2, (uint64_t)cv[l].k_head_stride * 2};
    if (dm.n_kv_heads == 1 && ks[1] == 0) ks[1] = ks[0] * rows_k;
    if (ks[1] == 0 || ks[1] % 16) return false;
    if (!encode_tile_map(&plan->tm_k[l], cv[l].k, false, 3, kd, ks, kSub)) return false;
  }
  const uint64_t qd[2] = {(uint64_t)kHeadDim, (uint64_t)n_layers * t.batch * dm.n_q_heads * dm.n_pseudo};
  const uint64_t qs[1] = {(uint64_t)kHeadDim * 2};
  return encode_tile_map(&plan->tm_q, q, true, 2, qd, qs, 128);
}

cudaError_t launch_score_flow(const FlowPlan& plan, const SeqTable& t, const Dims& dm, float2* part, int64_t max_chunks, const float* ref, float* slots,
                              float* scores, int64_t score_stride, uint32_t* sync, int n_sm, int* status, long long wait_limit, cudaStream_t s,
                              LaunchLog* log) {
  Args a = {};
  a.n_pseudo = dm.n_pseudo;
  a.group = dm.group;
  a.n_q_heads = dm.n_q_heads;
  a.n_kv_heads = dm.n_kv_heads;
  a.rows_total = dm.group * dm.n_pseudo;
  a.n_qgroups = plan.n_qgroups;
  a.rows_g = plan.rows_g;
  a.rows_pad = plan.rows_pad;
  a.n_units = plan.n_units;
  a.units_layer = plan.n_units / plan.n_layers;
  a.block = plan.block;
  a.score_stride = score_stride;
  a.layer_stride = (int64_t)dm.n_kv_heads * score_stride;
  a.slot_stride = a.layer_stride * plan.n_layers;
  a.wait_limit = wait_limit > 0 ? wait_limit : kWaitLimit;
  a.part = part;
  a.sums = reinterpret_cast<float*>(part + max_chunks * dm.n_kv_heads * plan.rows_pad);
  a.ref = ref;
  a.scores = plan.n_qgroups > 1 ? slots : scores;
  a.sync = sync;
  a.status = status;
  KeyMaps km;
  for (int l = 0; l < kMaxLayers; ++l) km.m[l] = plan.tm_k[l < plan.n_layers ? l : 0];
  auto run = [&](auto kernel, int smem) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const int64_t tickets = 2LL * plan.n_units;
    log->begin(kKindSweep1, s);
    e = launch_pdl(kernel, dim3((unsigned)(tickets < n_sm ? tickets : n_sm)), dim3(kThreads), smem, s, 1, km, plan.tm_q, t, plan.ct, a);
    log->end(s);
    return e;
  };
  cudaError_t e = plan.two ? run(flow_kernel<true>, Smem<true>::total) : run(flow_kernel<false>, Smem<false>::total);
  if (e != cudaSuccess) return e;
  if (plan.n_qgroups > 1 && (e = launch_slots_sum(slots, plan.n_qgroups, scores, a.slot_stride, s, log)) != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace dapq
