// Importance scoring on the tensor cores without rounding the operands (Section 4.2, Eq. 4): fp32 caches, and
// bf16 caches whose KV heads have fewer than 64 query rows (models without grouped queries, small windows), with
// the rotated queries in fp32.  The kernels are in score_split_kernel.cuh; the CUDA-core kernels (score_fma.cu)
// keep the calls that ask for the synthetic keys' mass, the callers without a context and DAPQ_FLAG_CUDA_CORE_SCORER.
//
// Why: the CUDA-core sweeps are bound by shared-memory reads (10 wavefronts per 32 FMA instructions) and stage every K
// tile once per query head.  Measured on B200, whole eviction of a layer, CUDA cores -> here: 32 heads without
// groups, 32 queries, 16 k bf16 keys 432 -> 70 us; 8 x 4 heads, 32 queries, 12 k fp32 keys 339 -> 66 us; 2 x 4 heads,
// 2 k fp32 keys 48 -> 25 us of device time.  Relative error of the scores against float64 on those inputs
// 3.04e-7 -> 1.64e-7, 1.62e-7 -> 1.57e-7, 1.53e-7 -> 0.90e-7 (the mean of six seeds each): a chain of four tensor-core
// additions per accumulator rounds less than one of 128 FMAs, and the products left out for fp32 keys are below all that.
//
// What bounds it.  fp32 keys: the MMAs, 2450 cycles per tile and 64 query rows (28 MMAs of 64 to 192 columns; the split
// of a tile into its parts takes four warps somewhat less).  bf16 keys: about 1200 cycles of MMAs per tile (9 of up
// to 96 columns, which one thread cannot issue faster) against 1400 for the tile's 32 KB at an SM's share of HBM.
// Score slots are needed beyond 128 query rows per KV head only (two sub-groups share a CTA in sweep 2).
#include "score_split_kernel.cuh"

namespace dapq {
namespace {

using namespace split;

constexpr int kMaxSmem = 232448;

// Ring and staging slots beside the queries of n_sub sub-groups of R rows; returns the shared memory they take.
// fp32 keys: two ring slots, and as many staging slots as still fit (two with 128 query rows).
int smem_of(int R, int n_sub, int key_parts, int* n_ring, int* n_stage) {
  const bool f32 = key_parts == 3;
  const int q = n_sub * (f32 ? Roles<3>::query_bytes(R) : Roles<1>::query_bytes(R)), slot = f32 ? Roles<3>::slot : Roles<1>::slot;
  const int room = kMaxSmem - State::total - q;
  *n_ring = f32 ? 2 : (room / slot < kMaxRing ? room / slot : kMaxRing);
  *n_stage = f32 ? (room - 2 * slot) / kQuarter : 0;
  if (*n_stage > kMaxStage) *n_stage = kMaxStage;
  return q + *n_ring * slot + *n_stage * kQuarter + State::total;
}
static_assert(kMaxSmem - State::total - 2 * Roles<3>::query_bytes(64) - 2 * Roles<3>::slot >= 2 * kQuarter, "two staging slots have to fit");

template <int kR, int kKeyParts>
cudaError_t run(const SplitPlan& plan, const SeqTable& t, Args a, int smem1, int smem2, bool after_own_kernel, cudaStream_t s,
                LaunchLog* log) {
  auto k1 = split_kernel<kR, kKeyParts, false>;
  auto k2 = split_kernel<kR, kKeyParts, true>;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k2, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem)) != cudaSuccess) return e;
  const int n_sub2 = a.n_sub;
  if (a.lse_in == nullptr) {
    a.n_sub = 1;
    a.n_qgroups = plan.n_qgroups;
    a.n_ring = plan.n_ring1;
    a.n_stage = plan.n_stage1;
    a.state_off = smem1 - State::total;
    a.early_loads = after_own_kernel ? 1 : 0;
    log->begin(kKindSweep1, s);
    e = launch_pdl(k1, dim3(plan.ct1.n_chunks * a.n_qgroups, a.n_kv_heads), dim3(Roles<kKeyParts>::threads), smem1, s, 1, plan.tm_k, t,
                   plan.ct1, plan.ct1, a);
    log->end(s);
    if (e != cudaSuccess) return e;
  }
  a.n_sub = n_sub2;
  a.n_qgroups = plan.n_qgroups2;
  a.n_ring = plan.n_ring2;
  a.n_stage = plan.n_stage2;
  a.state_off = smem2 - State::total;
  a.early_loads = (after_own_kernel || a.lse_in == nullptr) ? 1 : 0;   // (sweep 1, if it ran, waited for what came before)
  log->begin(kKindSweep2, s);
  e = launch_pdl(k2, dim3(plan.ct2.n_chunks * a.n_qgroups, a.n_kv_heads), dim3(Roles<kKeyParts>::threads), smem2, s, 1, plan.tm_k, t,
                 plan.ct2, plan.ct1, a);
  log->end(s);
  return e;
}

template <int kKeyParts>
cudaError_t run_rows(const SplitPlan& plan, const SeqTable& t, const Args& a, int smem1, int smem2, bool after, cudaStream_t s,
                     LaunchLog* log) {
  switch (plan.R) {
    case 16: return run<16, kKeyParts>(plan, t, a, smem1, smem2, after, s, log);
    case 32: return run<32, kKeyParts>(plan, t, a, smem1, smem2, after, s, log);
    case 48: return run<48, kKeyParts>(plan, t, a, smem1, smem2, after, s, log);
    default: return run<64, kKeyParts>(plan, t, a, smem1, smem2, after, s, log);
  }
}

}  // namespace

int split_groups(const Dims& dm) { return (dm.group * dm.n_pseudo + 2 * 64 - 1) / (2 * 64); }

bool split_plan(int dtype, const CacheDev& cv, const SeqTable& t, const Dims& dm, int n_sm, SplitPlan* plan) {
  const int rows = dm.group * dm.n_pseudo;
  plan->key_parts = dtype == DAPQ_F32 ? 3 : 1;
  plan->n_qgroups = (rows + 63) / 64;
  plan->R = ((rows + plan->n_qgroups - 1) / plan->n_qgroups + 15) & ~15;
  plan->n_sub2 = plan->n_qgroups > 1 ? 2 : 1;
  plan->n_qgroups2 = (plan->n_qgroups + plan->n_sub2 - 1) / plan->n_sub2;
  plan->smem1 = smem_of(plan->R, 1, plan->key_parts, &plan->n_ring1, &plan->n_stage1);
  plan->smem2 = smem_of(plan->R, plan->n_sub2, plan->key_parts, &plan->n_ring2, &plan->n_stage2);
  // (a CTA's set-up of some 6 k cycles weighs two to three fp32 tiles, and more of the bf16 ones of about 1.2 k)
  const double cost = dtype == DAPQ_F32 ? 3.0 : 6.0;
  if (!plan_chunks(t, dm.n_pseudo, kTile, dm.n_kv_heads * plan->n_qgroups, n_sm, &plan->ct1, cost)) return false;
  if (!plan_chunks(t, 0, kTile, dm.n_kv_heads * plan->n_qgroups2, n_sm, &plan->ct2, cost)) return false;
  const uint64_t rows_k = (uint64_t)t.cu_rows[t.batch], eb = dtype == DAPQ_F32 ? 4 : 2;
  const uint64_t kd[3] = {(uint64_t)kHeadDim, rows_k, (uint64_t)dm.n_kv_heads};
  uint64_t ks[2] = {(uint64_t)cv.k_row_stride * eb, (uint64_t)cv.k_head_stride * eb};
  if (dm.n_kv_heads == 1 && ks[1] == 0) ks[1] = ks[0] * rows_k;
  if (ks[1] == 0 || ks[1] % 16) return false;
  return dtype == DAPQ_F32 ? encode_rows_map_f32(&plan->tm_k, cv.k, kd, ks, 32, kTile) : encode_tile_map(&plan->tm_k, cv.k, false, 3, kd, ks, kTile);
}

cudaError_t launch_score_split(const SplitPlan& plan, int q_dtype, const void* q, const SeqTable& t, const Dims& dm,
                               const float* lse_in, float2* part, float* slots, float* scores, int64_t score_stride, float* lse_out,
                               int* status, long long wait_limit, bool after_own_kernel, cudaStream_t s, LaunchLog* log) {
  Args a = {};
  a.q = q;
  a.q_bf16 = q_dtype == DAPQ_BF16 ? 1 : 0;
  a.n_pseudo = dm.n_pseudo;
  a.group = dm.group;
  a.n_q_heads = dm.n_q_heads;
  a.n_kv_heads = dm.n_kv_heads;
  a.rows_total = dm.group * dm.n_pseudo;
  a.n_sub = plan.n_sub2;
  a.rows_pad = (a.rows_total + 255) / 256 * 256;
  a.scale_log2e = dm.scale_log2e;
  a.wait_limit = wait_limit > 0 ? wait_limit : ptx::kWaitLimit;
  a.part = part;
  a.lse_in = lse_in;
  a.lse_out = lse_out;
  a.scores = plan.n_qgroups2 > 1 ? slots : scores;
  a.score_stride = score_stride;
  a.slot_stride = (int64_t)dm.n_kv_heads * score_stride;
  a.status = status;
  cudaError_t e = plan.key_parts == 3 ? run_rows<3>(plan, t, a, plan.smem1, plan.smem2, after_own_kernel, s, log)
                                      : run_rows<1>(plan, t, a, plan.smem1, plan.smem2, after_own_kernel, s, log);
  if (e != cudaSuccess) return e;
  if (plan.n_qgroups2 > 1) e = launch_slots_sum(slots, plan.n_qgroups2, scores, a.slot_stride, s, log);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace dapq
