// Both sweeps of the tensor-core scorer as one stream of units over all sequences, KV heads and layers of a launch
// (host side in score_flow.cu).
//
// A unit is one sweep over a run of key pairs (256 keys) of one (layer, sequence, KV head, query group): sweep 1 leaves
// the run's partial row sums, sweep 2 the scores of its keys.  The CTAs, one per SM, take units in a fixed order from a
// ticket counter.  The order alternates blocks of units, sweep 2 two blocks behind sweep 1, so that a unit of sweep 2 finds
// the row sums of its item complete (they are counted per item) and, with short units, its keys still in L2.  A unit depends on units with lower tickets only, which
// other CTAs are already working on: whatever number of CTAs is resident, the lowest unfinished unit can always finish.
//
// Why one launch: two launches per layer spent a third (32 k keys, 8 heads x 256 query rows) to a half (8 k keys) of their
// time on set-up - barriers, tensor memory, the first copies, the merge of the partials, each a few microseconds that
// nothing else filled - and on the last wave.  Here the roles run ahead of one another across units: the next unit's ticket,
// keys, conversions and log-sum-exps come while the epilogue still works on the unit before.
//
// Keys come in pairs of 128-key sub-tiles whose halves lie side by side, [64 channels][256 keys] twice: sweep 1 takes the
// pair as one operand of 256 columns (a job is [128 query rows x 256 keys]), sweep 2 a sub-tile at a time (a job is
// [128 keys x 256 query rows]; with at most 128 query rows, both sub-tiles side by side, [2 x 128 keys x 128 rows]).
// So a job is always one accumulator of 256 columns of which every epilogue thread adds up 64.
//
// What bounds it: instruction issue (0.57 to 0.59 a cycle and scheduler) and, under a sustained load, power (1.62 GHz); the
// exponential pipe is 57 (128 query rows) to 69 % busy (256), the tensor pipe 34 to 40 %, DRAM 55 to 30 %.  Us a layer with selection
// and compaction, two launches a layer -> here, in bursts of 10 ms | over seconds: 32 k keys on 8 heads x 256 rows 71 -> 47 | 71 -> 54,
// a ragged batch of 150 k keys x 128 rows 189 -> 158 | 198 -> 176, 40 prompts of 8 k 371 -> 309 | 404 -> 357.  The code has one body per role on purpose: with all variants inlined (118 to 142 KB against 67 to 71) units of three
// pairs ran at 0.75 of this pace, waiting for instructions.
#pragma once
#include "score_qg_sweep1.cuh"
#include "score_qg_sweep2.cuh"

namespace dapq {
namespace flow {

using namespace ptx;
using qg::RowSum;

constexpr int kSub = 128, kPair = 2 * kSub;            // keys
constexpr int kSubs = 4;                               // sub-tiles in the ring: two pairs
constexpr int kSubHalf = kSub * 128, kPairHalf = 2 * kSubHalf, kPairBytes = 2 * kPairHalf;
constexpr int kConvWarps = 4, kFirstEpi = 2 + kConvWarps, kEpiWarps = 16, kSumWarp = kFirstEpi + kEpiWarps, kSchedWarp = kSumWarp + 1;
constexpr int kThreads = (kSchedWarp + 1) * 32;
constexpr int kSlots = 4;                              // posts of the epilogue on their way to the summing warp, 2 KB each
constexpr int kUnitRing = 2;                           // units announced and not yet read by every role
constexpr int kEndUnit = 0, kSweep1 = 1, kSweep2 = 2;

// One unit, as announced by the scheduling warp.
struct alignas(16) Unit {
  int32_t kind, layer, kvh, b;
  int32_t pair0, n_pairs, rows, qgrp;
  int32_t L, row_base, qrow, new_q;                    // prompt length, first cache row, first query row; the queries are not the unit's before
  int32_t chunk, first_chunk, n_chunks, item;          // rows of `part`: this run's, its item's; the item's counter
};

struct Args {
  int32_t n_pseudo, group, n_q_heads, n_kv_heads, rows_total, n_qgroups, rows_g, rows_pad;
  int32_t n_units, units_layer, block;                 // units of a sweep in all and of one layer; units of a block
  int64_t score_stride, slot_stride, layer_stride;     // floats between heads, query groups and layers of `scores`
  long long wait_limit;
  float* sums;                                         // [layers][chunks][H_kv][rows_pad] row sums relative to the references; -1: see `part`
  float2* part;                                        // the same as (base, sum), where a sum has left its range
  const float* ref;                                    // [layers][B, H_q, N] reference logits from the rotation
  float* scores;
  uint32_t* sync;                                      // [0] next ticket, [1 + item] runs of the item whose row sums are stored
  int* status;
};

template <bool kTwo>
struct Smem {                                          // kTwo: groups of 129 .. 256 query rows, else up to 128
  static constexpr int rows = kTwo ? 256 : 128, q_half = rows * 128;
  static constexpr int ring = 2 * q_half;
  static constexpr int slab = ring + kSubs / 2 * kPairBytes, slab_bytes = rows * 32;   // two: minus the references / log-sum-exps
  static constexpr int ones = slab + 2 * slab_bytes, ones_bytes = kPair * 32;
  static constexpr int exch = ones + ones_bytes;
  static constexpr int unit = exch + kSlots * 2048;
  static constexpr int bars = unit + kUnitRing * (int)sizeof(Unit);
  static constexpr int k_full = 0, k_conv = 4, k_empty = 8, acc_full = 12, acc_empty = 14, part_full = 16, part_empty = 20, unit_full = 24,
                       unit_empty = 26, slab_full = 28, slab_empty = 30, q_full = 32, drain = 33, go = 34, n_bars = 35;
  static constexpr int tmem_ptr = bars + n_bars * 8, abort_flag = tmem_ptr + 4, total = abort_flag + 4;
  static_assert(slab % 1024 == 0 && ones % 256 == 0 && exch % 16 == 0 && unit % 16 == 0 && bars % 8 == 0, "");
  static_assert(total <= 232448, "exceeds the shared memory a CTA can opt in to");
  static __device__ __forceinline__ uint32_t bar_count(int i) {
    if (i < k_conv) return 1u;
    if (i < k_empty) return kConvWarps;
    if (i < acc_empty) return 1u;                      // k_empty, acc_full: one tcgen05.commit
    if (i < part_empty) return kEpiWarps;              // acc_empty, part_full
    if (i < unit_empty) return 1u;                     // part_empty, unit_full
    if (i < slab_full) return 2u + kConvWarps + kEpiWarps + 1u;   // unit_empty: every role but the scheduling warp
    if (i < slab_empty) return 1u;
    if (i < q_full) return 1u + kEpiWarps;             // slab_empty: the MMAs' commit, the epilogue warps
    return 1u;
  }
};

__device__ __forceinline__ Unit read_unit(const uint8_t* smem, int at) {
  Unit u;
  const int4* p = reinterpret_cast<const int4*>(smem + at);
  int4* d = reinterpret_cast<int4*>(&u);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(Unit) / 16); ++i) d[i] = p[i];
  return u;
}

// Ticket -> sweep and number of a unit.  Blocks of `X` units (the last may be shorter): sweep 1 of blocks 0 and 1, sweep 2 of
// block 0, sweep 1 of block 2, sweep 2 of block 1, ...
__host__ __device__ __forceinline__ int unit_of_ticket(int x, int n, int X, int* kind) {
  const int nb = (n + X - 1) / X;
  if (nb <= 1) {
    *kind = x < n ? kSweep1 : kSweep2;
    return x < n ? x : x - n;
  }
  *kind = kSweep1;
  if (x < X) return x;
  x -= X;
  const int full = 2 * X * (nb - 2);
  if (x < full) {
    const int j = x / (2 * X), z = x - j * 2 * X;      // sweep 1 of block j + 1, sweep 2 of block j
    if (z < X) return (j + 1) * X + z;
    *kind = kSweep2;
    return j * X + z - X;
  }
  x -= full;
  const int last = n - (nb - 1) * X;
  if (x < last) return (nb - 1) * X + x;
  *kind = kSweep2;
  return (nb - 2) * X + x - last;
}

// The unit behind a ticket; n_pairs may be 0 (a run of sweep 2 that would hold synthetic keys only).
__device__ __forceinline__ void make_unit(Unit& u, int x, const SeqTable& t, const ChunkTable& ct, const Args& a) {
  const int n = unit_of_ticket(x, a.n_units, a.block, &u.kind);
  const int per_chunk = a.n_kv_heads * a.n_qgroups;
  u.layer = n / a.units_layer;
  const int r = n - u.layer * a.units_layer;
  u.b = find_segment(ct.cu_chunk, t.batch, r / per_chunk);
  const int c0 = ct.cu_chunk[u.b], r1 = r - c0 * per_chunk;
  u.n_chunks = ct.cu_chunk[u.b + 1] - c0;
  u.kvh = r1 / (u.n_chunks * a.n_qgroups);
  const int r2 = r1 - u.kvh * u.n_chunks * a.n_qgroups, c = r2 / a.n_qgroups;
  u.qgrp = r2 - c * a.n_qgroups;
  u.L = t.prompt_len[u.b];
  u.row_base = t.cu_rows[u.b];
  const int np1 = (u.L + a.n_pseudo + kPair - 1) / kPair;
  const int p1 = (int)((int64_t)np1 * (c + 1) / u.n_chunks);
  u.pair0 = (int)((int64_t)np1 * c / u.n_chunks);
  u.n_pairs = (u.kind == kSweep1 ? p1 : min(p1, (u.L + kPair - 1) / kPair)) - u.pair0;
  u.rows = min(a.rows_g, a.rows_total - u.qgrp * a.rows_g);
  u.qrow = ((u.layer * t.batch + u.b) * a.n_q_heads + u.kvh * a.group) * a.n_pseudo + u.qgrp * a.rows_g;
  u.first_chunk = u.layer * ct.n_chunks + c0;
  u.chunk = u.first_chunk + c;
  u.item = ((u.layer * t.batch + u.b) * a.n_kv_heads + u.kvh) * a.n_qgroups + u.qgrp;
}

// 32 key columns of an accumulator row into the row's sum (RowSum, score_qg_sweep1.cuh).
__device__ __forceinline__ void row_sum32(const uint32_t* v, RowSum& st) {
  const float* x = reinterpret_cast<const float*>(v);
  if (st.m - st.r < 100.f) {
    float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
      acc0 = __fadd2_rn(acc0, ex2_pair_mufu(make_float2(x[e], x[e + 1])));
      acc1 = __fadd2_rn(acc1, ex2_pair_mufu(make_float2(x[e + 2], x[e + 3])));
    }
    const float zj = (acc0.x + acc0.y) + (acc1.x + acc1.y);
    if (zj < 1e37f) {                                            // (false for inf and NaN too)
      st.z = fmaf(zj, st.sc, st.z);
      if (st.z > 1e30f) {                                        // keep z well inside the float range
        st.m += 64.f;
        st.z *= 0x1p-64f;
        st.sc *= 0x1p-64f;
      }
      return;
    }
  }
  // careful path: these columns' own maximum and sum (relative to r), merged into the row's
  float ml = x[0];
#pragma unroll
  for (int e = 1; e < 32; ++e) ml = fmaxf(ml, x[e]);
  if (ml > -CUDART_INF_F) {
    float zl = 0.f;
#pragma unroll
    for (int e = 0; e < 32; ++e) zl += ex2(x[e] - ml);
    const float2 mg = qg::merge_stats(make_float2(st.m, st.z), make_float2(st.r + ml, zl));
    st.m = mg.x;
    st.z = mg.y;
    st.sc = exp2f(st.r - st.m);
  }
}

__device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, long long limit) {
  return mbar_wait_limit(bar, parity, abort_flag, status, limit);
}
struct Waiter {
  volatile int* abort_flag;
  int* status;
  long long limit;
  __device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity) const {
    return mbar_try(bar, parity) || wait_slow(bar, parity, abort_flag, status, limit);
  }
  __device__ __forceinline__ bool aborting() const { return *abort_flag != 0; }
};

__device__ __forceinline__ void tma_load_3d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
      ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z), "l"(policy) : "memory");
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// A value as the MMAs subtract it: an fp16 pair.
__device__ __forceinline__ uint32_t half_pair(float v) {
  const __half hi = __float2half_rn(v), lo = __float2half_rn(v - __half2float(hi));
  return (uint32_t)__half_as_ushort(hi) | ((uint32_t)__half_as_ushort(lo) << 16);
}
__device__ __forceinline__ float half_pair_value(uint32_t w) {
  return __half2float(__ushort_as_half((uint16_t)(w & 0xffffu))) + __half2float(__ushort_as_half((uint16_t)(w >> 16)));
}

__device__ __noinline__ float merge_row(const float2* part, int64_t step, int n) {
  float2 s = make_float2(-CUDART_INF_F, 0.f);
#pragma unroll 1
  for (int c = 0; c < n; ++c) s = qg::merge_stats(s, __ldcg(part + c * step));
  return s.x + log2f(s.y);
}

// Base-2 log-sum-exps of four neighbouring query rows from the sums of the item's n runs, in order; l holds the rows' references
// as they were subtracted.  Written during this launch by other CTAs: read past L1.
__device__ __forceinline__ void merge_rows(const Args& a, int64_t at, int64_t step, int n, float (&l)[4]) {
  float z[4] = {0.f, 0.f, 0.f, 0.f};
  bool ordinary = true;
  for (int c0 = 0; c0 < n; c0 += 8) {
    float4 q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) q[u] = c0 + u < n ? __ldcg(reinterpret_cast<const float4*>(a.sums + at + (c0 + u) * step)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      ordinary = ordinary && q[u].x >= 0.f && q[u].y >= 0.f && q[u].z >= 0.f && q[u].w >= 0.f;
      z[0] += q[u].x; z[1] += q[u].y; z[2] += q[u].z; z[3] += q[u].w;
    }
  }
  if (ordinary) {
#pragma unroll
    for (int x = 0; x < 4; ++x) l[x] += log2f(z[x]);
    return;
  }
#pragma unroll
  for (int x = 0; x < 4; ++x) l[x] = merge_row(a.part + at + x, step, n);
}

constexpr int kMaxLayers = kFlowLayers;
struct KeyMaps { CUtensorMap m[kMaxLayers]; };

template <bool kTwo>
__global__ void __launch_bounds__(kThreads, 1)
flow_kernel(const __grid_constant__ KeyMaps tm_k, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ SeqTable t,
            const __grid_constant__ ChunkTable ct, const __grid_constant__ Args a) {
  extern __shared__ __align__(1024) uint8_t smem[];
  using S = Smem<kTwo>;
  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {                                           // (uniform over the CTA: nothing has been set up yet)
    if (threadIdx.x == 0) atomicOr(a.status, kStatusSmemAlign);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar0 = sbase + S::bars;
  auto bar = [&](int i) { return bar0 + 8u * i; };
  // ---- set-up, beside the end of the kernel before
  if (warp == 0) {
    for (int i = lane; i < S::n_bars; i += 32) mbar_init(bar(i), S::bar_count(i));
    if (lane == 0) *reinterpret_cast<volatile int*>(smem + S::abort_flag) = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  } else if (warp == 1) {                                        // tensor memory: all 512 columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sbase + S::tmem_ptr), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else if (warp >= kFirstEpi && warp < kSumWarp) {
    // the operand of ones: its two ones lie in both 16-byte halves of every row, so whichever way the 32-byte swizzle orders the
    // halves, the k-step adds exactly the hi + lo of the other operand's row
    sts128(sbase + S::ones + (threadIdx.x - kFirstEpi * 32) * 16, make_uint4(0x3c003c00u, 0u, 0u, 0u));
    static_assert(S::ones_bytes == kEpiWarps * 32 * 16, "");
    fence_proxy_async();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();                                                    // (queries, references and cleared counters: the rotation's)
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + S::tmem_ptr);
  const Waiter wt{reinterpret_cast<volatile int*>(smem + S::abort_flag), a.status, a.wait_limit};
  // Unit n for a role of one thread, or of whole warps (lane 0 reports the read).
  auto next_unit = [&](int n, Unit& u, bool whole_warp) -> bool {
    const int at = n % kUnitRing;
    const bool ok = wt.wait(bar(S::unit_full + at), (n / kUnitRing) & 1);
    if (whole_warp ? !__all_sync(0xffffffffu, ok) : !ok) return false;
    u = read_unit(smem, S::unit + at * (int)sizeof(Unit));
    if (whole_warp) __syncwarp();
    if (!whole_warp || lane == 0) mbar_arrive(bar(S::unit_empty + at));
    return u.kind != kEndUnit;
  };

  if (warp == 0) {
    // ================================================================================ keys, by TMA
    if (lane == 0) {
      int si = 0;                                                // sub-tiles issued
      uint64_t last_use;
      asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(last_use));
      bool ok = true;
      Unit u;
      for (int n = 0; ok && next_unit(n, u, false); ++n) {
        const CUtensorMap* map = &tm_k.m[u.layer];
#pragma unroll 1
        for (int j = 0; j < 2 * u.n_pairs; ++j, ++si) {
          const int s = si & 3;
          if (si >= kSubs) ok = wt.wait(bar(S::k_empty + s), ((si >> 2) - 1) & 1);
          if (!ok) break;
          const uint32_t dst = sbase + S::ring + (s >> 1) * kPairBytes + (s & 1) * kSubHalf;
          const int row = u.row_base + u.pair0 * kPair + j * kSub;
          mbar_expect_tx(bar(S::k_full + s), 2 * kSubHalf);
          if (u.kind == kSweep1) {
            tma_load_3d(dst, map, bar(S::k_full + s), 0, row, u.kvh);
            tma_load_3d(dst + kPairHalf, map, bar(S::k_full + s), 64, row, u.kvh);
          } else {
            // (nobody but the next query group, at once, and the compaction of the kept rows reads these keys again: L2 may drop them
            // first.  A plain policy for all groups but the last: +- 0.5 % on 448 to 1024 query rows, in bursts and over seconds)
            tma_load_3d_hint(dst, map, bar(S::k_full + s), 0, row, u.kvh, last_use);
            tma_load_3d_hint(dst + kPairHalf, map, bar(S::k_full + s), 64, row, u.kvh, last_use);
          }
        }
      }
      // every copy issued lands before this thread, and with it the CTA, returns
      for (int back = 1; back <= kSubs && back <= si; ++back) drain_wait(bar(S::k_full + ((si - back) & 3)), ((si - back) >> 2) & 1, kWaitLimit);
    }
  } else if (warp == 1) {
    // ================================================================================ MMAs
    if (lane == 0) {
      int si = 0, job = 0, q_loads = 0;
      bool ok = true;
      Unit u;
      const uint64_t qd = umma_desc(sbase), ones_d = umma_desc_rows32(sbase + S::ones);
      auto acc_free = [&] { return job < 2 || wt.wait(bar(S::acc_empty + (job & 1)), ((job >> 1) - 1) & 1); };
      for (int n = 0; ok && next_unit(n, u, false); ++n) {
        const uint64_t slab_d = umma_desc_rows32(sbase + S::slab + (n & 1) * S::slab_bytes);
        ok = wt.wait(bar(S::slab_full + (n & 1)), (n >> 1) & 1);
        if (ok && u.new_q) ok = wt.wait(bar(S::q_full), q_loads++ & 1);
        const int mb = kTwo ? (u.rows + 127) / 128 : 1, ncols = (u.rows + 15) & ~15;
        const uint32_t id1 = umma_idesc_f16(128, kPair), id2 = umma_idesc_f16(128, ncols);
#pragma unroll 1
        for (int p = 0; p < u.n_pairs && ok; ++p) {
          // (the next ticket is drawn when four pairs are left: late enough for a short launch's first units to go round the
          // CTAs, early enough for the next unit's keys and log-sum-exps)
          if (p == max(0, u.n_pairs - 4)) mbar_arrive(bar(S::go));
          const int s = si & 3;
          const uint64_t kd = umma_desc(sbase + S::ring + (s >> 1) * kPairBytes);
          const uint32_t ph = (si >> 2) & 1;
          if (u.kind == kSweep1) {
            ok = wt.wait(bar(S::k_conv + s), ph) && wt.wait(bar(S::k_conv + s + 1), ph);
#pragma unroll 1
            for (int m = 0; m < mb && ok; ++m, ++job) {
              if (!(ok = acc_free())) break;
              tc_fence_after();
              const uint32_t d = tmem + (job & 1) * 256;
#pragma unroll
              for (int ks = 0; ks < 8; ++ks) {
                const int half = ks >> 2, kk = ks & 3;
                umma_ss(d, desc_advance(qd, half * S::q_half + m * 128 * 128 + kk * 32), desc_advance(kd, half * kPairHalf + kk * 32), id1, ks ? 1u : 0u);
              }
              umma_ss(d, desc_advance(slab_d, m * 128 * 32), ones_d, id1, 1u);   // D[i, key] += (-r_i) * 1
              tc_commit(bar(S::acc_full + (job & 1)));
            }
            if (!ok) break;
            tc_commit(bar(S::k_empty + s));
            tc_commit(bar(S::k_empty + s + 1));
          } else {
#pragma unroll 1
            for (int j = 0; j < 2 && ok; ++j) {
              ok = wt.wait(bar(S::k_conv + s + j), ph);
              if (ok && (kTwo || j == 0)) ok = acc_free();
              if (!ok) break;
              tc_fence_after();
              const uint32_t d = tmem + (job & 1) * 256 + (kTwo ? 0 : j * 128);
              const uint64_t kj = desc_advance(kd, j * kSubHalf);
#pragma unroll
              for (int ks = 0; ks < 8; ++ks) {
                const int half = ks >> 2, kk = ks & 3;
                umma_ss(d, desc_advance(kj, half * kPairHalf + kk * 32), desc_advance(qd, half * S::q_half + kk * 32), id2, ks ? 1u : 0u);
              }
              umma_ss(d, ones_d, slab_d, id2, 1u);               // D[key, i] += 1 * (-lse_i)
              if (kTwo || j == 1) {
                tc_commit(bar(S::acc_full + (job & 1)));
                ++job;
              }
              tc_commit(bar(S::k_empty + s + j));
            }
          }
          si += 2;
        }
        if (ok) tc_commit(bar(S::slab_empty + (n & 1)));         // (and the queries are read)
      }
      // every MMA issued retires before tensor memory is given back
      tc_commit(bar(S::drain));
      drain_wait(bar(S::drain), 0, kWaitLimit);
    }
  } else if (warp < kFirstEpi) {
    // ================================================================================ keys from bf16 to fp16 in place
    const int cw = warp - 2;
    int si = 0;
    bool ok = true;
    Unit u;
    for (int n = 0; ok && next_unit(n, u, true); ++n) {
      for (int j = 0; j < 2 * u.n_pairs && ok; ++j, ++si) {
        const int s = si & 3;
        if (!__all_sync(0xffffffffu, wt.wait(bar(S::k_full + s), (si >> 2) & 1))) { ok = false; break; }
        // this warp: 64 channels of 64 keys
        const uint32_t p0 = sbase + S::ring + (s >> 1) * kPairBytes + (s & 1) * kSubHalf + (cw >> 1) * kPairHalf + (cw & 1) * (kSubHalf / 2) + lane * 16;
#pragma unroll 1
        for (int it = 0; it < 16; it += 8) {
          uint4 v[8];
#pragma unroll
          for (int x = 0; x < 8; ++x) v[x] = lds128(p0 + (it + x) * 512);
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            v[x].x = qg::bf16x2_to_f16x2(v[x].x);
            v[x].y = qg::bf16x2_to_f16x2(v[x].y);
            v[x].z = qg::bf16x2_to_f16x2(v[x].z);
            v[x].w = qg::bf16x2_to_f16x2(v[x].w);
            sts128(p0 + (it + x) * 512, v[x]);
          }
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(S::k_conv + s));
      }
    }
  } else if (warp < kSumWarp) {
    // ================================================================================ epilogue
    const int eg = (warp - kFirstEpi) >> 2;                      // epilogue group 0 .. 3: columns 64 eg .. 64 eg + 63 of an accumulator
    const int quad = warp & 3, r = quad * 32 + lane;             // tensor-memory lane of this thread
    const uint32_t lane_addr = tmem + ((uint32_t)(quad * 32) << 16);
    float* exch = reinterpret_cast<float*>(smem + S::exch);
    int job = 0, post = 0;
    bool ok = true;
    Unit u;
    auto take_job = [&](int b) { return __all_sync(0xffffffffu, wt.wait(bar(S::acc_full + b), (job >> 1) & 1)); };
    auto release = [&](int b) {                                  // the accumulator's columns are in registers
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(S::acc_empty + b));
    };
    auto slot_free = [&] { return post < kSlots || __all_sync(0xffffffffu, wt.wait(bar(S::part_empty + (post & 3)), ((post >> 2) - 1) & 1)); };
    for (int n = 0; ok && next_unit(n, u, true); ++n) {
      ok = __all_sync(0xffffffffu, wt.wait(bar(S::slab_full + (n & 1)), (n >> 1) & 1));
      if (!ok) break;
      if (u.kind == kSweep1) {
        const int mb = kTwo ? (u.rows + 127) / 128 : 1;
        // (the row of query block 0 and, kTwo, that of block 1: they change places after every job, so that there is one body)
        RowSum now, other;
        auto reference = [&](int row) {                          // as the MMAs see it
          return -half_pair_value(*reinterpret_cast<const volatile uint32_t*>(smem + S::slab + (n & 1) * S::slab_bytes + (row >> 3) * 256 + (row & 7) * 32));
        };
        now.init(reference(r));
        other.init(kTwo ? reference(128 + r) : 0.f);
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(S::slab_empty + (n & 1)));
        int i_now = (u.qgrp * a.rows_g + r) % a.n_pseudo, i_other = (u.qgrp * a.rows_g + 128 + r) % a.n_pseudo;
        auto change = [&] {
          const RowSum x = now;
          now = other;
          other = x;
          const int i = i_now;
          i_now = i_other;
          i_other = i;
        };
        int base = u.pair0 * kPair;
#pragma unroll 1
        for (int j = 0; j < u.n_pairs * mb; ++j, ++job) {
          const int b = job & 1;
          if (!(ok = take_job(b))) break;
          tc_fence_after();
          const uint32_t taddr = lane_addr + b * 256 + eg * 64;
#pragma unroll 1
          for (int h = 0; h < 2; ++h) {
            uint32_t v[32];
            tmem_ld32(taddr + h * 32, v);
            tmem_ld_wait_for(v);
            if (h == 1) release(b);
            if (base + kPair > u.L) {                            // holds synthetic (or foreign) rows
              const int last = u.L + i_now - base - eg * 64 - h * 32;   // visible columns: up to this one
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (e > last) v[e] = 0xff800000u;                // -inf
            }
            row_sum32(v, now);
          }
          if (kTwo && mb == 2) change();
          if (!kTwo || mb == 1 || (j & 1)) base += kPair;
        }
        // the four groups' sums of the same rows over different keys, 64 rows to a post; negative: not relative to the reference
#pragma unroll 1
        for (int h = 0; h < 2 * mb && ok; ++h, ++post) {
          if (!(ok = slot_free())) break;
          if ((quad >> 1) == (h & 1)) {
            const bool second = kTwo && h >= 2;
            const float m = second ? other.m : now.m, z = second ? other.z : now.z, ref = second ? other.r : now.r;
            reinterpret_cast<float2*>(exch + (post & 3) * 512)[eg * 64 + (r & 63)] = make_float2(m, m == ref ? z : -z);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(S::part_full + (post & 3)));
        }
      } else {
        if (lane == 0) mbar_arrive(bar(S::slab_empty + (n & 1)));
        // pieces of 16 query columns: kTwo: the four groups share out all of them; else two groups a sub-tile
        const int nch = (u.rows + 15) >> 4;
        const int part = kTwo ? eg : (eg & 1), parts = kTwo ? 4 : 2;
        const int p0 = (part * nch) / parts, np = ((part + 1) * nch) / parts - p0;
        const uint32_t col_addr = lane_addr + (kTwo ? 0 : (eg >> 1) * 128) + p0 * 16;
        const int cols = min(np * 16, u.rows - p0 * 16);         // this thread's columns
#pragma unroll 1
        for (int j = 0; j < (kTwo ? 2 : 1) * u.n_pairs; ++j, ++job, ++post) {
          const int b = job & 1;
          if (!(ok = take_job(b))) break;
          tc_fence_after();
          float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
          if (np == 0) release(b);
#pragma unroll 1
          for (int c = 0; c < cols; c += 32) {
            uint32_t v[32];
            tmem_ld16(col_addr + b * 256 + c, v);
            if (c + 16 < np * 16) tmem_ld16(col_addr + b * 256 + c + 16, v + 16);
            tmem_ld_wait_for(v);
            if (c + 32 >= cols) {
              release(b);
              if (c + 32 > cols) {
#pragma unroll
                for (int e = 0; e < 32; ++e)
                  if (c + e >= cols) v[e] = 0xff800000u;
              }
            }
            qg::colsum_piece<true, true>(v, nullptr, 16, 1.f, acc0, acc1);
            if (c + 16 < cols) qg::colsum_piece<true, true>(v + 16, nullptr, 16, 1.f, acc0, acc1);
          }
          if (!(ok = slot_free())) break;
          exch[(post & 3) * 512 + eg * 128 + r] = (acc0.x + acc0.y) + (acc1.x + acc1.y);
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(S::part_full + (post & 3)));
        }
      }
    }
  } else if (warp == kSumWarp) {
    // ================================================================================ what leaves the CTA
    const float* exch = reinterpret_cast<const float*>(smem + S::exch);
    int post = 0;
    bool ok = true;
    Unit u;
    auto take = [&] { return __all_sync(0xffffffffu, wt.wait(bar(S::part_full + (post & 3)), (post >> 2) & 1)); };
    auto give = [&] {
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(S::part_empty + (post & 3)));
    };
    for (int n = 0; ok && next_unit(n, u, true); ++n) {
      if (u.kind == kSweep1) {
        const int mb = kTwo ? (u.rows + 127) / 128 : 1;
        const int64_t out = ((int64_t)u.chunk * a.n_kv_heads + u.kvh) * a.rows_pad + u.qgrp * a.rows_g;
        for (int h = 0; h < 2 * mb; ++h, ++post) {
          if (!(ok = take())) break;
          const float2* e = reinterpret_cast<const float2*>(exch + (post & 3) * 512);
#pragma unroll 1
          for (int x = 0; x < 2; ++x) {
            const int row = x * 32 + lane;
            // (a fixed order: the result does not depend on timing)
            const float2 s0 = e[row], s1 = e[64 + row], s2 = e[2 * 64 + row], s3 = e[3 * 64 + row];
            const bool ordinary = s0.y >= 0.f && s1.y >= 0.f && s2.y >= 0.f && s3.y >= 0.f;
            float2 v = make_float2(s0.x, ((s3.y + s2.y) + s1.y) + s0.y);
            if (!ordinary) {
              v = qg::merge_stats(make_float2(s2.x, fabsf(s2.y)), make_float2(s3.x, fabsf(s3.y)));
              v = qg::merge_stats(make_float2(s1.x, fabsf(s1.y)), v);
              v = qg::merge_stats(make_float2(s0.x, fabsf(s0.y)), v);
            }
            if (h * 64 + row < u.rows) {
              __stcg(a.sums + out + h * 64 + row, ordinary ? v.y : -1.f);
              __stcg(a.part + out + h * 64 + row, v);
            }
          }
          give();
        }
        if (!ok) break;
        __threadfence();                                         // the partials are visible before the count
        __syncwarp();
        if (lane == 0) atomicAdd(a.sync + 1 + u.item, 1u);
      } else {
        float* out = a.scores + u.layer * a.layer_stride + u.qgrp * a.slot_stride + u.kvh * a.score_stride + t.cu_prompt[u.b];
        for (int j = 0; j < (kTwo ? 2 : 1) * u.n_pairs; ++j, ++post) {
          if (!(ok = take())) break;
          const float* e = exch + (post & 3) * 512;
          const int key0 = u.pair0 * kPair + j * (kTwo ? kSub : kPair);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int x = q * 32 + lane, key = key0 + x;
            if (kTwo) {
              if (key < u.L) out[key] = ((e[x] + e[128 + x]) + e[256 + x]) + e[384 + x];
            } else {
              if (key < u.L) out[key] = e[x] + e[128 + x];
              if (key + kSub < u.L) out[key + kSub] = e[256 + x] + e[384 + x];
            }
          }
          give();
        }
      }
    }
  } else {
    // ================================================================ tickets, queries and the extra operands
    int last_q = -1, q_loads = 0;
    for (int n = 0;; ++n) {
      bool ok = true;
      if (lane == 0) {
        ok = (n == 0 || wt.wait(bar(S::go), (n - 1) & 1)) && (n < kUnitRing || wt.wait(bar(S::unit_empty + n % kUnitRing), (n / kUnitRing - 1) & 1));
        if (ok) {
          Unit u = {};
          for (;;) {
            const uint32_t x = atomicAdd(a.sync, 1u);
            if (x >= 2u * (uint32_t)a.n_units) break;
            make_unit(u, (int)x, t, ct, a);
            if (u.n_pairs > 0) break;
            u.kind = kEndUnit;
          }
          u.new_q = u.kind != kEndUnit && u.qrow != last_q ? 1 : 0;
          int4* d = reinterpret_cast<int4*>(smem + S::unit + n % kUnitRing * (int)sizeof(Unit));
          const int4* src = reinterpret_cast<const int4*>(&u);
#pragma unroll
          for (int i = 0; i < (int)(sizeof(Unit) / 16); ++i) d[i] = src[i];
          mbar_arrive(bar(S::unit_full + n % kUnitRing));
        }
      }
      if (!__all_sync(0xffffffffu, ok)) break;
      __syncwarp();                                              // (a vote orders no memory: what lane 0 has announced)
      const Unit u = read_unit(smem, S::unit + n % kUnitRing * (int)sizeof(Unit));   // (stays until unit n + 2 is announced)
      if (u.kind == kEndUnit) break;
      last_q = u.qrow;
      // The unit's extra operand: row i holds minus the row's reference logit (sweep 1) or log-sum-exp (sweep 2) as an fp16 pair
      // in channels 0 and 1, zeros elsewhere and in the rows beyond the group.
      ok = n < 2 || __all_sync(0xffffffffu, wt.wait(bar(S::slab_empty + (n & 1)), ((n >> 1) - 1) & 1));
      if (ok && u.kind == kSweep2) {
        bool there = true;
        if (lane == 0) {
          const long long start = clock64();
          while (ld_acquire(a.sync + 1 + u.item) < (uint32_t)u.n_chunks) {
            if (wt.aborting()) { there = false; break; }
            if (clock64() - start > wt.limit) {
              *wt.abort_flag = 1;
              atomicOr(a.status, kStatusTimeout);
              there = false;
              break;
            }
          }
        }
        ok = __all_sync(0xffffffffu, there);
        __syncwarp();                                            // (lane 0 has acquired the row sums: for all lanes)
      }
      if (!ok) break;
#pragma unroll 1
      for (int row = 4 * lane; row < S::rows; row += 128) {
        float l[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) l[x] = row + x < u.rows ? __ldg(a.ref + u.qrow + row + x) : 0.f;
        if (u.kind == kSweep2 && row < u.rows) {
          const int64_t step = (int64_t)a.n_kv_heads * a.rows_pad;
#pragma unroll
          for (int x = 0; x < 4; ++x) l[x] = -half_pair_value(half_pair(-l[x]));
          merge_rows(a, u.first_chunk * step + u.kvh * a.rows_pad + u.qgrp * a.rows_g + row, step, u.n_chunks, l);
        }
        const uint32_t dst = sbase + S::slab + (n & 1) * S::slab_bytes + (row >> 3) * 256 + (row & 7) * 32;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          sts128(dst + x * 32, make_uint4(row + x < u.rows ? half_pair(-l[x]) : 0u, 0u, 0u, 0u));
          sts128(dst + x * 32 + 16, make_uint4(0u, 0u, 0u, 0u));
        }
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(S::slab_full + (n & 1)));
      if (u.new_q) {
        // (the queries of the unit before are read when its extra operand is given back)
        if (lane == 0) {
          ok = n == 0 || wt.wait(bar(S::slab_empty + ((n - 1) & 1)), ((n - 1) >> 1) & 1);
          if (ok) {
            const int mb = kTwo ? (u.rows + 127) / 128 : 1;
            mbar_expect_tx(bar(S::q_full), (uint32_t)mb * 2u * 128u * 128u);
            for (int half = 0; half < 2; ++half)
              for (int m = 0; m < mb; ++m) tma_load_2d(sbase + half * S::q_half + m * 128 * 128, &tm_q, bar(S::q_full), half * 64, u.qrow + m * 128);
            ++q_loads;
          }
        }
        if (!__all_sync(0xffffffffu, ok)) break;
      }
    }
    if (lane == 0 && q_loads) drain_wait(bar(S::q_full), (q_loads - 1) & 1, kWaitLimit);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

}  // namespace flow
}  // namespace dapq
