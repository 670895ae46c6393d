// The tensor-core scorer that loses nothing of 32-bit queries and keys (Section 4.2, Eq. 4); host side and
// the reasons for its shape in score_split.cu.
//
// Every fp32 number is the exact sum of three bf16 numbers (the nearest one, the one nearest to what is left, and the
// rest), and a product of two bf16 numbers is exact in fp32, so q.k is a short sum of bf16 MMAs:
//   bf16 keys   q0.k + q1.k + q2.k                                   (nothing left out)
//   fp32 keys   q0.k0 + (q1.k0 + q0.k1) + (q2.k0 + q1.k1 + q0.k2)
// What is left out for fp32 keys, q1.k2 + q2.k1 + q2.k2, is at most (2^-24 + 2^-34) |q||k|: |q1| <= 2^-8 |q| and
// |q2| <= 2^-17 |q| by rounding to nearest (truncated parts have the sign of their number and twice the size each: up to
// 2^-21 |q||k|, always of the product's own sign).  Its sign is either one, 0.05 * 2^-23 |q||k| in root mean square on
// N(0, 1) operands (truncated: 0.50), where one rounding of fp32 is 0.29 * 2^-23 of its result.
// The three parts of the R query rows are stacked along N ([q0; q1; q2], N = 3 R), so that one MMA per k-step
// multiplies all of them with a part of K.  D[key, query]: keys on tensor-memory lanes, and the products of one
// order of magnitude share R accumulator columns; the leading products, whose roundings are the ones that
// count, are kept in two halves (channels 0-63 and 64-127):
//   columns [0, R)   q0.k0 over channels 0-63      [3R, 4R)  q0.k0 over channels 64-127
//           [R, 2R)  the products of order 2^-8    [2R, 3R)  those of order 2^-16
// and the epilogue adds the four columns of a logit in fp32.  The queries are multiplied by softmax scale * log2(e) before
// they are split: what the epilogue adds up is the base-2 logit, the same number in both sweeps whatever its size (a
// product formed and rounded in one sweep and fused into the subtraction in the other differs by half an ulp of the logit,
// which an exponential of logits beyond 2^24 turns into any value).  Both sweeps use this layout:
//   sweep 1  a thread keeps a running maximum and sum for a quarter of the query columns over the keys of its
//            lane; the lanes are merged once, at the end of the CTA's chunk;
//   sweep 2  a thread sums its key's exponentials over all query columns: one score, no exchange.
#pragma once
#include "score_qg_common.cuh"

namespace dapq {
namespace split {

using namespace ptx;
using qg::Ring;
using qg::Waiter;

constexpr int kTile = 128;                     // keys per tile (tensor-memory lanes)
constexpr int kPart = kTile * 128;             // bytes of one bf16 part of a half tile (64 channels)
constexpr int kEpiWarps = 16, kConvWarps = 4;
constexpr int kQuarter = kTile * 128;           // bytes of a quarter of an fp32 tile (32 channels)
constexpr int kMaxRing = 6, kMaxStage = 6, kMaxSub = 2;
constexpr float kLowest = -1e38f;              // running maximum before the first key

template <int kKeyParts>
struct Roles {
  static constexpr bool f32 = kKeyParts == 3;
  static constexpr int first_epi = f32 ? 2 + kConvWarps : 2;
  static constexpr int threads = (first_epi + kEpiWarps) * 32;
  static constexpr int slot = f32 ? 3 * kPart : 2 * kPart;     // a ring slot: half a tile in three parts, or a whole bf16 tile
  // rows of a query sub-group in shared memory, in units of R: channels 0-63 of [q0; q1; q2], then channels 64-127
  // of [q0; q1; q2], with bf16 keys followed by q0 once more: [q1; q2; q0] is then one operand (one MMA less per
  // k-step).  fp32 keys need the room.
  static constexpr int q_units = f32 ? 6 : 7;
  static __host__ __device__ constexpr int query_bytes(int R) { return q_units * R * 128; }
};

// Shared memory: queries, K ring, fp32 staging slots, state.
struct State {                                 // offsets from the end of the staging slots
  static constexpr int k_full = 0, k_empty = k_full + 8 * kMaxRing, acc_full = k_empty + 8 * kMaxRing, acc_empty = acc_full + 8 * 8;
  static constexpr int st_full = acc_empty + 16, st_empty = st_full + 8 * kMaxStage, q_full = st_empty + 8 * kMaxStage, drain = q_full + 8;
  static constexpr int lse = (drain + 8 + 15) & ~15;                   // [128] floats: minus the base-2 lse (sweep 2)
  static constexpr int tmem_ptr = lse + kMaxSub * 64 * 4, abort_flag = tmem_ptr + 4;
  static constexpr int total = abort_flag + 4;
};

struct Args {
  const void* q;                 // [B, H_q, N, d] rotated queries
  int32_t q_bf16;                // the queries are bf16 in memory (else fp32)
  int32_t n_pseudo, group, n_q_heads, n_kv_heads, rows_total;
  int32_t n_qgroups, n_sub;      // CTAs that share a chunk; sub-groups of R rows per CTA (1 in sweep 1)
  int32_t rows_pad;              // row pitch of `part`
  int32_t n_ring, n_stage, state_off;   // ring slots, fp32 staging slots
  int32_t early_loads;           // keys may be read before the wait for the kernel before this one
  float scale_log2e;
  long long wait_limit;
  float2* part;                  // [chunks, H_kv, rows_pad] (maximum, sum) of sweep 1
  const float* lse_in;
  float* lse_out;
  float* scores;                 // [H_kv][score_stride], one slot per query group slot_stride apart
  int64_t score_stride, slot_stride;
  int* status;
};

// Two fp32 values -> their three bf16 parts, packed in pairs (lower half: a).
// kNearest (fp32 keys): values beyond the largest bf16 number keep it as their first part (the others hold the rest); an
// infinity ends up in the third part, and its products are infinite, of their sign, as in fp32.  Otherwise (bf16 keys:
// all products are formed) by truncation: the parts of a query have one sign, and an infinite key meets no
// infinities of both signs.  NaN stays NaN.
__device__ __forceinline__ uint32_t nearest_bf16x2(float a, float b) {
  uint32_t r;
  asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
  return r;
}
template <bool kNearest>
__device__ __forceinline__ void split2(float a, float b, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
  auto part = [](float x, float y) { return kNearest ? nearest_bf16x2(x, y) : __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632); };
  p0 = part(a, b);
  const float ra = a - __uint_as_float(p0 << 16), rb = b - __uint_as_float(p0 & 0xffff0000u);
  p1 = part(ra, rb);
  const float sa = ra - __uint_as_float(p1 << 16), sb = rb - __uint_as_float(p1 & 0xffff0000u);
  p2 = __byte_perm(__float_as_uint(sa), __float_as_uint(sb), 0x7632);   // (at most eight significant bits)
}
template <bool kNearest>
__device__ __forceinline__ void split8(const float4& x, const float4& y, uint4 (&p)[3]) {
  split2<kNearest>(x.x, x.y, p[0].x, p[1].x, p[2].x);
  split2<kNearest>(x.z, x.w, p[0].y, p[1].y, p[2].y);
  split2<kNearest>(y.x, y.y, p[0].z, p[1].z, p[2].z);
  split2<kNearest>(y.z, y.w, p[0].w, p[1].w, p[2].w);
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
}
// The four blocks of P columns from `taddr` on, summed: x[e] = the logit of column e.  `release` gives
// the accumulator back once its `last` columns are in registers.
template <int kR, int P, class Release>
__device__ __forceinline__ void load_logits(uint32_t taddr, float (&x)[P], bool last, Release release) {
  static_assert(P % 4 == 0, "");
  uint32_t v[P / 4][16];
#pragma unroll
  for (int q = 0; q < P / 4; ++q)
#pragma unroll
    for (int blk = 0; blk < 4; ++blk) tmem_ld4(taddr + blk * kR + q * 4, v[q] + blk * 4);
#pragma unroll
  for (int q = 0; q < P / 4; ++q) tmem_ld_wait_for16(v[q]);
  if (last) release();
#pragma unroll
  for (int q = 0; q < P / 4; ++q)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t* w = v[q] + e;
      x[q * 4 + e] = (__uint_as_float(w[0]) + __uint_as_float(w[12])) + (__uint_as_float(w[4]) + __uint_as_float(w[8]));
    }
}

__device__ __forceinline__ float4 as_float4(uint4 v) {
  return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}

// Two words of packed bf16 values as fp32.
__device__ __forceinline__ float4 from_bf16(uint32_t a, uint32_t b) {
  return as_float4(make_uint4(a << 16, a & 0xffff0000u, b << 16, b & 0xffff0000u));
}

// (maximum, sum of exp2) of two disjoint sets of logits -> of their union (either may be empty: sum 0).
__device__ __forceinline__ float2 merge2(float2 a, float2 b) {
  const float m = fmaxf(a.x, b.x);
  return make_float2(m, a.y * exp2f(a.x - m) + b.y * exp2f(b.x - m));
}

template <int kR, int kKeyParts, bool kSweep2>
__global__ void __launch_bounds__(Roles<kKeyParts>::threads, 1)
split_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ SeqTable t, const __grid_constant__ ChunkTable ct,
             const __grid_constant__ ChunkTable ct1, const Args a) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {                                          // (uniform over the CTA: nothing has been set up yet)
    if (threadIdx.x == 0) atomicOr(a.status, kStatusSmemAlign);
    return;
  }
  using Ro = Roles<kKeyParts>;
  constexpr bool kF32 = Ro::f32;
  constexpr int kAcc = 4 * kR;                                  // columns of an accumulator; two of them
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = blockIdx.x / a.n_qgroups, qgrp = blockIdx.x - chunk * a.n_qgroups, kvh = blockIdx.y;
  const int b = find_segment(ct.cu_chunk, t.batch, chunk);
  const int L = t.prompt_len[b], N = a.n_pseudo;
  const int n_keys = kSweep2 ? L : L + N;                       // keys that this sweep covers
  const int t0 = (chunk - ct.cu_chunk[b]) * ct.chunk_tiles;
  const int nt = min((n_keys + kTile - 1) / kTile, t0 + ct.chunk_tiles) - t0;
  if (nt <= 0) return;
  const int row0 = qgrp * a.n_sub * kR;                         // first query row (of the KV head) of this CTA
  const int n_sub = kSweep2 ? min(a.n_sub, (a.rows_total - row0 + kR - 1) / kR) : 1;
  const int rows = min(n_sub * kR, a.rows_total - row0);        // query rows of this CTA
  const int qrow_base = (b * a.n_q_heads + kvh * a.group) * N + row0;
  const uint32_t ring = sbase + a.n_sub * Ro::query_bytes(kR), staging = ring + a.n_ring * Ro::slot, st = sbase + a.state_off;
  uint8_t* stp = smem + a.state_off;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(stp + State::abort_flag);
  const Waiter wt{abort_flag, a.status, a.wait_limit};
  auto k_full = [&](int i) { return st + State::k_full + 8 * i; };
  auto k_empty = [&](int i) { return st + State::k_empty + 8 * i; };
  // Sweep 1: one per accumulator, every epilogue warp sees every phase.  Sweep 2: one per (epilogue group, sub-group),
  // so that a group, which takes every fourth tile only, sees every phase of its own barriers.
  auto acc_full = [&](int i) { return st + State::acc_full + 8 * i; };
  auto full_of = [&](int ti, int sub) { return acc_full(kSweep2 ? (ti & 3) * 2 + sub : ti & 1); };
  auto acc_empty = [&](int i) { return st + State::acc_empty + 8 * i; };
  const uint32_t q_full = st + State::q_full, drain = st + State::drain;
  const int S = a.n_ring;
  // Sweep 2 walks its chunk backwards: what sweep 1 read last is what the L2 cache still holds.
  auto tile_of = [&](int ti) { return t0 + (kSweep2 ? nt - 1 - ti : ti); };
  // The copies: whole bf16 tiles into the ring, quarters of fp32 tiles into the staging slots.
  const int n_in = kF32 ? a.n_stage : S, n_copies = kF32 ? 4 * nt : nt;
  auto in_full = [&](int i) { return kF32 ? st + State::st_full + 8 * i : k_full(i); };
  auto in_empty = [&](int i) { return kF32 ? st + State::st_empty + 8 * i : k_empty(i); };
  auto copy_in = [&](int u, int s) {
    const int row = t.cu_rows[b] + tile_of(kF32 ? u >> 2 : u) * kTile;
    if (kF32) {
      mbar_expect_tx(in_full(s), kQuarter);
      tma_load_3d(staging + s * kQuarter, &tm_k, in_full(s), (u & 3) * 32, row, kvh);
    } else {
      mbar_expect_tx(in_full(s), Ro::slot);
      tma_load_3d(ring + s * Ro::slot, &tm_k, in_full(s), 0, row, kvh);
      tma_load_3d(ring + s * Ro::slot + kPart, &tm_k, in_full(s), 64, row, kvh);
    }
  };

  // ---- prologue: barriers, the first K tiles, tensor memory
  const int n_pre = min(n_copies, n_in);
  if (warp == 0) {
    if (lane < S) {
      mbar_init(k_full(lane), kF32 ? kConvWarps : 1);
      mbar_init(k_empty(lane), 1);
    }
    if (kF32 && lane < n_in) {
      mbar_init(in_full(lane), 1);
      mbar_init(in_empty(lane), kConvWarps);
    }
    if (lane < 8) mbar_init(acc_full(lane), 1);
    if (lane < 2) mbar_init(acc_empty(lane), kSweep2 ? 4 : kEpiWarps);
    if (lane == 0) {
      mbar_init(q_full, kEpiWarps);
      mbar_init(drain, 1);
      *abort_flag = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    if (lane == 0 && a.early_loads)
      for (int u = 0; u < n_pre; ++u) copy_in(u, u);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(st + State::tmem_ptr), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(stp + State::tmem_ptr);

  if (warp == 0) {
    // ======================================================================================= TMA producer
    if (lane == 0) {
      if (!a.early_loads) {
        pdl_wait();
        for (int u = 0; u < n_pre; ++u) copy_in(u, u);
      }
      int u = n_pre;
      for (; u < n_copies; ++u) {
        if (!wt.wait(in_empty(u % n_in), ((u / n_in) - 1) & 1)) break;
        copy_in(u, u % n_in);
      }
      // see every copy land before the CTA returns
      for (int back = 1; back <= n_in && back <= u; ++back) drain_wait(in_full((u - back) % n_in), ((u - back) / n_in) & 1, kWaitLimit);
    }
  } else if (warp == 1) {
    // ========================================================================================= MMA issuer
    if (lane == 0) {
      constexpr uint32_t id1 = umma_idesc(128, kR), id2 = umma_idesc(128, 2 * kR), id3 = umma_idesc(128, 3 * kR);
      // the MMAs of half `h` of a tile (kd: its first part) for the sub-group whose queries of that half begin at qd
      auto half_mmas = [&](uint32_t d, uint64_t qd, int h, uint64_t kd) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const uint64_t k0 = desc_advance(kd, kk * 32), q0 = desc_advance(qd, kk * 32);
          if (h == 0) {
            umma_ss(d, k0, q0, id3, kk ? 1u : 0u);
          } else if (kF32 || kk == 0) {                         // (columns [3R, 4R) begin here, the others go on)
            umma_ss(d + kR, k0, desc_advance(q0, kR * 128), id2, 1u);
            umma_ss(d + 3 * kR, k0, q0, id1, kk ? 1u : 0u);
          } else {
            umma_ss(d + kR, k0, desc_advance(q0, kR * 128), id3, 1u);
          }
          if (kF32) {
            umma_ss(d + kR, desc_advance(k0, kPart), q0, id2, 1u);
            umma_ss(d + 2 * kR, desc_advance(k0, 2 * kPart), q0, id1, 1u);
          }
        }
      };
      bool ok = wt.wait(q_full, 0);
      tc_fence_after();
      const uint64_t qd = umma_desc(sbase);
      Ring rs(S), ra(2);
      for (int ti = 0; ti < nt && ok; ++ti) {
        if (kF32) {
          for (int h = 0; h < 2 && ok; ++h, rs.next()) {
            const int s = rs.i;
            ok = wt.wait(k_full(s), rs.phase);
            const uint64_t kd = umma_desc(ring + s * Ro::slot);
            for (int sub = 0; sub < n_sub && ok; ++sub) {
              const int job = ti * n_sub + sub, buf = job & 1;
              if (h == 0 && job >= 2) ok = wt.wait(acc_empty(buf), ((job >> 1) - 1) & 1);
              if (!ok) break;
              tc_fence_after();
              half_mmas(tmem_base + buf * kAcc, desc_advance(qd, sub * Ro::query_bytes(kR) + h * 3 * kR * 128), h, kd);
              if (h == 1) tc_commit(full_of(ti, sub));
            }
            if (!ok) break;
            tc_commit(k_empty(s));
          }
        } else {
          const int s = rs.i;
          ok = wt.wait(k_full(s), rs.phase);
          const uint64_t kd = umma_desc(ring + s * Ro::slot);
          for (int sub = 0; sub < n_sub && ok; ++sub) {
            const int job = ti * n_sub + sub, buf = job & 1;
            if (job >= 2) ok = wt.wait(acc_empty(buf), ((job >> 1) - 1) & 1);
            if (!ok) break;
            tc_fence_after();
            half_mmas(tmem_base + buf * kAcc, desc_advance(qd, sub * Ro::query_bytes(kR)), 0, kd);
            half_mmas(tmem_base + buf * kAcc, desc_advance(qd, sub * Ro::query_bytes(kR) + 3 * kR * 128), 1, desc_advance(kd, kPart));
            tc_commit(full_of(ti, sub));
          }
          if (!ok) break;
          tc_commit(k_empty(s));
          rs.next();
        }
      }
      tc_commit(drain);                                         // see every MMA retire before tensor memory is given back
      drain_wait(drain, 0, kWaitLimit);
    }
  } else if (warp < Ro::first_epi) {
    // ================================================= fp32 keys: quarters of a tile into three bf16 parts, half a tile per ring slot
    if (kF32) {
      // A round: 8 rows x 4 pieces of 8 channels per warp.  Eight neighbouring lanes take rows r and r ^ 5: with the
      // 128-byte swizzle on both sides, bit 0 of the row puts their loads, and bit 2 their stores, into different banks.
      // (Measured with four warps: 4700 cycles per tile when every quarter had its own fence and the staged rows were
      // not swizzled, against 2450 cycles of MMAs; one fence per half tile and no selects bring it below them.)
      const int cw = warp - 2, piece = lane & 3, r0 = cw * 32 + ((lane >> 3) ^ (lane & 4 ? 5 : 0)), sw = r0 & 7;
      Ring rp(S), ri(n_in);
      for (int u = 0; u < 2 * nt; ++u, rp.next()) {
        const int s = rp.i;
        bool ok = !rp.wrapped || wt.wait(k_empty(s), rp.phase ^ 1u);
        if (!__all_sync(0xffffffffu, ok)) break;
        const uint32_t dst = ring + s * Ro::slot + r0 * 128;
#pragma unroll
        for (int h = 0; h < 2; ++h, ri.next()) {
          ok = ok && __all_sync(0xffffffffu, wt.wait(in_full(ri.i), ri.phase));
          if (!ok) break;
          const uint32_t src = staging + ri.i * kQuarter + r0 * 128;
          uint4 x[4][2];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            x[i][0] = lds128(src + i * 1024 + (((2 * piece) ^ sw) << 4));
            x[i][1] = lds128(src + i * 1024 + (((2 * piece + 1) ^ sw) << 4));
          }
          const uint32_t at = dst + (((h * 4 + piece) ^ sw) << 4);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint4 p[3];
            split8<true>(as_float4(x[i][0]), as_float4(x[i][1]), p);
#pragma unroll
            for (int e = 0; e < 3; ++e) sts128(at + i * 1024 + e * kPart, p[e]);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(in_empty(ri.i));
        }
        if (!ok) break;
        fence_proxy_async();                                          // the MMAs read the parts through the async proxy
        __syncwarp();
        if (lane == 0) mbar_arrive(k_full(s));
      }
    }
  } else {
    // =========================================================================================== epilogue
    const int te = threadIdx.x - Ro::first_epi * 32;              // 0 .. 511
    const int eg = te >> 7, quad = warp & 3, r = quad * 32 + lane;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
    pdl_wait();                                                   // the rotation kernel (sweep 1) wrote the queries (partials)
    // (sweep 2 reads nothing that is not complete by now ahead of its own wait; its CTAs set up as this sweep's leave: 2 k
    // fp32 keys 24.0 -> 22.0 us a layer, 32 heads of 16 k bf16 keys 69.9 -> 68.0)
    if (!kSweep2) pdl_trigger();
    // ---- the CTA's queries, scaled, in three parts
    const float c = a.scale_log2e;
    auto scaled = [c](float4 v) { return make_float4(v.x * c, v.y * c, v.z * c, v.w * c); };
    for (int x = te; x < n_sub * kR * 16; x += kEpiWarps * 32) {
      const int row = x >> 4, ch = x & 15, sub = row / kR, rr = row - sub * kR, h = ch >> 3;
      uint4 p[3];
      const int64_t src_row = (int64_t)qrow_base + min(row, rows - 1);   // (rows that do not exist repeat the last one: zeros
                                                                         // would make NaN of an infinite key, here as in its sums)
      if (a.q_bf16) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(a.q) + src_row * 16 + ch);
        split8<kF32>(scaled(from_bf16(v.x, v.y)), scaled(from_bf16(v.z, v.w)), p);
      } else {
        const float4* src = reinterpret_cast<const float4*>(a.q) + src_row * 32 + ch * 2;
        split8<kF32>(scaled(__ldg(src)), scaled(__ldg(src + 1)), p);
      }
      const uint32_t at = sbase + sub * Ro::query_bytes(kR) + h * 3 * kR * 128 + rr * 128 + (((ch & 7) ^ (rr & 7)) << 4);
#pragma unroll
      for (int e = 0; e < 3; ++e) sts128(at + e * kR * 128, p[e]);
      if (h && !kF32) sts128(at + 3 * kR * 128, p[0]);
    }
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) mbar_arrive(q_full);

    if constexpr (!kSweep2) {
      constexpr int C = kR / 4, P = C % 8 == 0 ? 8 : 4;           // columns per thread, and per piece
      const int c0 = eg * C;
      float m[C], z[C];
#pragma unroll
      for (int e = 0; e < C; ++e) { m[e] = kLowest; z[e] = 0.f; }
      bool ok = true;
      Ring ra(2);
      for (int ti = 0; ti < nt && ok; ++ti, ra.next()) {
        ok = __all_sync(0xffffffffu, wt.wait(acc_full(ra.i), ra.phase));
        if (!ok) break;
        tc_fence_after();
        auto release = [&] {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty(ra.i));
        };
        const int beyond = tile_of(ti) * kTile + r - L;           // this thread's key is visible to pseudo query i iff beyond <= i
        const bool masked = (tile_of(ti) + 1) * kTile > L;
#pragma unroll
        for (int p = 0; p < C; p += P) {
          float x[P];
          load_logits<kR, P>(lane_addr + ra.i * kAcc + c0 + p, x, p + P == C, release);
#pragma unroll
          for (int e = 0; e < P; ++e) {
            float s = x[e];
            if (masked && beyond > (row0 + c0 + p + e) % N) s = -CUDART_INF_F;
            // one exponential per logit: the smaller of (logit, running maximum) against the larger
            const float dlt = s - m[p + e], f = ex2(-fabsf(dlt));
            const bool up = dlt > 0.f;
            z[p + e] = fmaf(z[p + e], up ? f : 1.f, up ? 1.f : f);
            m[p + e] = fmaxf(m[p + e], s);
          }
        }
      }
      // The lanes of a warp hold the same columns over different keys: halve the columns and exchange (fixed
      // order), then plain merges; then the four quadrants through shared memory.
      int col = c0;
      {
        int o = 16;
#pragma unroll
        for (int w = C; w > 1 && w % 2 == 0; w >>= 1) {
          const bool hi = (lane & o) != 0;
#pragma unroll
          for (int e = 0; e < w / 2; ++e) {
            const float2 keep = hi ? make_float2(m[e + w / 2], z[e + w / 2]) : make_float2(m[e], z[e]);
            const float2 give = hi ? make_float2(m[e], z[e]) : make_float2(m[e + w / 2], z[e + w / 2]);
            const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, give.x, o), __shfl_xor_sync(0xffffffffu, give.y, o));
            const float2 mg = hi ? merge2(got, keep) : merge2(keep, got);
            m[e] = mg.x;
            z[e] = mg.y;
          }
          if (hi) col += w / 2;
          o >>= 1;
        }
        constexpr int left = C % 3 == 0 ? 3 : 1;                  // columns per lane that the halving leaves
        for (; o > 0; o >>= 1) {
#pragma unroll
          for (int e = 0; e < left; ++e) {
            const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, m[e], o), __shfl_xor_sync(0xffffffffu, z[e], o));
            const float2 own = make_float2(m[e], z[e]);
            const float2 mg = (lane & o) ? merge2(got, own) : merge2(own, got);
            m[e] = mg.x;
            z[e] = mg.y;
          }
        }
        constexpr int mask = (C / left) == 1 ? 31 : 31 / (C / left);   // lanes that hold the same columns: one of them stores
        float2* red = reinterpret_cast<float2*>(smem + a.n_sub * Ro::query_bytes(kR));   // (the ring: every MMA that read it has retired)
        if ((lane & mask) == 0) {
#pragma unroll
          for (int e = 0; e < left; ++e) red[quad * 64 + col + e] = make_float2(m[e], z[e]);
        }
        epilogue_sync();
        if (te < rows) {
          float2 v = red[te];
#pragma unroll
          for (int q = 1; q < 4; ++q) v = merge2(v, red[q * 64 + te]);
          a.part[((int64_t)chunk * a.n_kv_heads + kvh) * a.rows_pad + row0 + te] = v;
        }
      }
    } else {
      // ---- base-2 log-sum-exp of the CTA's query rows: four threads per row merge sweep 1's partials
      float* lse_s = reinterpret_cast<float*>(stp + State::lse);
      {
        const int row = te >> 2, grow = row0 + row;
        float2 s = make_float2(kLowest, 0.f);
        if (row < rows && !a.lse_in) {
          const int c_end = ct1.cu_chunk[b + 1];
          const int64_t step = (int64_t)a.n_kv_heads * a.rows_pad;
          const float2* src = a.part + (int64_t)kvh * a.rows_pad + grow;
          for (int cc = ct1.cu_chunk[b] + (te & 3); cc < c_end; cc += 16) {
            float2 q[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) q[u] = cc + 4 * u < c_end ? __ldg(src + (cc + 4 * u) * step) : make_float2(kLowest, 0.f);
#pragma unroll
            for (int u = 0; u < 4; ++u) s = merge2(s, q[u]);
          }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, s.x, o), __shfl_xor_sync(0xffffffffu, s.y, o));
          s = (te & o) ? merge2(got, s) : merge2(s, got);
        }
        if ((te & 3) == 0) {
          float l2 = CUDART_INF_F;                                // rows that do not exist: 2^(x - inf) = 0
          if (row < rows) {
            l2 = a.lse_in ? a.lse_in[qrow_base + row] * 1.4426950408889634f : s.x + log2f(s.y);
            if (a.lse_out && chunk == ct.cu_chunk[b])
              a.lse_out[qrow_base + row] = a.lse_in ? a.lse_in[qrow_base + row] : l2 * 0.6931471805599453f;
          }
          lse_s[row] = -l2;
        }
        epilogue_sync();
      }
      // ---- epilogue group g takes the tiles g, g + 4, ...: a thread sums all query columns of its key
      float* out = a.scores + (int64_t)qgrp * a.slot_stride + (int64_t)kvh * a.score_stride + t.cu_prompt[b];
      bool ok = true;
      for (int ti = eg; ti < nt && ok; ti += 4) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int sub = 0; sub < n_sub && ok; ++sub) {
          const int job = ti * n_sub + sub, buf = job & 1;
          ok = __all_sync(0xffffffffu, wt.wait(full_of(ti, sub), (ti >> 2) & 1));
          if (!ok) break;
          tc_fence_after();
          auto release = [&] {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty(buf));
          };
#pragma unroll
          for (int p = 0; p < kR; p += 8) {
            float x[8];
            load_logits<kR, 8>(lane_addr + buf * kAcc + p, x, p + 8 == kR, release);
            const float4 l0 = *reinterpret_cast<const float4*>(lse_s + sub * kR + p), l1 = *reinterpret_cast<const float4*>(lse_s + sub * kR + p + 4);
            const float ls[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e & 3] += ex2(x[e] + ls[e]);
          }
        }
        if (!ok) break;
        const int j = tile_of(ti) * kTile + r;
        if (j < L) out[j] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

}  // namespace split
}  // namespace dapq
