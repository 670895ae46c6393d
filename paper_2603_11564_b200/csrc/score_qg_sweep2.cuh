// Sweep 2 of the tensor-core scorer (Section 4.2, Eq. 4): S(j) = sum_i exp(s_ij - lse_i),
// summed over the N pseudo queries and the G query heads of the KV head's group.
//
//   D[key, query] = K_tile Q_grp^T, keys on tensor-memory lanes, up to 256 query columns.
// CTA = (chunk of K tiles, query group, KV head): a KV head with more than 512 query rows is cut into
// groups of equal size (a CTA keeps up to 512 rows resident and then runs two jobs per K tile), each scored by a CTA of its own against the same K chunk (the CTAs of a chunk
// are neighbours in the grid, run at the same time and find each other's K tiles in L2, so K crosses
// DRAM once); the groups' scores go to separate slots that a small kernel sums in fixed order.
// A job is one [128 keys x <= 256 queries] accumulator (two fit; four of 128 columns for small groups).
// All four epilogue groups work on every job, a quarter of the query columns each, and give the
// accumulator back as soon as their columns are in registers.  No epilogue warp waits for another one:
// a warp posts its 32 partial sums into a ring of kExchDepth slots in shared memory and goes on to the
// next job; one more warp sums the four groups' entries (fixed order) and stores the keys' scores, one
// coalesced fp32 per lane.  Before the first job the epilogue threads merge the per-chunk partials of
// sweep 1 into the base-2 log-sum-exp of the resident query rows.
#pragma once
#include "score_qg_common.cuh"

namespace dapq {
namespace qg {

// 16 accumulator columns of one key row: sum of 2^(s c - lse) over the columns, as two packed pairs.
// kFull: all 16 columns exist (no per-column test).  kFold: the accumulator already holds s c - lse (the
// queries were scaled before the MMAs and -lse was added by the job's last k-step).
template <bool kFull, bool kFold>
__device__ __forceinline__ void colsum_piece(const uint32_t* v, const float* lse16, int valid, float c, float2& acc, float2& acc1) {
  if (kFull) {
    const float2 c2 = make_float2(c, c);
#pragma unroll
    for (int e = 0; e < 16; e += 4) {
      float2 x0, x1;
      if (kFold) {
        x0 = make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1]));
        x1 = make_float2(__uint_as_float(v[e + 2]), __uint_as_float(v[e + 3]));
      } else {
        const float4 l4 = *reinterpret_cast<const float4*>(lse16 + e);
        x0 = __ffma2_rn(make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), c2, make_float2(l4.x, l4.y));
        x1 = __ffma2_rn(make_float2(__uint_as_float(v[e + 2]), __uint_as_float(v[e + 3])), c2, make_float2(l4.z, l4.w));
      }
      acc = __fadd2_rn(acc, ((kPolyPairMask >> (e / 2)) & 1u) ? ex2_pair_poly(x0) : ex2_pair_mufu(x0));
      acc1 = __fadd2_rn(acc1, ((kPolyPairMask >> (e / 2 + 1)) & 1u) ? ex2_pair_poly(x1) : ex2_pair_mufu(x1));
    }
  } else {
#pragma unroll
    for (int e = 0; e < 16; ++e)
      if (e < valid) acc.x += kFold ? ex2(__uint_as_float(v[e])) : ex2(fmaf(__uint_as_float(v[e]), c, lse16[e]));
  }
}

// This warp's pieces [p0, p0 + np) of one accumulator (np <= 4), two at a time; `release` gives the
// accumulator back once the last piece is in registers.  kFull: every column of these pieces exists.
template <bool kFull, bool kFold, class Release>
__device__ __forceinline__ float colsum_job(uint32_t taddr, const float* lse_s, int p0, int np, int rows, float c, Release release) {
  float2 acc = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
  if (np == 0) release();
#pragma unroll
  for (int k = 0; k < 4; k += 2) {
    if (k < np) {
      const int ch = p0 + k;
      const int valid = rows - ch * 16;                         // >= 16 except in the last piece
      if (k + 1 < np) {
        uint32_t v[32];
        tmem_ld16(taddr + ch * 16, v);
        tmem_ld16(taddr + ch * 16 + 16, v + 16);
        tmem_ld_wait_for(v);
        if (k + 2 >= np) release();
        colsum_piece<kFull, kFold>(v, lse_s + ch * 16, valid, c, acc, acc1);
        colsum_piece<kFull, kFold>(v + 16, lse_s + ch * 16 + 16, valid - 16, c, acc, acc1);
      } else {
        uint32_t v[16];
        tmem_ld16(taddr + ch * 16, v);
        tmem_ld_wait_for16(v);
        release();
        colsum_piece<kFull, kFold>(v, lse_s + ch * 16, valid, c, acc, acc1);
      }
    }
  }
  return (acc.x + acc.y) + (acc1.x + acc1.y);
}

// Forms of sweep 2.
//   kPlain   every key of the CTA's chunk, rows' log-sum-exp from sweep 1's partials;
//   kOnePass (score_prune.cu) the log-sum-exp is an estimate from a sample of the keys.  Every exponential is added
//            twice: to its key's sum and to its query's, so that one pass yields the exact log-sum-exp and the scores up
//            to the estimates' errors;
//   kGather  the keys of a candidate list instead of a chunk; rows' log-sum-exp from the one-pass sweep's partials.  On
//            the full route: every key, log-sum-exp from sweep 1's, like kPlain.
//            A list of most of the prompt gives way to the whole prompt, whose tiles come in larger pieces (a listed tile
//            takes about 0.85 us to gather, a job of 256 query rows 1.1).
enum : int { kPlain = 0, kOnePass = 1, kGather = 2 };
template <int kForm> struct Layout2 {
  // (kOnePass: its epilogue keeps 64 sums per thread and takes registers from the other roles; that works on whole
  // groups of four warps)
  static constexpr int first_epi = kForm == kOnePass ? 8 : kFirstEpiWarp, sum_warp = kForm == kOnePass ? 6 : kFirstEpiWarp + 4 * kEpiGroups;
  static constexpr int threads = kForm == kOnePass ? kThreadsOne : kThreads2;
};
// Chunks behind the partials that a form merges; kGather: of the one-pass sweep, and of sweep 1 on the full route.
struct ChunkTables2 { ChunkTable pruned, full; };
template <int kForm> struct Chunks1 { using type = ChunkTable; };
template <> struct Chunks1<kGather> { using type = ChunkTables2; };
template <int kForm>
__device__ __forceinline__ const ChunkTable& chunks1(const typename Chunks1<kForm>::type& c, bool pruned) {
  if constexpr (kForm == kGather) return pruned ? c.pruned : c.full;
  else return c;
}

// One 16-column piece of the one-pass sweep: exponentials into the key's sum and into the columns' sums.
__device__ __forceinline__ void both_sums_piece(const uint32_t* v, float2* z, float2& acc, float2& acc1) {
#pragma unroll
  for (int e = 0; e < 16; e += 4) {
    const float2 e0 = ex2_pair_mufu(make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])));
    const float2 e1 = ex2_pair_mufu(make_float2(__uint_as_float(v[e + 2]), __uint_as_float(v[e + 3])));
    z[e / 2] = __fadd2_rn(z[e / 2], e0);
    z[e / 2 + 1] = __fadd2_rn(z[e / 2 + 1], e1);
    acc = __fadd2_rn(acc, e0);
    acc1 = __fadd2_rn(acc1, e1);
  }
}
// At the end of a sequence or of the query rows: column e counts if it is one of `valid` columns and the key, `beyond`
// rows behind the prompt, is visible to its pseudo query (index (i0 + e) mod n).
__device__ __forceinline__ void mask_piece(uint32_t* v, int valid, int beyond, int i0, int n) {
  int i = i0 % n;
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    if (e >= valid || beyond > i) v[e] = 0xff800000u;           // -inf (the prompt's keys have beyond < 0)
    i = i + 1 == n ? 0 : i + 1;
  }
}

// Sum and maximum of a query row over the keys [j0, j1) of a sequence with a running maximum: what the one-pass sweep
// does over again for a row whose sum has left the float range (an estimate that missed a key 2^120 above it).
// All 512 epilogue threads; the result is valid in thread 0.
__device__ __forceinline__ float2 careful_row(const Args& a, uint32_t q_row, uint32_t q_half, int row7, const __nv_bfloat16* k, int j0, int j1,
                                              int limit, float2* red, int te) {
  float m = -1e38f, z = 0.f;
  for (int j = j0 + te; j < j1 && j <= limit; j += kEpiThreads) {
    const uint4* kr = reinterpret_cast<const uint4*>(k + (int64_t)j * a.k_row_stride);
    float s = 0.f;
#pragma unroll 1
    for (int p = 0; p < 16; ++p) {
      const uint4 kv = __ldg(kr + p), qv = lds128(q_row + (p >> 3) * q_half + (((p & 7) ^ row7) << 4));
      const uint32_t kw[4] = {kv.x, kv.y, kv.z, kv.w}, qw[4] = {qv.x, qv.y, qv.z, qv.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t kh = bf16x2_to_f16x2(kw[e]);
        const float2 kf = __half22float2(*reinterpret_cast<const __half2*>(&kh)), qf = __half22float2(*reinterpret_cast<const __half2*>(&qw[e]));
        s = fmaf(qf.x, kf.x, s);
        s = fmaf(qf.y, kf.y, s);
      }
    }
    const float d = s - m, f = exp2f(-fabsf(d));
    z = d > 0.f ? fmaf(z, f, 1.f) : z + f;
    m = fmaxf(m, s);
  }
  float2 v = make_float2(m, z);
  auto merge = [](float2 x, float2 y) {
    const float mm = fmaxf(x.x, y.x);
    return make_float2(mm, x.y * exp2f(x.x - mm) + y.y * exp2f(y.x - mm));
  };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = merge(v, make_float2(__shfl_down_sync(0xffffffffu, v.x, o), __shfl_down_sync(0xffffffffu, v.y, o)));
  if ((te & 31) == 0) red[te >> 5] = v;
  epilogue_sync();
  if (te == 0)
    for (int w = 1; w < 4 * kEpiGroups; ++w) v = merge(v, red[w]);
  epilogue_sync();
  return v;
}

// The one-pass form's epilogue loop and the merge of its row sums.  kPieces: pieces of 16 query columns per thread (2 for
// groups of up to 128 rows, else 4).  sums: [rows] floats of this CTA's own (the lse merge is done with them).
template <int kPieces>
__device__ __forceinline__ void one_pass_epilogue(const Args& a, const Work& w, const Bars& bars, const Waiter& wt, int L, int nt, int kvh,
                                                  uint32_t sbase, uint32_t lane_addr, int acc_cols, int n_acc, int p0, int np, bool full,
                                                  int eg, int quad, int lane, float* lse_s, float* sums, float* exch, uint32_t q_half) {
  const int r = quad * 32 + lane, N = a.n_pseudo, col0 = p0 * 16;
  float2 z[8 * kPieces];                                        // this thread's columns over the keys of its lane
#pragma unroll
  for (int e = 0; e < 8 * kPieces; ++e) z[e] = make_float2(0.f, 0.f);
  bool ok = true;
  Ring ra(n_acc);
  for (int ti = 0; ti < nt && ok; ++ti, ra.next()) {
    const int buf = ra.i;
    ok = __all_sync(0xffffffffu, wt.wait(bars.acc_full(buf), ra.phase));
    if (!ok) break;
    tc_fence_after();
    const uint32_t taddr = lane_addr + buf * acc_cols + col0;
    const int beyond = (w.t0 + ti) * kTile2 + r - L;            // >= 0: a synthetic (or foreign) row
    const bool edge = !full || (w.t0 + ti + 1) * kTile2 > L;
    float2 acc = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
    auto release = [&] {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bars.acc_empty(buf));
    };
    if (np == 0) release();
    if (kPieces == 2) {
      if (np == 2) {
        uint32_t v[32];
        tmem_ld16(taddr, v);
        tmem_ld16(taddr + 16, v + 16);
        tmem_ld_wait_for(v);
        release();
        if (edge) {
          mask_piece(v, w.rows - col0, beyond, w.qgrp * a.rows_g + col0, N);
          mask_piece(v + 16, w.rows - col0 - 16, beyond, w.qgrp * a.rows_g + col0 + 16, N);
        }
        both_sums_piece(v, z, acc, acc1);
        both_sums_piece(v + 16, z + 8, acc, acc1);
      } else if (np == 1) {
        uint32_t v[16];
        tmem_ld16(taddr, v);
        tmem_ld_wait_for16(v);
        release();
        if (edge) mask_piece(v, w.rows - col0, beyond, w.qgrp * a.rows_g + col0, N);
        both_sums_piece(v, z, acc, acc1);
      }
    } else {
#pragma unroll
      for (int k = 0; k < kPieces; ++k) {
        if (k < np) {
          uint32_t v[16];
          tmem_ld16(taddr + k * 16, v);
          tmem_ld_wait_for16(v);
          if (k + 1 == np) release();
          if (edge) mask_piece(v, w.rows - col0 - k * 16, beyond, w.qgrp * a.rows_g + col0 + k * 16, N);
          both_sums_piece(v, z + k * 8, acc, acc1);
        }
      }
    }
    const int slot = ti % kExchDepth;
    if (ti >= kExchDepth) ok = __all_sync(0xffffffffu, wt.wait(bars.part_empty(slot), ((ti / kExchDepth) - 1) & 1));
    if (!ok) break;
    exch[(slot * kEpiGroups + eg) * 128 + r] = (acc.x + acc.y) + (acc1.x + acc1.y);
    __syncwarp();
    if (lane == 0) mbar_arrive(bars.part_full(slot));           // (release: the stores above are visible to the waiter)
  }
  // Row sums: the 32 lanes of a warp hold the same columns over different keys; halve the columns and exchange (fixed
  // order): every lane ends with one pair of columns, pair `c` (two lanes with the same pair if there are 16 pairs).
  int c = 0;
  if (kPieces == 2) {
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      z[e].x += __shfl_xor_sync(0xffffffffu, z[e].x, 1);
      z[e].y += __shfl_xor_sync(0xffffffffu, z[e].y, 1);
    }
  }
#pragma unroll
  for (int o = 16, n = 4 * kPieces; n > 0; o >>= 1, n >>= 1) {   // n column pairs stay
    const bool hi = (lane & o) != 0;
#pragma unroll
    for (int e = 0; e < n; ++e) {
      const float2 give = hi ? z[e] : z[e + n], keep = hi ? z[e + n] : z[e];
      const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, give.x, o), __shfl_xor_sync(0xffffffffu, give.y, o));
      z[e] = make_float2(keep.x + got.x, keep.y + got.y);
    }
    if (hi) c += n;
  }
  // The four quadrants through shared memory (the ring behind the queries: every MMA that read it has retired, unless a
  // wait ran out: then copies and conversions may still land there, and what is read back is as undefined as the results).
  // No decision that a barrier hangs on comes from the ring: whether a row is done over again is agreed on by all
  // epilogue threads at once, never in a CTA one of whose epilogue warps gave up (the others' waits are over by then),
  // and which rows from `sums`, which no other role writes.
  float* red = reinterpret_cast<float*>(__cvta_shared_to_generic(sbase + 2 * q_half));   // [4][256], then the scratch of careful_row
  if (c * 2 < np * 16) *reinterpret_cast<float2*>(red + quad * 256 + col0 + c * 2) = z[0];
  const int te = eg * 128 + r;
  const bool gave_up = epilogue_any(wt.aborting());
  float sum = 0.f;
  if (te < w.rows) {
    sum = (red[te] + red[256 + te]) + (red[512 + te] + red[768 + te]);
    sums[te] = sum;
    float2* out = a.part_out + ((int64_t)w.chunk * a.n_kv_heads + kvh) * a.rows_pad + w.qgrp * a.rows_g;
    out[te] = make_float2(lse_s[te], sum);
  }
  const bool again = epilogue_any(!(sum < 1e37f));              // (inf and NaN too)
  if (again && !gave_up) {
    const __nv_bfloat16* k = reinterpret_cast<const __nv_bfloat16*>(a.k) + (int64_t)kvh * a.k_head_stride + (int64_t)w.row_base * a.k_row_stride;
    float2* out = a.part_out + ((int64_t)w.chunk * a.n_kv_heads + kvh) * a.rows_pad + w.qgrp * a.rows_g;
    const int j0 = w.t0 * kTile2, j1 = j0 + nt * kTile2;
    for (int row = 0; row < w.rows; ++row) {
      if (sums[row] < 1e37f) continue;
      const float2 v = careful_row(a, sbase + (row >> 7) * 128 * 128 + (row & 127) * 128, q_half, row & 7, k, j0, j1,
                                   L + (w.qgrp * a.rows_g + row) % N, reinterpret_cast<float2*>(red + 4 * 256), te);
      if (te == 0) out[row] = v;
    }
  }
}

// The K tiles of a candidate list, to shared memory and from bf16 to fp16 there (kConvWarps warps).  The rows lie
// anywhere, so these warps copy them themselves, 16 bytes per lane, asynchronously and up to S tiles ahead, into the
// layout that a TMA box would have left; a lane converts what it has copied.  (Single rows by TMA gather took 75
// cycles per 128 bytes.)  Slots beyond the list take its last row: nobody stores their scores.
__device__ __forceinline__ void gather_tiles(const Work& w, const Args& a, int n_cand, const int32_t* cand, int kvh, uint32_t sbase,
                                             const Bars& bars, int cw, const Waiter& wt) {
  using T = TileGeo<kTile2>;
  const int lane = threadIdx.x & 31, S = a.n_stages, piece = lane & 15, r0 = cw * 32 + (lane >> 4);
  const uint32_t ring = sbase + (uint32_t)w.mb * 2u * 128u * 128u + (piece >> 3) * T::kHalf + r0 * 128;
  const __nv_bfloat16* kb = reinterpret_cast<const __nv_bfloat16*>(a.k) + (int64_t)kvh * a.k_head_stride + (int64_t)w.row_base * a.k_row_stride + piece * 8;
  // (row r0 + 2 i of the tile: its 16-byte pieces are permuted by the row's lowest three bits)
  auto slot_at = [&](int s, int i) { return ring + s * T::kStage + i * 256 + (((piece & 7) ^ ((r0 + 2 * i) & 7)) << 4); };
  auto issue = [&](int ti) {
    if (ti < w.nt) {
      const int own = __ldg(cand + min((w.t0 + ti) * kTile2 + cw * 32 + lane, n_cand - 1));
#pragma unroll
      for (int i = 0; i < 16; ++i)
        cp_async16(slot_at(ti % S, i), kb + (int64_t)__shfl_sync(0xffffffffu, own, 2 * i + (lane >> 4)) * a.k_row_stride);
    }
    cp_async_commit();
  };
  for (int ti = 0; ti < S; ++ti) issue(ti);
  for (int ti = 0; ti < w.nt; ++ti) {
    // tile ti has landed: S + ti - 1 groups have been committed by now (S before the first tile)
    if (S == 2) cp_async_wait<0>(); else if (S == 3) cp_async_wait<1>(); else cp_async_wait<2>();
    __syncwarp();
#pragma unroll
    for (int i0 = 0; i0 < 16; i0 += 4) {
      uint4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = lds128(slot_at(ti % S, i0 + u));
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        v[u].x = bf16x2_to_f16x2(v[u].x);
        v[u].y = bf16x2_to_f16x2(v[u].y);
        v[u].z = bf16x2_to_f16x2(v[u].z);
        v[u].w = bf16x2_to_f16x2(v[u].w);
        sts128(slot_at(ti % S, i0 + u), v[u]);
      }
    }
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) mbar_arrive(bars.k_conv(ti % S));
    if (ti >= 1 && ti - 1 + S < w.nt) {                         // the slot of the tile before is free once its MMAs have retired
      if (!__all_sync(0xffffffffu, wt.wait(bars.k_empty((ti - 1) % S), ((ti - 1) / S) & 1))) break;
    }
    if (ti >= 1) issue(ti - 1 + S);
  }
  cp_async_wait<0>();                                           // (no copy in flight when the CTA returns)
}

// kNarrow (kOnePass): groups of up to 128 query rows.  kWide: the CTA keeps up to 512 query rows resident and runs two jobs per K tile (query columns 0..255 and
// 256..); a thread adds its two jobs' sums before it posts them, so a tile is fetched, converted and stored once
// for twice the queries.
template <bool kConvert, bool kWide, int kForm = kPlain, bool kNarrow = false>
__global__ void __launch_bounds__(Layout2<kForm>::threads, 1)
colsum_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_q,
              const __grid_constant__ SeqTable t, const __grid_constant__ ChunkTable ct,
              const __grid_constant__ typename Chunks1<kForm>::type ct1s, const Args a) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {                                          // (uniform over the CTA: nothing has been set up yet)
    if (threadIdx.x == 0) atomicOr(a.status, kStatusSmemAlign);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  using T = TileGeo<kTile2>;
  constexpr bool kFold = kConvert;                              // the library's own fp16 queries arrive scaled: -lse rides on the MMAs
  static_assert(kForm == kPlain || (kConvert && (kForm == kGather || !kWide)), "");
  using Lay = Layout2<kForm>;
  constexpr int kFirstEpi = Lay::first_epi;
  const int kvh = blockIdx.y;
  Work w;
  int n_cand = 0;                                               // kGather: candidates of this (sequence, head)
  bool listed = kForm == kGather;                               // ... and whether the tiles are made of them
  bool pruned = true;                                           // this layer's route
  float credit = 0.f;
  if constexpr (kForm == kOnePass) {
    credit = route_of(a.route_in, a.most);
    pruned = credit >= 0.f;
  }
  if constexpr (kForm == kGather) {
    pruned = route_of(a.route_in, a.most) >= 0.f;
    if (pruned) pdl_wait();                                     // (the full route: set-up and first copies beside sweep 1's end)
    const int cta = blockIdx.x / a.n_qgroups;
    w.qgrp = blockIdx.x - cta * a.n_qgroups;
    w.b = find_segment(ct.cu_chunk, t.batch, cta);
    w.chunk = cta - ct.cu_chunk[w.b];
    const int n_ctas = ct.cu_chunk[w.b + 1] - ct.cu_chunk[w.b];
    w.L = t.prompt_len[w.b];
    n_cand = pruned ? (int)a.hist[(w.b * a.n_kv_heads + kvh) * kPruneHist + kPruneBins] : w.L;
    if (pruned && n_cand == t.cu_keep[w.b + 1] - t.cu_keep[w.b]) return;   // as many as are kept: they need no scores
    listed = kWide ? 8 * (int64_t)n_cand <= 7 * (int64_t)w.L : 3 * (int64_t)n_cand <= 2 * (int64_t)w.L;
    const int n_tiles = ((listed ? n_cand : w.L) + kTile2 - 1) / kTile2, per = (n_tiles + n_ctas - 1) / n_ctas;
    w.t0 = w.chunk * per;
    w.nt = min(per, n_tiles - w.t0);
    w.row_base = t.cu_rows[w.b];
    w.qrow_base = (w.b * a.n_q_heads + kvh * a.group) * a.n_pseudo;
    w.rows = min(a.rows_g, a.rows_total - w.qgrp * a.rows_g);
    w.mb = (w.rows + 127) / 128;
  } else {
    w = cta_work(t, ct, a, blockIdx.x, kvh, kTile2, kForm == kOnePass);
  }
  const int nt = w.nt, L = w.L, b = w.b;
  if constexpr (kForm == kOnePass) {
    if (!pruned) {                                              // nothing to do; the next layer goes the same way
      pdl_trigger();
      if (wait_in_one_cta() && threadIdx.x == 0) *a.route_out = {credit, a.most};
      return;
    }
  }
  if (nt <= 0) return;
  const ChunkTable& ct1 = chunks1<kForm>(ct1s, pruned);
  using Smem = SmemT<kWide>;
  const Bars bars{sbase + Smem::bars};
  const Waiter wt{reinterpret_cast<volatile int*>(smem + Smem::abort_flag), a.status, a.wait_limit};
  float* lse_s = reinterpret_cast<float*>(smem + Smem::lse);    // [rows] minus the base-2 lse of the resident query rows
  float* aux = reinterpret_cast<float*>(smem + Smem::aux);      // [rows] scratch of the lse merge
  float* exch = reinterpret_cast<float*>(smem + Smem::exch);    // [kExchDepth][4][128] partial sums on their way to the summing warp
  // The epilogue threads ask for sweep 1's partials of their query row first of all, before the CTA's copies of
  // queries and keys crowd the memory system (two threads per row: thread (eg, r) takes row (eg & 1) * 128 + r and
  // the chunks of parity eg >> 1; up to 16 partials per thread at once.  kWide: one thread per row, every chunk).
  const bool is_epi = warp >= kFirstEpi && warp < kFirstEpi + 4 * kEpiGroups;
  const int m_eg = (warp - kFirstEpi) >> 2, m_row = (kWide ? m_eg : (m_eg & 1)) * 128 + (warp & 3) * 32 + lane;
  constexpr int m_cs = kWide ? 1 : 2;                           // chunk stride of a thread
  const int m_c0 = kWide ? 0 : (m_eg >> 1);                     // its first chunk
  const bool m_live = is_epi && m_row < w.rows && !a.lse_in;
  const int m_nc = ct1.cu_chunk[b + 1] - ct1.cu_chunk[b];
  const int64_t m_step = (int64_t)a.n_kv_heads * a.rows_pad;
  const float2* m_p = (pruned ? a.part : a.part_full) + ((int64_t)ct1.cu_chunk[b] * a.n_kv_heads + kvh) * a.rows_pad + w.qgrp * a.rows_g + m_row;
  float2 m_q[16];
  float m_first = 0.f;                                          // kOnePass: the row's logit against the first key
  if (m_live) {
    pdl_wait();                                                 // (sweep 1 wrote them)
    if (kForm == kOnePass) m_first = __ldg(a.ref + w.qrow_base + w.qgrp * a.rows_g + m_row);
    if (kForm != kOnePass)                                      // (the sample's partials are few: read where they are merged)
#pragma unroll
    for (int u = 0; u < 16; ++u)
      m_q[u] = m_c0 + m_cs * u < m_nc ? __ldg(m_p + (m_c0 + m_cs * u) * m_step) : make_float2(-CUDART_INF_F, 0.f);
  }
  // (behind this library's own sweep 1 or rotation kernel, keys and queries were complete before that kernel
  // got past its wait: both go out at once)
  const uint32_t tmem_base = cta_prologue<Smem>(smem, sbase, bars, [&] {
    if (listed) tma_queries(&tm_q, w, a, sbase, bars);
    else if (a.early_loads) tma_first<kTile2, true>(&tm_k, &tm_q, w, a, sbase, bars, kvh);
  });
  // UMMA N: only the query columns that exist; job 1 (kWide) holds the rows from 256 on
  const int ncols = (min(w.rows, kGroupRows) + 15) & ~15, ncols1 = kWide ? ((max(w.rows - kGroupRows, 0) + 15) & ~15) : 0;
  const int n_jobs = ncols1 > 0 ? 2 : 1;                        // jobs per K tile
  const int acc_cols = ncols > 128 ? 256 : 128, n_acc = kTmemCols / acc_cols;
  const uint32_t q_half = (uint32_t)w.mb * 128u * 128u;         // bytes of one 64-channel half of the query group
  const int S = a.n_stages;

  if (is_epi) {
    // (kOnePass keeps 64 column sums per epilogue thread: 4 * 104 + 2 * 32 registers per lane of an SM sub-partition,
    // the 6 * 80 of the launch)
    if constexpr (kForm == kOnePass && !kNarrow) asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    // ============================================================================== epilogue
    const int eg = (warp - kFirstEpi) >> 2;                 // epilogue group 0 .. 3
    const int quad = warp & 3;                                  // TMEM lane quadrant of this warp
    const int r = quad * 32 + lane;                             // accumulator row (key) of this thread
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
    const float c = a.scale_log2e;
    // ---- base-2 log-sum-exp of the group's rows.  Two threads per row: thread (eg, r) merges the per-chunk
    // partials of row (eg & 1) * 128 + r over the chunks of parity eg >> 1, all of its loads in flight at
    // once; the odd half then crosses through shared memory and the even half finishes (fixed order).
    {
      const int row = m_row, grow = w.qgrp * a.rows_g + row;
      const bool live = row < w.rows;
      float mx = -CUDART_INF_F, z = 0.f;
      if (m_live) {
        for (int c0 = m_c0; c0 < m_nc; c0 += 16 * m_cs) {
          if (kForm == kOnePass || c0 > m_c0) {                                      // (more chunks than one batch of 16 per thread)
#pragma unroll
            for (int u = 0; u < 16; ++u)
              m_q[u] = c0 + m_cs * u < m_nc ? __ldg(m_p + (c0 + m_cs * u) * m_step) : make_float2(-CUDART_INF_F, 0.f);
          }
          float m16 = m_q[0].x;
#pragma unroll
          for (int u = 1; u < 16; ++u) m16 = fmaxf(m16, m_q[u].x);
          if (m16 > mx) {
            z *= exp2f(mx - m16);                               // exp2f(-inf) = 0 on the first round
            mx = m16;
          }
          if (mx > -CUDART_INF_F) {
#pragma unroll
            for (int u = 0; u < 16; ++u) z += m_q[u].y * exp2f(m_q[u].x - mx);
          }
        }
      }
      if (!kWide && eg >= 2) {
        aux[row] = mx;
        lse_s[row] = z;                                         // (the odd half's sums, until the even half has read them)
      }
      epilogue_sync();
      if (kWide || eg < 2) {
        float l2 = 0.f;
        if (live) {
          if (a.lse_in) {
            l2 = a.lse_in[w.qrow_base + grow] * 1.4426950408889634f;
          } else if (kWide) {
            l2 = mx + log2f(z);
          } else {
            const float mo = aux[row], zo = lse_s[row];
            const float m = fmaxf(mx, mo);
            l2 = m + log2f(z * exp2f(mx - m) + zo * exp2f(mo - m));
          }
          if (kForm == kOnePass) {
            // the estimate: the sample's sum times its stride, and the first key, which is not in the sample and may hold
            // most of a row's mass (its logit is the rotation's reference; it counts in full even where the sample's
            // logits, taken relative to it, have all underflowed)
            l2 += a.log2_sample;
            const float first = m_first, m = fmaxf(l2, first);
            l2 = m + log2f(exp2f(l2 - m) + exp2f(first - m));
          }
          if (kForm == kPlain && a.lse_out && w.chunk == ct.cu_chunk[b]) a.lse_out[w.qrow_base + grow] = l2 * 0.6931471805599453f;
        }
        lse_s[row] = -l2;                                       // negated: the epilogue adds it
        float seen = l2;                                        // the value that the MMAs subtract
        if (kFold) {
          // row `row` of the [256 x 16] operand: (-lse) as an fp16 pair in channels 0 and 1, zeros elsewhere.
          // The ones operand carries its two ones in BOTH 16-byte halves of every row, so whichever way the
          // 32-byte swizzle orders the halves of a row, the k-step adds exactly hi + lo.
          const __half hi = __float2half_rn(-l2);
          const __half lo = __float2half_rn(live ? -l2 - __half2float(hi) : 0.f);
          seen = -(__half2float(hi) + __half2float(lo));
          const uint32_t pair = (uint32_t)__half_as_ushort(hi) | ((uint32_t)__half_as_ushort(lo) << 16);
          const uint32_t dst = sbase + Smem::lse_slab + (row >> 3) * 256 + (row & 7) * 32;
          sts128(dst, make_uint4(live ? pair : 0u, 0u, 0u, 0u));
          sts128(dst + 16, make_uint4(0u, 0u, 0u, 0u));
        }
        if constexpr (kForm == kOnePass) {
          lse_s[row] = seen;                                      // (base of the row's sums, for the partials)
          if (live && w.chunk == ct.cu_chunk[b]) a.ref_out[w.qrow_base + grow] = seen;
        }
      }
      if (kForm == kOnePass && blockIdx.x == 0 && blockIdx.y == 0 && warp == kFirstEpi && lane == 0) *a.route_out = {credit, 0.f};
      if (kForm == kOnePass && w.qgrp == 0 && w.chunk == ct.cu_chunk[b]) {
        uint32_t* hist = a.hist + (int64_t)(b * a.n_kv_heads + kvh) * kPruneHist;
        for (int x = (warp - kFirstEpi) * 32 + lane; x < kPruneHist; x += kEpiThreads) hist[x] = 0u;
      }
      if (kFold) {
        const int tid_e = (warp - kFirstEpi) * 32 + lane;   // 0 .. 511: the ones operand, 256 pieces of 16 bytes
        if (tid_e < kOnesSlabBytes / 16) sts128(sbase + Smem::ones_slab + tid_e * 16, make_uint4(0x3c003c00u, 0u, 0u, 0u));
        fence_proxy_async();                                    // the MMAs read both operands through the async proxy
      }
      epilogue_sync();
      if (warp == kFirstEpi && lane == 0) mbar_arrive(bars.lse_ready());    // (the MMA issuer and the TMA producer wait for it)
    }
    // Pieces of a job (16 query columns): group g takes pieces [g nch / 4, (g + 1) nch / 4), at most four
    const int nch = ncols >> 4, nch1 = ncols1 >> 4;
    const int p0 = (eg * nch) / kEpiGroups, np = ((eg + 1) * nch) / kEpiGroups - p0;
    const int p1 = (eg * nch1) / kEpiGroups, np1 = ((eg + 1) * nch1) / kEpiGroups - p1;
    const bool full = (p0 + np) * 16 <= min(w.rows, kGroupRows);    // no column of this warp's pieces lies beyond the group
    const bool full1 = (p1 + np1) * 16 <= w.rows - kGroupRows;
    if constexpr (kForm == kOnePass) {
      one_pass_epilogue<(kForm == kOnePass && kNarrow) ? 2 : 4>(a, w, bars, wt, L, nt, kvh, sbase, lane_addr, acc_cols, n_acc, p0, np, full, eg, quad, lane, lse_s, aux, exch, q_half);
    } else {
      bool ok = true;
      Ring ra(n_acc);
      for (int ti = 0; ti < nt && ok; ++ti) {
        float sum = 0.f;
        for (int jb = 0; jb < n_jobs && ok; ++jb, ra.next()) {
          const int buf = ra.i;
          ok = __all_sync(0xffffffffu, wt.wait(bars.acc_full(buf), ra.phase));
          if (!ok) break;
          tc_fence_after();
          const uint32_t taddr = lane_addr + buf * acc_cols;
          // the accumulator goes back to the MMA issuer as soon as this warp's last piece is in registers
          auto release = [&] {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bars.acc_empty(buf));
          };
          if (jb == 0)
            sum = full ? colsum_job<true, kFold>(taddr, lse_s, p0, np, min(w.rows, kGroupRows), c, release)
                       : colsum_job<false, kFold>(taddr, lse_s, p0, np, min(w.rows, kGroupRows), c, release);
          else
            sum += full1 ? colsum_job<true, kFold>(taddr, lse_s + kGroupRows, p1, np1, w.rows - kGroupRows, c, release)
                         : colsum_job<false, kFold>(taddr, lse_s + kGroupRows, p1, np1, w.rows - kGroupRows, c, release);
        }
        if (!ok) break;
        const int slot = ti % kExchDepth;
        if (ti >= kExchDepth) ok = __all_sync(0xffffffffu, wt.wait(bars.part_empty(slot), ((ti / kExchDepth) - 1) & 1));
        if (!ok) break;
        exch[(slot * kEpiGroups + eg) * 128 + r] = sum;
        __syncwarp();
        if (lane == 0) mbar_arrive(bars.part_full(slot));         // (release: the stores above are visible to the waiter)
      }
    }
  } else {
    if constexpr (kForm == kOnePass && !kNarrow) asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (warp == 0) {
      if (lane == 0) {
        if (listed) {
          drain_wait(bars.q_full(), 0, kWaitLimit);             // (the only TMA copy of this form has landed)
        } else {
          if (!a.early_loads) tma_first<kTile2, true>(&tm_k, &tm_q, w, a, sbase, bars, kvh);
          tma_producer<kTile2, false, true>(&tm_k, &tm_q, w, a, sbase, bars, kvh, wt);
        }
      }
    } else if (warp == 1) {
      // ============================================================================= MMA issuer
      if (lane == 0) {
        bool ok = wt.wait(bars.q_full(), 0);
        if (ok && kFold) ok = wt.wait(bars.lse_ready(), 0);
        const uint32_t idesc = kConvert ? umma_idesc_f16(128, ncols) : umma_idesc(128, ncols);
        const uint32_t idesc1 = ncols1 ? (kConvert ? umma_idesc_f16(128, ncols1) : umma_idesc(128, ncols1)) : 0u;
        const uint64_t qd = umma_desc(sbase);
        const uint64_t ones_d = umma_desc_rows32(sbase + Smem::ones_slab), lse_d = umma_desc_rows32(sbase + Smem::lse_slab);
        const uint32_t ring = sbase + 2 * q_half;
        Ring rs(S), ra(n_acc);
        for (int ti = 0; ti < nt && ok; ++ti, rs.next()) {
          const int s = rs.i;
          ok = wt.wait(kConvert ? bars.k_conv(s) : bars.k_full(s), rs.phase);
          const uint64_t kd = umma_desc(ring + s * T::kStage);
          for (int jb = 0; jb < n_jobs && ok; ++jb, ra.next()) {
            const int buf = ra.i;
            if (ra.wrapped) ok = wt.wait(bars.acc_empty(buf), ra.phase ^ 1u);
            if (!ok) break;
            tc_fence_after();
            const uint32_t d = tmem_base + buf * acc_cols;
            const uint64_t qj = desc_advance(qd, jb * 2 * 128 * 128);          // query rows 256 jb ..: blocks 2 jb, 2 jb + 1
            const uint32_t id = jb ? idesc1 : idesc;
  #pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
              const int half = ks >> 2, kk = ks & 3;
              umma_ss(d, desc_advance(kd, half * T::kHalf + kk * 32), desc_advance(qj, half * q_half + kk * 32), id, ks ? 1u : 0u);
            }
            // D[key, i] += 1 * (-lse_i) (an fp16 pair against two ones)
            if (kFold) umma_ss(d, ones_d, desc_advance(lse_d, jb * kGroupRows * 32), id, 1u);
            tc_commit(bars.acc_full(buf));
          }
          if (!ok) break;
          tc_commit(bars.k_empty(s));                             // the K stage is free once these MMAs retire
        }
        mma_drain(bars);
      }
    } else if (warp < 2 + kConvWarps) {
      if (listed)
        gather_tiles(w, a, n_cand, a.cand + (int64_t)kvh * a.score_stride + t.cu_prompt[b], kvh, sbase, bars, warp - 2, wt);
      else if (kConvert) convert_tiles<kTile2>(w, a, sbase, bars, warp - 2, wt);
    } else if (warp == Lay::sum_warp) {
      // ====================================================================== sum of the four groups
      const int per_cta = kForm == kOnePass ? a.sum_groups : 1;   // sums that leave the CTA: groups 0..3, 0-1 and 2-3, or all
      float* out = a.scores + (int64_t)w.qgrp * per_cta * a.slot_stride + (int64_t)kvh * a.score_stride + t.cu_prompt[b];
      const int32_t* cand = kForm == kGather ? a.cand + (int64_t)kvh * a.score_stride + t.cu_prompt[b] : nullptr;
      for (int ti = 0; ti < nt; ++ti) {
        const int slot = ti % kExchDepth;
        if (!__all_sync(0xffffffffu, wt.wait(bars.part_full(slot), (ti / kExchDepth) & 1))) break;
        const float* e = exch + slot * kEpiGroups * 128;
  #pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int r = q * 32 + lane;
          if (listed) {
            const int c = (w.t0 + ti) * kTile2 + r;
            const float v = ((e[r] + e[128 + r]) + e[256 + r]) + e[384 + r];
            if (c < n_cand) out[cand[c]] = v;
          } else {
            const int j = (w.t0 + ti) * kTile2 + r;               // sequence-local key position
            if (j < L) {
              if (per_cta == 1) {
                out[j] = ((e[r] + e[128 + r]) + e[256 + r]) + e[384 + r];
              } else if (per_cta == 2) {
                out[j] = e[r] + e[128 + r];
                out[a.slot_stride + j] = e[256 + r] + e[384 + r];
              } else {
  #pragma unroll
                for (int g = 0; g < 4; ++g) out[g * a.slot_stride + j] = e[g * 128 + r];
              }
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bars.part_empty(slot));
      }
    }
  }
  cta_epilogue(tmem_base);
}

}  // namespace qg
}  // namespace dapq
