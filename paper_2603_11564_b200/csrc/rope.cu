// Rotation of the pseudo queries to their decode positions (Section 4.1: the N synthetic
// tokens take positions L_p .. L_p+N-1, so their queries carry the positional encodings of
// the first N decoding steps).
//
// Grid (pseudo queries i, layer and sequence b, block of query heads); thread (c, hy) owns the channel
// pair of frequency c of one head: (c, c + d/2), or (2c, 2c + 1) for the interleaved layout.  The angle pos * theta_c is formed and reduced in double
// precision: at positions near 131k a float angle has only ~7 fractional bits, which alone
// would cost half of the scorer's error budget.  The 64 angles of a query are evaluated once per block of heads.  The
// kernel is bound by the latency of its loads, angles and stores, block by block: batches take four queries per block
// (40 prompts of 8 k, 32 heads, 32 queries: 31 -> 23 us a layer).
#include <cuda_fp16.h>

#include "dapq_internal.cuh"

namespace dapq {
namespace {

constexpr int kHeadsPerBlock = 8;

template <typename T> __device__ __forceinline__ double to_double(T x);
template <> __device__ __forceinline__ double to_double<float>(float x) { return (double)x; }
template <> __device__ __forceinline__ double to_double<__nv_bfloat16>(__nv_bfloat16 x) {
  return (double)__bfloat162float(x);
}
template <> __device__ __forceinline__ double to_double<__half>(__half x) { return (double)__half2float(x); }
template <typename T> __device__ __forceinline__ T from_double(double x);
template <> __device__ __forceinline__ float from_double<float>(double x) { return (float)x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_double<__nv_bfloat16>(double x) {
  return __double2bfloat16(x);
}
// fp16 output (the query operand of the fp16 MMAs, stored times softmax scale * log2(e) so that the MMAs yield
// base-2 logits): values beyond the format's range saturate
template <> __device__ __forceinline__ __half from_double<__half>(double x) {
  return __double2half(fmin(fmax(x, -65504.0), 65504.0));
}

// kSplit: TO is bf16 and the rounding residual is stored as a second bf16 lo_offset elements on.
// rb.ref (optional, bf16 caches): also the logit of every rotated query against the FIRST key of its
// sequence, ref[layer, b, h, i] = out_scale * q_rot . K[h / G, cu_rows[b], :]: the first sweep of the
// tensor-core scorer measures every other logit of the row against it.
// kQ: consecutive pseudo queries per block.
// kLayers: 1, or up to kFlowLayers of them.
template <typename T, typename TO, bool kSplit, int kQ, int kLayers>
__global__ void __launch_bounds__(kHeadDim / 2 * kHeadsPerBlock)
rope_pseudo_q_kernel(const __grid_constant__ RopeLayers<kLayers> rb, TO* __restrict__ q_rot,
                     const double* __restrict__ inv_freq, const __grid_constant__ SeqTable t,
                     int n_q_heads, int n_pseudo, int64_t lo_offset, int late_wait,
                     int interleaved, double out_scale) {
  // late_wait: the kernel before this one in the stream neither writes q_pre nor still reads q_rot
  // (it is the compaction of the layer before), so the rotation runs beside it; the wait at the end
  // keeps this grid, and with it everything launched after it, ordered behind that kernel.
  // (the trigger comes behind the wait: the first sweep reads keys ahead of its own wait, so it may not start before
  // whatever wrote them has completed.  With late_wait the keys were complete before an earlier layer's rotation got past
  // its wait.)
  if (!late_wait) pdl_wait();
  pdl_trigger();
  const int layer = kLayers == 1 ? 0 : blockIdx.y / t.batch, b = blockIdx.y - layer * t.batch;
  const int i0 = blockIdx.x * kQ, c = threadIdx.x;
  // (the counters of the scorer behind this kernel; their last user completed before the kernel before this one could begin)
  for (int i = ((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * blockDim.x * blockDim.y + threadIdx.y * blockDim.x + c;
       kLayers > 1 && i < rb.n_clear; i += gridDim.x * gridDim.y * gridDim.z * blockDim.x * blockDim.y)
    rb.clear[i] = 0u;
  const T* __restrict__ q_pre = reinterpret_cast<const T*>(rb.q[layer]);
  const int h = blockIdx.z * kHeadsPerBlock + threadIdx.y, n = min(kQ, n_pseudo - i0);
  const bool active = h < n_q_heads;
  constexpr int half = kHeadDim / 2;
  static_assert(kQ <= kHeadsPerBlock, "row y of the block evaluates the angles of query y");
  const int c0 = interleaved ? 2 * c : c, c1 = interleaved ? 2 * c + 1 : c + half;
  const size_t base = (((size_t)b * n_q_heads + h) * n_pseudo + i0) * kHeadDim;         // of a layer's queries
  const size_t row0 = ((size_t)blockIdx.y * n_q_heads + h) * n_pseudo + i0, out = row0 * kHeadDim;
  double lo[kQ], hi[kQ];
#pragma unroll
  for (int u = 0; u < kQ; ++u) {
    lo[u] = hi[u] = 0.0;
    if (active && u < n) {
      lo[u] = to_double<T>(q_pre[base + u * kHeadDim + c0]);
      hi[u] = to_double<T>(q_pre[base + u * kHeadDim + c1]);
    }
  }
  __shared__ double2 angle[kQ][half];
  if (threadIdx.y < kQ) {
    double sn, cs;
    sincos((double)(t.pos_start[b] + i0 + (int)threadIdx.y) * inv_freq[c], &sn, &cs);
    angle[threadIdx.y][c] = make_double2(sn, cs);
  }
  float key0 = 0.f, key1 = 0.f;
  if (active && rb.ref != nullptr) {
    const __nv_bfloat16* k0 = rb.k[layer] + (int64_t)(h / rb.group) * rb.head_stride[layer] + (int64_t)t.cu_rows[b] * rb.row_stride[layer];
    key0 = __bfloat162float(k0[c0]);
    key1 = __bfloat162float(k0[c1]);
  }
  __syncthreads();
  float part[kQ];
#pragma unroll
  for (int u = 0; u < kQ; ++u) {
    const double sn = angle[u][c].x, cs = angle[u][c].y;
    const double r0 = (lo[u] * cs - hi[u] * sn) * out_scale, r1 = (hi[u] * cs + lo[u] * sn) * out_scale;
    part[u] = (float)r0 * key0 + (float)r1 * key1;
    if (active && u < n) {
      const size_t e0 = out + u * kHeadDim + c0, e1 = out + u * kHeadDim + c1;
      const TO h0 = from_double<TO>(r0), h1 = from_double<TO>(r1);
      q_rot[e0] = h0;
      q_rot[e1] = h1;
      if (kSplit) {
        q_rot[lo_offset + e0] = from_double<TO>(r0 - to_double<TO>(h0));
        q_rot[lo_offset + e1] = from_double<TO>(r1 - to_double<TO>(h1));
      }
    }
  }
  if (rb.ref != nullptr) {                                      // (uniform over the grid)
    __shared__ float red[kHeadsPerBlock][kQ][2];
#pragma unroll
    for (int u = 0; u < kQ; ++u) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) part[u] += __shfl_xor_sync(0xffffffffu, part[u], o);
      if ((c & 31) == 0) red[threadIdx.y][u][c >> 5] = part[u];   // the 64 threads of a head are two whole warps
    }
    __syncthreads();
    if (active && c < n) rb.ref[row0 + c] = red[threadIdx.y][c][0] + red[threadIdx.y][c][1];
  }
  if (late_wait) pdl_wait();
}

// The same for many queries (bf16 in, fp16 out): a warp per query head, a lane the channel pairs 2 l, 2 l + 1 of either half, so
// that a row moves in four-byte pieces, and a block evaluates the angles of its kRowsQ queries once for all heads.  The next head's
// rows are requested before this one's are computed.  Two layers of 40 prompts of 8 k, 32 heads, 32 queries: 37 -> 23 us,
// of which some 6 are double-precision arithmetic.
constexpr int kRowsQ = 4, kRowsWarps = 8;
__global__ void __launch_bounds__(kRowsWarps * 32)
rope_rows_kernel(const __grid_constant__ RopeBatch rb, __half2* __restrict__ q_rot, const double* __restrict__ inv_freq,
                 const __grid_constant__ SeqTable t, int n_q_heads, int n_pseudo, int late_wait, int interleaved, double out_scale) {
  if (!late_wait) pdl_wait();                                    // (as above)
  pdl_trigger();
  constexpr int half = kHeadDim / 2;
  const int layer = blockIdx.y / t.batch, b = blockIdx.y - layer * t.batch, i0 = blockIdx.x * kRowsQ;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n = min(kRowsQ, n_pseudo - i0);
  for (int i = (blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x; i < rb.n_clear; i += gridDim.x * gridDim.y * blockDim.x)
    rb.clear[i] = 0u;
  const __nv_bfloat162* q_pre = reinterpret_cast<const __nv_bfloat162*>(rb.q[layer]);
  const __nv_bfloat162* key = reinterpret_cast<const __nv_bfloat162*>(rb.k[layer] + (int64_t)t.cu_rows[b] * rb.row_stride[layer]);
  const int64_t key_step = rb.head_stride[layer] / 2;
  const size_t in_seq = (size_t)b * n_q_heads, out_seq = (size_t)blockIdx.y * n_q_heads;
  __nv_bfloat162 x[kRowsQ], y[kRowsQ], kx, ky;
  auto load = [&](int h) {
    const size_t row = ((in_seq + h) * n_pseudo + i0) * half;
#pragma unroll
    for (int u = 0; u < kRowsQ; ++u) {
      const size_t at = row + (size_t)min(u, n - 1) * half + lane;
      x[u] = q_pre[at];
      y[u] = q_pre[at + half / 2];
    }
    kx = key[(h / rb.group) * key_step + lane];
    ky = key[(h / rb.group) * key_step + half / 2 + lane];
  };
  if (warp < n_q_heads) load(warp);
  __shared__ double2 angle[kRowsQ][half];
  static_assert(kRowsQ * half == kRowsWarps * 32, "an angle per thread");
  {
    const int u = threadIdx.x / half, c = threadIdx.x % half;
    double sn, cs;
    sincos((double)(t.pos_start[b] + i0 + u) * inv_freq[c], &sn, &cs);
    angle[u][c] = make_double2(sn, cs);
  }
  __syncthreads();
  // the frequencies of a lane: pairs (c, c + d/2) of channels 2 l, 2 l + 1, or the pairs (2 l, 2 l + 1), (64 + 2 l, 65 + 2 l) themselves
  const int c0 = interleaved ? lane : 2 * lane, c1 = interleaved ? half / 2 + lane : 2 * lane + 1;
  for (int h = warp; h < n_q_heads; h += kRowsWarps) {
    float2 xs[kRowsQ], ys[kRowsQ];
#pragma unroll
    for (int u = 0; u < kRowsQ; ++u) {
      xs[u] = __bfloat1622float2(x[u]);
      ys[u] = __bfloat1622float2(y[u]);
    }
    const float2 fx = __bfloat1622float2(kx), fy = __bfloat1622float2(ky);
    if (h + kRowsWarps < n_q_heads) load(h + kRowsWarps);
    const size_t row0 = (out_seq + h) * n_pseudo + i0;
    float part[kRowsQ];
#pragma unroll
    for (int u = 0; u < kRowsQ; ++u) {
      const double2 s0 = angle[u][c0], s1 = angle[u][c1];
      // (lo, hi) of the two rotations
      const double lo0 = xs[u].x, hi0 = interleaved ? xs[u].y : ys[u].x, lo1 = interleaved ? ys[u].x : xs[u].y, hi1 = ys[u].y;
      const double r0 = (lo0 * s0.y - hi0 * s0.x) * out_scale, r1 = (hi0 * s0.y + lo0 * s0.x) * out_scale;
      const double r2 = (lo1 * s1.y - hi1 * s1.x) * out_scale, r3 = (hi1 * s1.y + lo1 * s1.x) * out_scale;
      // channels 2 l, 2 l + 1 of the first half, of the second
      const double a0 = r0, a1 = interleaved ? r1 : r2, b0 = interleaved ? r2 : r1, b1 = r3;
      part[u] = ((float)a0 * fx.x + (float)b0 * fy.x) + ((float)a1 * fx.y + (float)b1 * fy.y);
      if (u < n) {
        __half2* out = q_rot + (row0 + u) * half + lane;
        out[0] = __halves2half2(from_double<__half>(a0), from_double<__half>(a1));
        out[half / 2] = __halves2half2(from_double<__half>(b0), from_double<__half>(b1));
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < kRowsQ; ++u) part[u] += __shfl_xor_sync(0xffffffffu, part[u], o);
    float mine = part[0];
#pragma unroll
    for (int u = 1; u < kRowsQ; ++u) mine = lane == u ? part[u] : mine;
    if (lane < n) rb.ref[row0 + lane] = mine;
  }
  if (late_wait) pdl_wait();
}

// The queries may begin anywhere that an element may (the keys lie on 16-byte boundaries, like their strides).
bool aligned4(const RopeBatch& rb) {
  for (int l = 0; l < rb.n_layers; ++l)
    if ((uintptr_t)rb.q[l] & 3u) return false;
  return true;
}

}  // namespace

cudaError_t launch_rope(int dtype, int out_mode, int64_t lo_offset, const RopeBatch& rb, void* q_rot, const double* inv_freq_dev,
                        const SeqTable& t, const Dims& dm, bool late_wait, cudaStream_t s, LaunchLog* log) {
  const int lw = late_wait ? 1 : 0;
  log->begin(kKindRope, s);
  // One query per block keeps a short call's latency lowest; four where a block each would take several waves.
  const int heads = (dm.n_q_heads + kHeadsPerBlock - 1) / kHeadsPerBlock, seqs = t.batch * rb.n_layers;
  const bool many = (int64_t)dm.n_pseudo * seqs * heads > 2048;
  RopeLayers<1> one = {{rb.q[0]}, {rb.k[0]}, {rb.head_stride[0]}, {rb.row_stride[0]}, 1, rb.group, nullptr, nullptr, 0};   // (no reference)
  auto launch = [&](auto kernel1, auto kernel4, auto* out, int64_t offset, double scale, const auto& layers) {
    const dim3 block(kHeadDim / 2, kHeadsPerBlock), grid1(dm.n_pseudo, seqs, heads), grid4((dm.n_pseudo + 3) / 4, seqs, heads);
    launch_pdl(many ? kernel4 : kernel1, many ? grid4 : grid1, block, 0, s, 1, layers, out, inv_freq_dev, t, dm.n_q_heads, dm.n_pseudo, offset, lw,
               dm.rope_interleaved, scale);
  };
  using bf16 = __nv_bfloat16;
  if (dtype == DAPQ_BF16 && out_mode == kRopeOutSplitBf16) {
    launch(rope_pseudo_q_kernel<bf16, bf16, true, 1, 1>, rope_pseudo_q_kernel<bf16, bf16, true, 4, 1>, (bf16*)q_rot, lo_offset, 1.0, one);
  } else if (dtype == DAPQ_BF16 && out_mode == kRopeOutF16) {
    one.ref = rb.ref;
    if (many && rb.ref != nullptr && aligned4(rb))
      launch_pdl(rope_rows_kernel, dim3((dm.n_pseudo + kRowsQ - 1) / kRowsQ, seqs), dim3(kRowsWarps * 32), 0, s, 1, rb, (__half2*)q_rot, inv_freq_dev, t,
                 dm.n_q_heads, dm.n_pseudo, lw, dm.rope_interleaved, (double)dm.scale_log2e);
    else if (rb.n_layers > 1)
      launch(rope_pseudo_q_kernel<bf16, __half, false, 1, kFlowLayers>, rope_pseudo_q_kernel<bf16, __half, false, 4, kFlowLayers>, (__half*)q_rot, 0,
             (double)dm.scale_log2e, rb);
    else
      launch(rope_pseudo_q_kernel<bf16, __half, false, 1, 1>, rope_pseudo_q_kernel<bf16, __half, false, 4, 1>, (__half*)q_rot, 0, (double)dm.scale_log2e, one);
  } else if (dtype == DAPQ_BF16 && out_mode == kRopeOutBf16) {
    launch(rope_pseudo_q_kernel<bf16, bf16, false, 1, 1>, rope_pseudo_q_kernel<bf16, bf16, false, 4, 1>, (bf16*)q_rot, 0, 1.0, one);
  } else if (dtype == DAPQ_BF16) {
    launch(rope_pseudo_q_kernel<bf16, float, false, 1, 1>, rope_pseudo_q_kernel<bf16, float, false, 4, 1>, (float*)q_rot, 0, 1.0, one);
  } else {
    launch(rope_pseudo_q_kernel<float, float, false, 1, 1>, rope_pseudo_q_kernel<float, float, false, 4, 1>, (float*)q_rot, 0, 1.0, one);
  }
  log->end(s);
  return cudaGetLastError();
}

}  // namespace dapq
