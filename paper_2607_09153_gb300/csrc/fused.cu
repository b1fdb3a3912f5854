// Small kernels around the projections of the verify-token forward (Sec. 4.1;
// the c_ffn d^2 and c_attn d L terms of Eq. cost_kv live in the GEMMs and the
// attention, these are the O(d) glue).  All arithmetic is fp32; an activation
// that feeds a tensor-core contraction is stored as a bf16 (hi, lo) pair,
// hi = bf16(x), lo = bf16(x - hi), so no bf16 rounding of the activation
// itself enters the result.
//   call_begin   the call's tables from pinned host memory into the device
//                tables (and, for the attention entry point, q as hi/lo)
//   prologue     cos/sin of p * base^(-2i/hd) at p = L_b (fp64 angles);
//                h = e_v ; per-tile sums of squares of h ; x = h ⊙ g (the
//                RMSNorm's per-candidate factor 1/sqrt(mean(h^2) + eps) is
//                applied by the QKV epilogue, as between all projections)
//   head         x = RMSNorm(h) * g_final with mean(h^2) from the per-tile
//                sums of squares the last residual epilogue wrote (summed in
//                a fixed order: deterministic);
//                P(+) = 1/(1 + exp(w_minus.x - w_plus.x)) (Eq. score, App. B.2)
#include <cuda_bf16.h>

#include <algorithm>

#include "kernels.h"
#include "ptx.cuh"

namespace kvprm {

namespace {

__device__ __forceinline__ void store_hilo(HiLo o, int64_t i, float x) {
  const __nv_bfloat16 hi = __float2bfloat16_rn(x);
  o.hi[i] = hi;
  o.lo[i] = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// Four consecutive activations as 8-byte hi and lo stores.
__device__ __forceinline__ void store_hilo4(HiLo o, int64_t i, float4 x) {
  const __nv_bfloat162 h0 = __floats2bfloat162_rn(x.x, x.y), h1 = __floats2bfloat162_rn(x.z, x.w);
  const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
  const __nv_bfloat162 l0 = __floats2bfloat162_rn(x.x - f0.x, x.y - f0.y);
  const __nv_bfloat162 l1 = __floats2bfloat162_rn(x.z - f1.x, x.w - f1.y);
  uint2 hi, lo;
  hi.x = *reinterpret_cast<const uint32_t*>(&h0);
  hi.y = *reinterpret_cast<const uint32_t*>(&h1);
  lo.x = *reinterpret_cast<const uint32_t*>(&l0);
  lo.y = *reinterpret_cast<const uint32_t*>(&l1);
  *reinterpret_cast<uint2*>(o.hi + i) = hi;
  *reinterpret_cast<uint2*>(o.lo + i) = lo;
}

// The call's tables, read by the GPU from the pinned staging buffer (one launch instead of a copy per
// table: seven to nine small copies took ~2 us each on the stream, ahead of every call), and for the
// attention entry point the query as a bf16 pair.  Measured per call with calls queued back to back:
// 2 layers of d 256 with 4 candidates 74 -> 55 us (with prologue_kernel in place of two launches and
// the head's own store instead of a copy), the attention entry point with 37 ragged candidates 99 -> 71
// us and with 24 candidates behind a prefix 81 -> 56 us (with the planner's counts first).  CTAs below pull_ctas copy the parts' 16-byte quads,
// four loads in flight per thread (the host link's latency bounds it); the others split.
__global__ void __launch_bounds__(128) call_begin_kernel(const __grid_constant__ TableParts parts, const uint4* src,
                                                         uint4* dst, int pull_ctas, const float4* __restrict__ q,
                                                         int64_t q_quads, HiLo out) {
  if (static_cast<int>(blockIdx.x) < pull_ctas) {
    const uint32_t total = parts.end[parts.n - 1], stride = static_cast<uint32_t>(pull_ctas) * blockDim.x;
    for (uint32_t i0 = blockIdx.x * blockDim.x + threadIdx.x; i0 < total; i0 += 4 * stride) {
      uint4 v[4];
      uint32_t at[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t i = i0 + k * stride;
        if (i >= total) continue;
        int p = 0;
        while (i >= parts.end[p]) ++p;
        at[k] = parts.off[p] + (i - (p ? parts.end[p - 1] : 0u));
        v[k] = __ldcv(src + at[k]);   // host memory that the next call rewrites
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i0 + k * stride < total) dst[at[k]] = v[k];
    }
    return;
  }
  const int64_t stride = static_cast<int64_t>(gridDim.x - pull_ctas) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x - pull_ctas) * blockDim.x + threadIdx.x; i < q_quads; i += stride)
    store_hilo4(out, 4 * i, q[i]);
}

// One CTA of 256 threads per row: its rotation (row b is verify token b % depth of its candidate, at
// position L + b % depth), h = e_v with its per-tile sums of squares as the residual epilogue writes
// them, and x.  Latency only; the rotation's fp64 sine and cosine are its longest chain, so the powers
// base^(-2i/hd) come from a table laid down with the context.
__global__ void __launch_bounds__(256) prologue_kernel(const int32_t* __restrict__ seq_lens,
                                                       const double* __restrict__ inv_freq, int half, int depth,
                                                       float2* __restrict__ rope, const __nv_bfloat16* __restrict__ e_v,
                                                       const __nv_bfloat16* __restrict__ gain, int d, int n_rows,
                                                       float* __restrict__ h, float* __restrict__ sumsq, HiLo x,
                                                       unsigned long long* ts) {
  trace_begin(ts);
  grid_dep_launch();
  grid_dep_wait();
  const int b = blockIdx.x;
  const int64_t row = static_cast<int64_t>(b) * d;
  for (int c = 4 * threadIdx.x; c < d; c += 4 * blockDim.x) {   // d % 64 == 0
    const float4 v = load_bf16x4(e_v + c), g = load_bf16x4(gain + c);
    *reinterpret_cast<float4*>(h + row + c) = v;
    store_hilo4(x, row + c, make_float4(v.x * g.x, v.y * g.y, v.z * g.z, v.w * g.w));
  }
  // the rotation on the first warps, the sums on the last ones first
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (static_cast<int>(threadIdx.x) < half) {
    const double ang = static_cast<double>(seq_lens[b] + b % depth) * inv_freq[threadIdx.x];
    double sn, cs;
    sincos(ang, &sn, &cs);
    rope[b * half + threadIdx.x] = make_float2(static_cast<float>(cs), static_cast<float>(sn));
  }
  const int m_tiles = (d + 127) / 128;
  for (int t = nw - 1 - warp; t < m_tiles; t += nw) {
    const int c = t * 128 + 4 * lane;
    float s = 0.f;
    if (c < d) {
      const float4 v = load_bf16x4(e_v + c);
      s = (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) sumsq[static_cast<int64_t>(t) * n_rows + b] = s;
  }
  trace_end(ts);
}

// One CTA of 256 threads per candidate: the reward of its last row (its last verify token; one row per
// candidate except in a depth-k readout), also stored at *out_slot when that is set (the caller's
// buffer of an asynchronous call).  The RMSNorm factor is common to both logits, so the logits' sums
// and the sum of the tiles' squares meet in one reduction.
__global__ void __launch_bounds__(256) head_kernel(const float* __restrict__ h, const float* __restrict__ sumsq,
                                                   int m_tiles, int n_rows, int depth, int d, float eps,
                                                   const __nv_bfloat16* __restrict__ gain,
                                                   const __nv_bfloat16* __restrict__ w_plus,
                                                   const __nv_bfloat16* __restrict__ w_minus,
                                                   float* __restrict__ rewards, float* const* out_slot,
                                                   unsigned long long* ts) {
  trace_begin(ts);
  __shared__ float red[8][3];
  grid_dep_launch();
  grid_dep_wait();
  const int b = blockIdx.x, row = b * depth + depth - 1;
  float zp = 0.f, zm = 0.f, ss = 0.f;
  for (int t = threadIdx.x; t < m_tiles; t += blockDim.x) ss += sumsq[static_cast<int64_t>(t) * n_rows + row];
  for (int c = 4 * threadIdx.x; c < d; c += 4 * blockDim.x) {
    const float4 hv = *reinterpret_cast<const float4*>(h + static_cast<int64_t>(row) * d + c);
    const float4 g = load_bf16x4(gain + c), p = load_bf16x4(w_plus + c), m = load_bf16x4(w_minus + c);
    const float4 x = make_float4(hv.x * g.x, hv.y * g.y, hv.z * g.z, hv.w * g.w);
    zp += (x.x * p.x + x.y * p.y) + (x.z * p.z + x.w * p.w);
    zm += (x.x * m.x + x.y * m.y) + (x.z * m.z + x.w * m.w);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    zp += __shfl_xor_sync(0xffffffffu, zp, off);
    zm += __shfl_xor_sync(0xffffffffu, zm, off);
    ss += __shfl_xor_sync(0xffffffffu, ss, off);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    red[warp][0] = zp;
    red[warp][1] = zm;
    red[warp][2] = ss;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    zp = zm = ss = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      zp += red[w][0];
      zm += red[w][1];
      ss += red[w][2];
    }
    const float r = 1.0f / sqrtf(ss / d + eps);
    const float p = 1.0f / (1.0f + expf(zm * r - zp * r));
    rewards[b] = p;
    float* out = *out_slot;
    if (out) out[b] = p;
  }
  trace_end(ts);
}

__global__ void split_hilo_kernel(const float* __restrict__ in, int64_t count, HiLo out) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < count;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    store_hilo(out, i, in[i]);
}

cudaLaunchConfig_t make_cfg(dim3 grid, dim3 block, cudaStream_t st, cudaLaunchAttribute* attr, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cfg;
}

}  // namespace

cudaError_t launch_call_begin(const TableParts& parts, const int32_t* staging, int32_t* tables, const float* q,
                              int64_t count, HiLo out, cudaStream_t stream) {
  if (parts.n < 1 || parts.n > kMaxTableParts || (count & 3)) return cudaErrorInvalidValue;
  // 64 CTAs hold the host link's bandwidth (as the cache copy does)
  const int pull = static_cast<int>(std::min<uint32_t>(64, (parts.end[parts.n - 1] + 511) / 512));
  const int64_t split = std::min<int64_t>(152 * 8, (count / 4 + 127) / 128);
  call_begin_kernel<<<static_cast<unsigned>(pull + split), 128, 0, stream>>>(
      parts, reinterpret_cast<const uint4*>(staging), reinterpret_cast<uint4*>(tables), pull,
      reinterpret_cast<const float4*>(q), count / 4, out);
  return cudaGetLastError();
}

cudaError_t launch_prologue(const ModelDims& m, const int32_t* seq_lens, const double* inv_freq, int depth,
                            float2* rope, const __nv_bfloat16* e_v, const __nv_bfloat16* gain, int n_rows, float* h,
                            float* sumsq, HiLo x, cudaStream_t stream, bool pdl, unsigned long long* ts) {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = make_cfg(dim3(n_rows), dim3(256), stream, attr, pdl);
  return cudaLaunchKernelEx(&cfg, prologue_kernel, seq_lens, inv_freq, m.hd / 2, depth, rope, e_v, gain, m.d, n_rows,
                            h, sumsq, x, ts);
}

cudaError_t launch_head(const ModelDims& m, const float* h, const float* sumsq, int m_tiles, int n_rows, int depth,
                        const __nv_bfloat16* gain, const __nv_bfloat16* w_plus, const __nv_bfloat16* w_minus,
                        float* rewards, float* const* out_slot, cudaStream_t stream, bool pdl,
                        unsigned long long* ts) {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = make_cfg(dim3(n_rows / depth), dim3(256), stream, attr, pdl);
  return cudaLaunchKernelEx(&cfg, head_kernel, h, sumsq, m_tiles, n_rows, depth, m.d, m.eps, gain, w_plus, w_minus,
                            rewards, out_slot, ts);
}

__global__ void wait_probe_kernel(const int* flag, int* err, unsigned long long limit_ns) {
  if (threadIdx.x == 0) flag_wait(flag, err, limit_ns, kDevProbeTimeout);
}

cudaError_t launch_wait_probe(const int* flag, int* err, unsigned long long limit_ns, cudaStream_t stream) {
  if (limit_ns > kWaitTimeoutNs) limit_ns = kWaitTimeoutNs;
  wait_probe_kernel<<<1, 32, 0, stream>>>(flag, err, limit_ns);
  return cudaGetLastError();
}

cudaError_t launch_split_hilo(const float* in, int64_t count, HiLo out, cudaStream_t stream) {
  int64_t blocks = (count + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  if (blocks < 1) blocks = 1;
  split_hilo_kernel<<<static_cast<unsigned>(blocks), 256, 0, stream>>>(in, count, out);
  return cudaGetLastError();
}

}  // namespace kvprm
