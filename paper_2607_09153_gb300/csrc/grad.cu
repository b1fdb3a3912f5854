// Backward pass of the verify-token forward, for KV Steering (Sec. 6; App. C, Algorithm "KV Steering
// at agent handoff"): the gradient of l = sum_b -log P(+)_b with respect to every cached key and
// value.  The projections' transposed products run on the forward's tensor-core GEMM against
// transposed weight copies (kvprm_api.cu); this file holds the rest:
//   transpose       W [rows][cols] -> W^T (bf16), once per context
//   head_back       dh = d(-log P)/dh at the final RMSNorm: dx = (1 - P)(w_- - w_+)
//   rms_back        dh = dres + r g dy - h r^3 (sum_i g_i dy_i h_i) / d,  r = (mean h^2 + eps)^-1/2
//   silu_back       du = da t SiLU'(u),  dt = da SiLU(u)
//   attn_back_pre   per (candidate, kv head): D_h = do_h . o_h and the self entry's terms
//   attn_back_tc / attn_back_pages (G > 8)  per cached token:
//                   w_j = exp(q.K_j / sqrt(hd) - lse), ds_j = w_j (do.V_j - D),
//                   dK_j = sum_h ds_j q_h / sqrt(hd), dV_j = sum_h w_j do_h, dq_h += ds_j K_j / sqrt(hd)
//   rope_back       the rotation by the negative angle, and [dq; dk; dv] as the next GEMM's input
//   zero_pages      clears the gradient of pages several candidates read (they are accumulated)
//   steer_update    kv <- RNE_bf16(kv - eta grad) on the pages the block tables reference
// Every product runs in fp32; a gradient that feeds a tensor-core contraction is stored as a bf16
// (hi, lo) pair like the forward's activations.
#include <cuda_bf16.h>

#include <algorithm>
#include <functional>
#include <map>
#include <queue>
#include <utility>

#include "kernels.h"
#include "ptx.cuh"

namespace kvprm {

namespace {

typedef __nv_bfloat16 bf16;

// Four consecutive values (8-byte aligned hi and lo).
__device__ __forceinline__ void put_hilo4(bf16* hi, bf16* lo, int64_t i, float4 x) {
  const __nv_bfloat162 h0 = __floats2bfloat162_rn(x.x, x.y), h1 = __floats2bfloat162_rn(x.z, x.w);
  const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
  const __nv_bfloat162 l0 = __floats2bfloat162_rn(x.x - f0.x, x.y - f0.y);
  const __nv_bfloat162 l1 = __floats2bfloat162_rn(x.z - f1.x, x.w - f1.y);
  uint2 a, b;
  a.x = *reinterpret_cast<const uint32_t*>(&h0);
  a.y = *reinterpret_cast<const uint32_t*>(&h1);
  b.x = *reinterpret_cast<const uint32_t*>(&l0);
  b.y = *reinterpret_cast<const uint32_t*>(&l1);
  *reinterpret_cast<uint2*>(hi + i) = a;
  *reinterpret_cast<uint2*>(lo + i) = b;
}

// two block-wide sums at once (blockDim.x a multiple of 32, <= 1024); every thread gets both
__device__ __forceinline__ float2 block_sum2(float a, float b, float2* red) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, off);
    b += __shfl_xor_sync(0xffffffffu, b, off);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (l == 0) red[w] = make_float2(a, b);
  __syncthreads();
  float2 t = make_float2(0.f, 0.f);
  for (int i = 0; i < nw; ++i) {
    t.x += red[i].x;
    t.y += red[i].y;
  }
  return t;
}

__global__ void transpose_kernel(const bf16* __restrict__ in, bf16* __restrict__ out, int rows, int cols) {
  __shared__ bf16 tile[32][34];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int j = threadIdx.y; j < 32; j += blockDim.y) {
    const int r = r0 + j, c = c0 + threadIdx.x;
    if (r < rows && c < cols) tile[j][threadIdx.x] = in[static_cast<int64_t>(r) * cols + c];
  }
  __syncthreads();
  for (int j = threadIdx.y; j < 32; j += blockDim.y) {
    const int c = c0 + j, r = r0 + threadIdx.x;
    if (c < cols && r < rows) out[static_cast<int64_t>(c) * rows + r] = tile[threadIdx.x][j];
  }
}

// The RMSNorm backward of one row, one CTA: four consecutive elements per thread and step, the first
// step's inputs (all of them for d <= 4096) kept in registers between the two sums and the outputs, so
// that a row costs one round trip to memory (32 rows of 3,584: 17 -> 4.8 us against scalar loops that
// read everything twice; 16 of 1,536: 9.8 -> 4.1).  load(c) gives (h, g dy, dres) of elements c .. c + 3;
//   out = dres + r g dy - h r^3 (sum g dy h) / d,  r = (mean h^2 + eps)^-1/2
struct NormBack {
  float4 h, gdy, dres;
};
template <typename Load>
__device__ __forceinline__ void rms_back_row(Load load, int64_t row, int d, float eps, float* out, bf16* o_hi,
                                             bf16* o_lo, float2* red) {
  const int step = 4 * blockDim.x, c0 = 4 * threadIdx.x;
  float ss = 0.f, sd = 0.f;
  auto add = [&](const NormBack& v) {
    ss += (v.h.x * v.h.x + v.h.y * v.h.y) + (v.h.z * v.h.z + v.h.w * v.h.w);
    sd += (v.gdy.x * v.h.x + v.gdy.y * v.h.y) + (v.gdy.z * v.h.z + v.gdy.w * v.h.w);
  };
  NormBack first;
  if (c0 < d) {
    first = load(c0);
    add(first);
  }
#pragma unroll 1
  for (int c = c0 + step; c < d; c += step) add(load(c));
  const float2 t = block_sum2(ss, sd, red);
  const float r = rsqrtf(t.x / d + eps);
  const float k = r * r * r * t.y / d;
  auto put = [&](int c, const NormBack& v) {
    const float4 o = make_float4(v.dres.x + r * v.gdy.x - v.h.x * k, v.dres.y + r * v.gdy.y - v.h.y * k,
                                 v.dres.z + r * v.gdy.z - v.h.z * k, v.dres.w + r * v.gdy.w - v.h.w * k);
    *reinterpret_cast<float4*>(out + row + c) = o;
    if (o_hi) put_hilo4(o_hi, o_lo, row + c, o);
  };
  if (c0 < d) put(c0, first);
#pragma unroll 1
  for (int c = c0 + step; c < d; c += step) put(c, load(c));
}

// One CTA per row: the loss gradient at the final residual stream h.
__global__ void __launch_bounds__(1024) head_back_kernel(
    const float* __restrict__ h, const float* __restrict__ p_plus, const bf16* __restrict__ gain,
    const bf16* __restrict__ w_plus, const bf16* __restrict__ w_minus, int d, float eps, float* __restrict__ dh,
    bf16* __restrict__ dh_hi, bf16* __restrict__ dh_lo) {
  __shared__ float2 red[32];
  grid_dep_launch();
  grid_dep_wait();   // every input is written by earlier kernels of the stream
  const int64_t row = static_cast<int64_t>(blockIdx.x) * d;
  const float q = 1.f - p_plus[blockIdx.x];   // d(-log P)/dz_- = 1 - P = -d(-log P)/dz_+
  auto load = [&](int c) {
    const float4 g = load_bf16x4(gain + c), p = load_bf16x4(w_plus + c), m = load_bf16x4(w_minus + c);
    NormBack v;
    v.h = *reinterpret_cast<const float4*>(h + row + c);
    v.gdy = make_float4(g.x * q * (m.x - p.x), g.y * q * (m.y - p.y), g.z * q * (m.z - p.z), g.w * q * (m.w - p.w));
    v.dres = make_float4(0.f, 0.f, 0.f, 0.f);
    return v;
  };
  rms_back_row(load, row, d, eps, dh, dh_hi, dh_lo, red);
}

// One CTA per row: dh = dres + RMSNorm backward of (h, gain) applied to dy (may run in place:
// dres == out).  h_bf16 (when set) is one bf16 row shared by every row (the embedding of layer 0).
__global__ void __launch_bounds__(1024) rms_back_kernel(const float* __restrict__ h, const bf16* __restrict__ h_bf16,
                                                        const bf16* __restrict__ gain, const float* __restrict__ dy,
                                                        const float* dres, int d, float eps, float* out,
                                                        bf16* __restrict__ o_hi, bf16* __restrict__ o_lo) {
  __shared__ float2 red[32];
  grid_dep_launch();
  grid_dep_wait();
  const int64_t row = static_cast<int64_t>(blockIdx.x) * d;
  auto load = [&](int c) {
    const float4 g = load_bf16x4(gain + c), y = *reinterpret_cast<const float4*>(dy + row + c);
    NormBack v;
    v.h = h_bf16 ? load_bf16x4(h_bf16 + c) : *reinterpret_cast<const float4*>(h + row + c);
    v.gdy = make_float4(g.x * y.x, g.y * y.y, g.z * y.z, g.w * y.w);
    v.dres = *reinterpret_cast<const float4*>(dres + row + c);
    return v;
  };
  rms_back_row(load, row, d, eps, out, o_hi, o_lo, red);
}

// da [n][ff], gu [n][2 ff] (gate then up pre-activations) -> [du; dt] [n][2 ff] as hi/lo, four
// consecutive elements per thread (ff % 64 == 0)
__global__ void __launch_bounds__(256) silu_back_kernel(const float* __restrict__ da, const float* __restrict__ gu,
                                                        int n, int ff, bf16* __restrict__ o_hi,
                                                        bf16* __restrict__ o_lo) {
  grid_dep_launch();
  grid_dep_wait();
  const int per = ff / 4;
  const int total = n * per;
#pragma unroll 1
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int b = i / per, j = 4 * (i - b * per);
    const int64_t at = static_cast<int64_t>(b) * 2 * ff + j;
    const float4 a4 = *reinterpret_cast<const float4*>(da + static_cast<int64_t>(b) * ff + j);
    const float4 u4 = *reinterpret_cast<const float4*>(gu + at), t4 = *reinterpret_cast<const float4*>(gu + at + ff);
    const float a[4] = {a4.x, a4.y, a4.z, a4.w}, u[4] = {u4.x, u4.y, u4.z, u4.w}, t[4] = {t4.x, t4.y, t4.z, t4.w};
    float du[4], dt[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float sg = 1.f / (1.f + expf(-u[e]));
      du[e] = a[e] * t[e] * sg * (1.f + u[e] * (1.f - sg));
      dt[e] = a[e] * u[e] * sg;
    }
    put_hilo4(o_hi, o_lo, at, make_float4(du[0], du[1], du[2], du[3]));
    put_hilo4(o_hi, o_lo, at + ff, make_float4(dt[0], dt[1], dt[2], dt[3]));
  }
}

// One CTA of 8 warps per (row b, kv head g), a warp per query head: D_h = do_h . o_h, and the verify
// token's own entry: w_s = exp(q_h . k_s / sqrt(hd) - lse_h), ds_s = w_s (do_h . v_s - D_h),
// dk_s = sum_h ds_s q_h / sqrt(hd), dv_s = sum_h w_s do_h, dq_h = ds_s k_s / sqrt(hd) (the pages add on).
// With ops set (G <= 8) also the tensor-core backward's operands of this (b, g): q, then dO, each as a
// hi and a lo block of 8 rows (heads past G: the workspace's initial zeros) in the 128-byte swizzle,
// [q, dO][hi, lo][HD / 64][8 rows][128 B], and meta [8] = (lse, D) (heads past G: lse = inf, so that
// their weight is 0).  Latency only: every input is read once, in one round.
__global__ void __launch_bounds__(256) attn_back_pre_kernel(
    const float* __restrict__ q, const float* __restrict__ ks, const float* __restrict__ vs, const float* __restrict__ o,
    const float* __restrict__ dout, const float* __restrict__ lse, int n_q, int n_kv, int hd, float* __restrict__ D,
    float* __restrict__ dq, float* __restrict__ dks, float* __restrict__ dvs, uint8_t* __restrict__ ops,
    float2* __restrict__ meta) {
  __shared__ float s_w[kMaxGroup], s_ds[kMaxGroup];
  __shared__ float4 s_q[kMaxGroup][32], s_do[kMaxGroup][32];
  grid_dep_launch();
  grid_dep_wait();
  const int b = blockIdx.x / n_kv, g = blockIdx.x % n_kv, G = n_q / n_kv;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float scale = rsqrtf(static_cast<float>(hd));
  const int64_t hk = (static_cast<int64_t>(b) * n_kv + g) * hd;
  const int64_t row0 = static_cast<int64_t>(b) * n_q + static_cast<int64_t>(g) * G;
  const bool on = 4 * lane < hd;   // four elements a lane
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const float4 k4 = on ? reinterpret_cast<const float4*>(ks + hk)[lane] : zero;
  const float4 v4 = on ? reinterpret_cast<const float4*>(vs + hk)[lane] : zero;
  auto dot = [](float4 x, float4 y) { return (x.x * y.x + x.y * y.y) + (x.z * y.z + x.w * y.w); };
#pragma unroll 1
  for (int r = warp; r < G; r += 8) {
    const int64_t hq = (row0 + r) * hd;
    const float4 q4 = on ? reinterpret_cast<const float4*>(q + hq)[lane] : zero;
    const float4 d4 = on ? reinterpret_cast<const float4*>(dout + hq)[lane] : zero;
    const float4 o4 = on ? reinterpret_cast<const float4*>(o + hq)[lane] : zero;
    const float ls = lse[row0 + r];
    float dd = dot(d4, o4), sq = dot(q4, k4), dp = dot(d4, v4);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      dd += __shfl_xor_sync(0xffffffffu, dd, off);
      sq += __shfl_xor_sync(0xffffffffu, sq, off);
      dp += __shfl_xor_sync(0xffffffffu, dp, off);
    }
    s_q[r][lane] = q4;
    s_do[r][lane] = d4;
    if (lane == 0) {
      const float w = expf(sq * scale - ls);
      D[row0 + r] = dd;
      s_w[r] = w;
      s_ds[r] = w * (dp - dd);
      if (ops) meta[static_cast<int64_t>(blockIdx.x) * 8 + r] = make_float2(ls, dd);
    }
    if (ops && on) {   // 8 bytes of this head's hi and lo rows each: half a 16-byte chunk
      const int block = (hd / 64) * 1024, c = lane >> 1;
      const int64_t at = static_cast<int64_t>(blockIdx.x) * 4 * block + (c >> 3) * 1024 + r * 128 +
                         (((c & 7) ^ r) << 4) + (lane & 1) * 8;
      put_hilo4(reinterpret_cast<bf16*>(ops + at), reinterpret_cast<bf16*>(ops + at + block), 0, q4);
      put_hilo4(reinterpret_cast<bf16*>(ops + at + 2 * block), reinterpret_cast<bf16*>(ops + at + 3 * block), 0, d4);
    }
  }
  if (ops && static_cast<int>(threadIdx.x) >= G && threadIdx.x < 8)
    meta[static_cast<int64_t>(blockIdx.x) * 8 + threadIdx.x] = make_float2(INFINITY, 0.f);
  __syncthreads();
  // warp 0: dk_s, dv_s; then every warp dq of its heads
  if (warp == 0 && on) {
    float4 ak = zero, av = zero;
#pragma unroll 1
    for (int r = 0; r < G; ++r) {
      const float4 x = s_q[r][lane], y = s_do[r][lane];
      const float ds = s_ds[r] * scale, w = s_w[r];
      ak = make_float4(ak.x + ds * x.x, ak.y + ds * x.y, ak.z + ds * x.z, ak.w + ds * x.w);
      av = make_float4(av.x + w * y.x, av.y + w * y.y, av.z + w * y.z, av.w + w * y.w);
    }
    reinterpret_cast<float4*>(dks + hk)[lane] = ak;
    reinterpret_cast<float4*>(dvs + hk)[lane] = av;
  }
  if (on)
#pragma unroll 1
    for (int r = warp; r < G; r += 8) {
      const float ds = s_ds[r] * scale;
      reinterpret_cast<float4*>(dq + (row0 + r) * hd)[lane] = make_float4(ds * k4.x, ds * k4.y, ds * k4.z, ds * k4.w);
    }
}

// One CTA of 4 warps per unit {b, g, j0, j1}: candidate b's logical pages j0 .. j1 - 1 (at most
// kBackUnitPages) of kv head g.  Thread 0 bulk-copies the unit's K and V blocks (16 x HD bf16 each,
// contiguous in the pool) into shared memory at once, so every byte of the unit is in flight before
// any is used.  Warp w then takes tokens w, w + 4, .. of each page; each lane holds HD / 32
// consecutive elements of the token's key and value, of the G query rows and of their output
// gradients, so every dot product is a lane-local sum and one warp reduction.  dK and dV of a page
// only this candidate reads are stored; of a page several read (shared[page] != 0) they are added
// with atomics (zero_pages cleared them).  dq is summed over the CTA's warps (in the shared memory
// the pages occupied), then added atomically.
constexpr int kBackUnitPages = kBackUnitPagesMax;

template <int HD>
constexpr size_t back_pages_smem() {
  return static_cast<size_t>(kBackUnitPages) * 2 * 16 * HD * 2 + 16;   // the pages' K and V, the barrier
}

template <int HD, int GMAX>
__global__ void __launch_bounds__(128) attn_back_pages_kernel(
    const int4* __restrict__ units, const int32_t* __restrict__ seq_lens, const int32_t* __restrict__ block_table,
    int max_blocks, const bf16* __restrict__ pool_layer, const uint8_t* __restrict__ shared, const float* __restrict__ q,
    const float* __restrict__ dout, const float* __restrict__ lse, const float* __restrict__ D, int n_q, int n_kv,
    float* __restrict__ grad_layer, float* __restrict__ dq, int* err) {
  constexpr int kPer = HD / 32;   // 4 (hd 128) or 2 (hd 64)
  constexpr uint32_t kBlock = 16 * HD * 2;   // one page's K (or V) of one kv head, bytes
  extern __shared__ __align__(16) uint8_t smem[];
  bf16* s_kv = reinterpret_cast<bf16*>(smem);   // [page][K, V][16][HD]
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + static_cast<size_t>(kBackUnitPages) * 2 * kBlock);
  grid_dep_launch();
  grid_dep_wait();
  const int4 u = units[blockIdx.x];
  const int b = u.x, g = u.y, j0 = u.z, j1 = u.w;
  const int npg = j1 - j0;   // 1 .. kBackUnitPages
  const int G = n_q / n_kv;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float scale = rsqrtf(static_cast<float>(HD));
  const int L = seq_lens[b];
  const int64_t page_elems = static_cast<int64_t>(2) * n_kv * 16 * HD;   // one page of one layer
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    mbar_arrive_expect_tx(bar, static_cast<uint32_t>(npg) * 2 * kBlock);
    for (int i = 0; i < npg; ++i) {
      const int32_t p = block_table[static_cast<int64_t>(b) * max_blocks + j0 + i];
      const bf16* kp = pool_layer + p * page_elems + static_cast<int64_t>(g) * 16 * HD;
      bulk_load(s_kv + (2 * i) * 16 * HD, kp, kBlock, bar);
      bulk_load(s_kv + (2 * i + 1) * 16 * HD, kp + static_cast<int64_t>(n_kv) * 16 * HD, kBlock, bar);
    }
  }
  float qr[GMAX][kPer], dr[GMAX][kPer], acc[GMAX][kPer];
  float lse_r[GMAX], D_r[GMAX];
#pragma unroll
  for (int r = 0; r < GMAX; ++r) {
    if (r < G) {
      const int64_t row = static_cast<int64_t>(b) * n_q + g * G + r;
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        qr[r][k] = q[row * HD + lane * kPer + k];
        dr[r][k] = dout[row * HD + lane * kPer + k];
        acc[r][k] = 0.f;
      }
      lse_r[r] = lse[row];
      D_r[r] = D[row];
    }
  }
  __syncthreads();   // the barrier is initialised
  if (!mbar_wait(bar, 0, err)) {
    // gave up (the error word is set): wait, bounded again, for the copies still landing in this
    // CTA's shared memory before leaving
    mbar_wait(bar, 0, err);
    return;
  }
  for (int i = 0; i < npg; ++i) {
    const int j = j0 + i;
    const int32_t p = block_table[static_cast<int64_t>(b) * max_blocks + j];
    const int valid = min(16, L - 16 * j);
    const bf16* ks = s_kv + (2 * i) * 16 * HD;
    const bf16* vs = ks + 16 * HD;
    float* gk = grad_layer + p * page_elems + static_cast<int64_t>(g) * 16 * HD;
    float* gv = gk + static_cast<int64_t>(n_kv) * 16 * HD;
    const bool sh = shared[p] != 0;
    for (int t = warp; t < 16; t += 4) {
      float kf[kPer], vf[kPer];
      if constexpr (kPer == 4) {
        const uint2 kb = *reinterpret_cast<const uint2*>(ks + t * HD + lane * 4);
        const uint2 vb = *reinterpret_cast<const uint2*>(vs + t * HD + lane * 4);
        const float2 k01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&kb.x));
        const float2 k23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&kb.y));
        const float2 v01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&vb.x));
        const float2 v23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&vb.y));
        kf[0] = k01.x; kf[1] = k01.y; kf[2] = k23.x; kf[3] = k23.y;
        vf[0] = v01.x; vf[1] = v01.y; vf[2] = v23.x; vf[3] = v23.y;
      } else {
        const uint32_t kb = *reinterpret_cast<const uint32_t*>(ks + t * HD + lane * 2);
        const uint32_t vb = *reinterpret_cast<const uint32_t*>(vs + t * HD + lane * 2);
        const float2 k01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&kb));
        const float2 v01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&vb));
        kf[0] = k01.x; kf[1] = k01.y;
        vf[0] = v01.x; vf[1] = v01.y;
      }
      float dk[kPer], dv[kPer];
#pragma unroll
      for (int k = 0; k < kPer; ++k) dk[k] = dv[k] = 0.f;
      if (t < valid) {
        // the G heads' two dot products, reduced over the warp together
        float sv[GMAX], pv[GMAX];
#pragma unroll
        for (int r = 0; r < GMAX; ++r) {
          sv[r] = 0.f;
          pv[r] = 0.f;
          if (r < G) {
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
              sv[r] += qr[r][k] * kf[k];
              pv[r] += dr[r][k] * vf[k];
            }
          }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
          for (int r = 0; r < GMAX; ++r)
            if (r < G) {
              sv[r] += __shfl_xor_sync(0xffffffffu, sv[r], off);
              pv[r] += __shfl_xor_sync(0xffffffffu, pv[r], off);
            }
#pragma unroll
        for (int r = 0; r < GMAX; ++r) {
          if (r >= G) break;
          const float w = expf(sv[r] * scale - lse_r[r]);
          const float ds = w * (pv[r] - D_r[r]);
#pragma unroll
          for (int k = 0; k < kPer; ++k) {
            dk[k] += ds * scale * qr[r][k];
            dv[k] += w * dr[r][k];
            acc[r][k] += ds * scale * kf[k];
          }
        }
      }
      float* gkt = gk + t * HD + lane * kPer;
      float* gvt = gv + t * HD + lane * kPer;
      if constexpr (kPer == 4) {
        const float4 k4 = make_float4(dk[0], dk[1], dk[2], dk[3]);
        const float4 v4 = make_float4(dv[0], dv[1], dv[2], dv[3]);
        if (sh) {
          atomicAdd(reinterpret_cast<float4*>(gkt), k4);
          atomicAdd(reinterpret_cast<float4*>(gvt), v4);
        } else {
          *reinterpret_cast<float4*>(gkt) = k4;
          *reinterpret_cast<float4*>(gvt) = v4;
        }
      } else {
        if (sh) {
#pragma unroll
          for (int k = 0; k < kPer; ++k) {
            atomicAdd(gkt + k, dk[k]);
            atomicAdd(gvt + k, dv[k]);
          }
        } else {
          *reinterpret_cast<float2*>(gkt) = make_float2(dk[0], dk[1]);
          *reinterpret_cast<float2*>(gvt) = make_float2(dv[0], dv[1]);
        }
      }
    }
  }
  // dq: the four warps' sums (in the shared memory the pages occupied), then one atomic add each
  __syncthreads();
  float* s_dq = reinterpret_cast<float*>(smem);   // [4][GMAX][HD] <= the page buffer
#pragma unroll
  for (int r = 0; r < GMAX; ++r)
    if (r < G)
#pragma unroll
      for (int k = 0; k < kPer; ++k) s_dq[(warp * GMAX + r) * HD + lane * kPer + k] = acc[r][k];
  __syncthreads();
  for (int i = threadIdx.x; i < G * HD; i += blockDim.x) {
    const int r = i / HD, e = i - r * HD;
    const float v = s_dq[(0 * GMAX + r) * HD + e] + s_dq[(1 * GMAX + r) * HD + e] + s_dq[(2 * GMAX + r) * HD + e] +
                    s_dq[(3 * GMAX + r) * HD + e];
    atomicAdd(dq + (static_cast<int64_t>(b) * n_q + g * G + r) * HD + e, v);
  }
}

// ---------------------------------------------------------------- attention backward on the tensor cores
// G <= 8 query heads per kv head.  An item is a tile of up to 8 pages (128 tokens) of one kv head and
// the candidates that read all of them (one for private pages; a beam prefix or a tree edge has many);
// the candidates are taken up to four at a time, 8 rows (heads, padded) each.  Per item and four
// candidates, with tcgen05 MMAs (bf16 in, fp32 accumulators in TMEM, M = 128), every fp32 operand as a
// bf16 (hi, lo) pair:
//   S  = K [q_hi; q_lo]^T, dP = V [dO_hi; dO_lo]^T   lanes = tokens, N = 64: per candidate 8 hi rows,
//                                 then their 8 lo rows (the two are added when TMEM is read);
//   w = exp(S / sqrt(hd) - lse), ds = w (dP - D) / sqrt(hd)     two threads per token, to shared memory
//                                 as [token][32 hi | 32 lo] rows of 128 bytes in the 128-byte swizzle;
//   dV^T += dO^T w, dK^T += q^T ds  lanes = head dim, N = 128 tokens, K = the rows: hi hi + hi lo +
//                                 lo hi (the lo x lo term, ~2^-16 of the product, is left out); they
//                                 accumulate in TMEM over the item's candidates, so a page's gradient is
//                                 stored once however many candidates read it (no atomics, no zeroing);
//   dq^T = K^T [ds_hi | ds_lo]    lanes = head dim, added to dq by atomics.
// Keys and values serve K-major (S, dP) and MN-major (dq) operands as TMA left them; so do the rows.
// Persistent, one CTA per SM with an equal share of the work (plan_attn_back).  Warps 0 and 14 load (keys
// and values of the next item and the rows of the next steps while the current ones are used), warp 1 issues every MMA (S and dP of the next step before the products of this one, when
// their operands have landed), warps 2..9 compute w and ds, two threads per token, and add dq of the
// step before, warps 10..13 store the results, a warp's 32 lanes 128 contiguous bytes at a time.
// Bound: for private pages the stores (twice the K/V bytes in fp32, ~2.4 us of an item's ~2.8 us on an
// SM, which is why they have warps of their own and the next item is scored beside them), for widely
// shared ones the chain S -> w, ds -> products of a four-candidate step (~2 us).  A warp-MMA form that
// took a CTA per candidate and eight pages and added a shared page's gradient once per candidate was the
// form before: gradient call of 32 candidates of 4,096 shared + 500 own tokens, four 7B layers, 2,116 ->
// 1,363 us (its launch alone 226 -> 37 us a layer); 16 distinct caches of 2,048, 1.5B, 3,538 -> 3,420 us
// (30.5 -> 20.6 us a layer for 33 MB read and 67 MB written).
__device__ __forceinline__ BackItem back_item(const BackItem* __restrict__ items, int i) {
  const int4 a = __ldg(reinterpret_cast<const int4*>(items + i)), b = __ldg(reinterpret_cast<const int4*>(items + i) + 1);
  return BackItem{a.x, a.y, a.z, a.w, b.x, b.y, {0, 0}};
}

constexpr int kBackRowsCands = 4;    // candidates per step
constexpr uint32_t kBackRowStages = 3;
constexpr int kBackWarps = 15;       // 0 and 14 load, 1 issues MMAs, 2..9 w and ds, 10..13 results
constexpr int kBackThreads = 32 * kBackWarps;
constexpr uint32_t kBackTmemCols = 512;
constexpr uint32_t kBackColS = 0, kBackColP = 64, kBackColV = 128, kBackColK = 256, kBackColQ = 384;

template <int HD>
struct BackSmem {
  static constexpr uint32_t kSub = 128 * 128;                    // 64 columns of 128 tokens
  static constexpr uint32_t kTile = (HD / 64) * kSub;            // keys (or values) of an item
  static constexpr uint32_t kGroup = (HD / 64) * 1024;           // 8 rows
  static constexpr uint32_t kCand = 2 * kGroup;                  // hi and lo rows of a candidate
  static constexpr uint32_t kRows = kBackRowsCands * kCand;      // q (or dO) rows of a step
  // values are read by the first products of a step only, so one stage of them is free again early in
  // an item's last step; rows are released by the last ones and take ~2,000 cycles to reload: three
  static constexpr uint32_t kK = 0;                              // [2 stages]
  static constexpr uint32_t kV = kK + 2 * kTile;
  static constexpr uint32_t kRowBuf = kV + kTile;                // [kRowStages][q, dO]
  static constexpr uint32_t kW = kRowBuf + kBackRowStages * 2 * kRows;   // w [128 tokens][128 B]
  static constexpr uint32_t kDs = kW + kSub;                     // ds
  static constexpr uint32_t kMeta = kDs + kSub;                  // [kBackRowStages][32] (lse, D)
  static constexpr uint32_t kBars = kMeta + kBackRowStages * 32 * 8;
  static constexpr size_t kBytes = kBars + 256 + 1024;           // barriers and the TMEM address, alignment slack
};
static_assert(BackSmem<128>::kBytes <= 227 * 1024, "attention backward shared memory exceeds the per-block limit");

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~static_cast<uintptr_t>(1023));
}

// Eight values as 16-byte hi and lo chunks.
__device__ __forceinline__ void split8(const float (&x)[8], uint4* hi, uint4* lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(x[2 * e], x[2 * e + 1]);
    const float2 hf = __bfloat1622float2(h2);
    const __nv_bfloat162 l2 = __floats2bfloat162_rn(x[2 * e] - hf.x, x[2 * e + 1] - hf.y);
    h[e] = *reinterpret_cast<const uint32_t*>(&h2);
    l[e] = *reinterpret_cast<const uint32_t*>(&l2);
  }
  *hi = make_uint4(h[0], h[1], h[2], h[3]);
  *lo = make_uint4(l[0], l[1], l[2], l[3]);
}

template <int HD>
__global__ void __launch_bounds__(kBackThreads, 1) attn_back_tc_kernel(
    const __grid_constant__ CUtensorMap tm_pool_tc, int64_t layer_page0, const BackItem* __restrict__ items,
    const int32_t* __restrict__ cta_item, const uint32_t* __restrict__ pages, const int32_t* __restrict__ cands,
    const uint8_t* __restrict__ ops, const uint8_t* __restrict__ zero_rows, const float2* __restrict__ meta, int n_q,
    int n_kv, float* __restrict__ grad_layer, float* __restrict__ dq, int* err) {
  using SM = BackSmem<HD>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = align1024(smem_raw);
  uint64_t* k_full = reinterpret_cast<uint64_t*>(base + SM::kBars);   // [2] keys landed
  uint64_t* k_empty = k_full + 2;                                      // [2] every MMA that reads them done
  uint64_t* v_full = k_empty + 2;                                      // values landed
  uint64_t* v_empty = v_full + 1;
  uint64_t* r_full = v_empty + 1;                                      // [kBackRowStages] a step's rows landed
  uint64_t* r_empty = r_full + kBackRowStages;                         // [kBackRowStages]
  uint64_t* s_full = r_empty + kBackRowStages;                                      // S and dP in TMEM
  uint64_t* s_free = s_full + 1;                                       // read by the softmax warps
  uint64_t* p_full = s_free + 1;                                       // w and ds in shared memory
  uint64_t* o_full = p_full + 1;                                       // the step's products done
  uint64_t* acc_full = o_full + 1;                                     // [2] an item's dV, dK complete
  uint64_t* acc_free = acc_full + 2;                                   // [2] and read out
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_free + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = n_q / n_kv;
  const int item0 = cta_item[blockIdx.x], item1 = cta_item[blockIdx.x + 1];   // uploaded before the call
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
      mbar_init(&acc_full[s], 1);
      mbar_init(&acc_free[s], 4);
    }
    mbar_init(v_full, 1);
    mbar_init(v_empty, 1);
    for (uint32_t s = 0; s < kBackRowStages; ++s) {
      mbar_init(&r_full[s], 1);
      mbar_init(&r_empty[s], 1);
    }
    mbar_init(s_full, 1);
    mbar_init(s_free, 8);
    mbar_init(p_full, 8);
    mbar_init(o_full, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tm_pool_tc);
  }
  // The partner rows of an odd candidate meet zero weights, but 0 x Inf is NaN: they are zero, here and
  // (load_rows) whenever an earlier step left a candidate's rows there.
  for (uint32_t i = threadIdx.x; i < kBackRowStages * 2 * SM::kRows / 16; i += blockDim.x)
    reinterpret_cast<uint4*>(base + SM::kRowBuf)[i] = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async_smem();
  if (warp == 1) {
    tmem_alloc(tmem_slot, kBackTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_dep_launch();

  if (warp == 0 || warp == kBackWarps - 1) {
    // ------------------------------------------------ loads: warp 0 the rows and keys, the last warp the values
    // (a 2 KB box takes a thread ~110 cycles to issue: two threads keep up with an item)
    if (lane == 0) {
      const bool keys = warp == 0;
      const uint64_t pol = policy_evict_first();
      uint32_t it = 0, ki = 0;
      uint32_t filled = 0;   // bit 4 rb + i: candidate slot i of row stage rb holds some candidate's rows
      bool ok = true;
      auto load_pages = [&](const BackItem& w) -> bool {
        uint64_t* full = keys ? &k_full[ki & 1u] : v_full;
        if (keys ? ki >= 2 && !mbar_wait(&k_empty[ki & 1u], ((ki >> 1) - 1) & 1u, err)
                 : ki >= 1 && !mbar_wait(v_empty, (ki - 1) & 1u, err))
          return false;
        mbar_arrive_expect_tx(full, static_cast<uint32_t>(w.n_pages) * (HD / 64) * 2048);
        uint8_t* dst = base + (keys ? SM::kK + (ki & 1u) * SM::kTile : SM::kV);
#pragma unroll 1
        for (int i = 0; i < w.n_pages; ++i) {
          const int32_t unit =
              static_cast<int32_t>(2 * (layer_page0 + (__ldg(pages + w.page_off + i) & ~kBackAtomicPage))) + (keys ? 0 : 1);
#pragma unroll
          for (int sub = 0; sub < HD / 64; ++sub)
            tma_load_5d(dst + sub * SM::kSub + i * 2048, &tm_pool_tc, full, 0, 0, sub, w.g, unit, pol);
        }
        ++ki;
        return true;
      };
      auto load_rows = [&](const BackItem& w, int c0) -> bool {
        const uint32_t rb = it % kBackRowStages, use = it / kBackRowStages;
        if (use > 0 && !mbar_wait(&r_empty[rb], (use - 1) & 1u, err)) return false;
        const int nc = min(kBackRowsCands, w.n_cands - c0);
        // an odd candidate's partner in its 16-row MMA
        const uint32_t partner = (nc & 1) ? 1u << (kBackRowsCands * rb + nc) : 0u;
        const bool clear = (filled & partner) != 0u;
        mbar_arrive_expect_tx(&r_full[rb], static_cast<uint32_t>(nc) * (2 * SM::kCand + 64) + (clear ? 2 * SM::kCand : 0u));
        uint8_t* rows = base + SM::kRowBuf + rb * 2 * SM::kRows;
        if (clear) {
          bulk_load(rows + nc * SM::kCand, zero_rows, SM::kCand, &r_full[rb]);
          bulk_load(rows + SM::kRows + nc * SM::kCand, zero_rows, SM::kCand, &r_full[rb]);
        }
        filled = (filled & ~partner) | ((1u << nc) - 1u) << (kBackRowsCands * rb);
#pragma unroll 1
        for (int i = 0; i < nc; ++i) {
          const int64_t bg = static_cast<int64_t>(__ldg(cands + w.cand_off + c0 + i)) * n_kv + w.g;
          bulk_load(rows + i * SM::kCand, ops + bg * 2 * SM::kCand, SM::kCand, &r_full[rb]);
          bulk_load(rows + SM::kRows + i * SM::kCand, ops + bg * 2 * SM::kCand + SM::kCand, SM::kCand, &r_full[rb]);
          bulk_load(base + SM::kMeta + rb * 256 + i * 64, meta + bg * 8, 64, &r_full[rb]);
        }
        ++it;
        return true;
      };
      for (int item = item0; item < item1 && ok; ++item) {
        const BackItem w = back_item(items, item);
        // the pages are an input of the whole pass, the rows are not: the first item's pages go first,
        // later ones' after the rows, which the next step may be waiting for
        if (!keys || item == item0) ok = load_pages(w);
        if (!keys) continue;
        if (item == item0) grid_dep_wait();
#pragma unroll 1
        for (int c0 = 0; c0 < w.n_cands && ok; c0 += kBackRowsCands) {
          ok = load_rows(w, c0);
          if (ok && c0 == 0 && item > item0) ok = load_pages(w);
        }
      }
      // every copy issued above has landed before this CTA ends
      if (keys) {
        for (uint32_t v = ki > 2 ? ki - 2 : 0; v < ki; ++v)
          if (!mbar_wait(&k_full[v & 1u], (v >> 1) & 1u, err)) break;
        for (uint32_t v = it > kBackRowStages ? it - kBackRowStages : 0; v < it; ++v)
          if (!mbar_wait(&r_full[v % kBackRowStages], (v / kBackRowStages) & 1u, err)) break;
      } else if (ki > 0) {
        mbar_wait(v_full, (ki - 1) & 1u, err);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMAs (the whole warp; one elected lane issues)
    const uint32_t id_s = idesc_bf16_f32(128, 64);
    const uint32_t id_v = idesc_bf16_f32(128, 128) | kIdescMnMajorA;
    const uint32_t id_q = idesc_bf16_f32(128, 64) | kIdescMnMajorA | kIdescMnMajorB;
    // Each step's S and dP, then its products, in order; S and dP of the next step go first when they
    // can.  One copy of each sequence and rolled loops: the code of a step is fetched once per launch
    // (unrolled, with S at three places, the first product phase of a launch took ~7,000 cycles, the
    // later ones ~2,500).
    auto test_all = [&](uint64_t* bar, uint32_t phase) { return __all_sync(0xffffffffu, mbar_test(bar, phase & 1u)); };
    struct Step {   // a step: four candidates of an item
      int item, c0;
      uint32_t it, ki;
      BackItem w;
    };
    auto advance = [&](Step& s) {
      ++s.it;
      s.c0 += kBackRowsCands;
      if (s.c0 >= s.w.n_cands) {
        s.c0 = 0;
        ++s.ki;
        if (++s.item < item1) s.w = back_item(items, s.item);
      }
    };
    Step so;   // the next S, dP
    so.item = item0;
    so.c0 = 0;
    so.it = so.ki = 0;
    if (item0 < item1) so.w = back_item(items, item0);
    Step oo = so;   // the next products
    const uint32_t k0 = smem_u32(base + SM::kK), v0 = smem_u32(base + SM::kV), rows0 = smem_u32(base + SM::kRowBuf), w0 = smem_u32(base + SM::kW);
    uint32_t spins = 0;
    uint64_t idle = 0;
    while (oo.item < item1) {
      const uint32_t so_st = so.ki & 1u, so_rb = so.it % kBackRowStages;
      if (so.item < item1 && (so.it == oo.it || (so.it == oo.it + 1 && test_all(s_free, oo.it))) &&
          test_all(&r_full[so_rb], so.it / kBackRowStages) && test_all(&k_full[so_st], so.ki >> 1) &&
          test_all(v_full, so.ki)) {
        tc_fence_after();
#pragma unroll 1
        for (uint32_t x = 0; x < 2; ++x) {   // K q^T, then V dO^T
          const uint64_t a0 = desc_sw128_s(x ? v0 : k0 + so_st * SM::kTile, 1024, 1024);
          const uint64_t b0 = desc_sw128_s(rows0 + (2 * so_rb + x) * SM::kRows, 1024, SM::kGroup);
          const uint32_t d = tmem + (x ? kBackColP : kBackColS);
#pragma unroll
          for (int kk = 0; kk < HD / 16; ++kk)
            umma_bf16_w(d, a0 + (((kk >> 2) * SM::kSub + (kk & 3) * 32) >> 4),
                        b0 + (((kk >> 2) * 1024 + (kk & 3) * 32) >> 4), id_s, kk > 0 ? 1u : 0u);
        }
        umma_commit_w(s_full);
        if (so.c0 + kBackRowsCands >= so.w.n_cands) umma_commit_w(v_empty);
        advance(so);
        spins = 0;
      } else if (so.it > oo.it && test_all(p_full, oo.it)) {
        const uint32_t st = oo.ki & 1u, rb = oo.it % kBackRowStages;
        const int pairs = (min(kBackRowsCands, oo.w.n_cands - oo.c0) + 1) >> 1;   // 16 rows per MMA
        const bool last = oo.c0 + kBackRowsCands >= oo.w.n_cands;
        bool ok = true;
#pragma unroll 1
        for (uint32_t x = 0; x < 2 && ok; ++x) {   // dV from dO and w, then dK from q and ds
          // the first step of an item waits until the previous item's dV (dK) has been read out
          if (oo.c0 == 0 && oo.ki > 0) ok = __all_sync(0xffffffffu, mbar_wait(&acc_free[x], (oo.ki - 1) & 1u, err));
          tc_fence_after();
          uint64_t a0 = desc_sw128_s(rows0 + (2 * rb + 1 - x) * SM::kRows, 1024, SM::kCand);
          uint64_t b0 = desc_sw128_s(w0 + x * SM::kSub, 1024, 1024);
          const uint32_t d = tmem + (x ? kBackColK : kBackColV);
          uint32_t acc = oo.c0 > 0 ? 1u : 0u;
#pragma unroll 1
          for (int pr = 0; pr < pairs; ++pr) {
            umma_bf16_w(d, a0, b0, id_v, acc);
            umma_bf16_w(d, a0, b0 + (64 >> 4), id_v, 1u);
            umma_bf16_w(d, a0 + (SM::kGroup >> 4), b0, id_v, 1u);
            acc = 1u;
            a0 += (2 * SM::kCand) >> 4;
            b0 += 32 >> 4;
          }
          if (last) umma_commit_w(&acc_full[x]);
        }
        if (!ok) break;
        uint64_t a0 = desc_sw128_s(k0 + st * SM::kTile, SM::kSub, 1024);
        uint64_t b0 = desc_sw128_s(w0 + SM::kSub, SM::kSub, 1024);
#pragma unroll 1
        for (int ks = 0; ks < oo.w.n_pages; ++ks) {   // 16 tokens per MMA
          umma_bf16_w(tmem + kBackColQ, a0, b0, id_q, ks > 0 ? 1u : 0u);
          a0 += 2048 >> 4;
          b0 += 2048 >> 4;
        }
        umma_commit_w(o_full);
        umma_commit_w(&r_empty[rb]);
        if (last) umma_commit_w(&k_empty[st]);
        advance(oo);
        spins = 0;
      } else if ((++spins & 255u) == 0u) {   // bounded like every other wait
        const uint64_t now = global_timer_ns();
        if (spins == 256u) idle = now;
        if (now - idle > kErrPollNs && *(volatile int*)err != 0) break;
        if (now - idle > kWaitTimeoutNs) {
          if (lane == 0) atomicCAS(err, 0, kDevTimeout);
          break;
        }
      }
    }
  } else if (warp < 10) {
    // ------------------------------------------------ w and ds (two threads per token), and dq
    const int w4 = warp & 3;            // TMEM lane quadrant
    const int half = (warp - 2) >> 2;   // candidates 2 half, 2 half + 1 of a step
    const int t = w4 * 32 + lane;       // token (S, dP) or head-dim element (dq) of this thread
    const uint32_t trow = tmem + (static_cast<uint32_t>(w4 * 32) << 16);
    const float scale = rsqrtf(static_cast<float>(HD));
    const bool out_lane = HD == 128 || w4 < 2;   // lanes past HD hold nothing
    grid_dep_wait();
    // dq of a step (candidates c0 .. of item w): its sums out of TMEM, then added
    auto dq_load = [&](float (&v)[16]) {
      float a[16], b[16];
      tmem_ld16_nowait(trow + kBackColQ + 16 * half, a);
      tmem_ld16_nowait(trow + kBackColQ + 32 + 16 * half, b);
      tmem_wait_ld();
      tmem_hold(a);
      tmem_hold(b);
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = a[j] + b[j];
    };
    auto dq_add = [&](const float (&v)[16], const BackItem& w, int c0) {
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
        const int c = c0 + 2 * half + cc;
        if (c >= w.n_cands || !out_lane) break;
        float* dst = dq + (static_cast<int64_t>(__ldg(cands + w.cand_off + c)) * n_q + w.g * G) * HD + t;
#pragma unroll
        for (int r = 0; r < 8; ++r)
          if (r < G) atomicAdd(dst + r * HD, v[cc * 8 + r]);
      }
    };
    uint32_t it = 0;
    bool ok = true;
    BackItem next{}, prev{};
    int prev_c0 = 0;
    float dqv[16];
    if (item0 < item1) next = back_item(items, item0);
    for (int item = item0; item < item1; ++item) {
      const BackItem w = next;   // the item after this one: read now, used an item later
      if (item + 1 < item1) next = back_item(items, item + 1);
      for (int c0 = 0; c0 < w.n_cands; c0 += kBackRowsCands, ++it) {
        const uint32_t rb = it % kBackRowStages;
        // this thread's candidates; the second half has none when the step is one pair
        const int mine = min(2, w.n_cands - c0 - 2 * half);
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&r_full[rb], (it / kBackRowStages) & 1u, err));   // lse and D
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(s_full, it & 1u, err));
        tc_fence_after();
        uint4 whi[2], wlo[2], dhi[2], dlo[2];
        const bool live = ok && t < w.n_tokens;
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          whi[cc] = wlo[cc] = dhi[cc] = dlo[cc] = make_uint4(0u, 0u, 0u, 0u);
          if (cc >= mine || !ok) continue;   // (uniform)
          const int slot = 2 * half + cc;
          float s[16], p[16];
          tmem_ld16_nowait(trow + kBackColS + 16 * slot, s);
          tmem_ld16_nowait(trow + kBackColP + 16 * slot, p);
          tmem_wait_ld();
          tmem_hold(s);
          tmem_hold(p);
          const float2* ml = reinterpret_cast<const float2*>(base + SM::kMeta + rb * 256) + slot * 8;
          float wv[8], dv[8];
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const float2 m = ml[r];
            const float x = s[r] + s[8 + r], dp = p[r] + p[8 + r];
            // expf, not exp2 of the product with log2(e): one rounding less of an exponent that may be far
            // below zero (weights at -46 to -62 within 4.9e-7 in the mean instead of 1.75e-6), in the same time
            wv[r] = live ? expf(x * scale - m.x) : 0.f;
            dv[r] = live ? wv[r] * (dp - m.y) * scale : 0.f;
          }
          split8(wv, &whi[cc], &wlo[cc]);
          split8(dv, &dhi[cc], &dlo[cc]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(s_free);   // the next step's S and dP may overwrite these
        // the products that read the previous step's w and ds are done, and its dq is complete
        if (it > 0 && ok) ok = __all_sync(0xffffffffu, mbar_wait(o_full, (it - 1) & 1u, err));
        tc_fence_after();
        const bool add = it > 0 && ok;
        if (add) dq_load(dqv);
        if (mine > 0) {   // an odd candidate's partner in its pair is zero
#pragma unroll
          for (int cc = 0; cc < 2; ++cc) {
            const int ch = 2 * half + cc;
            uint8_t* wr = base + SM::kW + t * 128;
            uint8_t* dr = base + SM::kDs + t * 128;
            const int ohi = (ch ^ (t & 7)) << 4, olo = ((4 + ch) ^ (t & 7)) << 4;
            *reinterpret_cast<uint4*>(wr + ohi) = whi[cc];
            *reinterpret_cast<uint4*>(wr + olo) = wlo[cc];
            *reinterpret_cast<uint4*>(dr + ohi) = dhi[cc];
            *reinterpret_cast<uint4*>(dr + olo) = dlo[cc];
          }
          fence_proxy_async_smem();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(p_full);
        if (add) dq_add(dqv, prev, prev_c0);
        prev = w;
        prev_c0 = c0;
      }
    }
    if (it > 0 && ok && __all_sync(0xffffffffu, mbar_wait(o_full, (it - 1) & 1u, err))) {
      tc_fence_after();
      dq_load(dqv);
      dq_add(dqv, prev, prev_c0);
    }
  } else if (warp < 14) {
    // ------------------------------------------------ results (a thread per head-dim element; a column is a token)
    const int w4 = warp & 3;
    const uint32_t trow = tmem + (static_cast<uint32_t>(w4 * 32) << 16);
    const int64_t page_elems = static_cast<int64_t>(2) * n_kv * 16 * HD;
    const bool out_lane = HD == 128 || w4 < 2;
    grid_dep_wait();
    uint32_t ki = 0;
    bool ok = true;
    BackItem next{};
    if (item0 < item1) next = back_item(items, item0);
    for (int item = item0; item < item1; ++item, ++ki) {
      const BackItem w = next;
      if (item + 1 < item1) next = back_item(items, item + 1);
      // lane i: page i of the item
      const uint32_t my_page = lane < w.n_pages ? __ldg(pages + w.page_off + lane) : 0u;
#pragma unroll 1
      for (int x = 0; x < 2; ++x) {   // dV, then dK; the pool's layout: keys, then values
        float* const out0 = grad_layer + (x ? 0 : n_kv * 16 * HD) + w.g * 16 * HD + w4 * 32 + lane;
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[x], ki & 1u, err));
        tc_fence_after();
#pragma unroll 1
        for (int i = 0; i < w.n_pages && ok; ++i) {
          float v[16];
          tmem_ld16(trow + (x ? kBackColK : kBackColV) + 16 * i, v);
          const uint32_t page = __shfl_sync(0xffffffffu, my_page, i);
          if (!out_lane) continue;
          float* dst = out0 + (page & ~kBackAtomicPage) * page_elems;
          if (page & kBackAtomicPage) {
#pragma unroll
            for (int j = 0; j < 16; ++j) atomicAdd(dst + j * HD, v[j]);
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) dst[j * HD] = v[j];
          }
        }
        tc_fence_before();   // all read: the next item's products may overwrite them
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_free[x]);
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kBackTmemCols);
  }
}

// One CTA per row: [dq; dk; dv] before RoPE (the rotation by the negative angle of position L_b)
// as the bf16 hi/lo input of the W_qkv^T product, [n][(n_q + 2 n_kv) hd].
__global__ void rope_back_kernel(const float* __restrict__ dq, const float* __restrict__ dks,
                                 const float* __restrict__ dvs, const float2* __restrict__ rope, int n_q, int n_kv,
                                 int hd, bf16* __restrict__ o_hi, bf16* __restrict__ o_lo) {
  grid_dep_launch();
  grid_dep_wait();
  const int b = blockIdx.x, half = hd / 2, quads = half / 4;
  const int64_t ob = static_cast<int64_t>(b) * (n_q + 2 * n_kv) * hd;
#pragma unroll 1
  for (int e = threadIdx.x; e < (n_q + n_kv) * quads; e += blockDim.x) {   // four pairs i .. i + 3 of a head
    const int head = e / quads, i = 4 * (e - head * quads);
    const float* src = head < n_q ? dq + (static_cast<int64_t>(b) * n_q + head) * hd
                                  : dks + (static_cast<int64_t>(b) * n_kv + head - n_q) * hd;
    const float4* rp = reinterpret_cast<const float4*>(rope + static_cast<int64_t>(b) * half + i);
    const float4 r0 = rp[0], r1 = rp[1];   // (cos, sin) of pairs i, i + 1 / i + 2, i + 3
    const float4 x = *reinterpret_cast<const float4*>(src + i), y = *reinterpret_cast<const float4*>(src + i + half);
    put_hilo4(o_hi, o_lo, ob + head * hd + i,
              make_float4(x.x * r0.x + y.x * r0.y, x.y * r0.z + y.y * r0.w, x.z * r1.x + y.z * r1.y, x.w * r1.z + y.w * r1.w));
    put_hilo4(o_hi, o_lo, ob + head * hd + i + half,
              make_float4(y.x * r0.x - x.x * r0.y, y.y * r0.z - x.y * r0.w, y.z * r1.x - x.z * r1.y, y.w * r1.z - x.w * r1.w));
  }
  for (int e = 4 * threadIdx.x; e < n_kv * hd; e += 4 * blockDim.x)
    put_hilo4(o_hi, o_lo, ob + (n_q + n_kv) * hd + e,
              *reinterpret_cast<const float4*>(dvs + static_cast<int64_t>(b) * n_kv * hd + e));
}

// Zero every layer's gradient of the listed pages.
__global__ void zero_pages_kernel(float* __restrict__ grad, const int32_t* __restrict__ pages, int n_list,
                                  int n_layers, int64_t n_pages, int64_t page_elems) {
  grid_dep_launch();
  grid_dep_wait();
  const int64_t per = page_elems / 4;
  const int64_t total = static_cast<int64_t>(n_list) * n_layers * per;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t e = i % per, rest = i / per;
    const int64_t l = rest % n_layers, k = rest / n_layers;
    float4* dst = reinterpret_cast<float4*>(grad + (l * n_pages + pages[k]) * page_elems) + e;
    *dst = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// kv <- RNE_bf16(kv - eta grad) for every layer of the listed pages.
__global__ void steer_update_kernel(bf16* __restrict__ kv, const float* __restrict__ grad,
                                    const int32_t* __restrict__ pages, int n_list, int n_layers, int64_t n_pages,
                                    int64_t page_elems, float eta) {
  grid_dep_launch();
  grid_dep_wait();
  const int64_t per = page_elems / 4;
  const int64_t total = static_cast<int64_t>(n_list) * n_layers * per;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t e = i % per, rest = i / per;
    const int64_t l = rest % n_layers, k = rest / n_layers;
    const int64_t base = (l * n_pages + pages[k]) * page_elems + 4 * e;
    const float4 gr = *reinterpret_cast<const float4*>(grad + base);
    uint2 raw = *reinterpret_cast<const uint2*>(kv + base);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
    const float2 c = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
    const __nv_bfloat162 na = __floats2bfloat162_rn(a.x - eta * gr.x, a.y - eta * gr.y);
    const __nv_bfloat162 nc = __floats2bfloat162_rn(c.x - eta * gr.z, c.y - eta * gr.w);
    raw.x = *reinterpret_cast<const uint32_t*>(&na);
    raw.y = *reinterpret_cast<const uint32_t*>(&nc);
    *reinterpret_cast<uint2*>(kv + base) = raw;
  }
}

// Launch with programmatic dependent launch: the kernel may start while the previous one in the
// stream drains; every kernel here waits (griddepcontrol.wait) before touching what that one writes.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

unsigned grid_1d(int64_t total, int threads) {
  int64_t b = (total + threads - 1) / threads;
  if (b > 152 * 16) b = 152 * 16;
  return static_cast<unsigned>(b < 1 ? 1 : b);
}

// threads of a row's CTA: four elements each, at most 1024
dim3 row_threads(int d) { return dim3(static_cast<unsigned>(std::min(1024, (d / 4 + 31) / 32 * 32))); }

}  // namespace

cudaError_t launch_transpose(const __nv_bfloat16* in, __nv_bfloat16* out, int rows, int cols, cudaStream_t st) {
  const dim3 grid((cols + 31) / 32, (rows + 31) / 32);
  if (grid.y > 65535u) return cudaErrorInvalidValue;
  transpose_kernel<<<grid, dim3(32, 8), 0, st>>>(in, out, rows, cols);
  return cudaGetLastError();
}

cudaError_t launch_head_back(const float* h, const float* p_plus, const __nv_bfloat16* gain,
                             const __nv_bfloat16* w_plus, const __nv_bfloat16* w_minus, int n, int d, float eps,
                             float* dh, __nv_bfloat16* dh_hi, __nv_bfloat16* dh_lo, cudaStream_t st) {
  return launch_pdl(head_back_kernel, dim3(n), row_threads(d), 0, st, h, p_plus, gain, w_plus, w_minus, d, eps, dh, dh_hi,
                    dh_lo);
}

cudaError_t launch_rms_back(const float* h, const __nv_bfloat16* h_bf16, const __nv_bfloat16* gain, const float* dy,
                            const float* dres, int n, int d, float eps, float* out, __nv_bfloat16* o_hi,
                            __nv_bfloat16* o_lo, cudaStream_t st) {
  return launch_pdl(rms_back_kernel, dim3(n), row_threads(d), 0, st, h, h_bf16, gain, dy, dres, d, eps, out, o_hi, o_lo);
}

cudaError_t launch_silu_back(const float* da, const float* gu, int n, int ff, __nv_bfloat16* o_hi,
                             __nv_bfloat16* o_lo, cudaStream_t st) {
  return launch_pdl(silu_back_kernel, dim3(grid_1d(static_cast<int64_t>(n) * (ff / 4), 256)), dim3(256), 0, st, da, gu, n,
                    ff, o_hi, o_lo);
}

cudaError_t launch_attn_back(const AttnBackArgs& a, cudaStream_t st) {
  if (a.n_q / a.n_kv > kMaxGroup || (a.hd != 64 && a.hd != 128)) return cudaErrorInvalidValue;
  const int G = a.n_q / a.n_kv;
  const bool tc = G <= 8 && a.tm_pool_tc != nullptr;
  cudaError_t e = launch_pdl(attn_back_pre_kernel, dim3(a.n * a.n_kv), dim3(256), 0, st, a.q, a.kself, a.vself, a.o,
                             a.dout, a.lse, a.n_q, a.n_kv, a.hd, a.D, a.dq, a.dks, a.dvs, tc ? a.ops : nullptr, a.meta);
  if (e != cudaSuccess) return e;
  if (tc) {
    if (a.n_ctas == 0) return e;
    const dim3 grid(a.n_ctas);
    if (a.hd == 128)
      return launch_pdl(attn_back_tc_kernel<128>, grid, dim3(kBackThreads), BackSmem<128>::kBytes, st, *a.tm_pool_tc,
                        a.layer_page0, a.items, a.cta_item, a.item_pages, a.item_cands, a.ops, a.zero_rows, a.meta, a.n_q,
                        a.n_kv, a.grad_layer, a.dq, a.err);
    return launch_pdl(attn_back_tc_kernel<64>, grid, dim3(kBackThreads), BackSmem<64>::kBytes, st, *a.tm_pool_tc,
                      a.layer_page0, a.items, a.cta_item, a.item_pages, a.item_cands, a.ops, a.zero_rows, a.meta, a.n_q,
                      a.n_kv, a.grad_layer, a.dq, a.err);
  }
  if (a.n_units == 0) return e;
  const size_t smem = a.hd == 128 ? back_pages_smem<128>() : back_pages_smem<64>();
  cudaError_t le = cudaSuccess;
  auto go = [&](auto kern) {
    le = launch_pdl(kern, dim3(a.n_units), dim3(128), smem, st, a.units, a.seq_lens, a.block_table, a.max_blocks,
                    a.pool_layer, a.shared, a.q, a.dout, a.lse, a.D, a.n_q, a.n_kv, a.grad_layer, a.dq, a.err);
  };
  if (a.hd == 128) {
    if (G <= 4)
      go(attn_back_pages_kernel<128, 4>);
    else if (G <= 8)
      go(attn_back_pages_kernel<128, 8>);
    else
      go(attn_back_pages_kernel<128, 16>);
  } else {
    if (G <= 4)
      go(attn_back_pages_kernel<64, 4>);
    else if (G <= 8)
      go(attn_back_pages_kernel<64, 8>);
    else
      go(attn_back_pages_kernel<64, 16>);
  }
  return le;
}

cudaError_t grad_configure() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto kern, size_t bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
  };
  set(attn_back_pages_kernel<128, 4>, back_pages_smem<128>());
  set(attn_back_pages_kernel<128, 8>, back_pages_smem<128>());
  set(attn_back_pages_kernel<128, 16>, back_pages_smem<128>());
  set(attn_back_pages_kernel<64, 4>, back_pages_smem<64>());
  set(attn_back_pages_kernel<64, 8>, back_pages_smem<64>());
  set(attn_back_pages_kernel<64, 16>, back_pages_smem<64>());
  set(attn_back_tc_kernel<128>, BackSmem<128>::kBytes);
  set(attn_back_tc_kernel<64>, BackSmem<64>::kBytes);
  return e;
}

// Tensor cores: full pages that the same candidates (at least two) read, each once, form a group, cut
// into items of kBackTilePages pages per kv head; every other page of a candidate goes to items of its
// own, in logical order.  When the groups' items leave SMs idle, a group's candidates are split over
// several items (in fours, one step of the kernel each) whose pages then accumulate atomically.  The
// persistent CTAs get equal shares under a cost model: 9 units of 1/16 us a page and 8 an item (a
// private item moves 24 KB a page, ~0.56 us at an SM's share of HBM) and 22 every step after the first
// (measured ~1.4 us).  Items of several steps go to the least loaded CTA, longest first; the private
// pages then fill every CTA to the common level, cut wherever that falls.
// CUDA cores: units of kBackUnitPagesMax pages per candidate and kv head.
constexpr int64_t kBackPageCost = 9, kBackItemCost = 8, kBackStepCost = 22;

void plan_attn_back(const int32_t* bt, const int32_t* sl, int n, int max_blocks, int64_t n_pages, int n_kv,
                    bool tensor_cores, int n_sms, BackPlan& p) {
  p = BackPlan();
  const size_t np = static_cast<size_t>(std::max<int64_t>(n_pages, 1));
  std::vector<int32_t> refs(np + 1, 0);
  for (int b = 0; b < n; ++b)
    for (int j = 0, pg = (sl[b] + 15) / 16; j < pg; ++j) ++refs[bt[static_cast<int64_t>(b) * max_blocks + j]];
  p.atomic.assign(np, 0);
  std::vector<uint8_t> grouped(np, 0);
  std::vector<BackItem> shared;
  if (!tensor_cores) {
    for (int b = 0; b < n; ++b) {
      const int pages = (sl[b] + 15) / 16;
      for (int g = 0; g < n_kv; ++g)
        for (int j0 = 0; j0 < pages; j0 += kBackUnitPagesMax)
          p.units.push_back(make_int4(b, g, j0, std::min(pages, j0 + kBackUnitPagesMax)));
    }
  } else {
    // the full references of every page read at least twice, by page
    std::vector<int32_t> off(np + 1, 0), list;
    for (size_t i = 0; i < np; ++i) off[i + 1] = off[i] + (refs[i] > 1 ? refs[i] : 0);
    if (off[np] > 0) {
      list.assign(static_cast<size_t>(off[np]), -1);
      std::vector<int32_t> fill(off.begin(), off.end() - 1);
      for (int b = 0; b < n; ++b)
        for (int j = 0, full = sl[b] / 16; j < full; ++j) {
          const int32_t pg = bt[static_cast<int64_t>(b) * max_blocks + j];
          if (refs[pg] > 1) list[fill[pg]++] = b;
        }
      std::map<std::vector<int32_t>, std::vector<int32_t>> groups;   // candidates -> pages
      std::vector<int32_t> key;
      std::vector<int32_t>* last = nullptr;
      for (size_t i = 0; i < np; ++i) {
        const int32_t c = refs[i];
        if (c < 2 || fill[i] - off[i] != c) continue;   // some reference is partial
        const int32_t* r = list.data() + off[i];
        bool twice = false;
        for (int32_t k = 1; k < c; ++k) twice = twice || r[k] == r[k - 1];
        if (twice) continue;
        if (!last || key.size() != static_cast<size_t>(c) || !std::equal(key.begin(), key.end(), r)) {
          key.assign(r, r + c);
          last = &groups[key];
        }
        last->push_back(static_cast<int32_t>(i));
        grouped[i] = 1;
      }
      int64_t tiles = 0;
      for (const auto& kv : groups) tiles += (static_cast<int64_t>(kv.second.size()) + kBackTilePages - 1) / kBackTilePages;
      const int64_t room = std::max<int64_t>(1, tiles > 0 ? n_sms / (tiles * n_kv) : 1);   // items a group's tile may become
      for (const auto& kv : groups) {
        const std::vector<int32_t>&cs = kv.first, &pg = kv.second;
        const int steps = (static_cast<int>(cs.size()) + 3) / 4;
        const int parts = static_cast<int>(std::min<int64_t>(room, steps));
        const int page0 = static_cast<int>(p.item_pages.size()), cand0 = static_cast<int>(p.item_cands.size());
        p.item_pages.insert(p.item_pages.end(), pg.begin(), pg.end());
        p.item_cands.insert(p.item_cands.end(), cs.begin(), cs.end());
        for (size_t k = 0; k < pg.size(); k += kBackTilePages)
          for (int q = 0; q < parts; ++q) {
            const int c0 = 4 * (steps * q / parts), c1 = std::min<int>(4 * (steps * (q + 1) / parts), static_cast<int>(cs.size()));
            const int m = static_cast<int>(std::min<size_t>(kBackTilePages, pg.size() - k));
            for (int g = 0; g < n_kv; ++g)
              shared.push_back(BackItem{g, page0 + static_cast<int>(k), m, 16 * m, cand0 + c0, c1 - c0, {0, 0}});
          }
        if (parts > 1)
          for (int32_t x : pg) p.atomic[x] = 1;
      }
    }
    // private runs: every other page of a candidate
    struct Run {
      int32_t page_off, n_pages, last, cand_off;
    };
    std::vector<Run> runs;
    int64_t pages = 0;
    for (int b = 0; b < n; ++b) {
      const int32_t page0 = static_cast<int32_t>(p.item_pages.size());
      int32_t last = 0;   // valid tokens of the last page listed
      for (int j = 0, pg = (sl[b] + 15) / 16; j < pg; ++j) {
        const int32_t x = bt[static_cast<int64_t>(b) * max_blocks + j];
        if (grouped[x]) continue;
        p.item_pages.push_back(x);
        last = std::min(16, sl[b] - 16 * j);
      }
      const int32_t m = static_cast<int32_t>(p.item_pages.size()) - page0;
      if (m == 0) continue;
      runs.push_back(Run{page0, m, last, static_cast<int32_t>(p.item_cands.size())});
      p.item_cands.push_back(b);
      pages += static_cast<int64_t>(m) * n_kv;
    }
    // equal shares
    auto cost = [](int64_t m, int64_t steps) { return kBackItemCost + kBackPageCost * m + kBackStepCost * (steps - 1); };
    auto cost_of = [&](const BackItem& i) { return cost(i.n_pages, (i.n_cands + 3) / 4); };
    std::stable_sort(shared.begin(), shared.end(), [&](const BackItem& x, const BackItem& y) { return cost_of(x) > cost_of(y); });
    const int64_t most = static_cast<int64_t>(shared.size()) + pages;   // no more CTAs than items of a page
    const int C = static_cast<int>(std::min<int64_t>(n_sms, most));
    std::vector<std::vector<int32_t>> mine(static_cast<size_t>(C));   // shared items by CTA
    std::vector<int64_t> load(static_cast<size_t>(C), 0);
    {
      typedef std::pair<int64_t, int> Slot;   // (load, CTA), least first
      std::priority_queue<Slot, std::vector<Slot>, std::greater<Slot>> heap;
      for (int k = 0; k < C; ++k) heap.push({0, k});
      for (size_t i = 0; i < shared.size(); ++i) {
        Slot s = heap.top();
        heap.pop();
        s.first += cost_of(shared[i]);
        mine[s.second].push_back(static_cast<int32_t>(i));
        load[s.second] = s.first;
        heap.push(s);
      }
    }
    // the level that the private pages fill the CTAs below it to (an item more for each CTA's cut)
    int64_t priv = kBackPageCost * pages + kBackItemCost * C;
    for (const Run& x : runs) priv += kBackItemCost * n_kv * ((x.n_pages + kBackTilePages - 1) / kBackTilePages);
    std::vector<int64_t> sorted(load);
    std::sort(sorted.begin(), sorted.end());
    int64_t level = 0, sum = 0;
    for (int k = 0; k < C; ++k) {
      sum += sorted[k];
      level = (sum + priv + k) / (k + 1);
      if (k + 1 == C || level <= sorted[k + 1]) break;
    }
    size_t r = 0;
    int32_t at = 0, g = 0;   // next private page: run r, kv head g, page `at`
    int64_t left = pages, given = 0, want = 0;   // private cost laid, and due once CTA k is filled
    p.cta_item.push_back(0);
    for (int k = 0; k < C; ++k) {
      for (int32_t i : mine[k]) p.items.push_back(shared[i]);
      want += std::max<int64_t>(0, level - load[k]);
      const bool all = k + 1 == C;
      while (left > 0 && (all || given + kBackPageCost / 2 < want)) {
        const Run& run = runs[r];
        int64_t m = std::min<int64_t>(kBackTilePages, run.n_pages - at);
        if (!all) m = std::max<int64_t>(1, std::min<int64_t>(m, (want - given - kBackItemCost + kBackPageCost / 2) / kBackPageCost));
        const bool end = at + m == run.n_pages;
        p.items.push_back(BackItem{g, run.page_off + at, static_cast<int32_t>(m),
                                   static_cast<int32_t>(16 * (m - 1) + (end ? run.last : 16)), run.cand_off, 1, {0, 0}});
        given += cost(m, 1);
        left -= m;
        at += static_cast<int32_t>(m);
        if (end) {
          at = 0;
          if (++g == n_kv) {
            g = 0;
            ++r;
          }
        }
      }
      p.cta_item.push_back(static_cast<int32_t>(p.items.size()));
    }
  }
  for (size_t i = 0; i < np; ++i)
    if (refs[i] >= 2 && !grouped[i]) p.atomic[i] = 1;
  for (uint32_t& pg : p.item_pages)
    if (p.atomic[pg]) pg |= kBackAtomicPage;
  for (size_t i = 0; i < np; ++i)
    if (p.atomic[i]) p.lists.push_back(static_cast<int32_t>(i));
  p.n_atomic = static_cast<int>(p.lists.size());
  for (size_t i = 0; i < np; ++i)
    if (refs[i] >= 1) p.lists.push_back(static_cast<int32_t>(i));
}

cudaError_t launch_rope_back(const float* dq, const float* dks, const float* dvs, const float2* rope, int n, int n_q,
                             int n_kv, int hd, __nv_bfloat16* o_hi, __nv_bfloat16* o_lo, cudaStream_t st) {
  return launch_pdl(rope_back_kernel, dim3(n), dim3(256), 0, st, dq, dks, dvs, rope, n_q, n_kv, hd, o_hi, o_lo);
}

cudaError_t launch_zero_pages(float* grad, const int32_t* pages, int n_list, int n_layers, int64_t n_pages,
                              int64_t page_elems, cudaStream_t st) {
  if (n_list == 0) return cudaSuccess;
  return launch_pdl(zero_pages_kernel, dim3(grid_1d(static_cast<int64_t>(n_list) * n_layers * (page_elems / 4), 256)),
                    dim3(256), 0, st, grad, pages, n_list, n_layers, n_pages, page_elems);
}

cudaError_t launch_steer_update(__nv_bfloat16* kv, const float* grad, const int32_t* pages, int n_list, int n_layers,
                                int64_t n_pages, int64_t page_elems, float eta, cudaStream_t st) {
  if (n_list == 0) return cudaSuccess;
  return launch_pdl(steer_update_kernel, dim3(grid_1d(static_cast<int64_t>(n_list) * n_layers * (page_elems / 4), 256)),
                    dim3(256), 0, st, kv, grad, pages, n_list, n_layers, n_pages, page_elems, eta);
}

}  // namespace kvprm
