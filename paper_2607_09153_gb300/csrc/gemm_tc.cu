// Projection GEMMs of the verify-token forward, batched over candidates (the
// c_ffn * d^2 term of Eq. cost_kv): Y[n][m] = sum_k W[m][k] * X[n][k].
//
// The weight matrix is the streamed operand (read once from HBM per call), so
// it is the MMA's A operand: M = 128 weight rows per CTA, N = the candidate
// batch padded to a multiple of 16 (16..256), K in 64-element tiles.  A
// producer thread streams W and X tiles with TMA (128-byte swizzle) through a
// multi-stage mbarrier ring; one thread issues tcgen05.mma (kind::f16, bf16 x
// bf16 -> fp32) into a TMEM accumulator.  The activation X arrives as a bf16
// (hi, lo) pair, X = hi + lo to ~2^-17 relative, so the contraction sees the
// fp32 activation (the weights are bf16 by definition).  The hi and lo tiles
// sit back to back in shared memory and one MMA of N = 2 n_pad covers both
// (each weight K slice is read from shared memory once -- the MMA issue rate
// is bounded by those reads at this small N); the two accumulator halves are
// added when TMEM is read.  Beyond N = 256 each half takes its own MMA.  From
// 48 columns on two CTAs may share an M = 256 MMA (cta_group::2), each staging
// half of its activation rows.
//
// K is split across the CTAs of a thread-block cluster (one cluster per
// 128-row tile) so that every SM streams weights.  The splits are reduced
// inside the cluster through distributed shared memory in rank order
// (deterministic, no float atomics): each CTA parks its accumulator in its own
// shared memory, and CTA r sums the candidate columns [r*N/cs, (r+1)*N/cs)
// over all ranks and applies the epilogue of the step:
//   PLAIN  out[n][m] = y
//   QKV    RoPE on the q and k rows (rotate-half pairs inside a head) -> q
//          (fp32 and bf16 hi/lo), self k, self v (fp32)
//   RESID  h[n][m] += y, the tile's sum of squares of the new h per
//          candidate, and h ⊙ g (g = the next RMSNorm's gain) as the next
//          projection's bf16 hi/lo input
//   SILU   rows are 64 gate rows and the matching 64 up rows (two TMA boxes
//          per stage; CTA pairs: 128 and 128 as two tiles); a = SiLU(gate) * up
//          as a bf16 hi/lo pair
//   LOWRANK  t = s (A x) of a scorer adapter as a bf16 hi/lo pair, the next
//          projection's last K tiles
// An RMSNorm x = g ⊙ h / sqrt(mean(h^2) + eps) between two projections is
// thereby split: the per-candidate factor r = 1/sqrt(mean(h^2) + eps) is a
// scalar of the column, so W x = r (W (h ⊙ g)); the residual epilogue writes
// h ⊙ g and the per-tile sums of squares, and the QKV and SILU epilogues scale
// their accumulators by r before RoPE / SiLU.  No normalisation kernel runs
// between the projections.
#include <type_traits>
#include "kernels.h"
#include "ptx.cuh"

namespace kvprm {

namespace {

constexpr int kBM = 128;
constexpr int kBK = 64;
constexpr uint32_t kWTileBytes = kBM * kBK * 2;   // 16 KB
// after the ring: barriers, TMEM slot and 64 block-sum floats (512 B), then 256
// per-column RMSNorm factors (1 KB)
constexpr size_t kTailBytes = 512 + 1024 + 4096;   // barriers, RMSNorm factors, preloaded residual
constexpr int kLargeCols = 48;                      // padded columns from which the large-batch images run
constexpr int kHalfBoxCols = 96;                    // padded columns from which activation boxes hold half
constexpr int kHPreCols = 8;                        // residual columns preloaded per rank (128 rows each)
constexpr size_t kGemmMaxSmem = 200 * 1024;         // dynamic shared memory the kernel is configured for
constexpr size_t kAloneSmem = 120 * 1024;           // with which no second CTA fits on an SM

// The parked accumulator of a CTA with `cols` columns: 16 of them at a time, 128 fp32 rows each.
__host__ __device__ constexpr uint32_t park_bytes(int cols) { return static_cast<uint32_t>((cols + 15) / 16 * 16) * kBM * 4; }

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~static_cast<uintptr_t>(1023));
}

__device__ __forceinline__ void store_hilo(__nv_bfloat16* hi, __nv_bfloat16* lo, int64_t i, float x) {
  const __nv_bfloat16 h = __float2bfloat16_rn(x);
  hi[i] = h;
  lo[i] = __float2bfloat16_rn(x - __bfloat162float(h));
}

// LARGE (n_pad >= 48, one kernel image per batch class so that the small-batch code keeps its own
// register allocation): the residual epilogue issues a 16-column group's residual loads before
// using any and sums each column's squares in one pass over the parked tile, clusters reduce with
// 16-byte DSMEM loads, and the epilogues move 4 or 8 consecutive rows of a column per thread
// with 16-byte accesses (the 4-warp CTA is otherwise bound by 2- and 4-byte stores and by one load
// latency per column).
// MODE: the epilogue, an image each.  A CTA runs everything after its MMAs once, so those instructions
// are fetched cold in every launch, and their number is a good part of the ~3 us from the last MMA to
// the end of a small launch.  Hence the images, rolled outer loops, counters instead of divisions by the
// stage count and shifts by the head dimension: 51 KB of code in one small image became 20-33 KB each
// (large: 178 KB became 25-53), and a call of the 1.5B workload took 1,112 us instead of 1,155, with the
// rank-256 adapter 1,687 instead of 1,932, MCTS 9,814 instead of 10,110.
// PAIR (large batches; `plan_gemm` has the rule): a CTA pair's MMA multiplies both CTAs' weight tiles (M = 256)
// with a B operand that is half in either CTA, so a CTA stages half of the activation rows.  At 256
// columns a stage is 48 KB instead of 80, four fit instead of two, and a K tile's L2 reads fall from 80 KB
// to 48: with two stages an m-tile's eight MMAs (0.53 us) waited for loads 0.35 us of every K tile.
// LORA: the projection takes a scorer adapter's K tiles after its own (QKV, RESID, SILU).  Images of their own: in
// shared ones the loader's choices and the mark's acquire cost both kinds of call (1.5B, 16 candidates, rank 256:
// 1,518 us a call, apart 1,511; beam without an adapter 3,428, apart 3,418).
template <bool LARGE, int MODE, bool PAIR, bool LORA>
__global__ void __launch_bounds__(256, 2) gemm_cluster_kernel(const __grid_constant__ CUtensorMap tmW,
                                                           const __grid_constant__ CUtensorMap tmX,
                                                           const __grid_constant__ CUtensorMap tmXlo, int has_lo,
                                                           const __grid_constant__ CUtensorMap tmB,
                                                           const __grid_constant__ CUtensorMap tmT,
                                                           const __grid_constant__ CUtensorMap tmTlo, int k_main,
                                                           int k_tiles, int cs, int stages, uint32_t tmem_cols,
                                                           int n_pad, int n_split, GemmEpilogue ep, int* err,
                                                           unsigned long long* ts) {
  trace_begin(ts);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  constexpr bool silu = MODE == GemmEpilogue::SILU;
  // weight tiles of this CTA, which a stage holds ahead of the activation tile(s): a gate/up pair's CTA
  // has 128 gate rows and the matching 128 up rows, so that either is the other's TMEM lane for lane
  constexpr int mt = PAIR && silu ? 2 : 1;
  const uint32_t x_bytes = static_cast<uint32_t>(n_pad) * kBK * 2;
  const uint32_t w_bytes = kWTileBytes * static_cast<uint32_t>(mt);
  // PAIR: half of the pair's activation rows, i.e. one part's n_pad rows or half of each part's
  const uint32_t stage_bytes = w_bytes + x_bytes * (has_lo && !PAIR ? 2u : 1u);
  const uint32_t acc_bytes = park_bytes(n_pad);
  const uint32_t ring_bytes = stages * stage_bytes > acc_bytes ? stages * stage_bytes : acc_bytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + ring_bytes);
  uint64_t* empty = full + stages;
  uint64_t* done = empty + stages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  float* red = reinterpret_cast<float*>(tmem_slot + 4);   // 64 floats for per-column block sums
  float* rsc = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(full) + 512);   // RMSNorm factor per column
  float* hpre = rsc + 256;   // RESID: this rank's columns of h for the tile's rows, [c - cbeg][128]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // PAIR: cluster ranks 2 r and 2 r + 1 are split r's CTA pair, with an m-tile each
  const uint32_t crank = cluster_rank();
  const uint32_t rank = PAIR ? crank >> 1 : crank, side = PAIR ? crank & 1u : 0u;
  // of the two m-tiles' n_pad columns, or (n_split 2, n_pad then the half) of one half of the batch's
  const int pair_unit = static_cast<int>(blockIdx.x) / (2 * cs);
  const int m_tile = PAIR ? pair_unit / n_split * 2 + static_cast<int>(side)
                           : static_cast<int>(blockIdx.x) / cs;   // (gate/up pairs: of 128 gate rows)
  const int c_off = PAIR ? pair_unit % n_split * n_pad : 0;   // first column
  // the cluster rank of split r's CTA for this m-tile
  auto peer = [&](int r) { return PAIR ? 2u * static_cast<uint32_t>(r) + side : static_cast<uint32_t>(r); };
  const int kps = (k_tiles + cs - 1) / cs;
  const int kt0 = static_cast<int>(rank) * kps;
  const int kt1 = min(k_tiles, kt0 + kps);
  const int nk = kt1 > kt0 ? kt1 - kt0 : 0;
  // this rank's candidate columns in the reduction and the epilogue
  const int cols = n_pad / cs;
  const int cbeg = c_off + static_cast<int>(rank) * cols;
  const int cend = min(cbeg + cols, ep.n_valid);
  const int nc = cend > cbeg ? cend - cbeg : 0;
  const bool hpreload = MODE == GemmEpilogue::RESID && nc <= kHPreCols;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmW);
    tma_prefetch_desc(&tmX);
    if (has_lo) tma_prefetch_desc(&tmXlo);
    if constexpr (LORA) {
      tma_prefetch_desc(&tmB);
      tma_prefetch_desc(&tmT);
      if (has_lo) tma_prefetch_desc(&tmTlo);
    }
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      tmem_alloc_pair(tmem_slot, tmem_cols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, tmem_cols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  if constexpr (PAIR)
    cluster_sync();   // the pair uses each other's barriers and tensor memory
  else
    __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // Let the next kernel in the stream start its own independent prologue and
  // streaming now (or, with late_trigger, once the partials are parked); it
  // waits for this grid's completion before touching what this grid writes.
  // LOWRANK lets it start once the activations it reads are there (below).
  if (MODE != GemmEpilogue::LOWRANK && !ep.late_trigger) grid_dep_launch();

  if (warp == 0 && lane == 0 && nk > 0) {
    // ---------------- TMA producer
    const uint64_t pol_w = policy_evict_first();
    const uint64_t pol_x = policy_evict_last();
    // K tiles [0, k_main) come from W and x; a scorer adapter's tiles after them from B and t
    auto load = [&](uint8_t* dst, const CUtensorMap* map, int stage, int x, int y, uint64_t pol) {
      if constexpr (PAIR)   // both CTAs' copies complete on the even CTA's barrier, which its MMAs wait for
        tma_load_2d_pair(dst, map, cluster_addr(&full[stage], crank & ~1u), x, y, pol);
      else
        tma_load_2d(dst, map, &full[stage], x, y, pol);
    };
    auto load_w = [&](int stage, int kt) {
      if (!PAIR)
        mbar_arrive_expect_tx(&full[stage], stage_bytes);
      else if (side == 0)
        mbar_arrive_expect_tx(&full[stage], 2 * stage_bytes);
      const bool main = !LORA || kt < k_main;
      const CUtensorMap* wm = main ? &tmW : &tmB;
      const int kx = (main ? kt : kt - k_main) * kBK;
      uint8_t* wt = smem + stage * stage_bytes;
      if constexpr (!silu) {
        load(wt, wm, stage, kx, m_tile * kBM, pol_w);
      } else {   // mt x 64 gate rows, then the matching up rows, in boxes of 64
#pragma unroll 1
        for (int t = 0; t < 2 * mt; ++t)
          load(wt + t * (kWTileBytes / 2), wm, stage, kx,
               (t < mt ? 0 : ep.ff) + (m_tile * mt + (t < mt ? t : t - mt)) * 64, pol_w);
      }
    };
    // the activation maps' boxes hold the batch's columns, from 96 on half of them (gemm_x_box): a stage's
    // rows are then loaded as halves (hi, hi, lo, lo), of which a pair's CTA takes its own
    auto load_x = [&](int stage, int kt) {
      const bool main = !LORA || kt < k_main;
      const int kx = (main ? kt : kt - k_main) * kBK;
      const CUtensorMap *xh = main ? &tmX : &tmT, *xl = main ? &tmXlo : &tmTlo;
      uint8_t* xt = smem + stage * stage_bytes + w_bytes;
      if (PAIR && n_split == 2) {
        load(xt, side ? xl : xh, stage, kx, c_off, pol_x);
      } else if (!LARGE || n_pad < kHalfBoxCols) {
        if (!PAIR || side == 0) load(xt, xh, stage, kx, 0, pol_x);
        if (PAIR ? side == 1 : has_lo) load(PAIR ? xt : xt + x_bytes, xl, stage, kx, 0, pol_x);
      } else {
        const uint32_t hb = x_bytes / 2;
        const int hr = n_pad / 2;
#pragma unroll 1
        for (int q = 0; q < (PAIR || !has_lo ? 2 : 4); ++q) {
          // a pair's CTA: both halves of one part where an MMA covers both parts, else its half of each
          const bool lo_part = PAIR ? (n_pad <= 128 ? side : q) != 0 : q >= 2;
          const int y = PAIR ? (n_pad <= 128 ? q : static_cast<int>(side)) : (q & 1);
          load(xt + q * hb, lo_part ? xl : xh, stage, kx, y * hr, pol_x);
        }
      }
    };
    // Weights do not depend on the preceding kernel: start streaming the first
    // ring's worth of W before waiting for the activations it produces.
    const int pre = min(stages, nk);
#pragma unroll 1
    for (int i = 0; i < pre; ++i) load_w(i, kt0 + i);
    // With an adapter the preceding kernel is its A x, which starts this one after its own wait for the
    // kernel that wrote x: only the last K tiles, t's, wait for it.  The weights' products then run beside
    // A x (1.5B, 16 candidates: rank 256 1,582 -> 1,550 us a call, rank 64 414 -> 391 for eight layers; 48
    // candidates at rank 256 577 -> 542; ranks 512 and 1,024 -3 to +1 %).  Starting it from A x's last
    // landed tile instead: 1,607.  That A x has waited does not by itself order x before the reads here, so
    // one of its threads leaves a mark after its wait (1,506 -> 1,511; 8B, 4 candidates, rank 64,
    // four layers 375 -> 378; with x behind A x's end 1,563 and 395).
    bool waited = !LORA;
    if constexpr (LORA)
      mark_acquire(ep.x_ready, *ep.call, err);
    else
      grid_dep_wait();
    trace_event(ts, 0);   // the preceding kernel has completed (with an adapter: the one before A x)
    auto load_act = [&](int stage, int kt) {
      if (LORA && !waited && kt >= k_main) {
        grid_dep_wait();
        waited = true;
      }
      load_x(stage, kt);
    };
#pragma unroll 1
    for (int i = 0; i < pre; ++i) load_act(i, kt0 + i);
    int s = 0;   // stage of K tile i, and the parity of the release before its use
    uint32_t parity = 0u;
#pragma unroll 1
    for (int i = pre; i < nk; ++i) {
      if (!mbar_wait(&empty[s], parity, err)) break;
      load_w(s, kt0 + i);
      load_act(s, kt0 + i);
      if (++s == stages) {
        s = 0;
        parity ^= 1u;
      }
    }
  } else if (warp >= 2) {
    // ---------------- while the weights stream: the RMSNorm factor of each of this rank's columns
    // (QKV, SILU), from the residual stream's tile sums of squares the preceding kernel wrote; the
    // parking barrier below orders these writes before the epilogue reads them
    const bool marks = MODE == GemmEpilogue::LOWRANK && blockIdx.x == 0 && threadIdx.x == 64;
    const int call = marks ? *ep.call : 0;
    grid_dep_wait();
    if (MODE == GemmEpilogue::LOWRANK) {
      if (marks) mark_release(ep.x_ready, call);
      grid_dep_launch();
    }
    if ((MODE == GemmEpilogue::QKV || MODE == GemmEpilogue::SILU) && ep.rs_sumsq)
#pragma unroll 1
      for (int t0 = threadIdx.x - 64; t0 < nc; t0 += blockDim.x - 64) {   // nc <= 256 columns
        const int c = cbeg + t0;
        float ssum = 0.f;
        for (int t = 0; t < ep.rs_tiles; ++t) ssum += ep.rs_sumsq[static_cast<int64_t>(t) * ep.n_valid + c];
        rsc[t0] = 1.0f / sqrtf(ssum / ep.rs_d + ep.rs_eps);
      }
    // RESID: the residual values the epilogue adds to, read now rather than after the MMAs, when
    // the next kernel's weight stream may be competing for the memory system
    if (hpreload) {   // warps 2 and 3 take alternate columns, 16 bytes a lane, all in flight at once
      float4 v[kHPreCols / 2];
      const int gm = m_tile * kBM + 4 * lane;
#pragma unroll
      for (int k = 0; k < kHPreCols / 2; ++k) {
        const int cl = 2 * k + (warp & 1);
        v[k] = (warp < 4 && cl < nc && gm < ep.M)
                   ? *reinterpret_cast<const float4*>(ep.h + static_cast<int64_t>(cbeg + cl) * ep.M + gm)
                   : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < kHPreCols / 2; ++k) {
        const int cl = 2 * k + (warp & 1);
        if (warp < 4 && cl < nc) *reinterpret_cast<float4*>(hpre + cl * kBM + 4 * lane) = v[k];
      }
    }
  } else if (warp == 1 && nk > 0 && side == 0) {
    // ---------------- MMA issuer (the whole warp; one elected lane issues)
    // With the hi and lo activation tiles stored back to back (2 n_pad rows
    // under the same swizzle), one MMA of N = 2 n_pad reads each weight K
    // slice from shared memory once: columns [0, n_pad) accumulate W hi,
    // [n_pad, 2 n_pad) accumulate W lo, summed when the accumulator is read.
    // Beyond N = 256 the two halves take one MMA each into the same columns.
    // A gate/up pair's up tile accumulates in the second half of the allocation.
    const bool merged = has_lo && 2 * n_pad <= 256;
    const bool two = has_lo && !merged;
    // A pair's MMA (M = 256, both CTAs' weight tiles) takes half of its B rows from either CTA: one part
    // each when merged, else half of the hi and half of the lo rows.
    const uint32_t idesc = idesc_bf16_f32(PAIR ? 2 * kBM : kBM, merged ? 2 * n_pad : n_pad);
    const uint16_t pair_mask = static_cast<uint16_t>(3u << crank);
    // PAIR without gate/up: two accumulators, one of the hi and one of the lo part, or when merged one of the first and
    // one of the second half of the K tiles: half as many fp32 roundings in a row (without them rewards
    // were 10-20 % further off, a pair's CTA having twice the K tiles of the CTA it replaces).
    const uint32_t tile_cols = tmem_cols / (PAIR ? 2u : 1u);
    const int i_half = PAIR && !silu && merged ? (nk + 1) / 2 : nk;   // the second accumulator's first K tile
    int s = 0;
    uint32_t parity = 0u;
#pragma unroll 1
    for (int i = 0; i < nk; ++i) {
      if (!__all_sync(0xffffffffu, mbar_wait(&full[s], parity, err))) break;
      if (i == 0 && lane == 0) trace_event(ts, 1);   // first weight and activation tiles landed
      tc_fence_after();
      const uint64_t a0 = desc_sw128(smem_u32(smem + s * stage_bytes));   // K step kk: + 2 kk (32 bytes)
      const uint64_t b0 = a0 + (w_bytes >> 4);
      const uint64_t l0 = b0 + static_cast<uint64_t>((PAIR ? x_bytes / 2 : x_bytes) >> 4);
      const uint32_t acc0 = i > 0 && i != i_half ? 1u : 0u;
#pragma unroll 1
      for (int t = 0; t < mt; ++t) {
        const uint32_t d = tmem + (t > 0 || i >= i_half ? tile_cols : 0u);
        const uint64_t at = a0 + static_cast<uint64_t>(t) * (kWTileBytes >> 4);
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk) {
          if constexpr (PAIR) {
            umma_bf16_pair_w(d, at + 2 * kk, b0 + 2 * kk, idesc, kk > 0 ? 1u : acc0);
            if (two) {
              if constexpr (silu)
                umma_bf16_pair_w(d, at + 2 * kk, l0 + 2 * kk, idesc, 1u);
              else
                umma_bf16_pair_w(d + tile_cols, at + 2 * kk, l0 + 2 * kk, idesc, kk > 0 ? 1u : acc0);
            }
          } else {
            umma_bf16_w(d, at + 2 * kk, b0 + 2 * kk, idesc, kk > 0 ? 1u : acc0);
            if (LARGE && two) umma_bf16_w(d, at + 2 * kk, l0 + 2 * kk, idesc, 1u);   // n_pad > 128
          }
        }
      }
      if constexpr (PAIR)
        umma_commit_pair_w(&empty[s], pair_mask);
      else
        umma_commit_w(&empty[s]);
      if (++s == stages) {
        s = 0;
        parity ^= 1u;
      }
    }
    if constexpr (PAIR)
      umma_commit_pair_w(done, pair_mask);
    else
      umma_commit_w(done);
  }
  __syncwarp();

  // ---------------- accumulator -> own shared memory, acc[c][m] (fp32, c < n_pad, m < 128)
  const bool have = nk > 0 ? __all_sync(0xffffffffu, mbar_wait(done, 0, err)) : true;
  if (threadIdx.x == 0) trace_event(ts, 2);   // all MMAs of this CTA completed
  tc_fence_after();
  // the ring is idle once `done` has fired; indexed by the batch's column, this CTA's first at the start
  float* acc = reinterpret_cast<float*>(smem) - c_off * kBM;
  // 4 warps, or 8 (the large-batch image): warps w and w + 4 share TMEM lane quadrant w,
  // i.e. the tile's rows 32 w .. 32 w + 31, and take alternate 16-column groups (or columns)
  const int nw = LARGE ? static_cast<int>(blockDim.x >> 5) : 4, nwh = LARGE ? nw >> 2 : 1, wh = LARGE ? warp >> 2 : 0;
  const int m = (warp & 3) * 32 + lane;
  const bool merged = has_lo && 2 * n_pad <= 256;
  const uint32_t tile_cols = tmem_cols / (PAIR ? 2u : 1u);
  const uint32_t trow = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
  if constexpr (PAIR && silu) {
    // Gate and up of a row sit in the same TMEM lane, so their product needs no parked accumulator: 16
    // columns at a time to shared memory as (hi, lo) words, and from there 16 bytes of rows a thread to
    // global memory.  Bound by those stores: 8 us after the last MMA at 256 columns, 7 without any of the
    // arithmetic; storing from the lanes (4 bytes of two rows) took 9.3.
    const bool few = n_pad < 64;   // the exact functions at batches where their time does not show
    grid_dep_wait();    // outputs may still be read by kernels that precede this one
    __syncthreads();    // the columns' RMSNorm factors
    if (threadIdx.x == 0) trace_event(ts, 5);
    const int j = m_tile * kBM + m;
    // stores: 16 row groups of 8 x 8 columns a step; the halves are read in the order free of bank conflicts
    const int rg = static_cast<int>(threadIdx.x) & 15, tq = (static_cast<int>(threadIdx.x) & 127) >> 4;
    const int row = m_tile * kBM + 8 * rg, flip = (rg >> 2) & 1;   // ff % 8 == 0
    const uint32_t np = static_cast<uint32_t>(n_pad);
#pragma unroll 1
    for (int c0 = 16 * wh; c0 < cend; c0 += 16 * nwh) {
      float g[16], u[16];
      const uint32_t t = trow + static_cast<uint32_t>(c0);
      tmem_ld16_nowait(t, g);
      tmem_ld16_nowait(t + tile_cols, u);
      if (merged) {
        float gl[16], ul[16];
        tmem_ld16_nowait(t + np, gl);
        tmem_ld16_nowait(t + tile_cols + np, ul);
        tmem_wait_ld();
        tmem_hold(g);
        tmem_hold(u);
        tmem_hold(gl);
        tmem_hold(ul);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          g[k] += gl[k];
          u[k] += ul[k];
        }
      } else {
        tmem_wait_ld();
        tmem_hold(g);
        tmem_hold(u);
      }
      if (ep.rs_sumsq) {
#pragma unroll
        for (int k = 0; k < 16; k += 4) {   // columns past the batch: whatever the slot holds, and not stored
          const float4 rs = *reinterpret_cast<const float4*>(rsc + c0 + k);
          g[k] *= rs.x, g[k + 1] *= rs.y, g[k + 2] *= rs.z, g[k + 3] *= rs.w;
          u[k] *= rs.x, u[k + 1] *= rs.y, u[k + 2] *= rs.z, u[k + 3] *= rs.w;
        }
      }
      if (ep.gu_save && j < ep.ff) {   // pre-activations for a backward pass
        float* gs = ep.gu_save + static_cast<int64_t>(c0) * 2 * ep.ff + j;
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if (c0 + k < cend) {
            gs[static_cast<int64_t>(2 * k) * ep.ff] = g[k];
            gs[static_cast<int64_t>(2 * k + 1) * ep.ff] = u[k];
          }
      }
      uint32_t* xc = reinterpret_cast<uint32_t*>(smem) + c0 * kBM;   // (hi, lo) of 16 columns, in the idle ring
#pragma unroll
      for (int k = 0; k < 16; k += 2) {
        float a[2];
#pragma unroll
        for (int e = 0; e < 2; ++e)
          a[e] = (few ? g[k + e] / (1.0f + expf(-g[k + e]))
                      : g[k + e] * rcp_ftz(1.0f + ex2_ftz(-1.4426950408889634f * g[k + e]))) * u[k + e];
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(a[0], a[1]);
        const float2 hf = __bfloat1622float2(h2);
        const __nv_bfloat162 l2 = __floats2bfloat162_rn(a[0] - hf.x, a[1] - hf.y);
        const uint32_t h = *reinterpret_cast<const uint32_t*>(&h2), l = *reinterpret_cast<const uint32_t*>(&l2);
        xc[k * kBM + m] = __byte_perm(h, l, 0x5410);
        xc[(k + 1) * kBM + m] = __byte_perm(h, l, 0x7632);
      }
      named_bar_sync(1 + wh, 128);   // the four warps of these columns
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int cl = tq + 8 * k;
        const uint4* xp = reinterpret_cast<const uint4*>(xc + cl * kBM + 8 * rg);
        const uint4 w0 = xp[flip], w1 = xp[1 - flip], v0 = flip ? w1 : w0, v1 = flip ? w0 : w1;
        if (c0 + cl < cend && row < ep.ff) {
          const int64_t o = static_cast<int64_t>(c0 + cl) * ep.ff + row;
          *reinterpret_cast<uint4*>(ep.a_hi + o) = make_uint4(__byte_perm(v0.x, v0.y, 0x5410), __byte_perm(v0.z, v0.w, 0x5410),
                                                              __byte_perm(v1.x, v1.y, 0x5410), __byte_perm(v1.z, v1.w, 0x5410));
          *reinterpret_cast<uint4*>(ep.a_lo + o) = make_uint4(__byte_perm(v0.x, v0.y, 0x7632), __byte_perm(v0.z, v0.w, 0x7632),
                                                              __byte_perm(v1.x, v1.y, 0x7632), __byte_perm(v1.z, v1.w, 0x7632));
        }
      }
    }
    tc_fence_before();
    __syncwarp();
    cluster_arrive();
  } else {
    // park the tile, reduce it over the cluster, write its epilogue
    if constexpr (PAIR) {
      // the two accumulators, a group's loads in flight while the one before it is stored
      const uint32_t np = static_cast<uint32_t>(n_pad);
      const bool second = nk > 0 && have && (!merged || nk > 1), any = nk > 0 && have;
      float v[16], w[16], v2[16], w2[16];
      auto issue = [&](int c0) {
        const uint32_t t = trow + static_cast<uint32_t>(c0);
        tmem_ld16_nowait(t, v);
        tmem_ld16_nowait(t + tile_cols, v2);
        if (merged) {
          tmem_ld16_nowait(t + np, w);
          tmem_ld16_nowait(t + tile_cols + np, w2);
        }
      };
      if (16 * wh < n_pad) issue(16 * wh);
#pragma unroll 1
      for (int c0 = 16 * wh; c0 < n_pad; c0 += 16 * nwh) {
        float r[16];
        tmem_wait_ld();
        tmem_hold(v);
        tmem_hold(v2);
#pragma unroll
        for (int j = 0; j < 16; ++j) r[j] = (any ? v[j] : 0.f) + (second ? v2[j] : 0.f);
        if (merged) {
          tmem_hold(w);
          tmem_hold(w2);
#pragma unroll
          for (int j = 0; j < 16; ++j) r[j] += (any ? w[j] : 0.f) + (second ? w2[j] : 0.f);
        }
        if (c0 + 16 * nwh < n_pad) issue(c0 + 16 * nwh);
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[(c_off + c0 + j) * kBM + m] = r[j];
      }
    } else {
#pragma unroll 1
      for (int c0 = 16 * wh; c0 < n_pad; c0 += 16 * nwh) {
        float v[16];
        if (nk > 0 && have) {
          const uint32_t t = trow + static_cast<uint32_t>(c0);
          tmem_ld16(t, v);
          if (merged) {
            float w[16];
            tmem_ld16(t + static_cast<uint32_t>(n_pad), w);
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] += w[j];
          }
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = 0.f;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[(c0 + j) * kBM + m] = v[j];
      }
    }
    tc_fence_before();
    {
      cluster_sync();   // every rank's partial is parked
      if (threadIdx.x == 0) trace_event(ts, 3);
      if (ep.late_trigger) grid_dep_launch();
      // ---------------- reduce this rank's candidate columns over the cluster, then the epilogue
      grid_dep_wait();   // outputs may still be read by kernels that precede this one
      // Step 1: acc[c][m] <- sum over ranks of acc_r[c][m] for this rank's columns (only this rank reads
      // them, so it may overwrite its own copy), in a fixed order; all peer loads of a round in flight.  Without split K (cs = 1) the parked accumulator is already the sum.
      if (LARGE && cs > 1) {
        // four consecutive rows of one column per thread (a warp covers a column's 128 rows), 16 / cs
        // columns per round: 16 loads of 16 bytes, the ranks' copies of each; warp w takes columns cbeg + w,
        // cbeg + w + nw, ...  A rank begins with its own copy and takes the others in an order of its own,
        // so that the cluster's loads do not all meet in one CTA; exchanged operands leave the sums what
        // they are.  The 7B QKV projection as halves over two ranks, 256 columns: this step 4.5 us with
        // 4-byte loads, 1.4 now (19.8 -> 16.9 in all); with ranks in one order 16 of them took 0.3 longer.
        const int rq = static_cast<int>(threadIdx.x) & 31, lcs = 31 - __clz(cs);
        float* col = acc + (cbeg + warp) * kBM + 4 * rq;
#pragma unroll 1
        for (int c0 = cbeg + warp; c0 < cend; c0 += nw * (16 >> lcs), col += nw * (16 >> lcs) * kBM) {
          float4 v[16];
#pragma unroll
          for (int k = 0; k < 16; ++k) {   // rank (k ^ this one) % cs of column c0 + nw (k / cs)
            const int dc = nw * (k >> lcs);
            v[k] = c0 + dc < cend ? ld_cluster4(col + dc * kBM, peer((k ^ static_cast<int>(rank)) & (cs - 1))) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
#pragma unroll
          for (int w = 1; w < 16; w *= 2)
            if (w < cs)
#pragma unroll
              for (int k = 0; k < 16; k += 2 * w)
                v[k] = make_float4(v[k].x + v[k + w].x, v[k].y + v[k + w].y, v[k].z + v[k + w].z, v[k].w + v[k + w].w);
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const int dc = nw * (k >> lcs);
            if ((k & (cs - 1)) == 0 && c0 + dc < cend) *reinterpret_cast<float4*>(col + dc * kBM) = v[k];
          }
        }
      } else if (cs > 1) {   // two columns per round trip when the cluster has <= 8 ranks
        const int step = cs <= 8 ? 2 : 1;
#pragma unroll 1
        for (int c = cbeg; c < cend; c += step) {
          const bool two = step == 2 && c + 1 < cend;
          float v[16];
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const int r = step == 2 ? (k & 7) : k;
            const int cc = (step == 2 && k >= 8) ? c + 1 : c;
            const bool use = r < cs && (cc == c || two);
            v[k] = use ? ld_cluster(acc + cc * kBM + m, peer(r)) : 0.f;
          }
          if (step == 2) {
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              s0 += v[k];
              s1 += v[8 + k];
            }
            __syncwarp();
            acc[c * kBM + m] = s0;
            if (two) acc[(c + 1) * kBM + m] = s1;
          } else {
            float s0 = 0.f;
#pragma unroll
            for (int k = 0; k < 16; ++k) s0 += v[k];
            acc[c * kBM + m] = s0;
          }
        }
      }
      if (threadIdx.x == 0) trace_event(ts, 4);   // this rank's columns are reduced over the cluster
      // no peer reads this tile's partial any more once every rank has arrived here: arrive now and
      // wait only before the exit, so the barrier's latency hides behind the epilogue
      __syncwarp();
      cluster_arrive();
    }
    __syncthreads();   // every warp's reduced columns are in acc
    if (threadIdx.x == 0) trace_event(ts, 5);
    // QKV with the per-head q/k RMSNorm: the factor of each (column, head of this tile) over the
    // head's hd rows of the RMSNorm-scaled projection, 1/sqrt(mean(y^2) + eps) times the column's
    // RMSNorm factor (v heads keep the latter alone); parked where RESID preloads its residual
    float* qkf = hpre;   // [column][head of the tile]
    if (MODE == GemmEpilogue::QKV && ep.qn_gain) {
      const int hpt = ep.hd == 128 ? 1 : 2;   // heads per tile
#pragma unroll 1
      for (int it = warp; it < nc * hpt; it += nw) {
        const int cl = it >> (hpt - 1), hh = it & (hpt - 1);
        const float* col = acc + (cbeg + cl) * kBM + hh * ep.hd;
        float sq = 0.f;
        for (int r = lane; r < ep.hd; r += 32) sq += col[r] * col[r];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
        if (lane == 0) {
          const float rs = ep.rs_sumsq ? rsc[cl] : 1.f;
          const int head = m_tile * hpt + hh;
          qkf[cl * 2 + hh] = head < ep.n_q + ep.n_kv ? rs / sqrtf(rs * rs * sq / ep.hd + ep.rs_eps) : rs;
        }
      }
      __syncthreads();
    }
    // Step 2: the epilogue over (row, column) pairs, all threads in parallel
    if constexpr (MODE == GemmEpilogue::PLAIN) {
      const int gm = m_tile * kBM + m;
      if (gm < ep.M)
#pragma unroll 4
        for (int c = cbeg + wh; c < cend; c += nwh) ep.out[static_cast<int64_t>(c) * ep.M + gm] = acc[c * kBM + m];
    } else if constexpr (MODE == GemmEpilogue::LOWRANK) {   // t = s (A x), hi/lo [n][r]
      const int gm = m_tile * kBM + m;
      if (gm < ep.M)
#pragma unroll 2
        for (int c = cbeg + wh; c < cend; c += nwh)
          store_hilo(ep.t_hi, ep.t_lo, static_cast<int64_t>(c) * ep.M + gm, ep.lr_scale * acc[c * kBM + m]);
    } else if constexpr (MODE == GemmEpilogue::RESID && LARGE) {
      // pass 1, eight columns' residual loads in flight before the first use: h += acc, the next
      // projection's input, and hv^2 parked in place of acc (each (column, row) slot is this thread's own)
      {   // M = d_model, a multiple of 64
        // four consecutive rows of one column per thread (a warp covers one column's 128 rows):
        // 16-byte residual loads and stores, 8-byte hi/lo stores; eight columns' loads in flight
        const int rq = static_cast<int>(threadIdx.x) & 31, cg = static_cast<int>(threadIdx.x) >> 5;
        const int gm0 = m_tile * kBM + 4 * rq;
        const bool rows_ok = gm0 < ep.M;   // M % 4 == 0: the four rows are all valid or all past M
        float g4[4] = {0.f, 0.f, 0.f, 0.f};
        if (ep.gain_next && rows_ok) {
          const float4 g = load_bf16x4(ep.gain_next + gm0);
          g4[0] = g.x;
          g4[1] = g.y;
          g4[2] = g.z;
          g4[3] = g.w;
        }
#pragma unroll 1
        for (int c0 = cbeg + cg; c0 < cend; c0 += nw * 8) {
          float4 h_in[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int c = c0 + nw * k;
            h_in[k] = !(c < cend && rows_ok) ? make_float4(0.f, 0.f, 0.f, 0.f)
                      : hpreload ? *reinterpret_cast<const float4*>(hpre + (c - cbeg) * kBM + 4 * rq)
                                 : *reinterpret_cast<const float4*>(ep.h + static_cast<int64_t>(c) * ep.M + gm0);
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int c = c0 + nw * k;
            if (c >= cend) break;
            float4* ap = reinterpret_cast<float4*>(acc + c * kBM + 4 * rq);
            const float4 a = *ap;
            float4 hv = make_float4(0.f, 0.f, 0.f, 0.f);
            if (rows_ok) {
              hv = make_float4(h_in[k].x + a.x, h_in[k].y + a.y, h_in[k].z + a.z, h_in[k].w + a.w);
              const int64_t o = static_cast<int64_t>(c) * ep.M + gm0;
              *reinterpret_cast<float4*>(ep.h + o) = hv;
              if (ep.h_copy) *reinterpret_cast<float4*>(ep.h_copy + o) = hv;
              if (ep.gain_next) {
                const float x[4] = {hv.x * g4[0], hv.y * g4[1], hv.z * g4[2], hv.w * g4[3]};
                uint32_t hi[2], lo[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                  const __nv_bfloat162 h2 = __floats2bfloat162_rn(x[2 * e], x[2 * e + 1]);
                  const float2 hf = __bfloat1622float2(h2);
                  const __nv_bfloat162 l2 = __floats2bfloat162_rn(x[2 * e] - hf.x, x[2 * e + 1] - hf.y);
                  hi[e] = *reinterpret_cast<const uint32_t*>(&h2);
                  lo[e] = *reinterpret_cast<const uint32_t*>(&l2);
                }
                *reinterpret_cast<uint2*>(ep.x_hi + o) = make_uint2(hi[0], hi[1]);
                *reinterpret_cast<uint2*>(ep.x_lo + o) = make_uint2(lo[0], lo[1]);
              }
            }
            *ap = make_float4(hv.x * hv.x, hv.y * hv.y, hv.z * hv.z, hv.w * hv.w);
          }
        }
      }
      __syncthreads();
      // pass 2: each column's sum of squares over the tile's 128 rows, eight threads per column
      // (rows part + 8 q, the start of q rotated per column so that a warp's four columns hit
      // different banks), warp-uniform trip count for the shuffles
#pragma unroll 1
      for (int t0 = 0; t0 < nc * 8; t0 += blockDim.x) {
        const int t = t0 + static_cast<int>(threadIdx.x);
        const int cl = t >> 3, part = t & 7;
        float sq = 0.f;
        if (t < nc * 8) {
          const float* col = acc + (cbeg + cl) * kBM + part;
#pragma unroll
          for (int q = 0; q < 16; ++q) sq += col[8 * ((q + (cl & 3)) & 15)];
        }
        sq += __shfl_xor_sync(0xffffffffu, sq, 1);
        sq += __shfl_xor_sync(0xffffffffu, sq, 2);
        sq += __shfl_xor_sync(0xffffffffu, sq, 4);
        if (t < nc * 8 && part == 0) ep.sumsq[static_cast<int64_t>(m_tile) * ep.n_valid + cbeg + cl] = sq;
      }
    } else if constexpr (MODE == GemmEpilogue::RESID) {
      const int gm = m_tile * kBM + m;
      float* sq_s = red;   // [16 columns][4 warps]
#pragma unroll 1
      for (int c0 = cbeg; c0 < cend; c0 += 16) {
        const int c1 = min(cend, c0 + 16);
        {
#pragma unroll 1
          for (int c = c0; c < c1; ++c) {
            float hv = 0.f;
            if (gm < ep.M) {
              float* hp = ep.h + static_cast<int64_t>(c) * ep.M + gm;
              hv = (hpreload ? hpre[(c - cbeg) * kBM + m] : *hp) + acc[c * kBM + m];
              *hp = hv;
              if (ep.h_copy) ep.h_copy[static_cast<int64_t>(c) * ep.M + gm] = hv;
              if (ep.gain_next)
                store_hilo(ep.x_hi, ep.x_lo, static_cast<int64_t>(c) * ep.M + gm, hv * __bfloat162float(ep.gain_next[gm]));
            }
            float sq = hv * hv;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
            if (lane == 0) sq_s[(c - c0) * 4 + warp] = sq;
          }
        }
        __syncthreads();
        if (threadIdx.x < c1 - c0) {
          const float* q4 = sq_s + threadIdx.x * 4;
          ep.sumsq[static_cast<int64_t>(m_tile) * ep.n_valid + c0 + threadIdx.x] = (q4[0] + q4[1]) + (q4[2] + q4[3]);
        }
        __syncthreads();
      }
    } else if constexpr (MODE == GemmEpilogue::SILU && LARGE) {   // d_ff is a multiple of 64
      // eight consecutive rows of one column per thread (8 row groups x 16 column groups): 16-byte
      // loads from the parked tile and one 16-byte store for each of the hi and lo halves (2-byte
      // stores, 256 per warp and tile at B = 256, bound the scalar form); the exponential and the
      // divide take the fast intrinsics
      const int rg = static_cast<int>(threadIdx.x) & 7, cg = static_cast<int>(threadIdx.x) >> 3;
      const int j0 = m_tile * 64 + 8 * rg;   // ff % 8 == 0: a row group is all valid or all past ff
      const bool few = n_pad < 64;   // the exact functions at batches where their time does not show
      if (j0 < ep.ff) {
#pragma unroll 2
        for (int c = cbeg + cg; c < cend; c += 4 * nw) {   // 4 nw column groups of 8 threads
          const float rs = ep.rs_sumsq ? rsc[c - cbeg] : 1.f;
          const float4* gp = reinterpret_cast<const float4*>(acc + c * kBM + 8 * rg);
          const float4* up = reinterpret_cast<const float4*>(acc + c * kBM + 64 + 8 * rg);
          const float4 g0 = gp[0], g1 = gp[1], u0 = up[0], u1 = up[1];
          const float g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
          const float u[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float ga = g[2 * e] * rs, gb = g[2 * e + 1] * rs;
            const float a = (few ? ga / (1.0f + expf(-ga)) : __fdividef(ga, 1.0f + __expf(-ga))) * (u[2 * e] * rs);
            const float b = (few ? gb / (1.0f + expf(-gb)) : __fdividef(gb, 1.0f + __expf(-gb))) * (u[2 * e + 1] * rs);
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(a, b);
            const float2 hf = __bfloat1622float2(h2);
            const __nv_bfloat162 l2 = __floats2bfloat162_rn(a - hf.x, b - hf.y);
            hi[e] = *reinterpret_cast<const uint32_t*>(&h2);
            lo[e] = *reinterpret_cast<const uint32_t*>(&l2);
          }
          const int64_t o = static_cast<int64_t>(c) * ep.ff + j0;
          *reinterpret_cast<uint4*>(ep.a_hi + o) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(ep.a_lo + o) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
          if (ep.gu_save) {   // gate and up pre-activations (after the RMSNorm factor) for a backward pass
            float4* gs = reinterpret_cast<float4*>(ep.gu_save + static_cast<int64_t>(c) * 2 * ep.ff + j0);
            float4* us = reinterpret_cast<float4*>(ep.gu_save + static_cast<int64_t>(c) * 2 * ep.ff + ep.ff + j0);
            gs[0] = make_float4(g[0] * rs, g[1] * rs, g[2] * rs, g[3] * rs);
            gs[1] = make_float4(g[4] * rs, g[5] * rs, g[6] * rs, g[7] * rs);
            us[0] = make_float4(u[0] * rs, u[1] * rs, u[2] * rs, u[3] * rs);
            us[1] = make_float4(u[4] * rs, u[5] * rs, u[6] * rs, u[7] * rs);
          }
        }
      }
    } else if constexpr (MODE == GemmEpilogue::SILU) {
      // two column groups of 64 threads (rows m and m + 64 of a column share a group)
      const int r = m & 63;
      const int j = m_tile * 64 + r;
      if (j < ep.ff)
#pragma unroll 1
        for (int c = cbeg + (m >> 6); c < cend; c += 2) {
          const float rs = ep.rs_sumsq ? rsc[c - cbeg] : 1.f;
          const float g = acc[c * kBM + r] * rs, u = acc[c * kBM + 64 + r] * rs;
          store_hilo(ep.a_hi, ep.a_lo, static_cast<int64_t>(c) * ep.ff + j, g / (1.0f + expf(-g)) * u);
          if (ep.gu_save) {   // gate and up pre-activations for a backward pass
            ep.gu_save[static_cast<int64_t>(c) * 2 * ep.ff + j] = g;
            ep.gu_save[static_cast<int64_t>(c) * 2 * ep.ff + ep.ff + j] = u;
          }
        }
    } else if constexpr (LARGE) {   // QKV
      // QKV, four consecutive RoPE pairs (i .. i + 3, partners i + half ..) of one column per
      // thread (16 pair groups x 8 column groups): 16-byte loads of the parked tile and the
      // rotation, 16-byte fp32 and 8-byte hi/lo stores; two columns' operands in flight
      const int pq = 4 * (static_cast<int>(threadIdx.x) & 15), cg = static_cast<int>(threadIdx.x) >> 4;
      const int lhd = ep.hd == 128 ? 7 : 6;   // head_dim is 64 or 128
      const int hd = 1 << lhd, half = hd >> 1;
      const int row_a = ((pq >> (lhd - 1)) << lhd) + (pq & (half - 1));   // half % 4 == 0: the four pairs share a head
      const int row_b = row_a + half;
      const int grow = m_tile * kBM + row_a;
      const int head = grow >> lhd, i = grow & (hd - 1);
      const bool rot = head < ep.n_q + ep.n_kv;
      // per-head q/k RMSNorm: the gains of these rows (q heads: q_norm, k heads: k_norm)
      const bool qkn = ep.qn_gain != nullptr && rot;
      float gna[4] = {1.f, 1.f, 1.f, 1.f}, gnb[4] = {1.f, 1.f, 1.f, 1.f};
      if (qkn) {
        const __nv_bfloat16* gsrc = head < ep.n_q ? ep.qn_gain : ep.kn_gain;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          gna[e] = __bfloat162float(gsrc[i + e]);
          gnb[e] = __bfloat162float(gsrc[i + half + e]);
        }
      }
      const int hh_tile = row_a >> lhd;   // head of this tile
      auto store4 = [&](float* dst, __nv_bfloat16* dhi, __nv_bfloat16* dlo, int64_t o, const float (&x)[4]) {
        *reinterpret_cast<float4*>(dst + o) = make_float4(x[0], x[1], x[2], x[3]);
        if (dhi) {
          uint32_t hi[2], lo[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(x[2 * e], x[2 * e + 1]);
            const float2 hf = __bfloat1622float2(h2);
            const __nv_bfloat162 l2 = __floats2bfloat162_rn(x[2 * e] - hf.x, x[2 * e + 1] - hf.y);
            hi[e] = *reinterpret_cast<const uint32_t*>(&h2);
            lo[e] = *reinterpret_cast<const uint32_t*>(&l2);
          }
          *reinterpret_cast<uint2*>(dhi + o) = make_uint2(hi[0], hi[1]);
          *reinterpret_cast<uint2*>(dlo + o) = make_uint2(lo[0], lo[1]);
        }
      };
      if (head < ep.n_q + 2 * ep.n_kv) {
#pragma unroll 2
        for (int c = cbeg + cg; c < cend; c += 2 * nw) {   // 2 nw column groups of 16 threads
          const float rs = ep.qn_gain ? qkf[(c - cbeg) * 2 + hh_tile] : (ep.rs_sumsq ? rsc[c - cbeg] : 1.f);
          const float4 a4 = *reinterpret_cast<const float4*>(acc + c * kBM + row_a);
          const float4 b4 = *reinterpret_cast<const float4*>(acc + c * kBM + row_b);
          float4 r0 = make_float4(1.f, 0.f, 1.f, 0.f), r1 = r0;   // (cos, sin) of pairs i, i+1 / i+2, i+3
          if (rot) {
            const float4* rp = reinterpret_cast<const float4*>(ep.rope + c * half + i);
            r0 = rp[0];
            r1 = rp[1];
          }
          const float cs_[4] = {r0.x, r0.z, r1.x, r1.z}, sn_[4] = {r0.y, r0.w, r1.y, r1.w};
          const float av[4] = {a4.x * rs * gna[0], a4.y * rs * gna[1], a4.z * rs * gna[2], a4.w * rs * gna[3]};
          const float bv[4] = {b4.x * rs * gnb[0], b4.y * rs * gnb[1], b4.z * rs * gnb[2], b4.w * rs * gnb[3]};
          float oa[4], ob[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (rot) {
              oa[e] = av[e] * cs_[e] - bv[e] * sn_[e];
              ob[e] = bv[e] * cs_[e] + av[e] * sn_[e];
            } else {
              oa[e] = av[e];
              ob[e] = bv[e];
            }
          }
          if (head < ep.n_q) {
            const int64_t o = (static_cast<int64_t>(c) * ep.n_q + head) * hd + i;
            store4(ep.q, ep.q_hi, ep.q_lo, o, oa);
            store4(ep.q, ep.q_hi, ep.q_lo, o + half, ob);
          } else {
            const bool is_k = head < ep.n_q + ep.n_kv;
            const int kvh = is_k ? head - ep.n_q : head - ep.n_q - ep.n_kv;
            float* dst = is_k ? ep.kself : ep.vself;
            const int64_t o = (static_cast<int64_t>(c) * ep.n_kv + kvh) * hd + i;
            store4(dst, nullptr, nullptr, o, oa);
            store4(dst, nullptr, nullptr, o + half, ob);
          }
        }
      }
    } else {   // QKV: pair p = m & 63 of this tile, two column groups of 64 threads
      const int p = m & 63;
      const int lhd = ep.hd == 128 ? 7 : 6;               // head_dim is 64 or 128
      const int hd = 1 << lhd, half = hd >> 1;
      const int row_a = ((p >> (lhd - 1)) << lhd) + (p & (half - 1));   // first element of the pair, within the tile
      const int row_b = row_a + half;
      const int grow = m_tile * kBM + row_a;              // row of W_qkv
      const int head = grow >> lhd, i = grow & (hd - 1);  // i < half
      const bool rot = head < ep.n_q + ep.n_kv;   // q and k rows take RoPE, v rows do not
      // per-head q/k RMSNorm (q heads: q_norm, k heads: k_norm gains of these two rows)
      float gna = 1.f, gnb = 1.f;
      if (ep.qn_gain && rot) {
        const __nv_bfloat16* gsrc = head < ep.n_q ? ep.qn_gain : ep.kn_gain;
        gna = __bfloat162float(gsrc[i]);
        gnb = __bfloat162float(gsrc[i + half]);
      }
      const int hh_tile = row_a >> lhd;
#pragma unroll 1
      for (int c = cbeg + (m >> 6); c < cend; c += 2) {
        const float rs = ep.qn_gain ? qkf[(c - cbeg) * 2 + hh_tile] : (ep.rs_sumsq ? rsc[c - cbeg] : 1.f);
        float a = acc[c * kBM + row_a] * rs * gna, b = acc[c * kBM + row_b] * rs * gnb;
        if (rot) {
          const float2 cs2 = ep.rope[c * half + i];
          const float a2 = fmaf(a, cs2.x, -(b * cs2.y));
          const float b2 = fmaf(a, cs2.y, b * cs2.x);
          a = a2;
          b = b2;
        }
        if (head < ep.n_q) {
          const int64_t o = (static_cast<int64_t>(c) * ep.n_q + head) * hd + i;
          ep.q[o] = a;
          ep.q[o + half] = b;
          store_hilo(ep.q_hi, ep.q_lo, o, a);
          store_hilo(ep.q_hi, ep.q_lo, o + half, b);
        } else if (head < ep.n_q + 2 * ep.n_kv) {
          const bool is_k = head < ep.n_q + ep.n_kv;
          const int kvh = is_k ? head - ep.n_q : head - ep.n_q - ep.n_kv;
          float* dst = (is_k ? ep.kself : ep.vself) + (static_cast<int64_t>(c) * ep.n_kv + kvh) * hd + i;
          dst[0] = a;
          dst[half] = b;
        }
      }
    }
  }
  (void)nc;
  if (threadIdx.x == 0) trace_event(ts, 6);   // this thread's epilogue written
  __syncwarp();
  cluster_wait();   // peers have finished reading this CTA's partial
  if (threadIdx.x == 0) trace_event(ts, 7);
  if (warp == 1) {
    if constexpr (PAIR)
      tmem_dealloc_pair(tmem, tmem_cols);
    else
      tmem_dealloc(tmem, tmem_cols);
  }
  trace_end(ts);
}

}  // namespace

uint32_t gemm_x_box(int n_pad) { return static_cast<uint32_t>(n_pad >= kHalfBoxCols ? n_pad / 2 : n_pad); }

GemmPlan plan_gemm(int M, int K, int n_pad, int num_sms, bool has_lo, bool gate_up) {
  GemmPlan p;
  p.has_lo = has_lo;
  p.gate_up = gate_up;
  p.m_tiles = gate_up ? (M + 63) / 64 : (M + kBM - 1) / kBM;   // gate/up: M = d_ff, 64 pairs per tile
  p.k_tiles = (K + kBK - 1) / kBK;
  const uint32_t stage_bytes = kWTileBytes + static_cast<uint32_t>(n_pad) * kBK * 2 * (has_lo ? 2u : 1u);
  int stages = static_cast<int>((112u * 1024u) / stage_bytes);
  p.stages = stages < 2 ? 2 : (stages > 8 ? 8 : stages);
  // the parked accumulator (n_pad x 128 fp32) reuses the ring
  size_t ring = static_cast<size_t>(p.stages) * stage_bytes;
  const size_t acc = park_bytes(n_pad);
  if (ring < acc) ring = acc;
  p.smem_bytes = ring + 1024 /*align*/ + kTailBytes;
  // cluster size: the largest power of two <= 16 that keeps the CTA count within what fits on the
  // SMs at once (two per SM when two CTAs' shared memory fits, else one: at B = 256 a stage holds
  // 64 KB of activations) and gives every rank at least two K tiles
  constexpr size_t kHalfSm = 228u * 1024u / 2;
  int per_sm = p.smem_bytes + 1024 <= kHalfSm ? 2 : 1;
  // A cluster is placed whole on one GPC.  With two CTAs per SM, a grid that needs (nearly) every
  // slot cannot be placed in one wave while the preceding kernel still holds part of the SMs
  // (programmatic dependent launch places this grid's first clusters early, half-filling SMs in a
  // pattern that strands slots): the 7B QKV projection at B = 64, 36 clusters of 8 = 288 of 304
  // slots, had its last clusters start ~10 us after the preceding kernel ended.  Such grids keep
  // within 7/8 of the slots.  With one CTA per SM, the GPCs (of 18 to 20 SMs, one of fewer) take 36
  // clusters of 4, 15 of 8 and 7 of 16: what they cannot place starts when the first wave ends (16
  // clusters of 8 for the 1.5B QKV projection at 256 columns: 12 us later, 22.4 us in all; 12.1 in 4s).
  auto fit = [&](int c) {
    return c == 1 ? num_sms : (c == 2 ? num_sms / 2 : num_sms * (c == 4 ? 36 : (c == 8 ? 15 : 7)) / 152);
  };
  auto cluster_of = [&](int ctas_per_sm) {
    int c = 1;
    while (c < 16 && c * 4 <= p.k_tiles && c * 2 <= n_pad &&
           (ctas_per_sm == 2 ? p.m_tiles * c * 2 <= 2 * num_sms * 7 / 8 : p.m_tiles <= fit(2 * c)))
      c *= 2;
    return c;
  };
  int cs = cluster_of(per_sm);
  // One stage less can let two CTAs share an SM (48 and 80 padded columns: a few KB too many).  Taken
  // where it saves a second wave (the 296 CTAs of the 7B gate/up at 48 columns: 52 -> 46 us) or lets a
  // long K loop run on twice the CTAs (the 7B down projection 31 -> 26 us at 48 columns, 37 -> 35 at 80);
  // elsewhere the deeper ring of the single CTA is worth more (the 7B QKV at 80 columns: 12.4 us, 17.3
  // with a stage less).
  if (per_sm == 1 && p.stages > 2) {
    size_t less = static_cast<size_t>(p.stages - 1) * stage_bytes;
    if (less < acc) less = acc;
    const int cs2 = cluster_of(2);
    if (less + 1024 + kTailBytes + 1024 <= kHalfSm &&
        ((n_pad <= 64 && cs == 1 && p.m_tiles > num_sms) || (cs2 > cs && (p.k_tiles + cs - 1) / cs >= 16))) {
      --p.stages;
      p.smem_bytes = less + 1024 + kTailBytes;
      per_sm = 2;
      cs = cs2;
    }
  }
  p.cluster = p.ranks = cs;
  p.kt_per_rank = (p.k_tiles + cs - 1) / cs;
  // a ring deeper than the K tiles one CTA streams only holds shared memory
  // that overlapping kernels could use
  if (p.stages > p.kt_per_rank) p.stages = p.kt_per_rank < 2 ? 2 : p.kt_per_rank;
  ring = static_cast<size_t>(p.stages) * stage_bytes;
  if (ring < acc) ring = acc;
  p.smem_bytes = ring + 1024 /*align*/ + kTailBytes;
  uint32_t cols = 32;
  const int need = (has_lo && 2 * n_pad <= 256) ? 2 * n_pad : n_pad;   // merged hi/lo accumulator halves
  while (cols < static_cast<uint32_t>(need)) cols <<= 1;
  p.tmem_cols = cols;
  // A pair's CTA takes all shared memory it may (its ring and the parked accumulator are well below): its tensor
  // memory (up to 512 columns) is allocated in two SMs at once, and beside a cluster of another stream's launch
  // either could hold the columns the other's second CTA waits for.  What is left (26 KB) is too little for any
  // other launch that allocates tensor memory.
  // gate/up without split K, more tiles than SMs: pairs of CTAs with two tiles each.  The 7B gate/up, 296
  // tiles: one-tile CTAs two to an SM took 51.6 us at 96 columns and 56.5 at 144, two tiles a CTA without
  // pairs 47.5 at 80, 66.5 at 160 and 80.0 at 256; pairs take 44.1, 50.1, 44.7, 52.9 and 75.4 (the weights'
  // bytes alone 40.7, the MMAs 71 at 256).  At 64 columns 45.0 -> 43.7, at 48 45.6 -> 43.1.
  if (gate_up && has_lo && n_pad >= kLargeCols && cs == 1 && p.m_tiles % 2 == 0 && p.m_tiles > num_sms &&
      (p.m_tiles / 2 + 1) / 2 <= fit(2)) {
    const uint32_t st2 = 2 * kWTileBytes + static_cast<uint32_t>(n_pad) * kBK * 2;
    int stages2 = static_cast<int>((192u * 1024u) / st2);
    if (stages2 > 8) stages2 = 8;
    if (stages2 > p.k_tiles) stages2 = p.k_tiles < 2 ? 2 : p.k_tiles;
    p.pair = true;
    p.mt = 2;
    p.stages = stages2;
    p.smem_bytes = kGemmMaxSmem;
    p.tmem_cols = 2 * cols;
  }
  const int pc = cluster_of(1);
  auto take_pairs = [&](int ranks, int n_split) {
    const int cols2 = n_pad / n_split;
    const uint32_t st2 = kWTileBytes + static_cast<uint32_t>(cols2) * kBK * 2;
    const int kps = (p.k_tiles + ranks - 1) / ranks;
    int stages2 = static_cast<int>((192u * 1024u) / st2);
    if (stages2 > 8) stages2 = 8;
    if (stages2 > kps) stages2 = kps < 2 ? 2 : kps;
    p.pair = true;
    p.mt = 3 - n_split;
    p.cluster = 2 * ranks;
    p.ranks = ranks;
    p.kt_per_rank = kps;
    p.col_parts = n_split;
    p.stages = stages2;
    p.smem_bytes = kGemmMaxSmem;
    p.tmem_cols = 2 * cols;
  };
  // CTA pairs (see the kernel).  The CTAs that one m-tile each over pc ranks would take, as clusters of
  // 2 pc for two m-tiles; or, where such clusters of 8 do not fit, and without a cluster reduction where pc
  // is 2, as clusters of pc for two m-tiles and half of the columns.  7B at 256 columns: O 22.7 -> 18.7 us,
  // down 62.5 -> 51.0 (it was two m-tiles a CTA over 8 ranks), QKV 22.6 -> 19.3 (halves); 8B at 256: QKV
  // 35.1 -> 26.8 (halves; 35.1 too as whole pairs), O 24.3 -> 20.6 (halves).  Fewer columns, 7B: O 12.2 ->
  // 10.5 at 80 and 17.2 -> 13.4 at 144, down 35.5 -> 26 and 42.2 -> 32.5, QKV as halves 18.5 -> 13.9 at 96
  // (but 12.4 -> 13.7 at 80).  8B QKV at 112: whole pairs 19.1, halves 20.7, neither 21.9.  Below 80 only a
  // K loop over four ranks gains (7B O at 48: 11.4 -> 9.1; 8B QKV over two 14.4 -> 17.2).
  if (!gate_up && has_lo && n_pad >= kLargeCols && p.m_tiles % 2 == 0 && pc <= 4) {
    if ((n_pad > 128 && pc == 2) || (n_pad >= kHalfBoxCols && pc == 4 && p.m_tiles / 2 > fit(8)))
      take_pairs(pc / 2, 2);
    else if ((n_pad >= 80 || pc == 4) && p.m_tiles / 2 <= fit(2 * pc))
      take_pairs(pc, 1);
  }
  // the large-batch image runs eight warps instead of four (registers for two such CTAs per SM), so
  // that the parking, the cluster reduction and the epilogue after the MMAs run on twice the warps
  p.threads = n_pad >= 64 ? 256 : 128;
  return p;
}

// An adapter's A x keeps its few SMs (16 to 64 CTAs) to itself, over half of an SM's shared memory a CTA:
// beside CTAs of the projection that it lets start, its K loop and its parking took twice as long (gate/up's
// A x 8.8 us, 3.9 alone).  Eight 1.5B layers at rank 64 392 -> 370 us, rank 512 433 -> 411; four 7B layers,
// 16 candidates, rank 256 452 -> 431; rank 256 over 28 1.5B layers the same (1,550).
GemmPlan plan_lowrank(int rank, int K, int n_pad, int num_sms) {
  GemmPlan p = plan_gemm(rank, K, n_pad, num_sms, true, false);
  if (p.smem_bytes < kAloneSmem) p.smem_bytes = kAloneSmem;
  return p;
}

namespace {

typedef decltype(&gemm_cluster_kernel<false, GemmEpilogue::PLAIN, false, false>) GemmKernel;

enum GemmImage { kSmall, kLarge, kPair, kGemmImages };

template <int MODE, bool LORA = false>
GemmKernel image_of(GemmImage i) {
  if (i == kPair) return gemm_cluster_kernel<true, MODE, true, LORA>;
  return i == kLarge ? gemm_cluster_kernel<true, MODE, false, LORA> : gemm_cluster_kernel<false, MODE, false, LORA>;
}
// The kernel image of a batch class and epilogue, with an adapter's K tiles or without (null: none).
GemmKernel gemm_image(GemmImage i, int mode, bool lora) {
  switch (mode) {
    case GemmEpilogue::PLAIN: return lora ? nullptr : image_of<GemmEpilogue::PLAIN>(i);
    case GemmEpilogue::QKV: return lora ? image_of<GemmEpilogue::QKV, true>(i) : image_of<GemmEpilogue::QKV>(i);
    case GemmEpilogue::RESID: return lora ? image_of<GemmEpilogue::RESID, true>(i) : image_of<GemmEpilogue::RESID>(i);
    case GemmEpilogue::SILU: return lora ? image_of<GemmEpilogue::SILU, true>(i) : image_of<GemmEpilogue::SILU>(i);
    case GemmEpilogue::LOWRANK: return lora ? nullptr : image_of<GemmEpilogue::LOWRANK>(i);
  }
  return nullptr;
}

}  // namespace

cudaError_t gemm_configure(int n_pad_max, bool lora) {
  for (int i = 0; i < (n_pad_max >= kLargeCols ? kGemmImages : kLarge); ++i)
    for (int mode = GemmEpilogue::PLAIN; mode <= GemmEpilogue::LOWRANK; ++mode) {
      const bool ax = mode == GemmEpilogue::LOWRANK;   // an adapter's other launch
      const GemmKernel k = ax && !lora ? nullptr : gemm_image(static_cast<GemmImage>(i), mode, lora && !ax);
      if (!k) continue;
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kGemmMaxSmem));
      if (e == cudaSuccess && i != kPair) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

namespace {

// The image and launch configuration of a plan (null: none), but for the stream and its order; attr: two, the first
// of them set here.
GemmKernel gemm_config(const GemmPlan& p, int mode, int n_pad, bool lora, cudaLaunchConfig_t& cfg,
                       cudaLaunchAttribute* attr) {
  // the vector epilogues win from 48 padded columns on even with four warps (40 candidates of a 7B scorer
  // 564 -> 532 us for four layers; 24 candidates, 32 columns: 397 us small, 405 large)
  const bool large = n_pad >= kLargeCols;
  if (p.threads != 128 && (p.threads != 256 || !large)) return nullptr;
  if (p.pair && (!large || !p.has_lo || p.gate_up != (mode == GemmEpilogue::SILU))) return nullptr;
  const int units = (p.m_tiles + p.mt - 1) / p.mt;   // launched by the cluster, gate/up pairs' by two
  const bool gu_pair = p.pair && p.gate_up;
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3(gu_pair ? (units + 1) / 2 * 2 : units * p.cluster, 1, 1);
  cfg.blockDim = dim3(static_cast<unsigned>(p.threads), 1, 1);
  cfg.dynamicSmemBytes = p.smem_bytes;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = gu_pair ? 2 : p.cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return gemm_image(p.pair ? kPair : (large ? kLarge : kSmall), mode, lora);
}

}  // namespace

cudaError_t gemm_placement(const GemmPlan& p, int n_pad, int* clusters, int* placed) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  const GemmKernel kern = gemm_config(p, p.gate_up ? GemmEpilogue::SILU : GemmEpilogue::RESID, n_pad, false, cfg, attr);
  if (!kern) return cudaErrorInvalidValue;
  *clusters = static_cast<int>(cfg.gridDim.x / attr[0].val.clusterDim.x);
  return cudaOccupancyMaxActiveClusters(placed, kern, &cfg);
}

cudaError_t launch_gemm(const GemmPlan& p, const CUtensorMap* tmW, const CUtensorMap* tmX, const CUtensorMap* tmXlo,
                        const GemmEpilogue& ep, int n_pad, int* err, cudaStream_t stream, bool pdl,
                        unsigned long long* ts, const GemmLowRank* lr) {
  // without an adapter every K tile is W's and x's (the extra maps are never read)
  const bool with_lr = lr && lr->b && lr->t_hi && (!p.has_lo || lr->t_lo);
  if (with_lr && (lr->k_main < 1 || lr->k_main >= p.k_tiles)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  const GemmKernel kern = gemm_config(p, ep.mode, n_pad, with_lr, cfg, attr);
  if (!kern) return cudaErrorInvalidValue;
  cfg.stream = stream;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = pdl ? 2 : 1;
  const CUtensorMap& xlo = p.has_lo ? *tmXlo : *tmX;
  const CUtensorMap& mb = with_lr ? *lr->b : *tmW;
  const CUtensorMap& mt = with_lr ? *lr->t_hi : *tmX;
  const CUtensorMap& mtl = with_lr ? (p.has_lo ? *lr->t_lo : *lr->t_hi) : xlo;
  const int k_main = with_lr ? lr->k_main : p.k_tiles;
  GemmEpilogue e = ep;
  if (with_lr) {
    e.x_ready = lr->x_ready;
    e.call = lr->call;
  }
  return cudaLaunchKernelEx(&cfg, kern, *tmW, *tmX, xlo, p.has_lo ? 1 : 0, mb, mt, mtl, k_main, p.k_tiles,
                            p.ranks, p.stages, p.tmem_cols, n_pad / p.col_parts, p.col_parts, e, err, ts);
}

}  // namespace kvprm
