// sc_scores.cu -- the scores kernel of the per-layer route: each key's column
// sum from the rows kernel's partials, the threshold, the compaction, and the
// outputs of the global rows.
//
// One CTA per 128-key tile of a sequence, every head in it: no tensor-core
// work, no operand tiles, no hand-over between heads.  A key's sum is, per
// head, the band partials of the query tiles of its band in tile order, plus
// the global rows' probabilities (kept by the rows kernel relative to each key
// tile's maximum, rescaled here by 2^(m_tile - LSE)), plus the far rows of the
// global keys; four threads share a key, each with every fourth head in order.
// What bounds it is latency: about ten microseconds of a layer pass between the
// last rows CTA and the end of the compaction, in a chain of dependent loads of
// 0.6 to 1 us each.  So every load of a step is issued before the first is used,
// the factors of many global rows are found by a thread per (head, row) (a warp
// each, twelve after one another, took 8 us at 16 rows and 12 heads), and one
// acq_rel atomic counts the CTAs (two membars around a relaxed one: 0.4 us).  The
// last CTA of a sequence compacts the survivors.  The global rows' outputs are
// the key tiles' parts, rescaled the same way and added in tile order, spread
// over the sequence's CTAs after they have counted themselves done, with the
// first loads in flight while the last CTA compacts.  Against the chain with
// each of these after the other, a 12-layer stack of 3 x 1000 tokens (w = 64)
// takes 264 us instead of 280, a layer of 2 x 3000 tokens with 16 globals
// (w = 512) 83.6 instead of 90.4.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "sc_finalize.cuh"
#include "sc_internal.cuh"
#include "sc_layer_common.cuh"
#include "sm103_primitives.cuh"

namespace sc {

constexpr int kScoresThreads = 512;
constexpr int kScoresWarps = kScoresThreads / 32;
constexpr int kHeadBlock = 16;   // heads whose rescaling factors are held at once
constexpr int kHeadGroups = kScoresThreads / kTile;   // threads of one key: heads g, g + 4, ...
constexpr int kGroupHeads = kHeadBlock / kHeadGroups;
constexpr int kRowBatch = 4;    // global rows after the first, loaded together
constexpr int kPartBatch = 8;   // key tiles of a global row, likewise

struct ScoresSmem {
  float scale[kHeadBlock][kMaxGlobal];      // 2^(m_tile - LSE) of (head, global row)
  float far[kMaxGlobal][kScoresWarps];      // far rows of a global key, per warp's heads
  float group[kHeadGroups - 1][kTile];
  int gc[kMaxGlobal];
  int abort, last;
  FinalSmem<kScoresThreads> fin;
  alignas(16) uint8_t scratch[kFinalScratch];
};

// LSE of one global row of one head from its key tiles' (max, sum), one tile
// per lane (at most kMaxTiles = 32).
__device__ __forceinline__ float2 global_stat(const float2* st, int Tn, int lane) {
  return lane < Tn ? __ldcg(st + static_cast<size_t>(lane) * kMaxGlobal)
                   : make_float2(-INFINITY, 0.f);
}
__device__ __forceinline__ float global_lse(const float2 e) {
  const float M = warp_max(e.x);
  return M + lg2(warp_sum(e.x == -INFINITY ? 0.f : e.y * ex2(e.x - M)));
}
static_assert(kMaxTiles <= 32, "one key tile per lane");

// The band rows' sums of key j for heads h0, h0 + kHeadGroups, ... < h1: per
// head the query tiles qlo .. qhi (slot = tile mod kSlots), loaded together.
template <int kSlots>
__device__ __forceinline__ void band_load(float (&part)[kGroupHeads][kWideBandTiles],
                                          const LayerParams& p, size_t bH, int j, bool use, int h0,
                                          int h1, int qlo, int qhi) {
#pragma unroll
  for (int k = 0; k < kGroupHeads; ++k) {
    const int h = h0 + k * kHeadGroups;
    const float* cp = p.colpart + (bH + h) * kSlots * p.L + j;
    int slot = qlo % kSlots;
#pragma unroll
    for (int u = 0; u < kWideBandTiles; ++u) {
      part[k][u] = (u < kSlots && use && h < h1 && qlo + u <= qhi)
                       ? __ldcg(cp + static_cast<size_t>(slot) * p.L) : 0.f;
      slot = slot + 1 == kSlots ? 0 : slot + 1;
    }
  }
}

__global__ void __launch_bounds__(kScoresThreads)
    sc_scores_kernel(const __grid_constant__ LayerParams p) {
  // No grid-wide wait on the rows kernel: this kernel is scheduled only after
  // every rows CTA has passed its own wait (so the earlier kernels' results
  // are complete), and each CTA waits below for the rows CTAs of its own
  // sequence only, so that it can run beside the rows kernel's last CTAs.
  pdl_launch_dependents();
  const int kt = blockIdx.x % p.T, b = blockIdx.x / p.T;
  const LayerView v = layer_view(p);
  if (owned_by_tail(p, v, b)) return;
  const int n = __ldcg(v.len + b);
  if (n == 0) {
    if (kt == 0 && threadIdx.x == 0) {
      v.len_out[b] = 0;
      v.ng_out[b] = 0;
      v.ident_out[b] = 1;
    }
    return;
  }
  const int j0 = kt * kTile;
  if (j0 >= n) return;
  const int ng = min(__ldcg(v.ng + b), kMaxGlobal);
  const int Tn = (n + kTile - 1) / kTile;
  const int H = p.H;
  const size_t bH = static_cast<size_t>(b) * H;
  __shared__ ScoresSmem sm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < kMaxGlobal) sm.gc[tid] = tid < ng ? __ldcg(v.gcur + b * kMaxGlobal + tid) : -1;
  if (tid == 0) {
    sm.abort = 0;
    wait_count(p.rows_done + bH, static_cast<uint32_t>(H * Tn), &sm.abort);
  }
  __syncthreads();

  const int r = tid & (kTile - 1), grp = tid / kTile;   // key of the tile, heads grp, grp + 4, ...
  const int j = j0 + r;
  const int qlo = max(0, j0 - p.w) / kTile;
  const int qhi = min(n - 1, min(j0 + kTile, n) - 1 + p.w) / kTile;
  const float2* gst = reinterpret_cast<const float2*>(p.gstat);
  float acc = 0.f;
  // far rows of the global keys of this tile: one partial per (query tile,
  // 32-row slice) and head
  auto far_rows = [&]() {
    for (int g = 0; g < ng; ++g) {
      const int c = sm.gc[g];
      if (c < j0 || c >= j0 + kTile) continue;
      float s = 0.f;
      for (int h = warp; h < H; h += kScoresWarps) {
        const float* fp = p.gpart + (bH + h) * p.T * 4 * kMaxGlobal + g;
#pragma unroll
        for (int k = 0; k < 4 * kMaxTiles / 32; ++k) {
          const int e = lane + 32 * k;
          s += e < 4 * Tn ? __ldcg(fp + e * kMaxGlobal) : 0.f;
        }
      }
      s = warp_sum(s);
      if (lane == 0) sm.far[g][warp] = s;
    }
  };
  for (int hb = 0; hb < H; hb += kHeadBlock) {
    const int he = min(H, hb + kHeadBlock);
    // (head, global row) pairs: a warp each, loaded first, or a thread each
    const int pairs = (he - hb) * ng;
    float2 st = make_float2(-INFINITY, 0.f);
    if (pairs <= kScoresWarps && warp < pairs)
      st = global_stat(gst + (bH + hb + warp / ng) * p.T * kMaxGlobal + warp % ng, Tn, lane);
    float part[kGroupHeads][kWideBandTiles];
    if (p.band_slots == kMaxBandTiles)
      band_load<kMaxBandTiles>(part, p, bH, j, j < n, hb + grp, he, qlo, qhi);
    else
      band_load<kWideBandTiles>(part, p, bH, j, j < n, hb + grp, he, qlo, qhi);
    // the first global row's probabilities (most layers have one global token)
    float pg[kGroupHeads];
#pragma unroll
    for (int k = 0; k < kGroupHeads; ++k) {
      const int h = hb + grp + k * kHeadGroups;
      pg[k] = ng > 0 && h < he && j < n
                  ? __ldcg(p.gprob + (bH + h) * kMaxGlobal * p.L + j) : 0.f;
    }
    float pr[kRowBatch][kGroupHeads];
    auto load_rows = [&](int g0) {
#pragma unroll
      for (int u = 0; u < kRowBatch; ++u)
#pragma unroll
        for (int k = 0; k < kGroupHeads; ++k) {
          const int h = hb + grp + k * kHeadGroups;
          pr[u][k] = g0 + u < ng && h < he && j < n
                         ? __ldcg(p.gprob + ((bH + h) * kMaxGlobal + g0 + u) * p.L + j) : 0.f;
        }
    };
    if (ng > 1) load_rows(1);
    if (hb > 0) __syncthreads();   // the previous heads' factors are read
    if (hb == 0) far_rows();
    if (pairs <= kScoresWarps) {
      if (warp < pairs) {
        const float lse = global_lse(st);
        const float mt = __shfl_sync(0xffffffffu, st.x, kt);
        if (lane == 0) sm.scale[warp / ng][warp % ng] = ex2(mt - lse);
      }
    } else if (tid < pairs) {
      const int hh = tid / ng, g = tid - hh * ng;
      const float2* gs = gst + (bH + hb + hh) * p.T * kMaxGlobal + g;
      float M = -INFINITY, S = 0.f;
#pragma unroll 1
      for (int t = 0; t < Tn; t += kPartBatch) {
        float2 x[kPartBatch];
#pragma unroll
        for (int k = 0; k < kPartBatch; ++k)
          x[k] = t + k < Tn ? __ldcg(gs + static_cast<size_t>(t + k) * kMaxGlobal)
                            : make_float2(-INFINITY, 0.f);
        float m = M;
#pragma unroll
        for (int k = 0; k < kPartBatch; ++k) m = fmaxf(m, x[k].x);
        if (m == -INFINITY) continue;
        S *= ex2(M - m);
#pragma unroll
        for (int k = 0; k < kPartBatch; ++k)
          S += x[k].x == -INFINITY ? 0.f : x[k].y * ex2(x[k].x - m);
        M = m;
      }
      const float mt = __ldcg(gs + static_cast<size_t>(kt) * kMaxGlobal).x;
      sm.scale[hh][g] = ex2(mt - (M + lg2(S)));
    }
#pragma unroll
    for (int k = 0; k < kGroupHeads; ++k) {
      float s = 0.f;
#pragma unroll
      for (int u = 0; u < kWideBandTiles; ++u) s += part[k][u];
      acc += s;
    }
    if (ng == 0) continue;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kGroupHeads; ++k)
      if (hb + grp + k * kHeadGroups < he) acc += pg[k] * sm.scale[grp + k * kHeadGroups][0];
#pragma unroll 1
    for (int g0 = 1; g0 < ng; g0 += kRowBatch) {
      if (g0 > 1) load_rows(g0);
#pragma unroll
      for (int u = 0; u < kRowBatch; ++u)
#pragma unroll
        for (int k = 0; k < kGroupHeads; ++k)
          if (g0 + u < ng && hb + grp + k * kHeadGroups < he)
            acc += pr[u][k] * sm.scale[grp + k * kHeadGroups][g0 + u];
    }
  }
  if (grp > 0) sm.group[grp - 1][r] = acc;
  __syncthreads();
  if (grp == 0 && j < n) {
#pragma unroll
    for (int k = 0; k < kHeadGroups - 1; ++k) acc += sm.group[k][r];
    for (int g = 0; g < ng; ++g)
      if (sm.gc[g] == j)
#pragma unroll
        for (int k = 0; k < kScoresWarps; ++k) acc += sm.far[g][k];
    const float s = acc / static_cast<float>(H * n);
    v.scores[static_cast<size_t>(b) * p.L + j] = s;
    if (p.keep_rule != kKeepTopRatio) {   // the top-ratio cut needs every score first
      const float theta = p.theta ? __ldg(p.theta + b)
                          : p.keep_rule == kKeepAbsolute ? v.alpha
                                                         : v.alpha / static_cast<float>(n);
      p.keep[static_cast<size_t>(b) * p.L + j] = (j == 0 || s >= theta) ? 1 : 0;
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (sm.abort) atomicOr(p.status, kStatusTimeout);
    // the scores and flags of this CTA (ordered by the barrier) before it is counted
    sm.last = atom_acq_rel_add_u32(p.cnt_seq + b, 1u) == static_cast<uint32_t>(Tn - 1);
  }
  // the global rows' outputs: (head, global row) pairs kt, kt + Tn, ..., two
  // warps each (32 of the 64 features), the key tiles' parts in tile order.  The
  // first pair's loads are issued before the last CTA compacts.
  const int d = 32 * (warp & 1) + lane;
  const int pairs = v.O == nullptr ? 0 : H * ng;
  int e = kt + Tn * (warp >> 1);
  float2 st = make_float2(-INFINITY, 0.f);
  float x[kPartBatch] = {};
  size_t t0 = 0;
  auto load_pair = [&]() {
    const int h = e / ng, g = e - h * ng;
    t0 = (bH + h) * p.T * kMaxGlobal + g;
    st = global_stat(gst + t0, Tn, lane);
  };
  auto load_parts = [&](int t) {
#pragma unroll
    for (int k = 0; k < kPartBatch; ++k)
      x[k] = t + k < Tn
                 ? __ldcg(p.gog + (t0 + static_cast<size_t>(t + k) * kMaxGlobal) * kHeadDim + d)
                 : 0.f;
  };
  if (e < pairs) {
    load_pair();
    load_parts(0);
  }
  __syncthreads();
  if (sm.last) finalize_sequence<kScoresThreads>(p, v, b, n, ng, sm.fin, sm.gc, sm.scratch);
#pragma unroll 1
  while (e < pairs) {
    const float lse = global_lse(st);
    const float wt = lane < Tn ? ex2(st.x - lse) : 0.f;
    float o = 0.f;
#pragma unroll 1
    for (int t = 0; t < Tn; t += kPartBatch) {
      if (t > 0) load_parts(t);
#pragma unroll
      for (int k = 0; k < kPartBatch; ++k)
        o = fmaf(x[k], __shfl_sync(0xffffffffu, wt, (t + k) & 31), o);
    }
    const int h = e / ng, g = e - h * ng;
    v.O[((static_cast<size_t>(b) * p.L + sm.gc[g]) * H + h) * kHeadDim + d] =
        __bfloat16_as_ushort(__float2bfloat16_rn(o));
    e += Tn * (kScoresWarps / 2);
    if (e < pairs) {
      load_pair();
      load_parts(0);
    }
  }
}

cudaError_t launch_scores(const LayerParams& p, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(p.B * p.T));
  cfg.blockDim = dim3(kScoresThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, sc_scores_kernel, p);
}

}  // namespace sc
