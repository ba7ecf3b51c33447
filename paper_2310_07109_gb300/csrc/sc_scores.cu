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
// What bounds it is latency: every load of a step is issued before the first
// is used.  The last CTA of a
// sequence compacts the survivors.  The global rows' outputs are the key tiles'
// parts, rescaled the same way and added in tile order, spread over the
// sequence's CTAs after they have counted themselves done.
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
// per lane (at most kMaxTiles = 32): m is this lane's maximum.
__device__ __forceinline__ float global_lse(const float2* st, int Tn, int lane, float& m) {
  const float2 e = lane < Tn ? __ldcg(st + static_cast<size_t>(lane) * kMaxGlobal)
                             : make_float2(-INFINITY, 0.f);
  m = e.x;
  const float M = warp_max(m);
  return M + lg2(warp_sum(m == -INFINITY ? 0.f : e.y * ex2(m - M)));
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
  for (int hb = 0; hb < H; hb += kHeadBlock) {
    const int he = min(H, hb + kHeadBlock);
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
    if (hb > 0) __syncthreads();   // the previous heads' factors are read
#pragma unroll 2
    for (int e = warp; e < (he - hb) * ng; e += kScoresWarps) {
      const int hh = e / ng, g = e - hh * ng;
      float m;
      const float lse = global_lse(gst + (bH + hb + hh) * p.T * kMaxGlobal + g, Tn, lane, m);
      const float mt = __shfl_sync(0xffffffffu, m, kt);
      if (lane == 0) sm.scale[hh][g] = ex2(mt - lse);
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
    for (int g = 1; g < ng; ++g) {
#pragma unroll
      for (int k = 0; k < kGroupHeads; ++k) {
        const int h = hb + grp + k * kHeadGroups;
        pg[k] = h < he && j < n ? __ldcg(p.gprob + ((bH + h) * kMaxGlobal + g) * p.L + j) : 0.f;
      }
#pragma unroll
      for (int k = 0; k < kGroupHeads; ++k)
        if (hb + grp + k * kHeadGroups < he) acc += pg[k] * sm.scale[grp + k * kHeadGroups][g];
    }
  }
  // far rows of the global keys of this tile: one partial per (query tile,
  // 32-row slice) and head
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
    __threadfence();   // the scores and flags of this CTA, before it is counted
    if (sm.abort) atomicOr(p.status, kStatusTimeout);
    sm.last = atomicAdd(p.cnt_seq + b, 1u) == static_cast<uint32_t>(Tn - 1);
  }
  __syncthreads();
  if (sm.last) {
    __threadfence();
    finalize_sequence<kScoresThreads>(p, v, b, n, sm.fin, sm.gc, sm.scratch);
  }

  // the global rows' outputs: (head, global row) pairs kt, kt + Tn, ..., two
  // warps each (32 of the 64 features), the key tiles' parts in tile order
  if (v.O == nullptr) return;
  for (int e = kt + Tn * (warp >> 1); e < H * ng; e += Tn * (kScoresWarps / 2)) {
    const int h = e / ng, g = e - h * ng;
    const size_t t0 = (bH + h) * p.T;
    float m;
    const float lse = global_lse(gst + t0 * kMaxGlobal + g, Tn, lane, m);
    const float wt = lane < Tn ? ex2(m - lse) : 0.f;
    const int d = 32 * (warp & 1) + lane;
    const float* part = p.gog + (t0 * kMaxGlobal + g) * kHeadDim + d;
    float o = 0.f;
    constexpr int kBatch = 8;   // loads in flight before they are added
    for (int t = 0; t < Tn; t += kBatch) {
      float x[kBatch];
#pragma unroll
      for (int k = 0; k < kBatch; ++k)
        x[k] = t + k < Tn ? __ldcg(part + static_cast<size_t>(t + k) * kMaxGlobal * kHeadDim) : 0.f;
#pragma unroll
      for (int k = 0; k < kBatch; ++k) o = fmaf(x[k], __shfl_sync(0xffffffffu, wt, (t + k) & 31), o);
    }
    v.O[((static_cast<size_t>(b) * p.L + sm.gc[g]) * H + h) * kHeadDim + d] =
        __bfloat16_as_ushort(__float2bfloat16_rn(o));
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
