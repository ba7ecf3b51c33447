// sc_finalize.cuh -- the end of a layer's pruning for one sequence: the
// order-preserving compaction of the kept tokens and the state that the next
// layer reads, run by the CTA that finishes the sequence's scores last.
#pragma once

#include <cstdint>

#include "sc_internal.cuh"
#include "sc_layer_common.cuh"
#include "sc_select.cuh"

namespace sc {

// Per (round, warp) ballots of kept tokens and the exclusive prefix of their
// counts; the next layer's index of each global token.
template <int kThreads>
struct FinalSmem {
  static constexpr int kRounds = (kMaxLen + kThreads - 1) / kThreads;
  uint32_t kbits[kRounds][kThreads / 32];
  int kpre[kRounds][kThreads / 32];
  int gnew[kMaxGlobal];
  int last_pos;
  int total;
};
constexpr int kFinalScratch = sizeof(SelectSmem) + kMaxLen;   // used under the top-ratio rule

struct BlockSync {
  __device__ __forceinline__ void operator()() const { __syncthreads(); }
};

// Order-preserving compaction of sequence b's kept tokens, the next layer's
// global list, and the bf16 outputs of the global rows.  One CTA; token c is
// handled by thread c % kThreads in round c / kThreads (coalesced
// loads, all issued at once); output slots come from warp ballots and a
// fixed-order prefix over (round, warp).  Under the top-ratio rule the keep
// flags come from the cut over all n scores, found here (`scratch`: shared
// memory the CTA no longer uses, for the selection's histogram and tie flags).
template <int kThreads>
__device__ void finalize_sequence(const LayerParams& p, const LayerView& v, int b, int n, int ng,
                                  FinalSmem<kThreads>& sm, const int* gc, uint8_t* scratch) {
  constexpr int kRounds = FinalSmem<kThreads>::kRounds;
  constexpr int kWarps = kThreads / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint8_t* keep = p.keep + static_cast<size_t>(b) * p.L;
  const int32_t* pos = v.pos + static_cast<size_t>(b) * p.L;
  int32_t* pos_out = v.pos_out + static_cast<size_t>(b) * p.L;
  bool kf[kRounds];
  int32_t ps[kRounds];
  if (p.keep_rule == kKeepTopRatio) {
    const float* sc = v.scores + static_cast<size_t>(b) * p.L;
    uint32_t key[kRounds];
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      const int c = r * kThreads + tid;
      key[r] = (c >= 1 && c < n) ? select_key(__ldcg(sc + c)) : 0u;
      ps[r] = c < n ? __ldcg(pos + c) : 0;
    }
    SelectSmem& ss = *reinterpret_cast<SelectSmem*>(scratch);
    uint8_t* tie = scratch + sizeof(SelectSmem);
    uint32_t cut;
    int ties, eq;
    radix_cut<kThreads, kRounds>(key, top_count(v.alpha, n) - 1, n - 1, ss, tid, BlockSync(),
                                     cut, ties, eq);
    const bool split = eq > ties;   // an exact tie straddles the cut
    if (split) rank_ties<kThreads, kRounds>(key, cut, ties, n, tie, tid, BlockSync());
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      const int c = r * kThreads + tid;
      kf[r] = c < n && (c == 0 || key[r] > cut || (key[r] == cut && (!split || tie[c] == 2)));
    }
  } else {
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      const int c = r * kThreads + tid;
      kf[r] = c < n && __ldcg(keep + c) != 0;
      ps[r] = c < n ? __ldcg(pos + c) : 0;
    }
  }
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const uint32_t bits = __ballot_sync(0xffffffffu, kf[r]);
    if (lane == 0) sm.kbits[r][warp] = bits;
  }
  if (tid < kMaxGlobal) sm.gnew[tid] = -1;
  __syncthreads();
  if (warp == 0) {
    // prefix over (round, warp) in order: lane l covers entries l, l+32, ...
    constexpr int kEntries = kRounds * kWarps;
    int cnt[(kEntries + 31) / 32];
    int run = 0;
#pragma unroll
    for (int u = 0; u < (kEntries + 31) / 32; ++u) {
      const int e = u * 32 + lane;
      cnt[u] = e < kEntries ? __popc(sm.kbits[e / kWarps][e % kWarps]) : 0;
    }
#pragma unroll
    for (int u = 0; u < (kEntries + 31) / 32; ++u) {
      int x = cnt[u];
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
      }
      const int e = u * 32 + lane;
      if (e < kEntries) sm.kpre[e / kWarps][e % kWarps] = run + x - cnt[u];
      run += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) sm.total = run;
  }
  __syncthreads();
  const uint32_t below = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    if (!kf[r]) continue;
    const int out = sm.kpre[r][warp] + __popc(sm.kbits[r][warp] & below);
    pos_out[out] = ps[r];
    if (p.kept_cur) p.kept_cur[static_cast<size_t>(b) * p.L + out] = r * kThreads + tid;
    if (out == sm.total - 1) sm.last_pos = ps[r];
  }
  // next-layer index of each surviving global token
  if (tid < ng) {
    const int c = gc[tid], r = c / kThreads, t = c % kThreads;
    const uint32_t bits = sm.kbits[r][t >> 5];
    if ((bits >> (t & 31)) & 1u) sm.gnew[tid] = sm.kpre[r][t >> 5] + __popc(bits & ((1u << (t & 31)) - 1u));
  }
  __syncthreads();
  if (tid == 0) {
    const int total = sm.total;
    int m = 0;
    for (int g = 0; g < ng; ++g)
      if (sm.gnew[g] >= 0) v.gcur_out[b * kMaxGlobal + m++] = sm.gnew[g];
    v.ng_out[b] = m;
    v.len_out[b] = total;
    if (p.tail_from != nullptr && total <= p.tail_max) p.tail_from[b] = v.layer + 1;
    // the survivors are original positions 0..total-1 exactly when the last one is total-1
    v.ident_out[b] = (!p.no_ident && (total == 0 || sm.last_pos == total - 1)) ? 1 : 0;
    p.cnt_seq[b] = 0u;
  }
  for (int hh = tid; hh < p.H; hh += kThreads) p.rows_done[b * p.H + hh] = 0u;
}

}  // namespace sc
