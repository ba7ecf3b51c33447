// sc_kernels.cu -- device code of one sparse-attention + learned-token-pruning
// layer on sm_103a.
//
// Per layer, per sequence b (n current tokens, original positions pos[b][*]):
//
//   rows kernel   (one CTA per 128-row query tile of one (sequence, head), two
//                 CTAs per SM)
//     S = Q K^T over the band in items of 64 keys and one 16-wide item of global
//     keys on the tensor cores (tcgen05, bf16 -> fp32 in tensor memory); each
//     16 KB operand tile is one TMA copy.  Row softmax in fp32 (base 2, a
//     reference per row that is raised when it has to be); P (bf16) goes back
//     to tensor memory and P V accumulates there.  Then the band pass: S^T =
//     K Q^T of each key tile of the band and, per key column j, the sum over the
//     tile's rows of exp2(S_ij - LSE_i) (one thread per column, no cross-thread
//     reduction), one partial per (key, query tile).  Writes O, those partials,
//     the far-row column sums of the global keys, and, for the tile's own keys,
//     the global rows' probabilities and P V relative to the tile's maximum.
//
//   scores kernel (sc_scores.cu; one CTA per 128 keys of a sequence)
//     Each key's column sum: the band partials added in tile order, plus the
//     global rows' share, heads in a fixed order; the threshold; the last CTA of
//     a sequence compacts the survivors in order.  Each CTA waits (bounded) only
//     for the rows CTAs of its own sequence; the "last" CTA is found by an
//     atomic counter.
//
//   cols kernel   the same role behind the single-pass band kernel (sc_band.cu):
//     one CTA per pair of 128-key tiles and head.
//
//   gather kernel copies the survivors' next-layer Q, K, V rows into compacted
//   buffers (coalesced 16-byte vectors) when they are not already in place.
//
// The method (allowed sets, row softmax, vertical accumulation, >= threshold,
// order-preserving removal) is Sec. "Sparse Attention", Sec. "Extractor of
// Attention Scores in Sparse Attention Matrix" and Sec. "Token Pruning".
#include <algorithm>
#include <cuda_runtime.h>
#include <utility>
#include <cuda_bf16.h>
#include <cstddef>
#include <cstdint>

#include "sc_internal.cuh"
#include "sc_finalize.cuh"
#include "sc_layer_common.cuh"
#include "sm103_primitives.cuh"

namespace sc {

// The global rows' P is the A operand of an M = 128 MMA whose rows past the 16
// global rows are never used: each 64-key block of that A tile holds its 16
// valid rows (2 KB) and lets the MMA read the following rows from whatever
// shared memory comes next, so only 2 KB is reserved.
constexpr uint32_t kPgBlock = 2 * 1024;

// ---------------------------------------------------------------------------
// rows kernel
// ---------------------------------------------------------------------------
// One CTA per 128-row query tile of one (sequence, head), two CTAs per SM, so
// that one CTA's start and end hide behind the other's exponentials.  Warps 0-3
// (one thread per row) are the softmax; warp 4 issues the MMAs, warp 5 the
// copies, warps 6 and 7 evaluate the global rows over the tile's keys beside
// the softmax.
//
// The softmax warps take one item after the other from three 64-column buffers
// in tensor memory, filled in order by warp 4, three items ahead:
//   row pass    S of 64 keys of the band (the blocks that some row attends to),
//               then S_G of the 16 global keys: P (bf16) goes over the first
//               columns of the item's own buffer, and P V reads it there
//   band pass   S^T of a 128-key tile against 64 queries, last tile first (the
//               last three are still in shared memory): per key column the sum
//               over the rows of exp2(S - LSE); after the diagonal tile S_Gt,
//               its keys against the global queries
// Handing an item back (P stored, or S^T read) lets warp 4 issue P V and the
// item three further on into the same buffer: what overwrites columns that an
// earlier product reads is issued after it.  32-column chunks that no row of a
// warp attends to are not evaluated.
//
// Tensor memory (256 columns a CTA): the buffers [0, 192), O [192, 256); once O
// is out, its columns take the global rows' P V.
//
// What bounds it: each allowed (row, key) pair costs two exponentials, one in
// each pass, and about eight further issue slots; with one softmax warp of each
// CTA on an SM sub-partition the in-order issue of two warps (IPC 0.4 of 1),
// not the exponential unit (a fifth busy) or the tensor cores (a quarter).  So
// the gains lie in instructions and latencies: three items in flight, narrow
// bands by 64-key items and 32-column chunks, two independent CTAs.  Code size
// counts as much: every section but the two item loops runs once a CTA, and at
// 78 KB of code instead of 55 KB the kernel missed the instruction caches and
// took 14% longer.
// Layer 0 of 2 x 4096 tokens (w 256, 12 heads, 9 global tokens), rows and scores
// together: 80 us, against 89 us for pairs of query tiles in one CTA per SM
// with whole-tile items and a tensor-core scores kernel; 4 x 4096, one global
// token: 117 against 145 us; 8 x 1024 at w 64: 45 against 71 us.
constexpr int kRowsThreads = 256;
constexpr int kKSlots = 3, kVSlots = 2;          // 16 KB operand slots
constexpr int kRowsSlots = kKSlots + kVSlots;    // K tiles 0..2, V tiles 3..4
constexpr int kBufs = 3;
constexpr int kHalf = 64;                        // columns of a buffer: keys (queries) of an item
constexpr uint32_t kColO = kBufs * kHalf;
constexpr uint32_t kColPG = kMaxGlobal;          // P_G in its buffer, after S_G
constexpr float kRefSlack = 6.f;                 // base 2 (see the softmax)

struct RowsSmem {
  alignas(16) float nlse[kTile];         // -LSE of the tile's rows (read as float4)
  float gm[kMaxGlobal][2];               // global rows: maximum over 64 of the tile's keys
  float gs[kMaxGlobal][2];               // ... and sum of exponentials
  // in this order: first those with one arrival per softmax warp
  uint64_t bar_back[kBufs];              // a buffer's item is handed back
  uint64_t bar_stage, bar_gx;
  uint64_t bar_q, bar_g, bar_vd;
  uint64_t full[kRowsSlots], empty[kRowsSlots];
  uint64_t bar_full[kBufs];              // a buffer's item is there
  uint64_t bar_pv[kBufs];                // P V of the buffer's item is complete
  uint64_t bar_og, bar_fin;
  uint64_t bar_stall;                    // test hook: nothing ever completes it
  uint32_t tmem_base;
  int abort;
  int gc[kMaxGlobal];
};

constexpr int kRowsBars4 = kBufs + 2;
constexpr int kRowsBars = kRowsBars4 + 3 + 2 * kRowsSlots + 2 * kBufs + 3;
static_assert(kRowsBars <= 32, "one barrier a lane at start");
static_assert(offsetof(RowsSmem, bar_stall) - offsetof(RowsSmem, bar_back) == 8 * (kRowsBars - 1),
              "the barriers are consecutive");

// dynamic shared memory: the Q tile, the global rows' P blocks, the operand
// slots, the global rows (whose space takes S_Gt in the band pass).  The P
// blocks' 16 rows are rows 64..79 of the A operand of an M = 128 product (so
// that its result lies in warp 6's lanes); the other rows read the shared
// memory around them.
constexpr uint32_t kGxBytes = kMaxGlobal * kTile * 4;
static_assert(kGxBytes >= 3 * kGTileBytes, "S_Gt takes the global rows' space");
constexpr uint32_t kPgRow0 = 64;
static_assert(kTileBytes >= kPgRow0 * 128 && kRowsSlots * kTileBytes >= 8 * 1024,
              "the A operand's unused rows stay inside the shared memory");
constexpr uint32_t kRowsDyn = kTileBytes * (1 + kRowsSlots) + 2 * kPgBlock + kGxBytes + 1024;

// Where key tile u of the band pass (counted from the last tile of the row
// pass, nk tiles in all) sits: the last three are still in their K slots; the
// others are loaded again, into the V slot of the last tile but one, then the K
// slots in the order in which the band pass frees them.
struct SlotFill {
  int slot, fill;   // fill-th filling of the slot
};
__device__ __forceinline__ SlotFill band_slot(int u, int nk) {
  if (u < kKSlots) {
    const int t = nk - 1 - u;
    return {t % kKSlots, t / kKSlots};
  }
  const int r = u - kKSlots, c = r & 3;
  if (c == 0) return {kKSlots + (nk & 1), (nk - 2) / kVSlots + 1 + (r >> 2)};
  const int t = nk - c;
  return {t % kKSlots, t / kKSlots + 1 + (r >> 2)};
}

// Which of a warp's 32 rows may attend to keys c0 .. c0 + 31 (rows i0 .. i0 + 31):
// 0 none, 1 some, 2 all of them to all keys.
__device__ __forceinline__ int chunk_kind(int i0, int c0, int w, int n) {
  if (c0 + 31 < i0 - w || c0 > min(n - 1, i0 + 31 + w)) return 0;
  return (c0 >= i0 + 31 - w && c0 + 31 <= min(n - 1, i0 + w)) ? 2 : 1;
}

// x[k] = -inf outside lo..hi (columns of the chunk).
__device__ __forceinline__ void mask_range(float* x, int lo, int hi) {
  const uint32_t in = bit_range32(lo, hi);
#pragma unroll
  for (int k = 0; k < 32; ++k) x[k] = (in & (1u << k)) ? x[k] : -INFINITY;
}

__global__ void __launch_bounds__(kRowsThreads, 2)
    sc_rows_kernel(const __grid_constant__ TensorMaps maps, const __grid_constant__ LayerParams p) {
  // the scores kernel is scheduled once every CTA here is past this wait (and
  // holds its tensor memory), so what the kernels before this one wrote is
  // complete when it starts (with p.gathered, the gather kernel before this
  // one lets it start only once the kernels before the gather are complete,
  // and each CTA waits below for its own sequence's rows)
  if (p.gathered == nullptr) pdl_wait();
  // grid: query tiles, (sequence, head)-major, so that the CTAs of a sequence
  // finish together and its scores CTAs can start early
  const int qt = blockIdx.x % p.T, bh = blockIdx.x / p.T;
  const int h = bh % p.H, b = bh / p.H;
  const LayerView v = layer_view(p);
  // the sequence's state, loaded together
  const bool tailed = owned_by_tail(p, v, b);
  const int n = __ldcg(v.len + b);
  const int ng_raw = __ldcg(v.ng + b);
  const int gc_raw = threadIdx.x < kMaxGlobal ? __ldcg(v.gcur + b * kMaxGlobal + threadIdx.x) : -1;
  const RowSource rs = row_source(p, v, b);
  if (tailed) return;
  const int q0 = qt * kTile;
  if (q0 >= n) return;
  const int ng = min(ng_raw, kMaxGlobal);
  const bool glob = ng > 0;

  extern __shared__ uint8_t dyn_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dyn_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* Qs = base;
  uint8_t* Pg = Qs + kTileBytes;                   // 2 blocks of 16 rows
  uint8_t* Slots = Pg + 2 * kPgBlock;              // K slots, V slots
  uint8_t* KG = Slots + kRowsSlots * kTileBytes;
  uint8_t* VG = KG + kGTileBytes;
  uint8_t* QG = VG + kGTileBytes;
  float* const gx = reinterpret_cast<float*>(KG);  // S_Gt [kMaxGlobal][kTile]
  __shared__ RowsSmem sm;

  // the warp index, uniform over the warp
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int w = p.w;
  // keys that some row of the tile attends to, and their key tiles
  const int q1 = min(q0 + kTile - 1, n - 1);
  const int jlo = max(0, q0 - w), jhi = min(n - 1, q1 + w);
  const int klo = jlo / kTile;
  const int nk = jhi / kTile - klo + 1;            // <= 9; window checked on the host
  const int blo = jlo / kHalf;                     // 64-key blocks of the row pass
  const int nrow = jhi / kHalf - blo + 1 + (glob ? 1 : 0);   // its items
  const int u_d = nk - 1 - (qt - klo);             // the diagonal tile in the band pass
  // the last tile's V slot: O leaves through it, then it takes V of the
  // diagonal tile, for the global rows
  const int vd_slot = kKSlots + ((nk - 1) & 1);
  // the band pass: some key of tile u attends to some query of the half
  auto reaches = [&](int u, int qh) {
    const int j0 = (klo + nk - 1 - u) * kTile, i0 = q0 + kHalf * qh;
    return i0 < n && min(j0 + kTile, n) - 1 + w >= i0 && j0 - w <= min(i0 + kHalf, n) - 1;
  };

  uint32_t fills = 0;   // warp 5: how often each slot has been filled (four bits a slot)
  if (warp == 5) {
    // the barriers, one a lane; then the first copies, ahead of the block's start
    if (lane < kRowsBars) mbar_init(sm.bar_back + lane, lane < kRowsBars4 ? 4 : 1);
    if (lane == 0) sm.abort = 0;
    fence_mbar_init();
    __syncwarp();
    if (lane == 0) {
      // this sequence's rows may still be crossing the host link
      if (p.gathered != nullptr) {
        wait_count(p.gathered + b, p.gather_target, &sm.abort);
        fence_proxy_async_global();   // the copies, before any TMA load
      }
      mbar_arrive_expect_tx(&sm.bar_q, kTileBytes);
      load_tile(maps, 0, rs, h, q0, Qs, &sm.bar_q);
      for (int t = 0; t < min(nk, 2); ++t) {
        mbar_arrive_expect_tx(&sm.full[t], kTileBytes);
        load_tile(maps, 1, rs, h, (klo + t) * kTile, Slots + t * kTileBytes, &sm.full[t]);
      }
      mbar_arrive_expect_tx(&sm.full[kKSlots], kTileBytes);
      load_tile(maps, 2, rs, h, klo * kTile, Slots + kKSlots * kTileBytes, &sm.full[kKSlots]);
    }
    __syncwarp();
    fills = 1u | (nk > 1 ? 1u << 4 : 0u) | 1u << (4 * kKSlots);
  }
  if (tid < kMaxGlobal) sm.gc[tid] = tid < ng ? gc_raw : -1;
  if (warp == 4) tmem_alloc(&sm.tmem_base, 256);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_launch_dependents();
  const uint32_t tm = __shfl_sync(0xffffffffu, sm.tmem_base, 0);
  volatile int* abort_flag = &sm.abort;
  const size_t tile = (static_cast<size_t>(b) * p.H + h) * p.T + qt;   // of the partial results

  if (warp >= 4) {
    if (warp == 4) {
      // ----------------------------------------------------------- MMA issue
      const uint32_t q_d = sdesc_lo(smem_u32(Qs)), slot_d = sdesc_lo(smem_u32(Slots));
      constexpr uint32_t kTileD = kTileBytes >> 4;   // in descriptors
      constexpr uint32_t kIdS = idesc_bf16(128, kHalf, false, false);
      constexpr uint32_t kIdG = idesc_bf16(128, 16, false, false);
      constexpr uint32_t kIdPV = idesc_bf16(128, 64, false, true);
      constexpr uint32_t kHalfD = kTileD / 2;
      const uint32_t kg_d = sdesc_lo(smem_u32(KG)), vg_d = sdesc_lo(smem_u32(VG)),
                     qg_d = sdesc_lo(smem_u32(QG));
      const int nblk = nrow - (glob ? 1 : 0);
      bool ok = true;
      if (p.stall_ns != 0)   // test hook: this bounded wait expires
        ok = __all_sync(0xffffffffu, mbar_wait(&sm.bar_stall, 0, abort_flag, p.stall_ns));
      ok = ok && warp_wait_poll(&sm.bar_q, 0, abort_flag);
      // the next item of the sequence, into buffer ib
      int is = 0, ib = 0, u = 0, qh = nk > 0 && !reaches(0, 0) ? 1 : 0;
      bool sgt = false, more = true;
      auto issue_next = [&]() {
        uint32_t a_d, b_d;
        uint64_t *wait = nullptr, *release = nullptr;
        uint32_t par = 0, id = kIdS;
        if (is < nblk) {                            // S of block is
          const int kb = blo + is, t = kb / 2 - klo, slot = t % kKSlots;
          wait = &sm.full[slot];
          par = (t / kKSlots) & 1;
          a_d = q_d;
          b_d = slot_d + slot * kTileD + (kb & 1) * kHalfD;
          // a tile's slot is free after its last block; the last three tiles stay
          if (t < nk - kKSlots && (kb & 1)) release = &sm.empty[slot];
          ++is;
        } else if (is < nrow) {                     // S_G
          wait = &sm.bar_g;
          a_d = q_d;
          b_d = kg_d;
          id = kIdG;
          ++is;
        } else {
          const SlotFill f = band_slot(u, nk);
          wait = &sm.full[f.slot];
          par = f.fill & 1;
          a_d = slot_d + f.slot * kTileD;
          const bool last = qh == 1 || !reaches(u, 1);
          if (sgt) {                                // S_Gt of the diagonal tile
            b_d = qg_d;
            id = kIdG;
          } else {                                  // S^T of tile u, query half qh
            b_d = q_d + qh * kHalfD;
          }
          if (!sgt && last && glob && u == u_d) {
            sgt = true;                             // the next item
          } else if (sgt || last) {
            release = &sm.empty[f.slot];
            sgt = false;
            ++u;
            qh = u < nk && !reaches(u, 0) ? 1 : 0;
          } else {
            qh = 1;
          }
          more = u < nk;
        }
        if (!(ok = warp_wait_poll(wait, par, abort_flag))) return;
        tc_fence_after();
        const uint32_t d = tm + kHalf * ib;
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < kHeadDim / 16; ++k)
            umma_bf16_lo(d, a_d + 2 * k, b_d + 2 * k, id, k > 0);
          umma_commit(&sm.bar_full[ib]);
          if (release != nullptr) umma_commit(release);
        }
        __syncwarp();
        ib = ib == kBufs - 1 ? 0 : ib + 1;
      };
      // kBufs items ahead of the one whose hand-over is awaited
      int left = kBufs;   // items issued and not handed back (from it = 0 on)
#pragma unroll 1
      for (int it = -kBufs, buf = 0, use = 0; ok && (it < 0 || left > 0); ++it) {
        if (it >= 0) {
          if (!(ok = warp_wait_poll(&sm.bar_back[buf], use & 1, abort_flag))) break;
          --left;
          if (it < nrow) {                          // P V
            const int kb = blo + it, t = kb / 2 - klo;
            const bool g = it >= nblk;
            const int slot = kKSlots + (t & 1);
            if (!g && !(ok = warp_wait_poll(&sm.full[slot], (t / kVSlots) & 1, abort_flag))) break;
            if (!g && (kb + 1) * kHalf > n) {   // (the last block)
              zero_rows(Slots + slot * kTileBytes, n - (klo + t) * kTile, kHalf * ((kb & 1) + 1),
                        lane, 32);
              __syncwarp();
            }
            tc_fence_after();
            const uint32_t v_d = g ? vg_d : slot_d + slot * kTileD + (kb & 1) * kHalfD;
            if (elect_one()) {
              umma_bf16_ts_lo(tm + kColO, tm + kHalf * buf + (g ? kColPG : 0), v_d, kIdPV, it > 0);
              if (!g)
#pragma unroll
                for (int k = 1; k < kHalf / 16; ++k)
                  umma_bf16_ts_lo(tm + kColO, tm + kHalf * buf + 8 * k, v_d + 128 * k, kIdPV, 1u);
              umma_commit(&sm.bar_pv[buf]);
              if (!g && ((kb & 1) || it == nblk - 1)) umma_commit(&sm.empty[slot]);
            }
            __syncwarp();
          }
          if (++buf == kBufs) {
            buf = 0;
            ++use;
          }
        }
        if (more) {
          issue_next();
          if (it >= 0) ++left;
        } else if (it < 0) {
          --left;                                   // fewer items than buffers
        }
      }
      if (elect_one()) umma_commit(&sm.bar_fin);
      __syncwarp();
      drain_wait(&sm.bar_fin, 0);
    } else if (warp == 5) {
      // ----------------------------------------------------------- copies
      if (p.gathered != nullptr) fence_proxy_async_global();   // every lane that issues copies
      bool ok = true, vd = false;
      auto load_slot = [&](int t, int tensor, int slot, bool vdl) {
        const uint32_t f = (fills >> (4 * slot)) & 15u;
        if (f > 0 && !(ok = warp_wait_poll(&sm.empty[slot], (f - 1) & 1, abort_flag))) return;
        uint64_t* bar = vdl ? &sm.bar_vd : &sm.full[slot];
        if (elect_one()) {
          mbar_arrive_expect_tx(bar, kTileBytes);
          load_tile(maps, tensor, rs, h, (klo + t) * kTile, Slots + slot * kTileBytes, bar);
        }
        __syncwarp();
        if (vdl) vd = true;
        else fills += 1u << (4 * slot);
      };
      if (glob) {
        if (elect_one()) mbar_arrive_expect_tx(&sm.bar_g, 3 * kGTileBytes);
        __syncwarp();
#pragma unroll 1
        for (int k = 0; k < 3; ++k)   // K, V, Q
          load_globals(maps, k == 2 ? 0 : k + 1, rs, h, p.H, sm.gc, ng, KG + k * kGTileBytes,
                       &sm.bar_g, lane);
        __syncwarp();
      }
      // in this order: V of tile 1, K of tile 2, V of tile 2, ...; then the
      // band pass's K tiles that are no longer here, after the first of them V
      // of the diagonal tile for the global rows
#pragma unroll 1
      for (int i = 0; ok && i < 2 * nk; ++i) {
        const int r = i - 2 * (nk - 1);   // 0, 1: the first band tile, V of the diagonal tile
        int t = 1 + i / 2, tensor = 2, slot = kKSlots + (t & 1);
        bool vdl = false;
        if (r < 0 && (i & 1)) {
          if (++t >= nk) continue;
          tensor = 1;
          slot = t % kKSlots;
        } else if (r == 0) {
          if (nk <= kKSlots) continue;
          t = nk - 1 - kKSlots;
          tensor = 1;
          slot = band_slot(kKSlots, nk).slot;
        } else if (r == 1) {
          if (!glob) continue;
          if (!(ok = warp_wait_poll(&sm.bar_stage, 0, abort_flag))) break;
          t = qt - klo;
          slot = vd_slot;
          vdl = true;
        }
        load_slot(t, tensor, slot, vdl);
      }
#pragma unroll 1
      for (int u = kKSlots + 1; ok && u < nk; ++u) load_slot(nk - 1 - u, 1, band_slot(u, nk).slot, false);
      // nothing may still be landing in shared memory when the CTA exits
#pragma unroll 1
      for (int s = 0; s < kRowsSlots + 3; ++s) {
        const uint32_t f = s < kRowsSlots ? (fills >> (4 * s)) & 15u
                           : s == kRowsSlots || (s == kRowsSlots + 1 ? glob : vd) ? 1u : 0u;
        uint64_t* bar = s < kRowsSlots ? &sm.full[s] : &sm.bar_q + (s - kRowsSlots);
        if (f > 0) drain_wait(bar, (f - 1) & 1);
      }
    } else if (glob) {
      // ----------------------------------------------------------- global rows
      // over this tile's keys (two a thread): their probabilities relative to
      // the tile's maximum, and P V
      const int x = tid & 63, half = warp & 1;
      bool ok = warp_wait_poll(&sm.bar_gx, 0, abort_flag);
#pragma unroll 1
      for (int g = 0; ok && g < ng; ++g) {
        const float m = warp_max(fmaxf(gx[g * kTile + x], gx[g * kTile + 64 + x]));
        if (lane == 0) sm.gm[g][half] = m;
      }
      asm volatile("bar.sync 2, 64;" ::: "memory");
      float* gp = p.gprob + (static_cast<size_t>(b) * p.H + h) * kMaxGlobal * p.L + q0 + x;
#pragma unroll 1
      for (int g = 0; ok && g < ng; ++g) {
        const float m = fmaxf(sm.gm[g][0], sm.gm[g][1]);
        // (a key past the end has S_Gt = -inf; m is finite: the tile has a key)
        const float a = ex2(gx[g * kTile + x] - m), c = ex2(gx[g * kTile + 64 + x] - m);
        if (q0 + x < n) gp[static_cast<size_t>(g) * p.L] = a;
        if (q0 + 64 + x < n) gp[static_cast<size_t>(g) * p.L + 64] = c;
        // transposed into the A tile: row g, column (key)
        const uint32_t at = sw128_offset(g, x >> 3) + (x & 7) * 2;
        *reinterpret_cast<uint16_t*>(Pg + at) = __bfloat16_as_ushort(__float2bfloat16_rn(a));
        *reinterpret_cast<uint16_t*>(Pg + kPgBlock + at) =
            __bfloat16_as_ushort(__float2bfloat16_rn(c));
        const float s = warp_sum(a + c);
        if (lane == 0) sm.gs[g][half] = s;
      }
      fence_proxy_async_smem();
      asm volatile("bar.sync 2, 64;" ::: "memory");
      if (warp == 6) {
        ok = ok && warp_wait_poll(&sm.bar_vd, 0, abort_flag);
        if (ok) {
          if (q0 + kTile > n) {
            zero_rows(Slots + vd_slot * kTileBytes, n - q0, kTile, lane, 32);
            __syncwarp();
          }
          tc_fence_after();   // O is out: its columns take the product
          if (elect_one()) {
            mma_pv(tm + kColO, smem_u32(Pg) - kPgRow0 * 128, kPgBlock,
                   smem_u32(Slots) + vd_slot * kTileBytes, kTile / 16, false);
            umma_commit(&sm.bar_og);
          }
          __syncwarp();
          ok = warp_wait_poll(&sm.bar_og, 0, abort_flag);
          tc_fence_after();
          float* part = p.gog + (tile * kMaxGlobal + lane) * kHeadDim;
#pragma unroll 1
          for (int c = 0; ok && c < 64; c += 16) {
            float o[16];
            tmem_ld16(tm + kColO + (kPgRow0 << 16) + c, o);
            tmem_ld_wait();
            if (lane < ng)
#pragma unroll
              for (int k = 0; k < 16; k += 4)
                *reinterpret_cast<float4*>(part + c + k) =
                    make_float4(o[k], o[k + 1], o[k + 2], o[k + 3]);
          }
          if (!ok) drain_wait(&sm.bar_og, 0);
        }
      } else if (ok && lane < ng) {
        reinterpret_cast<float2*>(p.gstat)[tile * kMaxGlobal + lane] = make_float2(
            fmaxf(sm.gm[lane][0], sm.gm[lane][1]), sm.gs[lane][0] + sm.gs[lane][1]);
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------- softmax
    const int r = tid;                    // row inside the tile == TMEM lane
    const int i = q0 + r;                 // current index of this query row
    const int iw = q0 + 32 * warp;        // first row of this warp
    const uint32_t lane_off = static_cast<uint32_t>(warp * 32) << 16;
    const uint32_t tB = tm + lane_off, tO = tB + kColO;
    bool row_global = false;
#pragma unroll 1
    for (int g = 0; g < ng; ++g) row_global |= (sm.gc[g] == i);
    const bool valid = (i < n) && !row_global;
    // allowed band keys of this row, inclusive (current index); the same band
    // is used for rows whose results are discarded (global rows, rows >= n)
    const int lo = max(0, i - w), hi = min(n - 1, i + w);
    const uint64_t c2 = f2_pack(kLogitScale2, kLogitScale2);
    bool ok = true;
    int buf = 0;                          // of the current item, and which use of it
    uint32_t use = 0;
    auto wait_item = [&]() {
      ok = ok && warp_wait_poll(&sm.bar_full[buf], use & 1, abort_flag);
      tc_fence_after();
    };
    auto hand_back = [&]() {
      tc_fence_before();
      warp_arrive(&sm.bar_back[buf]);
      if (++buf == kBufs) {
        buf = 0;
        ++use;
      }
    };

    // Softmax with a running reference m_ref (base-2 units): P = exp2(x - ref).
    // Where some row's maximum over the item lies more than kRefSlack above its
    // reference, every row of the warp that lies below its own maximum takes that
    // as its reference, and the row sums and O are rescaled: O after the item's
    // exponentials, when the P V before it is long complete.  So P stays below
    // 2^kRefSlack.  (The reference of a row, and with it the last bits of its O,
    // thus depends on the 31 rows of its warp too.)
    // Only the element the reference comes from is exact in bf16, so a reference
    // nearer to the maximum makes O's error smaller; at 6 the error against 64
    // bits is that of whole-tile items raised past 2^8.  12 layers of 8 x 1024
    // and 4 x 4096 tokens (w = 256) and a layer of 2 x 3000 (w = 512): 283, 1368
    // and 86 us; at 8 with errors 1 to 2 % larger 281, 1350 and 85.5; with no
    // maximum unless the exponentials of an item sum to 2^24, 3 to 4 % larger,
    // 279, 1329 and 84; the same past 2^8 by a second evaluation of the item
    // and O rescaled before it, 314, 1628 and 99.
    // lsum: the row sum of the exponentials (fp32), which gives the row's LSE
    // for the column sums; osum: the sum of the same values rounded to the
    // bf16 that P V multiplies, which normalises O (so that O is a weighted
    // mean of V rows whatever the rounding of P)
    float m_ref = i < n ? -INFINITY : 0.f, lsum = 0.f, osum = 0.f;
    // raise_to returns the factor that the row's O takes (see rescale)
    auto raise_to = [&](float tmax) {
      float f = 1.f;
      if (__any_sync(0xffffffffu, i < n && tmax > m_ref + kRefSlack) && i < n && tmax > m_ref) {
        f = m_ref == -INFINITY ? 0.f : ex2(m_ref - tmax);
        m_ref = tmax;
        lsum *= f;
        osum *= f;
      }
      return f;
    };
    auto rescale = [&](float f) {
      if (!__any_sync(0xffffffffu, f != 1.f)) return;
      // the item before this one: its P V, hence every earlier one
      const int pb = buf == 0 ? kBufs - 1 : buf - 1;
      ok = ok && warp_wait_poll(&sm.bar_pv[pb], (buf == 0 ? use - 1 : use) & 1, abort_flag);
      tc_fence_after();
#pragma unroll 1
      for (int c = 0; c < 64; c += 32) {
        float o[32];
        tmem_ld32(tO + c, o);
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 32; ++k) o[k] *= f;
        tmem_st32(tO + c, o);
      }
      tmem_st_wait();
    };
#pragma unroll 1
    for (int it = 0; it < nrow - (glob ? 1 : 0); ++it) {
      const int j0 = (blo + it) * kHalf;
      const int kind0 = chunk_kind(iw, j0, w, n), kind1 = chunk_kind(iw, j0 + 32, w, n);
      wait_item();
      if (!ok) break;
      const uint32_t tS = tB + kHalf * buf;
      float x[kHalf];
      tmem_ld32(tS, x);
      tmem_ld32(tS + 32, x + 32);
      tmem_ld_wait();
      if (kind0 == 1) mask_range(x, lo - j0, hi - j0);
      if (kind1 == 1) mask_range(x + 32, lo - j0 - 32, hi - j0 - 32);
      uint32_t pk[kHalf / 2];
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int ch = 0; ch < 2; ++ch)
        if (ch ? kind1 : kind0)
#pragma unroll
          for (int k = 32 * ch; k < 32 * ch + 32; k += 8)
#pragma unroll
            for (int e = 0; e < 4; ++e) mx[e] = fmax3(mx[e], x[k + 2 * e], x[k + 2 * e + 1]);
      const float f = raise_to(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * kLogitScale2);
      const float nref = m_ref == -INFINITY ? 0.f : -m_ref;
      const uint64_t n2 = f2_pack(nref, nref);
      uint64_t s2a = f2_pack(0.f, 0.f), s2b = s2a;
      float sq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int ch = 0; ch < 2; ++ch) {
        if (ch ? kind1 : kind0) {
#pragma unroll
          for (int k = 32 * ch; k < 32 * ch + 32; k += 2) {
            float u, e;
            f2_unpack(f2_fma(f2_pack(x[k], x[k + 1]), c2, n2), u, e);
            u = ex2(u);
            e = ex2(e);
            const uint32_t q = pack_bf16x2(u, e);
            pk[k >> 1] = q;
            if (k & 2) s2b = f2_add(s2b, f2_pack(u, e));
            else s2a = f2_add(s2a, f2_pack(u, e));
            const int c = (k >> 1) & 1;
            sq[2 * c] = add_bf16_lo(sq[2 * c], q);
            sq[2 * c + 1] = add_bf16_hi(sq[2 * c + 1], q);
          }
        } else {
#pragma unroll
          for (int k = 16 * ch; k < 16 * ch + 16; ++k) pk[k] = 0u;
        }
      }
      float sa, sb, sc2, sd;
      f2_unpack(s2a, sa, sb);
      f2_unpack(s2b, sc2, sd);
      lsum += (sa + sb) + (sc2 + sd);
      osum += (sq[0] + sq[1]) + (sq[2] + sq[3]);
      if (it > 0) rescale(f);
      tmem_st16(tS, pk);
      tmem_st16(tS + 16, pk + 16);
      tmem_st_wait();
      hand_back();
    }
    // the global keys outside each row's band, and, with the row's LSE, the
    // far-row column sums of the global keys (one partial per warp, merged
    // later in a fixed order)
    float lse = INFINITY;
    if (glob) {
      wait_item();
      if (ok) {
        // four global keys at a time; x = -inf where the band reaches the key
        const uint32_t tS = tB + kHalf * buf;
        auto load4 = [&](int g0, float* x) {
          tmem_ld4(tS + g0, x);
          tmem_ld_wait();
#pragma unroll
          for (int k = 0; k < 4; ++k)
            x[k] = g0 + k < ng && abs(i - sm.gc[g0 + k]) > w ? x[k] * kLogitScale2 : -INFINITY;
        };
        float x[4], mx = -INFINITY;
#pragma unroll 1
        for (int g0 = 0; g0 < ng; g0 += 4) {
          load4(g0, x);
          mx = fmaxf(fmax3(mx, x[0], x[1]), fmaxf(x[2], x[3]));
        }
        rescale(raise_to(mx));
        const float nref = m_ref == -INFINITY ? 0.f : -m_ref;
#pragma unroll 1
        for (int g0 = 0; g0 < kMaxGlobal; g0 += 4) {
          uint32_t pk[2] = {0u, 0u};
          if (g0 < ng) {
            load4(g0, x);
#pragma unroll
            for (int k = 0; k < 4; k += 2) {
              const float a = ex2(x[k] + nref), c = ex2(x[k + 1] + nref);
              pk[k / 2] = pack_bf16x2(a, c);
              lsum += a + c;
              osum = add_bf16_hi(add_bf16_lo(osum, pk[k / 2]), pk[k / 2]);
            }
          }
          tmem_st2(tS + kColPG + g0 / 2, pk);
        }
        if (valid) lse = m_ref + lg2(lsum);
#pragma unroll 1
        for (int g0 = 0; g0 < ng; g0 += 4) {
          load4(g0, x);
#pragma unroll
          for (int k = 0; k < 4; ++k) x[k] = valid ? ex2(x[k] - lse) : 0.f;
          // two steps of a reduce-scatter, then plain sums: lane l holds key l >> 3
#pragma unroll
          for (int half = 2, bit = 16; half >= 1; half >>= 1, bit >>= 1)
#pragma unroll
            for (int k = 0; k < half; ++k) {
              const bool upper = (lane & bit) != 0;
              const float send = upper ? x[k] : x[k + half], mine = upper ? x[k + half] : x[k];
              x[k] = mine + __shfl_xor_sync(0xffffffffu, send, bit);
            }
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) x[0] += __shfl_xor_sync(0xffffffffu, x[0], o);
          if ((lane & 7) == 0 && g0 + (lane >> 3) < ng)
            p.gpart[(tile * 4 + warp) * kMaxGlobal + g0 + (lane >> 3)] = x[0];
        }
        tmem_st_wait();
        hand_back();
      }
    } else if (valid) {
      lse = m_ref + lg2(lsum);
    }
    const int last_pv = buf == 0 ? kBufs - 1 : buf - 1;   // P V of the row pass's last item
    const uint32_t last_pv_use = buf == 0 ? use - 1 : use;
    sm.nlse[r] = -lse;
    named_sync_softmax();                 // every -LSE of the tile is in shared memory

    // Band pass (the column sums of Sec. "Extractor of Attention Scores"):
    // for each key j of the band, the sum over this tile's rows i of
    // exp2(S_ij scaled - LSE_i); global rows (LSE = +inf) and rows past the
    // end add nothing.  One thread per key column of S^T; written per query
    // tile, summed over query tiles and heads in a fixed order by the scores
    // kernel.
    float* const part = p.colpart + ((static_cast<size_t>(b) * p.H + h) * p.band_slots +
                                     qt % p.band_slots) * p.L + r;
    bool o_out = false;
#pragma unroll 1
    for (int u = 0; ok && u < nk; ++u) {
      const int j0 = (klo + nk - 1 - u) * kTile, j = j0 + r, jw = j0 + 32 * warp;
      uint64_t a2a = f2_pack(0.f, 0.f), a2b = a2a;
#pragma unroll 1
      for (int qh = 0; qh < 2; ++qh) {
        if (!reaches(u, qh)) continue;
        const int i0 = q0 + kHalf * qh;
        // a warp's 32 keys against 32 queries: the relation is symmetric
        const int kind0 = chunk_kind(jw, i0, w, n), kind1 = chunk_kind(jw, i0 + 32, w, n);
        wait_item();
        if (!ok) break;
        const uint32_t tS = tB + kHalf * buf;
        float x[kHalf];
        tmem_ld32(tS, x);
        tmem_ld32(tS + 32, x + 32);
        tmem_ld_wait();
        hand_back();
        const float* lw = sm.nlse + kHalf * qh;
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          const int kind = ch ? kind1 : kind0;
          if (kind == 0) continue;
          // query columns of the chunk that are in j's band (and in the sequence)
          if (kind == 1)
            mask_range(x + 32 * ch, j - w - i0 - 32 * ch, min(j + w, n - 1) - i0 - 32 * ch);
#pragma unroll
          for (int k = 32 * ch; k < 32 * ch + 32; k += 4) {
            const float4 l4 = *reinterpret_cast<const float4*>(lw + k);
            float e0, e1, e2, e3;
            f2_unpack(f2_fma(f2_pack(x[k], x[k + 1]), c2, f2_pack(l4.x, l4.y)), e0, e1);
            f2_unpack(f2_fma(f2_pack(x[k + 2], x[k + 3]), c2, f2_pack(l4.z, l4.w)), e2, e3);
            a2a = f2_add(a2a, f2_pack(ex2(e0), ex2(e1)));
            a2b = f2_add(a2b, f2_pack(ex2(e2), ex2(e3)));
          }
        }
      }
      float sa, sb, sc2, sd;
      f2_unpack(a2a, sa, sb);
      f2_unpack(a2b, sc2, sd);
      if (ok && j < n) part[j0] = (sa + sc2) + (sb + sd);
      if (!o_out) {
        // ---- O: its rows leave through the last tile's V slot
        o_out = true;
        ok = ok && warp_wait_poll(&sm.bar_pv[last_pv], last_pv_use & 1, abort_flag);
        tc_fence_after();
        if (ok && v.O != nullptr) {
          const float inv = 1.f / osum;
          uint8_t* stage = Slots + vd_slot * kTileBytes + warp * 4096;
#pragma unroll 1
          for (int c = 0; c < 64; c += 8) {
            float o[8];
            tmem_ld8(tO + c, o);
            tmem_ld_wait();
            stage_row_piece<8>(stage, c >> 3,
                               make_uint4(pack_bf16x2(o[0] * inv, o[1] * inv),
                                          pack_bf16x2(o[2] * inv, o[3] * inv),
                                          pack_bf16x2(o[4] * inv, o[5] * inv),
                                          pack_bf16x2(o[6] * inv, o[7] * inv)));
          }
          __syncwarp();
          // four rows an instruction, eight lanes a row
          const uint32_t rows = __ballot_sync(0xffffffffu, valid) >> (lane >> 3);
          uint16_t* dst = v.O + ((static_cast<size_t>(b) * p.L + iw + (lane >> 3)) * p.H + h) *
                                    kHeadDim + 8 * (lane & 7);
#pragma unroll 2
          for (int k = 0; k < 32; k += 4, dst += static_cast<size_t>(4) * p.H * kHeadDim) {
            const uint4 val = *reinterpret_cast<const uint4*>(
                stage + stage_offset<8>(k + (lane >> 3), lane & 7));
            if ((rows >> k) & 1u) *reinterpret_cast<uint4*>(dst) = val;
          }
        }
        fence_proxy_async_smem();         // ... before the copy of V into it
        tc_fence_before();
        warp_arrive(&sm.bar_stage);
      }
      if (glob && u == u_d) {             // S_Gt of the tile's keys, for warps 6 and 7
        wait_item();
        if (!ok) break;
        const uint32_t tS = tB + kHalf * buf;
#pragma unroll 1
        for (int g0 = 0; g0 < ng; g0 += 4) {
          float y[4];
          tmem_ld4(tS + g0, y);
          tmem_ld_wait();
#pragma unroll
          for (int k = 0; k < 4; ++k)   // key i
            gx[(g0 + k) * kTile + r] = i < n ? y[k] * kLogitScale2 : -INFINITY;
        }
        hand_back();
        tc_fence_before();
        warp_arrive(&sm.bar_gx);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 4) {
    tc_fence_after();
    tmem_dealloc(tm, 256);
  }
  if (tid == 0) {
    if (sm.abort) atomicOr(p.status, kStatusTimeout);
    // O, the partial sums and statistics of this CTA (ordered before this by
    // the barrier) are visible to the scores CTAs that see the count
    red_release_add_u32(p.rows_done + b * p.H, 1u);
  }
}

// ---------------------------------------------------------------------------
// cols kernel
// ---------------------------------------------------------------------------
// One CTA per pair of 128-key tiles (2p, 2p+1) of one (sequence, head), one
// warpgroup per key tile.  The band rows' column sums come from the rows
// kernel (one partial per query tile); here: the global rows' P over the
// pair's keys and their P V, the keys' column sums, and the finalisation.
// Tensor memory (256 columns, so that two CTAs share an SM) per warpgroup X:
// S^T against the global queries [16 X, +16), the global rows' P V
// [64 + 64 X, +64).
constexpr int kColsThreads = 320;
struct ColsSmem {
  uint64_t bar_kv;
  uint64_t bar_sfull[2], bar_sfree[2], bar_sg[2], bar_pg[2], bar_og[2], bar_fin;
  uint32_t tmem_base;
  int abort;
  int gc[kMaxGlobal];
  float lse_g[kMaxGlobal];
  int flag, flag2;
  FinalSmem<kColsThreads> fin;
  // each key tile's part of the global rows' P V (warpgroup X), added in
  // tile order into the pair's part
  alignas(16) float ogx[2][kMaxGlobal][kHeadDim];   // read and written as float4
};

// dynamic shared memory: the global rows' P blocks (2 per warpgroup), K and V
// of both key tiles, the global queries
constexpr uint32_t kColsDyn = 4 * kPgBlock + kTileBytes * 4 + kGTileBytes + 1024;
static_assert(3 * kPgBlock + kTileBytes <= 4 * kPgBlock + 4 * kTileBytes,
              "the A operand's unused rows stay inside the shared memory");

__global__ void __launch_bounds__(kColsThreads, 2)
    sc_cols_kernel(const __grid_constant__ TensorMaps maps, const __grid_constant__ LayerParams p) {
  // No grid-wide wait on the rows kernel: this kernel is scheduled only after
  // every rows CTA has passed its own wait (so the earlier kernels' results
  // are complete), and each CTA waits below for the rows CTAs of its own
  // (sequence, head) only, so that it can run beside the rows kernel's last CTAs.
  pdl_launch_dependents();
  const int T2 = (p.T + 1) / 2;
  const int pr = blockIdx.x % T2, bh = blockIdx.x / T2;
  const int h = bh % p.H, b = bh / p.H;
  const LayerView v = layer_view(p);
  if (owned_by_tail(p, v, b)) return;
  const int n = __ldcg(v.len + b);
  if (n == 0) {
    if (pr == 0 && h == 0 && threadIdx.x == 0) {
      v.len_out[b] = 0;
      v.ng_out[b] = 0;
      v.ident_out[b] = 1;
    }
    return;
  }
  if (2 * pr * kTile >= n) return;
  const int ng = min(__ldcg(v.ng + b), kMaxGlobal);
  const int ngp = ng > 0 ? kMaxGlobal : 0;
  const int Tn = (n + kTile - 1) / kTile;
  const int Tp = (Tn + 1) / 2;
  const bool hasB = (2 * pr + 1) * kTile < n;

  extern __shared__ uint8_t dyn_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dyn_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* Pg = base;                              // 2 x 2 blocks of 16 rows
  uint8_t* Ks = Pg + 4 * kPgBlock;                 // 2 tiles
  uint8_t* Vs = Ks + 2 * kTileBytes;               // 2 tiles
  uint8_t* QG = Vs + 2 * kTileBytes;
  __shared__ ColsSmem sm;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int qlo[2], qhi[2];
#pragma unroll
  for (int X = 0; X < 2; ++X) {
    const int j0 = (2 * pr + X) * kTile, j1 = min(j0 + kTile - 1, n - 1);
    qlo[X] = max(0, j0 - p.w) / kTile;
    qhi[X] = min(n - 1, j1 + p.w) / kTile;
  }

  if (tid == 0) {
    mbar_init(&sm.bar_kv, 1);
    for (int X = 0; X < 2; ++X) {
      mbar_init(&sm.bar_sfull[X], 1);
      mbar_init(&sm.bar_sfree[X], 4);   // one arrival per warp
      mbar_init(&sm.bar_sg[X], 1);
      mbar_init(&sm.bar_pg[X], 4);
      mbar_init(&sm.bar_og[X], 1);
    }
    mbar_init(&sm.bar_fin, 1);
    sm.abort = 0;
    fence_mbar_init();
  }
  if (tid < kMaxGlobal) sm.gc[tid] = tid < ng ? __ldcg(v.gcur + b * kMaxGlobal + tid) : -1;
  if (warp == 9) tmem_alloc(&sm.tmem_base, 256);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = sm.tmem_base;
  volatile int* abort_flag = &sm.abort;

  if (warp == 8) {
    const RowSource rs = row_source(p, v, b);
    // this sequence's rows may still be crossing the host link
    if (p.gathered != nullptr) {
      if (lane == 0) wait_count(p.gathered + b, p.gather_target, abort_flag);
      __syncwarp();
      fence_proxy_async_global();
    }
    if (lane == 0) {
      mbar_arrive_expect_tx(&sm.bar_kv, (hasB ? 4 : 2) * kTileBytes + ngp * 128);
      for (int X = 0; X < (hasB ? 2 : 1); ++X) {
        load_tile(maps, 1, rs, h, (2 * pr + X) * kTile, Ks + X * kTileBytes, &sm.bar_kv);
        load_tile(maps, 2, rs, h, (2 * pr + X) * kTile, Vs + X * kTileBytes, &sm.bar_kv);
      }
    }
    __syncwarp();
    if (ngp) load_globals(maps, 0, rs, h, p.H, sm.gc, ng, QG, &sm.bar_kv, lane);
    if (lane == 0) drain_wait(&sm.bar_kv, 0);
  } else if (warp == 9) {
    if (lane == 0) {
      const uint32_t k_a = smem_u32(Ks), v_a = smem_u32(Vs);
      const int nX = hasB ? 2 : 1;
      bool ok = mbar_wait(&sm.bar_kv, 0, abort_flag);
      if (ok) {
        tc_fence_after();
        if (ngp)
          for (int X = 0; X < nX; ++X) {
            mma_qk(tm + 16 * X, k_a + X * kTileBytes, smem_u32(QG), 16);
            umma_commit(&sm.bar_sg[X]);
          }
      }
      if (ok && ngp)
        for (int X = 0; ok && X < nX; ++X) {
          if (!(ok = mbar_wait(&sm.bar_pg[X], 0, abort_flag))) break;
          int steps = kTile / 16;
          const int left = n - (2 * pr + X) * kTile;   // the tile's keys before the end
          if (left < kTile) {
            steps = (left + 15) / 16;
            zero_rows(Vs + X * kTileBytes, left, 16 * steps, 0, 1);
          }
          tc_fence_after();
          mma_pv(tm + 64 + 64 * X, smem_u32(Pg) + X * 2 * kPgBlock, kPgBlock, v_a + X * kTileBytes,
                 steps, false);
          umma_commit(&sm.bar_og[X]);
        }
      umma_commit(&sm.bar_fin);
      drain_wait(&sm.bar_fin, 0);
    }
    __syncwarp();
  } else {
    const int X = warp >> 2, wq = warp & 3;
    const int qloX = X ? qlo[1] : qlo[0], qhiX = X ? qhi[1] : qhi[0];
    const int r = tid & 127;
    const int kt = 2 * pr + X;
    const int j0 = kt * kTile;
    const int j = j0 + r;             // key column owned by this thread
    const bool active = X == 0 || hasB;
    const uint32_t lane_off = static_cast<uint32_t>(wq * 32) << 16;
    const uint32_t tSG = tm + 16 * X, tOG = tm + 64 + 64 * X;
    // the rows CTAs of this (sequence, head) have finished (their partial
    // sums, statistics and the cleared global-row outputs are read below)
    if (tid == 0)
      wait_count(p.rows_done + b * p.H + h,
                 static_cast<uint32_t>(Tn), abort_flag);
    asm volatile("bar.sync 3, 256;" ::: "memory");
    // every load of the prologue is issued before any is used: this key's
    // band-row column sums of the query tiles of its band (one per tile, from
    // the rows kernel) and, per warp, the (max, sum) pieces of global rows
    // warp and warp + 8
    float part[kMaxBandTiles];   // (slot = query tile mod kMaxBandTiles)
    const float* cp = p.colpart + ((static_cast<size_t>(b) * p.H + h) * p.L + j) * kMaxBandTiles;
#pragma unroll
    for (int u = 0; u < kMaxBandTiles; ++u)
      part[u] = (active && j < n && qloX + u <= qhiX) ? __ldcg(cp + (qloX + u) % kMaxBandTiles) : 0.f;
    // lane k takes entries k, k+32, k+64, k+96 of the 4 Tn (key tile, warp
    // slice) pieces; the warp combines them in a fixed order
    const size_t base_slot = (static_cast<size_t>(b) * p.H + h) * p.T * 4 * kMaxGlobal;
    float me[2][4], se[2][4];
    // the far-row sums (rows whose band does not reach the key) of a global
    // key among this warp's 32 keys, over the (query tile, warp slice) pieces
    // of this head: lane k loads pieces k, k+32, k+64, k+96 (at most one
    // global key per warp is usual; more are summed one after another below)
    const int wk0 = j0 + 32 * wq;
    float far[4] = {0.f, 0.f, 0.f, 0.f};
    int far_g = -1;
    if (active && ngp) {
#pragma unroll 1
      for (int g = 0; g < ng; ++g)
        if (sm.gc[g] >= wk0 && sm.gc[g] < wk0 + 32) {
          far_g = g;
          break;
        }
      if (far_g >= 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int ent = lane + 32 * k;
          far[k] = ent < 4 * Tn ? __ldcg(p.gpart + base_slot + ent * kMaxGlobal + far_g) : 0.f;
        }
      }
    }
#pragma unroll
    for (int gg = 0; gg < 2; ++gg) {
      const int g = warp + 8 * gg;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int ent = lane + 32 * k;
        const bool use = ngp && g < ng && ent < 4 * Tn;
        me[gg][k] = use ? __ldcg(p.gstat + 2 * (base_slot + ent * kMaxGlobal + g)) : -INFINITY;
        se[gg][k] = use ? __ldcg(p.gstat + 2 * (base_slot + ent * kMaxGlobal + g) + 1) : 0.f;
      }
    }
#pragma unroll
    for (int gg = 0; gg < 2; ++gg) {
      const int g = warp + 8 * gg;
      if (!ngp || g >= ng) continue;   // warp-uniform
      const float m = fmaxf(fmaxf(me[gg][0], me[gg][1]), fmaxf(me[gg][2], me[gg][3]));
      float sacc = 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        sacc += (me[gg][k] == -INFINITY) ? 0.f : se[gg][k] * ex2(me[gg][k] - m);
      const float M = warp_max(m);
      const float S = warp_sum(m == -INFINITY ? 0.f : sacc * ex2(m - M));
      if (lane == 0) sm.lse_g[g] = M + lg2(S);
    }
    asm volatile("bar.sync 3, 256;" ::: "memory");

    // band rows: the query tiles' sums in tile order
    float acc = 0.f;
#pragma unroll
    for (int u = 0; u < kMaxBandTiles; ++u) acc += part[u];
    // far rows of the global keys among this warp's keys (gc increases with
    // g, so they are consecutive entries of the list)
    if (far_g >= 0) {
#pragma unroll 1
      for (int g = far_g; g < ng; ++g) {
        const int cg = sm.gc[g];
        if (cg >= wk0 + 32) break;
        if (g != far_g) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int ent = lane + 32 * k;
            far[k] = ent < 4 * Tn ? __ldcg(p.gpart + base_slot + ent * kMaxGlobal + g) : 0.f;
          }
        }
        const float fs = warp_sum((far[0] + far[1]) + (far[2] + far[3]));
        if (j == cg) acc += fs;
      }
    }
    const bool ok = active;
    float x[16];

    if (active && ngp) {
      bool ok2 = ok && warp_wait(&sm.bar_sg[X], 0, abort_flag);
      if (ok2) {
        tc_fence_after();
        tmem_ld16(tSG + lane_off, x);
        tmem_ld_wait();
      }
      uint16_t pb[kMaxGlobal];
      float s = 0.f;
#pragma unroll
      for (int g = 0; g < kMaxGlobal; ++g) {
        const float v =
            (ok2 && g < ng && j < n) ? ex2(fmaf(x[g], kLogitScale2, -sm.lse_g[g])) : 0.f;
        s += v;
        pb[g] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
      }
      acc += s;
      // P of the global rows, transposed into this warpgroup's A tile: row g,
      // column (key) r
      uint8_t* col = Pg + X * 2 * kPgBlock + (r >> 6) * kPgBlock;
      const int ch = (r & 63) >> 3, wi = (r & 7) * 2;
#pragma unroll
      for (int g = 0; g < kMaxGlobal; ++g)
        *reinterpret_cast<uint16_t*>(col + sw128_offset(g, ch) + wi) = pb[g];
      fence_proxy_async_smem();
      tc_fence_before();
      warp_arrive(&sm.bar_pg[X]);
      bool ok3 = ok2 && warp_wait(&sm.bar_og[X], 0, abort_flag);
      if (wq == 0) {
        // this key tile's part of the global rows' outputs (TMEM lane g = global g)
        if (ok3) tc_fence_after();
        float* mine = &sm.ogx[X][lane & (kMaxGlobal - 1)][0];
#pragma unroll 1
        for (int c = 0; c < 64; c += 16) {
          float o[16];
          if (ok3) {
            tmem_ld16(tOG + lane_off + c, o);
            tmem_ld_wait();
          } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) o[k] = 0.f;
          }
          if (lane < kMaxGlobal)
#pragma unroll
            for (int k = 0; k < 16; k += 4)
              *reinterpret_cast<float4*>(mine + c + k) = make_float4(o[k], o[k + 1], o[k + 2], o[k + 3]);
        }
        // warps 0 and 4 (the first warp of each warpgroup) meet here when the
        // pair has two key tiles; warp 0 adds the parts in tile order and
        // stores the pair's part (plain stores: no order-dependent atomics)
        if (hasB) asm volatile("bar.sync 5, 64;" ::: "memory");
        else __syncwarp();
        if (X == 0) {
          float* part = p.og + (((static_cast<size_t>(b) * p.H + h) * T2 + pr) * kMaxGlobal) *
                                   kHeadDim;
          for (int k = lane; k < ng * (kHeadDim / 4); k += 32) {
            const int g = k / (kHeadDim / 4), d = 4 * (k % (kHeadDim / 4));
            float4 a4 = *reinterpret_cast<const float4*>(&sm.ogx[0][g][d]);
            if (hasB) {
              const float4 b4 = *reinterpret_cast<const float4*>(&sm.ogx[1][g][d]);
              a4.x += b4.x; a4.y += b4.y; a4.z += b4.z; a4.w += b4.w;
            }
            *reinterpret_cast<float4*>(part + g * kHeadDim + d) = a4;
          }
        }
      }
    }
    if (active && j < n) p.acc[(static_cast<size_t>(b) * p.H + h) * p.L + j] = acc;
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tm, 256);
  }
  if (tid == 0 && sm.abort) atomicOr(p.status, kStatusTimeout);

  // One hand-over for both roles below: this CTA's part of the global rows'
  // outputs and its column sums are visible before either counter is raised.
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    sm.flag = ngp && atomicAdd(p.cols_done + b * p.H + h, 1u) == static_cast<uint32_t>(Tp - 1);
    sm.flag2 = atomicAdd(p.cnt_tile + b * p.T + pr, 1u) == static_cast<uint32_t>(p.H - 1);
  }
  __syncthreads();

  // ---- last pair of this (sequence, head): the global rows' outputs, the
  // pairs' parts added in pair order
  if (ngp) {
    if (sm.flag) {
      __threadfence();
      const float* part0 =
          p.og + (static_cast<size_t>(b) * p.H + h) * T2 * kMaxGlobal * kHeadDim;
      for (int k = tid; k < ng * (kHeadDim / 4); k += kColsThreads) {
        const int g = k / (kHeadDim / 4), d = 4 * (k % (kHeadDim / 4));
        constexpr int kBatch = 8;   // loads in flight before they are added
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q0 = 0; q0 < Tp; q0 += kBatch) {
          float4 x[kBatch];
#pragma unroll
          for (int u = 0; u < kBatch; ++u)
            x[u] = q0 + u < Tp ? __ldcg(reinterpret_cast<const float4*>(
                                     part0 + ((q0 + u) * kMaxGlobal + g) * kHeadDim + d))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int u = 0; u < kBatch; ++u) {
            acc.x += x[u].x; acc.y += x[u].y; acc.z += x[u].z; acc.w += x[u].w;
          }
        }
        if (v.O != nullptr)
          *reinterpret_cast<uint2*>(v.O + ((static_cast<size_t>(b) * p.L + sm.gc[g]) * p.H + h) *
                                              kHeadDim + d) =
              make_uint2(pack_bf16x2(acc.x, acc.y), pack_bf16x2(acc.z, acc.w));
      }
      if (tid == 0) p.cols_done[b * p.H + h] = 0u;
    }
  }

  // ---- last head of this pair of key tiles: scores and keep flags (fixed head order)
  if (!sm.flag2) return;
  __threadfence();
  const int j0 = 2 * pr * kTile;
  const int jn = min(n, j0 + 2 * kTile);
  // this thread's key column: every head's column sum, loaded first (in
  // flight while the global keys' partial sums are reduced below)
  const int jj = j0 + tid;
  const bool my_key = tid < 2 * kTile && jj < jn;
  float hs[kTailMaxHeads];
  float a = 0.f;
  const float* ap = p.acc + static_cast<size_t>(b) * p.H * p.L + jj;
#pragma unroll
  for (int u = 0; u < kTailMaxHeads; ++u)
    hs[u] = my_key && u < p.H ? __ldcg(ap + static_cast<size_t>(u) * p.L) : 0.f;
  for (int h0 = kTailMaxHeads; my_key && h0 < p.H; ++h0)   // more than 16 heads
    a += __ldcg(ap + static_cast<size_t>(h0) * p.L);
  if (my_key) {
    float hsum = 0.f;
#pragma unroll
    for (int u = 0; u < kTailMaxHeads; ++u) hsum += hs[u];   // heads in order
    a = hsum + a;
    const float s = a / static_cast<float>(p.H * n);
    v.scores[static_cast<size_t>(b) * p.L + jj] = s;
    if (p.keep_rule != kKeepTopRatio) {   // the top-ratio cut needs every score first
      const float theta = p.theta ? __ldg(p.theta + b)
                          : p.keep_rule == kKeepAbsolute ? v.alpha
                                                         : v.alpha / static_cast<float>(n);
      p.keep[static_cast<size_t>(b) * p.L + jj] = (jj == 0 || s >= theta) ? 1 : 0;
    }
  }
  if (tid == 0) p.cnt_tile[b * p.T + pr] = 0u;
  __threadfence();
  __syncthreads();
  if (tid == 0) sm.flag = (atomicAdd(p.cnt_seq + b, 1u) == static_cast<uint32_t>(Tp - 1));
  __syncthreads();
  if (!sm.flag) return;
  __threadfence();
  finalize_sequence<kColsThreads>(p, v, b, n, ng, sm.fin, sm.gc, base);
}

// ---------------------------------------------------------------------------
// gather kernel: the next layer's Q, K, V rows of the kept tokens, compacted
// ---------------------------------------------------------------------------
constexpr int kGatherTokens = 8;
constexpr int kGatherThreads = 256;

// One item: tokens 8 ch .. 8 ch + 7 of sequence b, 3 tensors; with H = 12 each
// thread moves at most nine 16-byte vectors, all loads issued before any store.
__device__ __forceinline__ void gather_item(const GatherParams& g, int b, int ch, int layer,
                                            long long src_base, const int32_t* lenp,
                                            const int32_t* posp, const int32_t* identp) {
  if (g.tail_from != nullptr && __ldcg(g.tail_from + b) <= layer) return;
  const int n = __ldcg(lenp + b);
  const int c0 = ch * kGatherTokens;
  if (__ldcg(identp + b) != 0 || c0 >= n) return;
  const int cnt = min(kGatherTokens, n - c0);
  const int vec = g.H * kHeadDim / 8;  // 16-byte vectors per token row
  const int total = cnt * vec;
  const long long dst_tok0 = static_cast<long long>(b) * g.L + c0;
  const long long src_tok0 = src_base + static_cast<long long>(b) * g.L;
  constexpr int kPer = 4;   // vectors per thread and tensor per round
  for (int k0 = threadIdx.x; k0 < total; k0 += kGatherThreads * kPer) {
    uint4 v[3][kPer];
    long long so[kPer], doff[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int k = k0 + u * kGatherThreads;
      const int tk = k / vec, e = k - tk * vec;
      so[u] = k < total ? (src_tok0 + __ldcg(posp + static_cast<size_t>(b) * g.L + c0 + tk)) * vec + e
                        : -1;
      doff[u] = (dst_tok0 + tk) * vec + e;
    }
#pragma unroll
    for (int t = 0; t < 3; ++t)
#pragma unroll
      for (int u = 0; u < kPer; ++u)
        if (so[u] >= 0) v[t][u] = __ldg(reinterpret_cast<const uint4*>(g.src[t]) + so[u]);
#pragma unroll
    for (int t = 0; t < 3; ++t)
#pragma unroll
      for (int u = 0; u < kPer; ++u)
        if (so[u] >= 0) reinterpret_cast<uint4*>(g.dst[t])[doff[u]] = v[t][u];
  }
}

// The per-layer gather: one CTA per item (grid: chunks x sequences).
__global__ void __launch_bounds__(kGatherThreads)
    sc_gather_kernel(const GatherParams g) {
  pdl_launch_dependents();
  pdl_wait();
  int layer = g.layer;
  long long src_base = g.src_base;
  const int32_t* lenp = g.len;
  const int32_t* posp = g.pos;
  const int32_t* identp = g.ident;
  if (g.dev_layer != nullptr) {
    layer = __ldcg(g.dev_layer) + 1;
    if (layer >= g.n_layers) return;
    src_base = layer * g.tok_stride;
    lenp += static_cast<size_t>(layer) * g.len_stride;
    posp += layer * g.row_stride;
    identp = g.ident_slot[layer & 1];
  }
  gather_item(g, blockIdx.y, blockIdx.x, layer, src_base, lenp, posp, identp);
}

// The gather with per-sequence counts (g.gathered): a grid-stride walk over
// the items sequence by sequence; gathered[b] is raised (release) once an item
// of sequence b is copied.  Its successor is launched once every CTA has
// passed the grid wait, so what the kernels before this one wrote is complete
// by then.  Used for the layer (given explicitly) whose rows cross the host link.
__global__ void __launch_bounds__(kGatherThreads)
    sc_gather_seq_kernel(const GatherParams g) {
  pdl_wait();
  pdl_launch_dependents();
  const int nch = (g.L + kGatherTokens - 1) / kGatherTokens;
  for (int it = blockIdx.x; it < g.B * nch; it += gridDim.x) {
    const int b = it / nch;
    gather_item(g, b, it - b * nch, g.layer, g.src_base, g.len, g.pos, g.ident);
    __syncthreads();   // every copy of the item is stored ...
    if (threadIdx.x == 0) {
      __threadfence();
      red_release_add_u32(g.gathered + b, 1u);   // ... before it is counted
    }
  }
}

// ---------------------------------------------------------------------------
// export kernel: a stack's results to page-locked host memory
// ---------------------------------------------------------------------------
constexpr int kExportTokens = 32;
constexpr int kExportThreads = 256;

// Work items of 32 current slots of one (layer, sequence), walked by a
// grid-stride loop; only the slots below the layer's length are copied.  Loads
// from device memory are issued in groups of four before the stores, which
// cross the host link.
__global__ void __launch_bounds__(kExportThreads)
    sc_export_kernel(const ExportParams e) {
  // part 1 runs beside the cluster kernel, which lets it start once every one
  // of its CTAs has passed its own grid wait: what part 1 reads is complete
  if (e.part != 1) pdl_wait();
  const int nch = (e.L + kExportTokens - 1) / kExportTokens;
  const int items = (e.n_layers + 1) * e.B * nch;
  const int vec = e.H * kHeadDim / 8;   // 16-byte vectors per row
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const int ch = it % nch, lb = it / nch;
    const int b = lb % e.B, l = lb / e.B;
    if (e.part != 0) {
      // a sequence that first gets short after the last layer has no layer in the
      // cluster kernel: its last slot is the per-layer kernels' too
      const int from = __ldcg(e.tail_from + b);
      if ((e.part == 1) != (l < from || from >= e.n_layers)) continue;
    }
    const size_t li = static_cast<size_t>(l) * e.B + b;
    const int n = __ldcg(e.len + li);
    if (ch == 0 && threadIdx.x == 0) e.hlen[li] = n;
    const int c0 = ch * kExportTokens;
    if (c0 >= n) continue;
    const int cnt = min(kExportTokens, n - c0);
    const size_t row0 = li * e.L + c0;
    if (threadIdx.x < cnt) {
      e.hpos[row0 + threadIdx.x] = __ldcg(e.pos + row0 + threadIdx.x);
      if (l < e.n_layers) e.hscores[row0 + threadIdx.x] = __ldcg(e.scores + row0 + threadIdx.x);
    }
    if (l >= e.n_layers) continue;
    uint4* dst;
    if (e.hO != nullptr) dst = reinterpret_cast<uint4*>(e.hO) + row0 * vec;
    else if (l == e.n_layers - 1 && e.hO_last != nullptr)
      dst = reinterpret_cast<uint4*>(e.hO_last) + (static_cast<size_t>(b) * e.L + c0) * vec;
    else continue;
    const int total = cnt * vec;
    const uint4* src = reinterpret_cast<const uint4*>(e.O) + row0 * vec;
    constexpr int kPer = 4;
    for (int k0 = threadIdx.x; k0 < total; k0 += kExportThreads * kPer) {
      uint4 v[kPer];
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int k = k0 + u * kExportThreads;
        if (k < total) v[u] = __ldcg(src + k);
      }
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int k = k0 + u * kExportThreads;
        if (k < total) dst[k] = v[u];
      }
    }
  }
  // part 1 completes only after the cluster kernel (which writes its own
  // layers' results to the host buffers), so that the call's last kernel
  // ends after every result is written
  if (e.part == 1) pdl_wait();
}

// ---------------------------------------------------------------------------
// prep kernel: padding removal (stack) or global-token lookup (single layer)
// ---------------------------------------------------------------------------
constexpr int kPrepThreads = 1024;

__global__ void __launch_bounds__(kPrepThreads)
    sc_prep_kernel(const PrepParams pp) {
  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ int wsum[kPrepThreads / 32];
  __shared__ int spos[kMaxLen];
  __shared__ int gfound[kMaxGlobal];
  __shared__ int s_n;
  if (pp.pos_in == nullptr) {
    const int L = pp.L;
    int32_t* out = pp.pos_out + static_cast<size_t>(b) * L;
    if (pp.pad_mask == nullptr) {
      // no padding: the current tokens are positions 0..L-1
      for (int c = tid; c < L; c += kPrepThreads) {
        out[c] = c;
        spos[c] = c;
      }
      if (tid == 0) {
        s_n = L;
        pp.len_out[b] = L;
      }
    } else {
      // stack mode with padding: the real tokens in order; thread tid takes
      // one contiguous run, runs are placed by a scan of their counts
      const uint8_t* mask = pp.pad_mask + static_cast<size_t>(b) * L;
      const int per = (L + kPrepThreads - 1) / kPrepThreads;
      const int c0 = min(L, tid * per), c1 = min(L, c0 + per);
      int cnt = 0;
      for (int c = c0; c < c1; ++c) cnt += mask[c] != 0;
      int x = cnt;   // inclusive scan within the warp
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
      }
      if (lane == 31) wsum[warp] = x;
      __syncthreads();
      if (warp == 0) {
        int w = wsum[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, w, off);
          if (lane >= off) w += y;
        }
        wsum[lane] = w;
      }
      __syncthreads();
      int at = (warp > 0 ? wsum[warp - 1] : 0) + x - cnt;
      for (int c = c0; c < c1; ++c) {
        if (!mask[c]) continue;
        out[at] = c;
        spos[at] = c;
        ++at;
      }
      if (tid == 0) {
        s_n = wsum[kPrepThreads / 32 - 1];
        pp.len_out[b] = s_n;
      }
    }
  } else {
    if (tid == 0) s_n = pp.len_in[b];
    __syncthreads();
    for (int c = tid; c < s_n; c += kPrepThreads)
      spos[c] = pp.pos_in[static_cast<size_t>(b) * pp.L + c];
  }
  __syncthreads();
  const int n = s_n;
  // current index of each global position (one thread each; binary search:
  // positions increase with the current index)
  if (tid < kMaxGlobal) {
    int found = -1;
    if (tid < pp.n_global) {
      const int target = pp.global_pos[tid];
      int lo = 0, hi = n - 1;
      while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        if (spos[mid] < target) lo = mid + 1;
        else hi = mid - 1;
      }
      if (lo < n && spos[lo] == target) found = lo;
    }
    gfound[tid] = found;
  }
  __syncthreads();
  if (tid == 0) {
    // global positions are sorted, so the matches come out in increasing order
    int m = 0;
    for (int g = 0; g < kMaxGlobal; ++g)
      if (gfound[g] >= 0) pp.gcur[b * kMaxGlobal + m++] = gfound[g];
    pp.ng[b] = m;
    // single-layer calls read their (already current-order) inputs in place
    pp.ident[b] = (!pp.no_ident && (pp.pos_in != nullptr || n == 0 || spos[n - 1] == n - 1))
                      ? 1 : 0;
    if (pp.tail_from != nullptr) pp.tail_from[b] = n <= pp.tail_max ? 0 : 0x7fffffff;
    if (pp.has_cond && n > pp.tail_max) cudaGraphSetConditional(pp.cond, 1u);
    if (pp.dev_layer != nullptr && b == 0) *pp.dev_layer = 0;
  }
}

// ---------------------------------------------------------------------------
// advance kernel: one step of the device-driven layer loop
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) sc_advance_kernel(const AdvanceParams a) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ int s_layer;
  if (threadIdx.x == 0) s_layer = a.dev_layer != nullptr ? __ldcg(a.dev_layer) + 1 : a.layer;
  __syncthreads();
  const int l = s_layer;
  int big = 0;
  for (int b = threadIdx.x; b < a.B; b += blockDim.x) big |= __ldcg(a.tail_from + b) > l;
  big = __syncthreads_or(big);
  if (threadIdx.x == 0) {
    if (a.dev_layer != nullptr) *a.dev_layer = l;
    cudaGraphSetConditional(a.cond, (big && l < a.n_layers) ? 1u : 0u);
  }
}

}  // namespace sc

// ---------------------------------------------------------------------------
// launch helpers used by the C ABI
// ---------------------------------------------------------------------------
namespace sc {

// Every kernel of the chain is launched with programmatic stream serialisation:
// it may be scheduled while its predecessor finishes and waits for it on the
// device (pdl_wait) before touching global memory.
template <typename... KArgs, typename... Args>
static cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t st, Args&&... args) {
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
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

cudaError_t launch_prep(const PrepParams& pp, cudaStream_t st) {
  return launch_chained(sc_prep_kernel, dim3(pp.B), dim3(kPrepThreads), 0, st, pp);
}

cudaError_t configure_band();

cudaError_t configure_kernels() {
  // the attention kernels use most of an SM's shared memory
  cudaError_t e = configure_band();
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(sc_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kRowsDyn));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(sc_rows_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(sc_cols_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kColsDyn));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(sc_cols_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  return e;
}

cudaError_t launch_band(const TensorMaps& m, const LayerParams& p, int sms, cudaStream_t st);

cudaError_t launch_rows(const TensorMaps& m, const LayerParams& p, cudaStream_t st) {
  if (p.band) return launch_band(m, p, p.sms, st);
  return launch_chained(sc_rows_kernel, dim3(p.B * p.H * p.T), dim3(kRowsThreads), kRowsDyn, st, m,
                        p);
}

cudaError_t launch_scores(const LayerParams& p, cudaStream_t st);

cudaError_t launch_cols(const TensorMaps& m, const LayerParams& p, cudaStream_t st) {
  if (!p.band) return launch_scores(p, st);
  dim3 grid(p.B * p.H * ((p.T + 1) / 2));
  return launch_chained(sc_cols_kernel, grid, dim3(kColsThreads), kColsDyn, st, m, p);
}

cudaError_t launch_advance(const AdvanceParams& a, cudaStream_t st) {
  return launch_chained(sc_advance_kernel, dim3(1), dim3(256), 0, st, a);
}

cudaError_t launch_export(const ExportParams& e, int ctas, cudaStream_t st) {
  const int items = (e.n_layers + 1) * e.B * ((e.L + kExportTokens - 1) / kExportTokens);
  return launch_chained(sc_export_kernel, dim3(std::max(1, std::min(items, ctas))),
                        dim3(kExportThreads), 0, st, e);
}

cudaError_t launch_gather(const GatherParams& g, cudaStream_t st) {
  const int nch = (g.L + kGatherTokens - 1) / kGatherTokens;
  if (g.gathered != nullptr) {
    // enough CTAs to keep the host link busy (about 2 MB in flight), few
    // enough that the items complete nearly in order, so that the first
    // sequences are in well before the last (measured on config 4 end to end:
    // 608 CTAs 0.489 ms, 152 0.484, 96 0.468, 64 0.469, 32 0.472)
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int items = g.B * nch;
    return launch_chained(sc_gather_seq_kernel,
                          dim3(std::max(1, std::min(items, std::max(32, sms / 2)))),
                          dim3(kGatherThreads), 0, st, g);
  }
  dim3 grid(nch, g.B);
  return launch_chained(sc_gather_kernel, grid, dim3(kGatherThreads), 0, st, g);
}

}  // namespace sc
