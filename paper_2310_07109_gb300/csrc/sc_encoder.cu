// sc_encoder.cu -- device code of the encoder layer around the sparse
// attention: the projections and the feed-forward block as tcgen05 GEMMs with
// a row gather on the A operand, and the post-layer norms.
//
// RoBERTa-style post-LN layer (the encoder SparseCoder prunes, Fig.
// "sparsecoder"), hidden size D = 64 H, on the n current tokens of a sequence:
//   Q, K, V = X W_{q,k,v}^T + b                     (one GEMM, N = 3D, split output)
//   O, s, keep = sparse attention + token pruning   (sc_kernels.cu)
//   S1 = X[kept] + O[kept] W_o^T + b_o              (GEMM: A and the residual gathered
//                                                    by the kept tokens' current index)
//   H1 = LN(S1);  F = GELU(H1 W_1^T + b_1);  S2 = H1 + F W_2^T + b_2;  Y = LN(S2)
// so everything after the attention runs on the kept tokens only, and the
// compaction of the kept rows is the A-operand gather of the output
// projection (Y is the next layer's X, already compacted).
//
// GEMM: output tiles of 128 rows of one sequence (rows are (sequence, row)
// pairs, row < rows[b] read on the device) by 256, 192, 128 or 64 columns (chosen
// on the device from the rows there are), one persistent CTA per SM walking the
// tiles that hold rows; K in steps of 64 through a TMA ring of four to eight
// stages: A's 128 rows by one tiled copy, or by
// four-row gathers (tile::gather4, any row order) when A is gathered, W's rows
// by one tiled copy, both 128B-swizzled and K-major; one thread issues the
// MMAs (M = 128) into one of two 256-column fp32 accumulators in tensor memory
// while eight warps read the other back, apply bias, GELU and the residual,
// and store each 32-column chunk through shared memory as whole row segments.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "sc_internal.cuh"
#include "sm103_primitives.cuh"

namespace sc {

constexpr int kGemmThreads = 320;   // warp 0 loads, warp 1 issues, warps 2-9 write back
constexpr int kGemmEpiWarps = 8;    // two per tensor-memory lane quarter, every other chunk
constexpr int kGemmChunkStep = 32 * (kGemmEpiWarps / 4);   // columns between a warp's chunks
constexpr int kGemmMinStages = 4;   // ring stages of 256-column tiles
constexpr int kGemmMaxStages = 8;   // ... of 64-column tiles, in the same shared memory
constexpr int kGemmMinBN = 64;      // narrowest tile
constexpr int kGemmSeqs = 128;      // most sequences whose tiles are counted out
constexpr int kGemmBK = 64;         // K per stage: one 128-byte swizzle atom of bf16
constexpr int kGemmBN = 256;        // most output columns per tile (one MMA, N <= 256)
constexpr uint32_t kGemmABytes = kTileBytes;              // 128 rows x 64
constexpr uint32_t kGemmWBytes = kGemmBN * kGemmBK * 2;   // 256 rows x 64
constexpr uint32_t kGemmRingBytes = kGemmMinStages * (kGemmABytes + kGemmWBytes);
// after the ring: a 4 KB staging area per write-back warp (32 rows of 128 bytes),
// through which the stores of a chunk leave as whole row segments
constexpr uint32_t kGemmStageOut = 4096;
constexpr uint32_t kGemmDyn = kGemmRingBytes + kGemmEpiWarps * kGemmStageOut + 1024;

struct GemmSmem {
  uint64_t full[kGemmMaxStages], empty[kGemmMaxStages];
  uint64_t tfull[2], tempty[2];   // accumulator buffers: written by the MMAs, read back
  uint32_t tmem_base;
  int abort;
  // per sequence: row tiles of the sequences before it (up to all)
  int tile0[kGemmSeqs + 1];
  uint8_t pad[kGemmSeqs];   // rows missing in the last tile
  int bn;
  alignas(16) float bias[kGemmBN];   // of the tile being written back
};

static_assert(sizeof(GemmSmem) + kGemmDyn <= 227 * 1024, "one CTA's shared memory");

// Bounded wait that ignores the abort flag (teardown: no copy or MMA may still
// write into this CTA's memory when it exits).
__device__ __forceinline__ void drain_wait_gemm(uint64_t* bar, uint32_t parity) {
  int dummy = 0;
  mbar_wait(bar, parity, &dummy, 1000000000ull);
}

// Nothing may still be landing in shared memory when the CTA exits: the last
// fill of every stage.  `use` rounds of the ring and s stages have been filled.
__device__ __forceinline__ void gemm_drain_full(GemmSmem& sm, int stages, int s, int use) {
#pragma unroll 1
  for (int q = 0; q < stages; ++q) {
    const int fills = use + (q < s ? 1 : 0);
    if (fills > 0) drain_wait_gemm(&sm.full[q], (fills - 1) & 1);
  }
}

__device__ __forceinline__ bool warp_wait_gemm(uint64_t* bar, uint32_t parity, volatile int* abort) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort));
}

// The write-back warps meet (barrier 1).
__device__ __forceinline__ void gemm_sync_epilogue() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * kGemmEpiWarps) : "memory");
}

__device__ __forceinline__ uint16_t bf16_bits(float x) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}

// GELU(x) = x/2 (1 + erf(x / sqrt 2)) with erf from Abramowitz & Stegun
// 7.1.26 (|error| <= 1.5e-7): erf(z) = 1 - (a1 t + ... + a5 t^5) exp(-z^2),
// t = 1 / (1 + p z), z >= 0, extended as an odd function.  With
// h = (1 - erf(|x| / sqrt 2)) / 2:  GELU(x) = x (1 - h) for x >= 0, x h below.
// Two values at once: the polynomial, the products and the exponent in packed
// fp32 pairs (the coefficients carry the factor 1/2), with
// exp(-z^2) = 2^(-z^2 log2 e).
__device__ __forceinline__ void gelu_erf2(float& x0, float& x1) {
  const float z0 = fabsf(x0) * 0.70710678118654752f, z1 = fabsf(x1) * 0.70710678118654752f;
  const uint64_t z = f2_pack(z0, z1);
  float d0, d1;
  f2_unpack(f2_fma(z, f2_pack(0.3275911f, 0.3275911f), f2_pack(1.f, 1.f)), d0, d1);
  const uint64_t t = f2_pack(__fdividef(1.f, d0), __fdividef(1.f, d1));
  uint64_t poly = f2_fma(f2_pack(0.5307027145f, 0.5307027145f), t,
                         f2_pack(-0.7265760135f, -0.7265760135f));
  poly = f2_fma(poly, t, f2_pack(0.7107068705f, 0.7107068705f));
  poly = f2_fma(poly, t, f2_pack(-0.142248368f, -0.142248368f));
  poly = f2_fma(poly, t, f2_pack(0.127414796f, 0.127414796f));
  float e0, e1;
  f2_unpack(f2_mul(f2_mul(z, z), f2_pack(-1.44269504088896341f, -1.44269504088896341f)), e0, e1);
  float h0, h1;
  f2_unpack(f2_mul(f2_mul(poly, t), f2_pack(ex2(e0), ex2(e1))), h0, h1);
  x0 *= x0 >= 0.f ? 1.f - h0 : h0;
  x1 *= x1 >= 0.f ? 1.f - h1 : h1;
}

// Tile t of the launch: column block nt of width bn (fastest, so that the
// CTAs of a wave share A rows), row tile rt of sequence b.  Where the tiles that
// hold rows are counted out (rows given, at most kGemmSeqs sequences) t counts
// only these; a role's tiles come in increasing order, so `b` is advanced.
struct GemmTile {
  int b, r0, n0, nw, rows;
  bool skip;
};

__device__ __forceinline__ bool gemm_counted(const GemmParams& p) {
  return p.rows != nullptr && p.B <= kGemmSeqs;
}

__device__ __forceinline__ void gemm_tile(const GemmParams& p, const GemmSmem& sm, int bn, int t,
                                          GemmTile& g) {
  const int tiles_n = (p.N + bn - 1) / bn;
  const int nt = t % tiles_n, rest = t / tiles_n;
  if (gemm_counted(p)) {
    while (sm.tile0[g.b + 1] <= rest) ++g.b;
    g.r0 = (rest - sm.tile0[g.b]) * kTile;
    g.rows = (sm.tile0[g.b + 1] - sm.tile0[g.b]) * kTile - sm.pad[g.b];
  } else {
    const int tiles_r = (p.L + kTile - 1) / kTile;
    g.b = rest / tiles_r;
    g.r0 = (rest % tiles_r) * kTile;
    g.rows = p.rows ? min(__ldcg(p.rows + g.b), p.L) : p.L;
  }
  g.n0 = nt * bn;
  g.nw = min(bn, p.N - g.n0);
  g.skip = g.r0 >= g.rows;
}

// Counts out the row tiles of every sequence and chooses the tile width; warp 0.
__device__ __forceinline__ void gemm_plan(const GemmParams& p, GemmSmem& sm, int lane) {
  int total = p.B * ((p.L + kTile - 1) / kTile);
  if (gemm_counted(p)) {
    total = 0;
#pragma unroll 1
    for (int b0 = 0; b0 < p.B; b0 += 32) {
      const int b = b0 + lane;
      const int n = b < p.B ? max(min(__ldcg(p.rows + b), p.L), 0) : 0;
      int x = (n + kTile - 1) / kTile;   // inclusive scan
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
      }
      if (b < p.B) {
        sm.pad[b] = static_cast<uint8_t>(-n & (kTile - 1));
        sm.tile0[b + 1] = total + x;
      }
      total += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) sm.tile0[0] = 0;
  }
  // The width with the least (whole rounds of tiles over the CTAs) x (width + 32),
  // the 32 a per-tile cost in columns' worth of time: the tiles run in rounds of
  // one per SM, so a width that leaves a last round mostly empty costs a whole
  // round.  Widths divide N and the split blocks; with a gathered A, 256 (A is
  // fetched again for every column tile).  One width per lane.  A short batch
  // leaves most SMs idle and each busy one fetches at its own L2 rate, so there
  // the narrowest tiles win: a layer of one sequence of 200 tokens takes 60.9 us
  // with 64-column tiles and 67.9 with 128 as the narrowest.  Counting the rows
  // that are there, not the L there may be, gives a layer of 8 x 1024 tokens with
  // a third pruned 172 us instead of 178.
  uint32_t key = 0xffffffffu;
  const int c = kGemmBN - 64 * lane;
  if (c > 0 && (p.a_idx == nullptr || c == kGemmBN)) {
    const bool fits = p.N % c == 0 && (p.out_split <= 0 || p.out_split % c == 0);
    const uint32_t tiles = static_cast<uint32_t>(total) * ((p.N + c - 1) / c);
    const uint32_t cost = (tiles + gridDim.x - 1) / gridDim.x * (c + 32);
    if (fits) key = min(cost, 0x0fffffffu) * 4 + lane;
    else if (c == kGemmBN) key = 0xfffffff0u;   // where nothing fits: masked last columns
  }
  key = __reduce_min_sync(0xffffffffu, key);
  if (lane == 0) sm.bn = kGemmBN - 64 * static_cast<int>(key & 3);
}

// Persistent: each CTA walks tiles blockIdx.x, blockIdx.x + gridDim.x, ...;
// the accumulator alternates between two 256-column buffers, so that the
// write-back of one tile overlaps the MMAs of the next.
// kPlain: bf16 out without a residual.  The fp32 staging and the residual are
// another instance: with both in one, the write-back loop of a feed-forward
// product with GELU (8 x 1024 rows, 768 -> 3072) took 45.2 us, without 38.5.
template <bool kPlain>
__global__ void __launch_bounds__(kGemmThreads, 1)
    sc_gemm_kernel(const __grid_constant__ GemmParams p) {
  extern __shared__ uint8_t dyn_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dyn_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  __shared__ GemmSmem sm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ksteps = p.K / kGemmBK;

  if (tid == 0) {
    for (int s = 0; s < kGemmMaxStages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&sm.tfull[a], 1);
      mbar_init(&sm.tempty[a], kGemmEpiWarps);   // one arrival per write-back warp
    }
    sm.abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc(&sm.tmem_base, 512);
  // what the launch before this one writes is read from here on
  pdl_wait();
  pdl_launch_dependents();
  if (warp == 0) gemm_plan(p, sm, lane);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = sm.tmem_base;
  volatile int* abort_flag = &sm.abort;
  const int bn = sm.bn;
  // A's rows and W's of one K step; as many stages as the ring holds (4 to 8)
  const uint32_t stage_bytes = kGemmABytes + bn * kGemmBK * 2;
  const int stages = min(kGemmMaxStages, static_cast<int>(kGemmRingBytes / stage_bytes));
  const int tiles = (gemm_counted(p) ? sm.tile0[p.B] : p.B * ((p.L + kTile - 1) / kTile)) *
                    ((p.N + bn - 1) / bn);
  GemmTile g;
  g.b = 0;

  if (warp == 0) {
    // ------------------------------------------------------------- loads
    const CUtensorMap* map_w = &p.map_w[bn / 64 - 1];
    const uint32_t w_bytes = min(bn, p.N) * kGemmBK * 2;   // rows past N: zeros
    bool ok = true;
    int s = 0, use = 0;
    if (p.a_idx == nullptr) {
      // one lane: a tiled copy of 128 consecutive rows, and one of W's rows (a
      // second W copy per step would cost 190 cycles: this loop paces short calls)
      if (elect_one()) {
        for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
          gemm_tile(p, sm, bn, t, g);
          if (g.skip) continue;
          const int row = g.b * p.L + g.r0;
#pragma unroll 1
          for (int kt = 0; kt < ksteps; ++kt) {
            if (use > 0 && !(ok = mbar_wait(&sm.empty[s], (use - 1) & 1, abort_flag))) break;
            uint8_t* As = base + s * stage_bytes;
            mbar_arrive_expect_tx(&sm.full[s], kGemmABytes + w_bytes);
            tma_load_2d(As + kGemmABytes, map_w, kt * kGemmBK, g.n0, &sm.full[s]);
            tma_load_2d(As, &p.map_a, kt * kGemmBK, row, &sm.full[s]);
            if (++s == stages) {
              s = 0;
              ++use;
            }
          }
        }
        gemm_drain_full(sm, stages, s, use);
      }
    } else {
      for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
        gemm_tile(p, sm, bn, t, g);
        if (g.skip) continue;
        // this lane's four rows (rows past the sequence read row 0: discarded)
        int ar[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int r = g.r0 + 4 * lane + k;
          ar[k] = g.b * p.L +
                  (r < g.rows ? __ldcg(p.a_idx + static_cast<size_t>(g.b) * p.L + r) : 0);
        }
#pragma unroll 1
        for (int kt = 0; kt < ksteps; ++kt) {
          if (use > 0 && !(ok = warp_wait_gemm(&sm.empty[s], (use - 1) & 1, abort_flag))) break;
          uint8_t* As = base + s * stage_bytes;
          if (lane == 0) {
            mbar_arrive_expect_tx(&sm.full[s], kGemmABytes + w_bytes);
            tma_load_2d(As + kGemmABytes, map_w, kt * kGemmBK, g.n0, &sm.full[s]);
          }
          __syncwarp();
          tma_gather4(As + 512 * lane, &p.map_a, kt * kGemmBK, ar[0], ar[1], ar[2], ar[3],
                      &sm.full[s]);
          if (++s == stages) {
            s = 0;
            ++use;
          }
        }
      }
      if (lane == 0) gemm_drain_full(sm, stages, s, use);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------- MMA issue
    if (elect_one()) {
      bool ok = true;
      int s = 0, use = 0, j = 0;
      const uint32_t ring = smem_u32(base);
      for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
        gemm_tile(p, sm, bn, t, g);
        if (g.skip) continue;
        const int acc = j & 1;
        // the buffer's previous tile has been read back
        if (j >= 2 && !(ok = mbar_wait(&sm.tempty[acc], ((j >> 1) - 1) & 1, abort_flag)))
          break;
        tc_fence_after();
        const uint32_t d = tm + acc * kGemmBN, idesc = idesc_bf16(128, g.nw, false, false);
#pragma unroll 1
        for (int kt = 0; kt < ksteps; ++kt) {
          if (!(ok = mbar_wait(&sm.full[s], use & 1, abort_flag))) break;
          tc_fence_after();
          const uint32_t a = sdesc_lo(ring + s * stage_bytes), w = a + (kGemmABytes >> 4);
#pragma unroll
          for (int k = 0; k < kGemmBK / 16; ++k)
            umma_bf16_lo(d, a + 2 * k, w + 2 * k, idesc, (kt | k) != 0);
          umma_commit(&sm.empty[s]);   // the stage is free once these MMAs are done
          if (++s == stages) {
            s = 0;
            ++use;
          }
        }
        umma_commit(&sm.tfull[acc]);
        ++j;
      }
      // every MMA has completed before the tensor memory is freed
      if (use > 0 || s > 0) {
        const int q = (s + stages - 1) % stages;
        const int fills = use + (q < s ? 1 : 0);
        drain_wait_gemm(&sm.empty[q], (fills - 1) & 1);
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------- write back
    // This part paces the products with K = 768: the copies of the next tile fill
    // the L2 ports, so anything it loads on the way costs up to a microsecond a
    // chunk.  Hence the bias through shared memory, the residual two chunks ahead
    // and in the layout of the stores (one row per lane touched 32 lines a load),
    // and one rolled loop.  8 x 1024 rows: 768 -> 2304 30.1 -> 24.4 us,
    // 768 -> 3072 with GELU 52.3 -> 38.6, 768 -> 768 with residual 22.1 -> 18.2.
    // Sixteen warps were slower (27.4, 50.1, 22.8).
    const int q = warp & 3;                  // tensor-memory lane quarter of this warp
    const int c0 = (warp - 2) / 4 * 32;      // its first chunk of 32 columns
    const int et = tid - 64;
    uint8_t* const stg = base + kGemmRingBytes + (warp - 2) * kGemmStageOut;
    bool ok = true;
    int j = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
      gemm_tile(p, sm, bn, t, g);
      if (g.skip) continue;
      const int acc = j & 1;
      const int r = g.r0 + 32 * q + lane;
      const bool in_rows = r < g.rows;
      // the residual of a chunk as the lanes store it (four columns of rows
      // lane / 8 + 4 k), loaded two chunks ahead: under the copies of the products
      // a load takes up to a microsecond
      [[maybe_unused]] uint2 rv[2][8];
      [[maybe_unused]] int rsrc = 0;
      [[maybe_unused]] auto load_res = [&](uint2 (&to)[8], int c) {
        if (p.res == nullptr || c >= g.nw) return;
        const uint16_t* res =
            p.res + static_cast<size_t>(g.b) * p.L * p.N + g.n0 + 4 * (lane & 7) + c;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int row = __shfl_sync(0xffffffffu, rsrc, 4 * k + lane / 8);
          to[k] = __ldcg(reinterpret_cast<const uint2*>(res + static_cast<size_t>(row) * p.N));
        }
      };
      if constexpr (!kPlain) {
        if (in_rows) rsrc = p.res_idx ? __ldcg(p.res_idx + static_cast<size_t>(g.b) * p.L + r) : r;
        load_res(rv[0], c0);
        load_res(rv[1], c0 + kGemmChunkStep);
      }
      // the tile's bias, once every warp is done with the previous one's
      const float bias = p.bias && et < g.nw ? __ldg(p.bias + g.n0 + et) : 0.f;
      gemm_sync_epilogue();
      if (et < kGemmBN) sm.bias[et] = bias;
      gemm_sync_epilogue();
      ok = ok && warp_wait_gemm(&sm.tfull[acc], (j >> 1) & 1, abort_flag);
      const uint32_t rows_mask = __ballot_sync(0xffffffffu, ok && in_rows);
      const size_t orow0 = static_cast<size_t>(g.b) * p.L + g.r0 + 32 * q;   // the warp's row 0
      int nb = g.n0, ldo = p.N;
      void* outp = p.out;
      if (p.out_split > 0) {
        const int sj = g.n0 / p.out_split;
        outp = p.outs[sj];
        nb = g.n0 - sj * p.out_split;
        ldo = p.out_split;
      }
      tc_fence_after();
#pragma unroll 1
      for (int c = c0; rows_mask != 0u && c < g.nw; c += kGemmChunkStep) {
        float v[32];
        tmem_ld32(tm + acc * kGemmBN + (static_cast<uint32_t>(32 * q) << 16) + c, v);
        tmem_ld_wait();
        const float4* bp = reinterpret_cast<const float4*>(sm.bias + c);
#pragma unroll
        for (int k = 0; k < 32; k += 4) {
          const float4 b4 = bp[k / 4];
          v[k] += b4.x;
          v[k + 1] += b4.y;
          v[k + 2] += b4.z;
          v[k + 3] += b4.w;
        }
        if (p.gelu)
#pragma unroll
          for (int k = 0; k < 32; k += 2) gelu_erf2(v[k], v[k + 1]);
        // the warp's 32 rows leave as row segments of 128 bytes (fp32) or 64 (bf16);
        // rows past the sequence are not written
        if constexpr (kPlain) {
#pragma unroll
          for (int k = 0; k < 32; k += 8)
            stage_row_piece<4>(stg, k / 8,
                               make_uint4(pack_bf16x2(v[k], v[k + 1]), pack_bf16x2(v[k + 2], v[k + 3]),
                                          pack_bf16x2(v[k + 4], v[k + 5]),
                                          pack_bf16x2(v[k + 6], v[k + 7])));
          flush_staged_rows<4>(stg, static_cast<uint16_t*>(outp) + orow0 * ldo + nb + c,
                               static_cast<size_t>(ldo), rows_mask);
          continue;
        }
#pragma unroll
        for (int k = 0; k < 32; k += 4)
          stage_row_piece<8>(stg, k / 4,
                             make_uint4(__float_as_uint(v[k]), __float_as_uint(v[k + 1]),
                                        __float_as_uint(v[k + 2]), __float_as_uint(v[k + 3])));
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int rr = 4 * k + lane / 8;
          float4 o = *reinterpret_cast<const float4*>(stg + stage_offset<8>(rr, lane & 7));
          if (p.res != nullptr) {
            o.x += __uint_as_float(rv[0][k].x << 16);
            o.y += __uint_as_float(rv[0][k].x & 0xffff0000u);
            o.z += __uint_as_float(rv[0][k].y << 16);
            o.w += __uint_as_float(rv[0][k].y & 0xffff0000u);
            rv[0][k] = rv[1][k];
          }
          if ((rows_mask >> rr) & 1u) {
            const size_t at = (orow0 + rr) * ldo + nb + c + 4 * (lane & 7);
            if (p.out_f32)
              *reinterpret_cast<float4*>(static_cast<float*>(outp) + at) = o;
            else
              *reinterpret_cast<uint2*>(static_cast<uint16_t*>(outp) + at) =
                  make_uint2(pack_bf16x2(o.x, o.y), pack_bf16x2(o.z, o.w));
          }
        }
        load_res(rv[1], c + 2 * kGemmChunkStep);
        __syncwarp();   // the staging area may be written again
      }
      // the buffer may take the tile after next
      tc_fence_before();
      warp_arrive(&sm.tempty[acc]);
      ++j;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
  if (tid == 0 && sm.abort) atomicOr(p.status, kStatusTimeout);
}

// ---------------------------------------------------------------------------
// row gather: the kept rows of a bf16 matrix, consecutive (8 rows per CTA,
// 16-byte vectors, every load of a thread issued before its stores)
// ---------------------------------------------------------------------------
constexpr int kRgRows = 8;
constexpr int kRgThreads = 256;

__global__ void __launch_bounds__(kRgThreads)
    sc_row_gather_kernel(const __grid_constant__ RowGatherParams p) {
  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.y, r0 = blockIdx.x * kRgRows;
  const int n = __ldcg(p.rows + b);
  if (r0 >= n) return;
  const int cnt = min(kRgRows, n - r0);
  const int vec = p.D / 8;
  const int total = cnt * vec;
  constexpr int kPer = 4;
  const size_t base = static_cast<size_t>(b) * p.L;
  for (int k0 = threadIdx.x; k0 < total; k0 += kRgThreads * kPer) {
    uint4 v[kPer];
    size_t dofs[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int k = k0 + u * kRgThreads;
      if (k < total) {
        const int rr = k / vec, e = k - rr * vec;
        const int src = __ldcg(p.idx + base + r0 + rr);
        v[u] = __ldcg(reinterpret_cast<const uint4*>(p.src + (base + src) * p.D) + e);
        dofs[u] = (base + r0 + rr) * vec + e;
      }
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u)
      if (k0 + u * kRgThreads < total) reinterpret_cast<uint4*>(p.dst)[dofs[u]] = v[u];
  }
}

// ---------------------------------------------------------------------------
// layer norm over D features, one warp per row: fp32 in, bf16 out
// ---------------------------------------------------------------------------
constexpr int kLnThreads = 256;
constexpr int kLnMaxPer = 32;   // features per lane: D <= 1024

__global__ void __launch_bounds__(kLnThreads)
    sc_layernorm_kernel(const __grid_constant__ LayerNormParams p) {
  pdl_wait();
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long row = static_cast<long long>(blockIdx.x) * (kLnThreads / 32) + warp;
  if (row >= static_cast<long long>(p.B) * p.L) return;
  const int b = static_cast<int>(row / p.L), r = static_cast<int>(row % p.L);
  if (r >= (p.rows ? min(__ldcg(p.rows + b), p.L) : p.L)) return;
  const float* x = p.in + row * p.D;
  uint16_t* y = p.out + row * p.D;
  if (p.vec) {
    // lane covers features 4 lane + 128 k .. + 3: 16-byte loads, 8-byte stores
    constexpr int kMaxChunks = kLnMaxPer / 4;
    const int chunks = p.D / 128;
    float4 v[kMaxChunks];
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < kMaxChunks; ++k) {
      v[k] = k < chunks ? __ldcg(reinterpret_cast<const float4*>(x) + lane + 32 * k)
                        : make_float4(0.f, 0.f, 0.f, 0.f);
      s += (v[k].x + v[k].y) + (v[k].z + v[k].w);
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    const float mean = s / static_cast<float>(p.D);
    float q = 0.f;
#pragma unroll
    for (int k = 0; k < kMaxChunks; ++k)
      if (k < chunks) {
        const float a = v[k].x - mean, b2 = v[k].y - mean, c = v[k].z - mean, d = v[k].w - mean;
        q += (a * a + b2 * b2) + (c * c + d * d);
      }
    for (int off = 16; off > 0; off >>= 1) q += __shfl_xor_sync(0xffffffffu, q, off);
    const float inv = 1.f / sqrtf(q / static_cast<float>(p.D) + p.eps);
#pragma unroll
    for (int k = 0; k < kMaxChunks; ++k)
      if (k < chunks) {
        const int f4 = lane + 32 * k;
        const float4 g = __ldg(reinterpret_cast<const float4*>(p.gamma) + f4);
        const float4 be = __ldg(reinterpret_cast<const float4*>(p.beta) + f4);
        const uint2 o = make_uint2(pack_bf16x2((v[k].x - mean) * inv * g.x + be.x,
                                               (v[k].y - mean) * inv * g.y + be.y),
                                   pack_bf16x2((v[k].z - mean) * inv * g.z + be.z,
                                               (v[k].w - mean) * inv * g.w + be.w));
        reinterpret_cast<uint2*>(y)[f4] = o;
      }
    return;
  }
  const int per = p.D / 32;   // features of this lane: lane, lane + 32, ...
  float v[kLnMaxPer];
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < kLnMaxPer; ++k) {
    v[k] = k < per ? __ldcg(x + lane + 32 * k) : 0.f;
    s += v[k];
  }
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  const float mean = s / static_cast<float>(p.D);
  float q = 0.f;
#pragma unroll
  for (int k = 0; k < kLnMaxPer; ++k)
    if (k < per) {
      const float d = v[k] - mean;
      q += d * d;
    }
  for (int off = 16; off > 0; off >>= 1) q += __shfl_xor_sync(0xffffffffu, q, off);
  const float inv = 1.f / sqrtf(q / static_cast<float>(p.D) + p.eps);
#pragma unroll
  for (int k = 0; k < kLnMaxPer; ++k)
    if (k < per) {
      const int f = lane + 32 * k;
      const float o = (v[k] - mean) * inv * __ldg(p.gamma + f) + __ldg(p.beta + f);
      y[f] = bf16_bits(o);
    }
}

// ---------------------------------------------------------------------------
// launch helpers used by the C ABI
// ---------------------------------------------------------------------------
cudaError_t configure_encoder() {
  const cudaError_t e =
      cudaFuncSetAttribute(sc_gemm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(kGemmDyn));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(sc_gemm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(kGemmDyn));
}

template <typename... KArgs>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, const KArgs&... args) {
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
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

cudaError_t launch_gemm(const GemmParams& p, cudaStream_t st) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
  }
  const int least = p.a_idx != nullptr ? kGemmBN : kGemmMinBN;   // narrowest tiles possible
  const long long tiles = static_cast<long long>(p.B) * ((p.L + kTile - 1) / kTile) *
                          ((p.N + least - 1) / least);
  const unsigned grid = static_cast<unsigned>(tiles < sms ? tiles : sms);
  const bool plain = p.res == nullptr && !p.out_f32;
  return launch_pdl(plain ? sc_gemm_kernel<true> : sc_gemm_kernel<false>, dim3(grid),
                    dim3(kGemmThreads), kGemmDyn, st, p);
}

cudaError_t launch_row_gather(const RowGatherParams& p, cudaStream_t st) {
  dim3 grid((p.L + kRgRows - 1) / kRgRows, p.B);
  return launch_pdl(sc_row_gather_kernel, grid, dim3(kRgThreads), 0, st, p);
}

cudaError_t launch_layernorm(const LayerNormParams& p, cudaStream_t st) {
  const long long rows = static_cast<long long>(p.B) * p.L;
  const unsigned blocks = static_cast<unsigned>((rows + kLnThreads / 32 - 1) / (kLnThreads / 32));
  auto al = [](const void* q, unsigned a) { return (reinterpret_cast<uintptr_t>(q) % a) == 0; };
  LayerNormParams q = p;
  q.vec = (p.D % 128 == 0 && al(p.in, 16) && al(p.gamma, 16) && al(p.beta, 16) && al(p.out, 8))
              ? 1 : 0;
  return launch_pdl(sc_layernorm_kernel, dim3(blocks), dim3(kLnThreads), 0, st, q);
}

}  // namespace sc
