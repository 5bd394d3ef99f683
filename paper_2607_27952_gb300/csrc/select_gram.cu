// Eq. 9-12 (Sec. 3.4): the greedy selection from a Gram matrix.
//
// Three launches.  norms_kernel: 1/|x_i| of every token (canonical order).
// gram_kernel or gram_pair_kernel: every request's dot products x_i . x_j on the tensor
// cores, fp32, to the workspace (lower triangle computed, mirrored on the way out); or
// gram_exact_kernel: the same in the canonical order (fp32 features, small batches).
// select_gram_kernel: the greedy, one thread-block cluster of C CTAs per request,
// in rounds that accept a batch of consecutive picks at once and give exactly the
// sequential Eq. 10-11 sequence:
//   1. every warp publishes its `mc` best live keys (w~_i delta_i, index) and its
//      (mc+1)-th key to every CTA of the cluster (DSMEM; one cluster barrier);
//   2. the published entries above U = the largest (mc+1)-th key form the candidate
//      list (at most kGlist; U rises to the first key cut off).  No token outside
//      the list has a key above U, and keys never increase;
//   3. the members' pairwise distances come from the Gram matrix;
//   4. warp 0 replays the greedy on the list alone while its best key is above U;
//   5. meanwhile the other warps fold the accepted centres' Gram rows into their
//      tokens, eight centres at a time as the replay posts them.
// The Gram distances d~ are only known to within eps, the decisions are canonical, so
// a token carries an interval: the minimum e over the centres evaluated so far, and up
// to four pending centres whose d~ lies within eps of being the minimum.  Tokens are
// ranked by the upper end; a member of the list has its pending centres evaluated in
// the canonical order (by the CTA that owns it, which sends the member's values to the
// others; a second cluster barrier), and during
// the replay a member is evaluated again only when the order of the picks depends on
// it.  A token far from the lead is never evaluated at all: evaluating every pair that
// the certificate leaves open, at the moment it appears, took 185K of 400K cycles a
// round on requests of 4096 tokens.
// Every CTA of a cluster does the rest of steps 2-4 alike.
//
// Against the rounds that stream X (select_impl.cuh) a round reads 4 bytes per token
// and centre instead of a whole row per token, so its cost no longer grows with
// d_v, and the N^2 d_v contraction runs once, at tensor-core rates, on every SM.
//
// A round is bound by latency: about 30K cycles on a request of 576 tokens (k = 192, 14
// rounds), of which the replay takes 650 a pick, 40K on 16384 tokens in 12 CTAs (k =
// 2048, 76 rounds).  Measured against the rounds that stream X (GB300, whole last_prune
// call): 64 requests of 576 x 2048, k 64/128/192: 1.71 -> 0.39 ms; 32 of 2880, k = 360:
// 5.27 -> 1.14; 128 of 256..4096 x 1536, k = N/8: 10.3 -> 2.41; 8 of 16384 x 2048, k =
// 2048: 16.9 -> 4.83 (3.0 of it the Gram matrix).
//
// Tokens are dealt to the cluster in blocks of 32: block k belongs to CTA k % C,
// worker warp (k / C) % 15, so neighbouring tokens (tiles, frames, near-duplicates) spread
// over all warps and both the ranking and the exact pairs stay balanced.
//
// Arithmetic of every decision is the canonical fp32 of the public header: the kept
// indices are bit-identical to the sequential definition.
#include "gram_schedule.h"
#include "select_impl.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace last {

namespace {

constexpr int kGwarps = 16;
constexpr int kGthreads = kGwarps * 32;
constexpr int kGwork = kGwarps - 1;        // worker warps own the tokens, warp 0 replays
constexpr int kGtok = kGwork * 32;
constexpr int kGbatch = 8;                 // accepted centres handed to the workers at a time
constexpr int kGlist = 64;                 // candidate list: two members per lane of the replay
constexpr int kGper = kGlist / 32;
constexpr int kGmaxAccept = 64;            // one bit per accepted centre
constexpr int kGpairLd = kGlist + 1;
constexpr int kGcand = 1024;               // published entries above U kept before the cut

// ---- Gram tiles: 128 rows x 256 columns, the lower triangle of each request ----
constexpr int kGM = 128, kGN = 256, kGK = 64;
constexpr int kGramStages = 4;
constexpr int kGramStageBytes = (kGM + kGN) * kGK * 2;   // 48 KB
constexpr int kPairStages = 3;
constexpr int kPairStageBytes = 2 * 2 * kGM * kGK * 2;   // two K blocks, 64 KB per CTA of a pair
constexpr int kGramThreads = 320;          // 8 epilogue warps, TMA producer, MMA issuer
constexpr int kGroupRows = 16;             // row blocks per tile group (L2 reuse of both operands)

}  // namespace

// Tiles of a request with R row blocks, in groups of 16 row blocks: group g has 16
// rows of 8g full column blocks and a triangular part of 8 more.
__host__ __device__ inline int gram_group_tiles(int g, int h) {
  int n = h * 8 * g;
  for (int c = 0; 2 * c < h; ++c) n += h - 2 * c;
  return n;
}
int gram_tiles(int n_tokens, bool pair) {
  if (pair) {
    const int R = (n_tokens + kGN - 1) / kGN;
    return R * (R + 1) / 2;
  }
  const int R = (n_tokens + kGM - 1) / kGM;
  int n = 0;
  for (int g = 0; 16 * g < R; ++g) n += gram_group_tiles(g, std::min(kGroupRows, R - 16 * g));
  return n;
}

// Bound on |d~ - d| between a distance from the Gram matrix and the canonical one.  A
// chunk of products is one chain of tensor-core accumulations: a sum of n exact
// products in any order, each addition rounded or truncated once to fp32, errs by at
// most n 2^-23 sum|x_i,k x_j,k|, and aligning groups of 16 products to the group's
// largest exponent by 17/16 of that; taken twice.  The chunks are added in fp32 (8 u at
// most), the canonical order adds 80 u (see tc_distance_eps) and the scalings 1e-6.
inline float gram_distance_eps(int dv, int chunk) {
  return (float)((std::min(dv, chunk) * 0x1p-22 + 88 * 0x1p-24) * 1.01 + 1e-6);
}
// Requests of at least this many tokens take CTA pairs; below, the pairs' 256-row tiles
// waste more than they gain (64 requests of 576: 0.111 against 0.090 ms).
bool gram_long(int max_vis) { return max_vis >= 2048; }
// Products per chain.  Short chains narrow the bound, so fewer distances are evaluated
// in the canonical order, but each costs the Gram kernel a pass over its accumulators,
// and long requests spend most of their time there.  Whole calls, pairs with chains of
// 256 / 512 / 1024 / 2048: 32 requests of 2880 1.22 / 1.17 / - / - ms, 128 of 256..4096
// 2.51 / 2.53, 8 of 16384 - / 5.45 / 5.00 / 5.18.
int gram_chunk(int max_vis) { return max_vis >= 8192 ? 1024 : max_vis >= 2048 ? 512 : 256; }

struct GramArgs {
  CUtensorMap tmap;        // X as [total_vis][dv] bf16, box 64 x 128, 128-byte swizzle
  float *gram;
  const int32_t *meta;
  const int32_t *tile0;    // [B + 1] first tile of each request
  int B, dv, total_tiles, chunk_kb;   // chunk_kb: K blocks per accumulation chain
  unsigned *err;
};

// An epilogue thread adds a tile row's 128 values up in registers: the ten warps are
// allocated like twelve, 168 registers each, and both kernels spill 40 and 32 bytes.

// Row i, columns j0 .. j0 + 127 of a request's matrix, and the same values as a column
// when `mirror`.
__device__ __forceinline__ void store_tile(const GramArgs &a, int b, int i, int j0, bool mirror,
                                           const float *v) {
  const int32_t *m = a.meta + b * kMetaFields;
  const int N = m[kNumVis], ld = gram_ld(N);
  float *G = a.gram + (long long)m[kGramOff] * 32;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int j = j0 + 32 * c;
    if (j < N) {
      if (i < N) {
        float *row = G + (long long)i * ld + j;
#pragma unroll
        for (int q = 0; q < 32; q += 8) st_global_v8(row + q, v + 32 * c + q);
      }
      if (mirror && i < ld) {
        float *col = G + (long long)j * ld + i;
#pragma unroll
        for (int q = 0; q < 32; ++q)
          if (j + q < N) col[(long long)q * ld] = v[32 * c + q];
      }
    }
  }
}

__global__ void __launch_bounds__(kGramThreads, 1) gram_kernel(const __grid_constant__ GramArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  __shared__ unsigned long long full[kGramStages], empty[kGramStages], afull[2], aempty[2], never;
  __shared__ uint32_t tslot;   // TMEM base
  __shared__ volatile int gave_up;   // a role's wait has expired
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkb = tc_kblocks(a.dv);
  if (threadIdx.x == 0) {
    for (int i = 0; i < kGramStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&afull[i], 1);
      mbar_init(&aempty[i], 8);
    }
    mbar_init(&never, 1);
    fence_mbar_init();
    gave_up = 0;
  }
  if (warp == 0) tmem_alloc(&tslot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot;
  // a role's waits: after one has expired the others return at once and the call reports it
  bool dead = false;
  auto twait = [&](unsigned long long *bar, uint32_t par) -> bool {
    if (!dead && !mbar_wait_bounded(bar, par, a.err, kErrTimeout)) {
      dead = true;
      gave_up = 1;
    }
    return !dead;
  };
  // tile -> (request, row block, column block)
  auto decode = [&](int tile, int *b_, int *ti, int *tj) {
    int lo = 0, hi = a.B - 1;
    while (lo < hi) {   // the last request whose first tile is at or before `tile`
      const int mid = (lo + hi + 1) >> 1;
      if (a.tile0[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    *b_ = lo;
    int rem = tile - a.tile0[lo];
    const int R = (a.meta[lo * kMetaFields + kNumVis] + kGM - 1) / kGM;
    int g = 0;
    while (16 * (g + 1) < R && rem >= 128 * g + 72) rem -= 128 * g++ + 72;   // whole groups
    const int h = min(kGroupRows, R - 16 * g);
    if (rem < h * 8 * g) {
      *tj = rem / h;
      *ti = 16 * g + rem % h;
    } else {
      rem -= h * 8 * g;
      int c = 0;
      while (rem >= h - 2 * c) rem -= h - 2 * c++;
      *tj = 8 * g + c;
      *ti = 16 * g + 2 * c + rem;
    }
  };

  if (warp == 8) {
    if (lane == 0) {
      int st = 0;
      uint32_t ph = 1;   // (the first pass over the ring waits for nothing)
      for (int tile = blockIdx.x; tile < a.total_tiles; tile += gridDim.x) {
        int b, ti, tj;
        decode(tile, &b, &ti, &tj);
        const int row0 = a.meta[b * kMetaFields + kVisOff];
        for (int kb = 0; kb < nkb; ++kb) {
          if (!twait(&empty[st], ph)) break;
          unsigned char *dst = smem + st * kGramStageBytes;
          mbar_expect_tx(&full[st], kGramStageBytes);
          tma_load_2d(dst, &a.tmap, kb * kGK, row0 + ti * kGM, &full[st]);
          tma_load_2d(dst + kGM * kGK * 2, &a.tmap, kb * kGK, row0 + tj * kGN, &full[st]);
          tma_load_2d(dst + 2 * kGM * kGK * 2, &a.tmap, kb * kGK, row0 + tj * kGN + 128, &full[st]);
          if (++st == kGramStages) {
            st = 0;
            ph ^= 1u;
          }
        }
      }
    }
  } else if (warp == 9) {
    if (lane == 0) {
      const uint32_t idesc = umma_idesc_bf16(kGM, kGN);
      // the operands' descriptors: a stage further is kGramStageBytes, 16 elements 32 bytes
      const uint64_t da = umma_desc_sw128(smem_addr(smem)), db = umma_desc_sw128(smem_addr(smem) + kGM * kGK * 2);
      int st = 0;
      uint32_t ph = 0, ab = 0, aph = 1;
      for (int tile = blockIdx.x; tile < a.total_tiles; tile += gridDim.x)
        for (int kb = 0; kb < nkb; kb += a.chunk_kb) {
          const int end = min(kb + a.chunk_kb, nkb);
          twait(&aempty[ab], aph);
          for (int k = kb; k < end; ++k) {
            const bool ok = twait(&full[st], ph);
            tc_fence_after();
            const uint64_t off = (uint64_t)(uint32_t)(st * (kGramStageBytes >> 4));
            if (ok) {
#pragma unroll
              for (int q = 0; q < kGK / 16; ++q)
                umma_bf16(tmem + ab * kGN, da + off + 2 * q, db + off + 2 * q, idesc, (k != kb || q) ? 1u : 0u);
            }
            umma_commit(&empty[st]);
            if (++st == kGramStages) {
              st = 0;
              ph ^= 1u;
            }
          }
          umma_commit(&afull[ab]);
          ab ^= 1u;
          aph ^= ab ^ 1u;   // flips when the first accumulator comes round again
        }
    }
  } else {
    // warps 0-7: 32 rows (the warp's TMEM lanes) x 128 columns each; the chains of a
    // tile are added in registers
    const int half = warp >> 2, quad = warp & 3;
    uint32_t nc = 0;
    for (int tile = blockIdx.x; tile < a.total_tiles; tile += gridDim.x) {
      int b, ti, tj;
      decode(tile, &b, &ti, &tj);
      float v[128];
#pragma unroll
      for (int q = 0; q < 128; ++q) v[q] = 0.f;
      for (int kb = 0; kb < nkb; kb += a.chunk_kb, ++nc) {
        const int ab = nc & 1;
        twait(&afull[ab], (nc >> 1) & 1);
        __syncwarp();
        tc_fence_after();
        const uint32_t tb = tmem + ab * kGN + half * 128 + ((uint32_t)(32 * quad) << 16);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          uint32_t raw[16];
          tmem_ld16(tb + 16 * c, raw);
#pragma unroll
          for (int q = 0; q < 16; ++q) v[16 * c + q] = __fadd_rn(v[16 * c + q], __uint_as_float(raw[q]));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&aempty[ab]);
      }
      // the transposed 128 x 128 block too, unless a tile of its own computes it
      const int j0 = tj * kGN + half * 128;
      store_tile(a, b, ti * kGM + 32 * quad + lane, j0, j0 / kGM < 2 * (ti / 2), v);
    }
  }
  __syncthreads();
  if (gave_up) {   // an aborted call: time for copies and MMAs in flight before the CTA may exit
    if (threadIdx.x == 0) wait_out(&never);
    __syncthreads();
  }
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the norms too are done when this grid is
}

// The same tiles for a pair of CTAs (a cluster of two): 256 rows x 256 columns, each CTA
// holding 128 rows of the accumulator and loading its half of either operand: 32 KB per
// K block of 128 x 256 products instead of 48, into and out of a shared memory that the
// single-CTA kernel saturates.  A stage holds two K blocks: handing a stage over costs
// about 750 cycles however small it is (copies alone, 2 x 16384 tokens: 0.64 ms with one
// K block a stage, 0.38 with two).  Copies and MMAs without the epilogue 0.59 ms, 1.86
// PFLOP/s over the lower triangle (single CTA 0.78); with it 0.79 in chains of 1024
// products, 0.91 of 512, 1.08 of 256 (single CTA 1.00 in one chain, 1.15 of 256): the
// epilogue's stores only overlap the chains that fit in tensor memory.  Both kernels'
// issuing threads keep the stage, its phase and the descriptors in registers: deriving
// them from a counter took 3.47 instead of 2.99 ms on 8 requests of 16384.
__global__ void __launch_bounds__(kGramThreads, 1) gram_pair_kernel(const __grid_constant__ GramArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  // full, aempty: of the even CTA (its barriers count both CTAs); empty, afull: each CTA's
  __shared__ unsigned long long full[kPairStages], empty[kPairStages], afull[2], aempty[2], never;
  __shared__ uint32_t tslot;   // TMEM base
  __shared__ volatile int gave_up;   // a role's wait has expired, in either CTA
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int nkb = tc_kblocks(a.dv);
  if (threadIdx.x == 0) {
    for (int i = 0; i < kPairStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&afull[i], 1);
      mbar_init(&aempty[i], 16);
    }
    mbar_init(&never, 1);
    fence_mbar_init();
    gave_up = 0;
  }
  if (warp == 0) tmem_alloc_pair(&tslot, 512);
  tc_fence_before();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem = tslot;
  bool dead = false;
  auto twait = [&](unsigned long long *bar, uint32_t par) -> bool {
    if (!dead && !mbar_wait_bounded(bar, par, a.err, kErrTimeout)) {
      dead = true;
      for (int r = 0; r < 2; ++r) st_cluster_s32(map_shared(const_cast<int *>(&gave_up), r), 1);
    }
    return !dead;
  };
  auto decode = [&](int tile, int *b_, int *ti, int *tj) {
    int lo = 0, hi = a.B - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (a.tile0[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    *b_ = lo;
    int rem = tile - a.tile0[lo];
    const int R = (a.meta[lo * kMetaFields + kNumVis] + kGN - 1) / kGN;
    int g = 0;
    while (8 * (g + 1) < R && rem >= 64 * g + 36) rem -= 64 * g++ + 36;   // whole groups
    const int h = min(8, R - 8 * g);
    if (rem < h * 8 * g) {
      *tj = rem / h;
      *ti = 8 * g + rem % h;
    } else {
      rem -= h * 8 * g;
      int c = 0;
      while (rem >= h - c) rem -= h - c++;
      *tj = 8 * g + c;
      *ti = 8 * g + c + rem;
    }
  };
  const int tile_first = blockIdx.x >> 1, tile_step = gridDim.x >> 1;

  if (warp == 8) {
    if (lane == 0) {
      int st = 0;
      uint32_t ph = 1;   // (the first pass over the ring waits for nothing)
      for (int tile = tile_first; tile < a.total_tiles; tile += tile_step) {
        int b, ti, tj;
        decode(tile, &b, &ti, &tj);
        const int row0 = a.meta[b * kMetaFields + kVisOff] + 128 * rank;
        for (int kb = 0; kb < nkb; kb += 2) {
          if (!twait(&empty[st], ph)) break;
          unsigned char *dst = smem + st * kPairStageBytes;
          const uint32_t bar = map_shared(&full[st], 0);
          if (rank == 0) mbar_expect_tx(&full[st], 2 * kPairStageBytes);
          for (int y = 0; y < 2; ++y) {   // (columns past d_v land as zeros)
            tma_load_2d_pair(dst + 2 * y * kGM * kGK * 2, &a.tmap, (kb + y) * kGK, row0 + ti * kGN, bar);
            tma_load_2d_pair(dst + (2 * y + 1) * kGM * kGK * 2, &a.tmap, (kb + y) * kGK, row0 + tj * kGN, bar);
          }
          if (++st == kPairStages) {
            st = 0;
            ph ^= 1u;
          }
        }
      }
    }
  } else if (warp == 9) {
    if (lane == 0 && rank == 0) {
      const uint32_t idesc = umma_idesc_bf16(2 * kGM, kGN);
      const uint64_t da = umma_desc_sw128(smem_addr(smem)), db = umma_desc_sw128(smem_addr(smem) + kGM * kGK * 2);
      int st = 0;
      uint32_t ph = 0, ab = 0, aph = 1;
      for (int tile = tile_first; tile < a.total_tiles; tile += tile_step)
        for (int kb = 0; kb < nkb; kb += a.chunk_kb) {
          const int end = min(kb + a.chunk_kb, nkb);
          twait(&aempty[ab], aph);
          for (int k = kb; k < end; k += 2) {
            const bool ok = twait(&full[st], ph);
            tc_fence_after();
            const uint64_t off = (uint64_t)(uint32_t)(st * (kPairStageBytes >> 4));
            if (ok) {
#pragma unroll
              for (int q = 0; q < 2 * kGK / 16; ++q) {
                const int at = (q / 4) * (2 * kGM * kGK * 2 >> 4) + 2 * (q % 4);
                umma_bf16_pair(tmem + ab * kGN, da + off + at, db + off + at, idesc, (k != kb || q) ? 1u : 0u);
              }
            }
            umma_commit_pair(&empty[st]);
            if (++st == kPairStages) {
              st = 0;
              ph ^= 1u;
            }
          }
          umma_commit_pair(&afull[ab]);
          ab ^= 1u;
          aph ^= ab ^ 1u;
        }
    }
  } else {
    const int half = warp >> 2, quad = warp & 3;
    uint32_t nc = 0;
    for (int tile = tile_first; tile < a.total_tiles; tile += tile_step) {
      int b, ti, tj;
      decode(tile, &b, &ti, &tj);
      float v[128];
#pragma unroll
      for (int q = 0; q < 128; ++q) v[q] = 0.f;
      for (int kb = 0; kb < nkb; kb += a.chunk_kb, ++nc) {
        const int ab = nc & 1;
        twait(&afull[ab], (nc >> 1) & 1);
        __syncwarp();
        tc_fence_after();
        const uint32_t tb = tmem + ab * kGN + half * 128 + ((uint32_t)(32 * quad) << 16);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          uint32_t raw[16];
          tmem_ld16(tb + 16 * c, raw);
#pragma unroll
          for (int q = 0; q < 16; ++q) v[16 * c + q] = __fadd_rn(v[16 * c + q], __uint_as_float(raw[q]));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_shared(&aempty[ab], 0));
      }
      store_tile(a, b, ti * kGN + 128 * rank + 32 * quad + lane, tj * kGN + half * 128, ti != tj, v);
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync();   // both CTAs are done with either's barriers, operands and accumulators
  if (gave_up) {   // an aborted call: time for copies and MMAs in flight before either may exit
    if (threadIdx.x == 0) wait_out(&never);
    __syncwarp();
    cluster_sync();
  }
  tc_fence_after();
  if (warp == 0) tmem_dealloc_pair(tmem, 512);
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// 1/|x_i| in the canonical order, one warp per token: one read of X at the copy rate (24
// us on 64 requests of 576 x 2048).  The Gram kernel starts beside it.
template <typename T, int NCH>
__global__ void __launch_bounds__(256) norms_kernel(const char *x, float *rn, int dv, int row_bytes,
                                                    long long total) {
  asm volatile("griddepcontrol.launch_dependents;");
  const int lane = threadIdx.x & 31;
  const long long nw = (long long)gridDim.x * 8;
  for (long long t = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); t < total; t += nw) {
    const char *row = x + t * row_bytes;
    const float ss = dot_rows<T, NCH>(row, false, row, false, dv, lane);
    if (lane == 0) rn[t] = ss > 0.f ? __fdiv_rn(1.0f, __fsqrt_rn(ss)) : 0.f;
  }
}

// The same matrix in the canonical order on CUDA cores: every distance the greedy reads
// from it is then exact.  For fp32 features (the tensor cores' tf32 would leave almost
// every pair open) and for bf16 batches small enough that the evaluations it saves the
// greedy outweigh it.  A warp's 32 lanes are the canonical order's: each holds the
// partial sums of 8 x 8 pairs over its own coordinate groups, rows staged 256
// coordinates at a time (three buffers), and the lanes' sums are added by the canonical
// butterfly with the pairs dealt out on the way (62 shuffles for 64 pairs instead of
// 320).  Bound by the fmas and the shared-memory reads that feed them: 15 T fma/s in fp32
// on 4096 x 1024, 21 in bf16.  A CTA takes 32 x 32 pairs in fp32, whose copies limit
// narrower tiles (six requests of 800 x 1000: 231 us at 32 x 16, 147 at 32 x 32), and 32 x
// 16 in bf16, which only comes here in small batches that must be spread over the SMs
// (one image of 576 x 2048: 27 against 32 us).
constexpr int kExRows = 32, kExBufs = 3;
template <typename T> constexpr int kExCols = sizeof(T) == 4 ? 32 : 16;
int gram_exact_tiles(int n_tokens, bool f32) {
  const int R = (n_tokens + kExRows - 1) / kExRows;
  return f32 ? R * (R + 1) / 2 : R * (R + 1);
}

struct GramExactArgs {
  const char *x;
  float *gram;
  const int32_t *meta;
  const int32_t *tile0;
  int B, dv, row_bytes;
};

template <typename T>
__global__ void __launch_bounds__(16 * kExCols<T>, kExRows / kExCols<T>) gram_exact_kernel(const GramExactArgs a) {
  constexpr int kCols = kExCols<T>, kThreads = 16 * kCols, kPer = kExRows / kCols;   // kPer column blocks a row block
  constexpr int kVec = (int)sizeof(T) / 2;            // 16-byte pieces per 8 coordinates
  constexpr int kRowBytes = 256 * (int)sizeof(T);     // a row's staged part
  constexpr int kBuf = (kExRows + kCols) * kRowBytes;
  asm volatile("griddepcontrol.launch_dependents;");   // the greedy waits for this grid's end
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int lo = 0, hi = a.B - 1;
  const int tile = blockIdx.x;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.tile0[mid] <= tile) lo = mid; else hi = mid - 1;
  }
  const int rem = tile - a.tile0[lo];
  // row block ti has kPer (ti + 1) column blocks
  int ti = (int)((sqrtf(8.0f * (float)(rem / kPer) + 1.0f) - 1.0f) * 0.5f);
  while (kPer * (ti * (ti + 1) / 2) > rem) --ti;
  while (kPer * ((ti + 1) * (ti + 2) / 2) <= rem) ++ti;
  const int tj = rem - kPer * (ti * (ti + 1) / 2);
  const int32_t *m = a.meta + lo * kMetaFields;
  const int N = m[kNumVis], ld = gram_ld(N);
  float *G = a.gram + (long long)m[kGramOff] * 32;
  const char *xreq = a.x + (long long)m[kVisOff] * a.row_bytes;
  const int i0 = ti * kExRows, j0 = tj * kCols;
  const uint32_t sbase = smem_addr(smem);
  const int nchunk = (a.dv + 255) / 256;

  // a thread copies the same 16-byte piece of every (threads / pieces per row)-th row:
  // piece q is lane q / kVec's part q % kVec.  fp32 lanes read every other piece; swapping
  // the two pieces of every second group of four lanes spreads them over all banks.
  constexpr int kPieces = 32 * kVec, kStep = kThreads / kPieces;
  const int q0 = tid % kPieces, r0 = tid / kPieces, col0 = (q0 / kVec) * 8;
  const char *src0 = xreq + 16 * q0;
  const int swap = kVec == 2 ? (lane >> 2) & 1 : 0;
  const uint32_t dst_q = sbase + r0 * kRowBytes + 16 * (kVec == 2 ? q0 ^ ((q0 >> 3) & 1) : q0);
  auto stage = [&](int c) {
    const uint32_t dst = dst_q + (c % kExBufs) * kBuf;
    const char *src = src0 + (size_t)c * kRowBytes;
    const bool in = 256 * c + col0 < a.dv;
#pragma unroll
    for (int i = 0; i < (kExRows + kCols) / kStep; ++i) {
      const int r = r0 + i * kStep;   // (a step never straddles the two operands)
      const int t = min(i * kStep < kExRows ? i0 + r : j0 + r - kExRows, N - 1);
      if (in)
        cp_async16(dst + i * kStep * kRowBytes, src + (size_t)(uint32_t)t * (uint32_t)a.row_bytes);
      else
        asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" :: "r"(dst + i * kStep * kRowBytes), "r"(0u) : "memory");
    }
    cp_async_commit();
  };
  float acc[64];
#pragma unroll
  for (int q = 0; q < 64; ++q) acc[q] = 0.f;
  constexpr int kWj = kCols / 8;   // warps along the columns
  const uint32_t row_i = 8 * (warp / kWj), row_j = kExRows + 8 * (warp % kWj);
  stage(0);
  if (nchunk > 1) stage(1);
  else cp_async_commit();
  for (int c = 0; c < nchunk; ++c) {
    cp_async_wait<1>();
    __syncthreads();   // chunk c has landed; its predecessor's buffer is free
    if (c + 2 < nchunk) stage(c + 2);
    else cp_async_commit();
#pragma unroll 1
    for (int h = 0; h < kVec; ++h) {
      const uint32_t base = sbase + (c % kExBufs) * kBuf + 16 * (lane * kVec + (h ^ swap));
      U4 xi[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) xi[i] = lds32(base + (row_i + i) * kRowBytes);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const U4 xj = lds32(base + (row_j + j) * kRowBytes);
        const uint32_t jw[4] = {xj.x, xj.y, xj.z, xj.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint32_t iw = q == 0 ? xi[i].x : q == 1 ? xi[i].y : q == 2 ? xi[i].z : xi[i].w;
            float &s = acc[i * 8 + j];
            if constexpr (sizeof(T) == 2) {
              s = fma_bf16_lo(iw, jw[q], s);
              s = fma_bf16_hi(iw, jw[q], s);
            } else {
              s = __fmaf_rn(__uint_as_float(iw), __uint_as_float(jw[q]), s);
            }
          }
      }
    }
  }
  // butterfly over the lanes (offsets 16 .. 1); at each step a lane keeps half of the
  // pairs, so lane l ends with pairs 2 l, 2 l + 1: row l / 4, columns 2 (l % 4) ..
#pragma unroll
  for (int o = 16, n = 32; o > 0; o >>= 1, n >>= 1) {
#pragma unroll
    for (int q = 0; q < n; ++q) {
      const float send = (lane & o) ? acc[q] : acc[q + n];
      const float keep = (lane & o) ? acc[q + n] : acc[q];
      acc[q] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, o));
    }
  }
  const int i = i0 + (int)row_i + (lane >> 2), j = j0 + 8 * (warp % kWj) + 2 * (lane & 3);
  if (i < N) {
    if (j < ld) *reinterpret_cast<float2 *>(G + (long long)i * ld + j) = make_float2(acc[0], acc[1]);
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (j + r < N) G[(long long)(j + r) * ld + i] = acc[r];
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the norms too are done when this grid is
}

struct GramSelArgs {
  const char *x;
  const float *w, *rn, *gram;
  int32_t *idx_out;
  char *x_out;             // nullable
  const int32_t *meta, *order;
  int dv, row_bytes, csize, mc, slots, words;
  float eps;               // bound on |distance from the Gram matrix - canonical distance|
  unsigned *err;
};

// Centres of a token whose distance is only known to within eps.  With two, tokens of
// tight clusters were evaluated again and again as a third came near: 2 / 4 took 2.53 /
// 2.44 ms on 128 requests of 256..4096, 1.29 / 1.20 on one video request.
constexpr int kGpend = 4;

// Shared memory of select_gram_kernel (host sizing and device carve-up alike).
struct GramSelSmem {
  size_t ks, w, r, e, hi, p, ids, hot, sel, pkey, pwr, ckey, cidx, pm, lidx, lr, res, top, acc, cen,
      crow, bars, misc, total;
};
__host__ __device__ inline GramSelSmem gram_sel_smem(int slots, int words, int csize, int mc) {
  GramSelSmem s;
  size_t o = 0;
  const size_t cap = (size_t)slots * kGtok;       // token slots of a CTA
  s.ks = o; o += 4 * cap;                         // high word of the upper key, 0 = not live
  s.w = o; o += 4 * cap;
  s.r = o; o += 4 * cap;
  s.e = o; o += 4 * cap;
  s.hi = o; o += 4 * cap;                         // upper end of delta
  s.p = o; o += 4 * kGpend * cap;                 // pending centres: distance
  s.ids = o; o += 2 * kGpend * cap;               // and token
  s.hot = o; o += 4 * cap;                        // tokens a batch may lower: slot, centres
  s.sel = o; o += align16(4 * (size_t)words);     // selected bits of the whole request
  s.pkey = o; o += (size_t)2 * kGwork * csize * (mc + 1) * 8;   // published keys
  s.pwr = o; o += (size_t)2 * kGwork * csize * (mc + 1) * 8;    // and their w~, 1/|x|
  s.ckey = o = align16(o); o += 8 * (kGcand + 2);
  s.cidx = o; o += 2 * kGcand;
  s.pm = o; o += align16(4 * kGlist * kGpairLd);  // the list's pairwise distances
  s.lidx = o; o += 4 * kGlist;                    // the list: token, 1/|x|
  s.lr = o; o += 4 * kGlist;
  s.res = o = align16(o); o += 16 * kGlist;       // key and delta (from its owner), w~, 1/|x|
  s.top = o; o += 8 * kGwarps * 16;               // a warp's leading keys
  s.acc = o; o += 4 * kGmaxAccept;
  s.cen = o; o += 8 * kGmaxAccept;                // accepted centres: token, 1/|x|
  s.crow = o; o += 4 * kGmaxAccept;               // and their Gram rows' offsets
  s.bars = o; o += 8 * (kGmaxAccept / kGbatch);   // batch i of the round's centres is posted
  s.misc = o; o += 8 * 48;
  s.total = align16(o);
  return s;
}

__device__ __forceinline__ unsigned long long gram_key(uint32_t kh, uint32_t idx) {
  return ((unsigned long long)kh << 32) | (0xffffffffu - idx);
}
// high word of the key of w delta
__device__ __forceinline__ uint32_t key_high(float w, float delta) {
  return (uint32_t)(argmax_key(__fmul_rn(w, delta), 0) >> 32);
}

// EX: the matrix holds canonical dot products (gram_exact_kernel, eps = 0): every
// distance is final, nothing is pending and no row is read before the epilogue.
template <int NCH, bool EX>
__global__ void __launch_bounds__(kGthreads, 1)
select_gram_kernel(const __grid_constant__ GramSelArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int C = a.csize, rank = (int)cluster_ctarank();
  // a programmatic dependent of the canonical matrix's kernel: nothing is read before it
  // (and what precedes it) has completed
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int b = a.order[cluster_id_x()];
  const int32_t *m = a.meta + b * kMetaFields;
  const int voff = m[kVisOff], N = m[kNumVis], koff = m[kKeepOff], K = m[kNumKeep];
  if (K == 0) return;   // the whole cluster leaves together
  const GramSelSmem S = gram_sel_smem(a.slots, a.words, C, a.mc);
  {
    uint32_t dyn;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
    if (S.total > dyn) {   // host and device plans disagree: every CTA leaves before any barrier
      if (tid == 0) atomicOr(a.err, kErrConfig);
      return;
    }
  }
  const int widx = warp - 1;   // worker or -1
  uint32_t *ks = reinterpret_cast<uint32_t *>(smem + S.ks);
  float *w_s = reinterpret_cast<float *>(smem + S.w);
  float *r_s = reinterpret_cast<float *>(smem + S.r);
  float *e_s = reinterpret_cast<float *>(smem + S.e);
  float *hi_s = reinterpret_cast<float *>(smem + S.hi);
  const int cap = a.slots * kGtok;
  float *p_s = reinterpret_cast<float *>(smem + S.p);            // [kGpend][cap]
  uint16_t *id_s = reinterpret_cast<uint16_t *>(smem + S.ids);   // [kGpend][cap]
  uint32_t *hot = reinterpret_cast<uint32_t *>(smem + S.hot) + widx * a.slots * 32;   // workers
  uint32_t *sel = reinterpret_cast<uint32_t *>(smem + S.sel);
  unsigned long long *pkey = reinterpret_cast<unsigned long long *>(smem + S.pkey);
  unsigned long long *ckey = reinterpret_cast<unsigned long long *>(smem + S.ckey);
  float *pm = reinterpret_cast<float *>(smem + S.pm);
  int *lidx = reinterpret_cast<int *>(smem + S.lidx);
  float *lr = reinterpret_cast<float *>(smem + S.lr);
  float2 *pwr = reinterpret_cast<float2 *>(smem + S.pwr);
  uint16_t *cidx = reinterpret_cast<uint16_t *>(smem + S.cidx);
  float4 *res = reinterpret_cast<float4 *>(smem + S.res);
  unsigned long long *top_s = reinterpret_cast<unsigned long long *>(smem + S.top) + warp * 16;
  int *acc_s = reinterpret_cast<int *>(smem + S.acc);
  float2 *cen = reinterpret_cast<float2 *>(smem + S.cen);
  uint32_t *crow = reinterpret_cast<uint32_t *>(smem + S.crow);
  unsigned long long *misc = reinterpret_cast<unsigned long long *>(smem + S.misc);
  unsigned long long *bars = reinterpret_cast<unsigned long long *>(smem + S.bars);
  int *cnt = reinterpret_cast<int *>(misc + 32);   // [0] kept tokens, [1] candidates, [2] picks, [4 + i] batch i

  const int rb = a.row_bytes, dv = a.dv, ld = gram_ld(N);
  const float eps = a.eps;
  const int nblk = (N + 31) >> 5;
  const char *xreq = a.x + (long long)voff * rb;
  const float *rreq = a.rn + voff, *wreq = a.w + voff;
  const float *G = a.gram + (long long)m[kGramOff] * 32;
  const int P = kGwork * C;                           // publishing warps of the cluster
  const int step = C * kGwork;                        // blocks between a warp's slots
  const int blk0 = rank + C * widx;             // a worker's first block
  const int nslot = widx < 0 ? 0 : (nblk - blk0 + step - 1) / step;   // and its blocks (<= a.slots)
  const int li0 = widx * 32 + lane;                           // a worker thread's first token slot
  // block k (< 2^12): owner CTA and slot in shared memory, by multiplication
  const uint32_t inv_c = (0xffffffffu / (uint32_t)C) + 1u, inv_step = (0xffffffffu / (uint32_t)step) + 1u;
  auto over_c = [&](int k) { return C == 1 ? k : (int)__umulhi((uint32_t)k, inv_c); };
  auto owned = [&](int k) { return k - over_c(k) * C == rank; };
  auto slot_of = [&](int t) {   // of an owned token
    const int k = t >> 5, z = (int)__umulhi((uint32_t)k, inv_step);
    return z * kGtok + (over_c(k) - z * kGwork) * 32 + (t & 31);
  };

  if (tid < kGmaxAccept / kGbatch) mbar_init(&bars[tid], 1);
  if (tid == 0) fence_mbar_init();
  for (int v = tid; v < nblk; v += kGthreads) sel[v] = K == N ? 0xffffffffu : 0u;
  for (int s = 0; s < nslot; ++s) {
    const int t = 32 * (blk0 + s * step) + lane, li = s * kGtok + li0;
    const bool in = t < N;
    w_s[li] = in ? wreq[t] : 0.f;
    r_s[li] = in && K < N ? rreq[t] : 0.f;
    hi_s[li] = INFINITY;
    if constexpr (!EX) {
      e_s[li] = INFINITY;
#pragma unroll
      for (int q = 0; q < kGpend; ++q) p_s[q * cap + li] = INFINITY;
    }
    ks[li] = in ? 1u : 0u;   // live; the first update sets the key
  }

  if (K < N) {
    auto csync = [&]() {
      if (C == 1) __syncthreads();
      else cluster_sync();
    };
    // 8 coordinates per lane of each chunk of row t
    auto load_row = [&](int t, U4 *v) {
      const char *row = xreq + (long long)t * rb;
#pragma unroll
      for (int g = 0; g < NCH; ++g) {
        const int col = 256 * g + 8 * lane;
        v[g] = col < dv ? ldg_nc(row + col * 2) : U4{0, 0, 0, 0};
      }
    };
    // canonical distance of two rows with reciprocal norms ri (the token's) and rc
    auto distance = [&](const U4 *x, const U4 *c, float ri, float rc) {
      float acc = 0.f;
#pragma unroll
      for (int g = 0; g < NCH; ++g) {
        if (256 * g + 8 * lane < dv) {
          const uint32_t xw[4] = {x[g].x, x[g].y, x[g].z, x[g].w};
          const uint32_t cw[4] = {c[g].x, c[g].y, c[g].z, c[g].w};
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            acc = fma_bf16_lo(xw[h], cw[h], acc);
            acc = fma_bf16_hi(xw[h], cw[h], acc);
          }
        }
      }
      return __fsub_rn(1.0f, __fmul_rn(__fmul_rn(butterfly_sum(acc), ri), rc));
    };

    // A worker folds the accepted centres cen[j0 .. j0 + n) (n <= kGbatch) into its
    // tokens.  A centre with d~ - eps at or above the token's upper bound cannot lower
    // its delta.  Any other becomes one of the token's pending centres; entries that a new
    // upper bound excludes leave.  Pairs outside the certificate's norm range, NaN and a
    // centre too many are evaluated at once.
    auto update = [&](int j0, int n) {
      const uint32_t all = (1u << n) - 1u;
      // centres whose pairs the certificate does not cover
      const uint32_t wide = __ballot_sync(0xffffffffu, lane < n && !tri_in_range(cen[j0 + min(lane, n - 1)].y));
      int nq = 0;
      // this batch's part of the rows starts towards L2 (a line per block and centre)
      for (int i = lane; i < kGbatch * nslot; i += 32)
        if (i % kGbatch < n)
          prefetch_l2(G + crow[j0 + i % kGbatch] + 32 * (blk0 + (i / kGbatch) * step));
      // Four blocks at a time, 32 loads in flight per thread.  d~ - eps < hi is tested as
      // g rc >= (1 - eps - hi) / ri with a slack of 1e-6 for the roundings; what passes
      // is queued and tested again below.  (Dead tokens load too: a row holds whole blocks.)
      for (int s0 = 0; s0 < nslot; s0 += 4) {
        float g[4][kGbatch];
        const float *gt = G + 32 * (blk0 + s0 * step) + lane;
#pragma unroll
        for (int j = 0; j < kGbatch; ++j) {
          const float *gr = gt + crow[j0 + min(j, n - 1)];
#pragma unroll
          for (int z = 0; z < 4; ++z) g[z][j] = __ldg(gr + (s0 + z < nslot ? 32 * z * step : 0));
        }
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          if (s0 + z >= nslot) break;
          const int li = (s0 + z) * kGtok + li0;
          const float ri = r_s[li], hi = hi_s[li];
          const float thr = __fdiv_rn(1.0f - eps - hi - 1e-6f, ri);
          uint32_t low = tri_in_range(ri) ? wide : all;
#pragma unroll
          for (int j = 0; j < kGbatch; ++j)
            if (!(g[z][j] * cen[j0 + min(j, n - 1)].y < thr)) low |= 1u << j;   // NaN: tested again
          low = ks[li] != 0u ? low & all : 0u;
          const unsigned bal = __ballot_sync(0xffffffffu, low != 0u);
          if (low) hot[nq + __popc(bal & ((1u << lane) - 1u))] = (uint32_t)li | (low << 16);
          nq += __popc(bal);
        }
      }
      __syncwarp();
      for (int q0 = 0; q0 < nq; q0 += 32) {
        uint32_t now = 0u;   // centres to evaluate at once
        int li = 0, t = 0;
        float ri = 0.f;
        if (q0 + lane < nq) {
          const uint32_t h = hot[q0 + lane];
          uint32_t bt = h >> 16;
          li = (int)(h & 0xffffu);
          const int z = li / kGtok;   // (a constant divisor)
          t = 32 * (blk0 + z * step) + (li & 31);
          ri = r_s[li];
          const bool in_range = tri_in_range(ri);
          float hi = hi_s[li], pp[kGpend];
          if constexpr (!EX)
#pragma unroll
            for (int q = 0; q < kGpend; ++q) pp[q] = p_s[q * cap + li];
          while (bt) {
            const int j = __ffs(bt) - 1;
            bt &= bt - 1;
            const float2 cc = cen[j0 + j];
            const float d = __fsub_rn(1.0f, __fmul_rn(__fmul_rn(__ldg(G + crow[j0 + j] + t), ri), cc.y));
            if constexpr (EX) {
              hi = fminf(hi, d);   // NaN leaves it
            } else if (!in_range || ((wide >> j) & 1u) || d != d) {
              now |= 1u << j;
            } else if (!(__fsub_rd(d, eps) >= hi)) {
              hi = fminf(hi, __fadd_ru(d, eps));
              bool placed = false;
#pragma unroll
              for (int q = 0; q < kGpend; ++q) {
                if (__fsub_rd(pp[q], eps) >= hi) pp[q] = INFINITY;
                if (!placed && pp[q] == INFINITY) {
                  pp[q] = d;
                  id_s[q * cap + li] = (uint16_t)__float_as_uint(cc.x);
                  placed = true;
                }
              }
              if (!placed) now |= 1u << j;
            }
          }
          hi_s[li] = hi;
          ks[li] = key_high(w_s[li], hi);
          if constexpr (!EX) {
#pragma unroll
            for (int q = 0; q < kGpend; ++q) p_s[q * cap + li] = pp[q];
          }
        }
        __syncwarp();
        // the whole warp per token to evaluate
        if constexpr (!EX) {
          for (unsigned todo = __ballot_sync(0xffffffffu, now != 0u); todo != 0u; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int lt = __shfl_sync(0xffffffffu, li, src);
            uint32_t bt = __shfl_sync(0xffffffffu, now, src);
            U4 xv[NCH], xc[NCH];
            load_row(__shfl_sync(0xffffffffu, t, src), xv);
            const float rt = __shfl_sync(0xffffffffu, ri, src);
            float e = e_s[lt];
            while (bt) {
              const int j = __ffs(bt) - 1;
              bt &= bt - 1;
              const float2 cc = cen[j0 + j];
              load_row(__float_as_int(cc.x), xc);
              e = fminf(e, distance(xv, xc, rt, cc.y));
            }
            __syncwarp();
            if (lane == 0) {   // (hi holds d~ + eps of these centres already)
              const float hi = fminf(e, hi_s[lt]);
              e_s[lt] = e;
              hi_s[lt] = hi;
              ks[lt] = key_high(w_s[lt], hi);
            }
            __syncwarp();
          }
        }
      }
    };

    // ---- seed (Eq. 9): argmax w~ over the request, every CTA alike ----
    {
      unsigned long long best = 0ull;
      for (int t = tid; t < N; t += kGthreads) best = max(best, argmax_key(wreq[t], t));
      best = warp_max_u64(best);
      if (lane == 0) misc[warp] = best;
      __syncthreads();
      best = warp_max_u64(lane < kGwarps ? misc[lane] : 0ull);
      const int seed = key_index(best);
      if (tid == 0) {
        cen[0] = make_float2(__int_as_float(seed), rreq[seed]);
        crow[0] = (uint32_t)seed * (uint32_t)ld;
        sel[seed >> 5] |= 1u << (seed & 31);
      }
      if (tid == 0 && owned(seed >> 5)) ks[slot_of(seed)] = 0u;
      __syncthreads();
    }
    int taken = 1;
    if (taken < K && widx >= 0) update(0, 1);
    csync();   // every CTA of the cluster runs before the first remote write

    // ---- rounds (Eq. 10-11) ----
    const int ent = a.mc + 1;
    for (int round = 0; taken < K; ++round) {
      const int par = round & 1;
      unsigned long long *keyp = pkey + (size_t)par * P * ent;
      float2 *pwrp = pwr + (size_t)par * P * ent;
      // 1. this warp's best live tokens by upper key, best first, into top_s: each lane
      // queues its three best.  A lane whose third is taken may hide a fourth, which is
      // below it: the third then becomes the bound.
      if (widx >= 0) {
        unsigned long long k1 = 0ull, k2 = 0ull, k3 = 0ull, bound = 0ull;
        for (int s = 0; s < nslot; ++s) {
          const uint32_t v = ks[s * kGtok + li0];
          const unsigned long long k = v ? gram_key(v, (uint32_t)(32 * (blk0 + s * step) + lane)) : 0ull;
          const unsigned long long m1 = min(k, k1), m2 = min(m1, k2);
          k1 = max(k, k1);
          k2 = max(m1, k2);
          k3 = max(m2, k3);
        }
        int left = 3;
        if (lane < ent) top_s[lane] = 0ull;
        __syncwarp();
        for (int e = 0; e < ent; ++e) {
          const uint32_t mx = __reduce_max_sync(0xffffffffu, (uint32_t)(k1 >> 32));
          if (mx == 0u) break;
          bool win = (uint32_t)(k1 >> 32) == mx;
          const unsigned bal = __ballot_sync(0xffffffffu, win);
          if (bal & (bal - 1u)) {   // equal values: the lowest token
            const uint32_t lo = __reduce_max_sync(0xffffffffu, win ? (uint32_t)k1 : 0u);
            win = win && (uint32_t)k1 == lo;
          }
          if (win) {
            top_s[e] = k1;
            if (--left == 0) bound = k1;
            k1 = k2;
            k2 = k3;
            k3 = 0ull;
          }
        }
        __syncwarp();   // the winners' entries, before lane 0 reads and rewrites the last one
        if (nslot > 3 && __any_sync(0xffffffffu, left == 0)) {
          bound = warp_max_u64(bound);
          if (lane == 0) top_s[a.mc] = max(top_s[a.mc], bound);
        }
        __syncwarp();
        // entry lane % 4, 8 or 16 to CTAs lane / 4, 8 or 16, ..
        const int esh = ent <= 4 ? 2 : ent <= 8 ? 3 : 4, e = lane & ((1 << esh) - 1);
        if (e < ent) {
          const unsigned long long kk = top_s[e];
          const int slot = (rank * kGwork + widx) * ent + e;
          const int li = slot_of(key_index(kk));   // (kk == 0: unused)
          const float2 wr = kk != 0ull ? make_float2(w_s[li], r_s[li]) : make_float2(0.f, 0.f);
          for (int q = lane >> esh; q < C; q += 32 >> esh) {
            st_cluster_u64(map_shared(&keyp[slot], q), kk);
            st_cluster_v2f(map_shared(&pwrp[slot], q), wr);
          }
        }
      }
      if (tid == 0) cnt[1] = 0;
      csync();
      // 2. the list: published entries above U
      unsigned long long U = 0ull;
      for (int q = lane; q < P; q += 32) U = max(U, keyp[q * ent + a.mc]);
      U = warp_max_u64(U);
      for (int e0 = warp * 32; e0 < P * ent; e0 += kGthreads) {
        const int e = e0 + lane;
        const unsigned long long kk = e < P * ent ? keyp[e] : 0ull;
        const bool up = kk > U;
        const unsigned bal = __ballot_sync(0xffffffffu, up);
        if (bal) {
          int base = 0;
          if (lane == 0) base = atomicAdd(&cnt[1], __popc(bal));
          base = __shfl_sync(0xffffffffu, base, 0);
          if (up) {
            const int pos = base + __popc(bal & ((1u << lane) - 1u));
            ckey[pos] = kk;
            cidx[pos] = (uint16_t)e;
          }
        }
      }
      __syncthreads();
      const int nc = cnt[1];
      if (warp == 0) ckey[nc] = 0ull;
      __syncthreads();
      // the best kGlist of them in key order (the same in every CTA); U' = the first
      // key cut off
      for (int c0 = warp * 32; c0 < nc; c0 += kGthreads) {
        const int c = c0 + lane;
        const unsigned long long kk = c < nc ? ckey[c] : 0ull;
        int pos = 0;
#pragma unroll 4
        for (int q = 0; q < nc; q += 2) {   // (ckey[nc] is zero)
          const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(&ckey[q]);
          pos += (x.x > kk ? 1 : 0) + (x.y > kk ? 1 : 0);
        }
        if (c < nc) {
          if (pos < kGlist) {
            const float2 wr = pwrp[cidx[c]];
            lidx[pos] = key_index(kk);
            lr[pos] = wr.y;
            res[pos].z = wr.x;
            res[pos].w = wr.y;
            if constexpr (EX) res[pos].x = __uint_as_float((uint32_t)(kk >> 32));   // final: no owner is asked
          } else if (pos == kGlist) {
            misc[20] = kk;
          }
        }
      }
      __syncthreads();
      if (nc == 0) {   // cannot happen (the best live key is above U): every CTA leaves alike
        if (tid == 0) atomicOr(a.err, kErrConfig);
        break;
      }
      const int nL = min(nc, kGlist);
      const unsigned long long Up = nc > kGlist ? misc[20] : U;
      unsigned long long need = 0ull;   // this warp's share of the CTA's members to evaluate
      if constexpr (!EX) {
        int before = 0;
#pragma unroll
        for (int h = 0; h < kGper; ++h) {
          const int u = lane + 32 * h;
          const bool mine = u < nL && owned(lidx[min(u, nL - 1)] >> 5);
          const unsigned bal = __ballot_sync(0xffffffffu, mine);
          const int at = before + __popc(bal & ((1u << lane) - 1u));
          // a member without a pending centre is exact: sent as it is
          bool open = false;
          if (mine && at % kGwarps == warp) {
            const int li = slot_of(lidx[u]);
#pragma unroll
            for (int q = 0; q < kGpend; ++q) open |= p_s[q * cap + li] != INFINITY;
            if (!open) {
              const float2 v = make_float2(__uint_as_float(ks[li]), e_s[li]);
              for (int q = 0; q < C; ++q) st_cluster_v2f(map_shared(&res[u], q), v);
            }
          }
          need |= (unsigned long long)__ballot_sync(0xffffffffu, open) << (32 * h);
          before += __popc(bal);
        }
      }
      // the rows to evaluate start towards L2
      if constexpr (!EX)
        for (unsigned long long n = need; n != 0ull; n &= n - 1) {
          const int t = lidx[__ffsll((long long)n) - 1], li = slot_of(t);
          if (lane * 128 < rb) {
            prefetch_l2(xreq + (long long)t * rb + lane * 128);
#pragma unroll
            for (int q = 0; q < kGpend; ++q)
              if (p_s[q * cap + li] != INFINITY)
                prefetch_l2(xreq + (long long)id_s[q * cap + li] * rb + lane * 128);
          }
        }
      // 3. pairwise distances from the Gram matrix (NaN: outside the certificate): a warp
      // takes rows u and kGlist - 1 - u together, 63 pairs; the loads are in flight while
      // members are evaluated
      constexpr int kRows = kGlist / 2 / kGwarps;
      float g[kRows][kGper];
      auto pair_of = [&](int i, int h, int *u, int *v) {
        const int r = warp + i * kGwarps, x = lane + 32 * h, len = kGlist - 1 - r;
        *u = x < len ? r : len;
        *v = x < len ? r + 1 + x : x + 1;
        return *u < *v && *v < nL;
      };
#pragma unroll
      for (int i = 0; i < kRows; ++i)
#pragma unroll
        for (int h = 0; h < kGper; ++h) {
          int u, v;
          g[i][h] = pair_of(i, h, &u, &v) ? __ldg(G + (long long)lidx[u] * ld + lidx[v]) : 0.f;
        }
      // the CTA that owns a member evaluates its pending centres in the canonical order,
      // keeps the result and sends (key, delta) to every CTA: every member's delta is exact
      // from here on
      if constexpr (!EX) {
        for (; need != 0ull; need &= need - 1) {
          const int u = __ffsll((long long)need) - 1, t = lidx[u], li = slot_of(t);
          float e = e_s[li];
          const float w = w_s[li], r = r_s[li];
          // nearest first: a centre whose d~ - eps is at or above e cannot lower it
          U4 xv[NCH], xc[NCH];
          load_row(t, xv);
          float pq = INFINITY;
          int first = 0;
#pragma unroll
          for (int q = 0; q < kGpend; ++q)
            if (p_s[q * cap + li] < pq) {
              pq = p_s[q * cap + li];
              first = q;
            }
#pragma unroll 1
          for (int it = 0; it < kGpend; ++it) {
            const int q = it == 0 ? first : it <= first ? it - 1 : it;
            const float pd = p_s[q * cap + li];
            if (pd == INFINITY || __fsub_rd(pd, eps) >= e) continue;
            const int c = id_s[q * cap + li];
            const float rc = rreq[c];
            load_row(c, xc);
            e = fminf(e, distance(xv, xc, r, rc));
          }
          const uint32_t kh = key_high(w, e);
          __syncwarp();
          if (lane == 0) {
            e_s[li] = e;
            hi_s[li] = e;
            ks[li] = kh;
          }
          if (lane < kGpend) p_s[lane * cap + li] = INFINITY;
          if (lane < C) st_cluster_v2f(map_shared(&res[u], lane), make_float2(__uint_as_float(kh), e));
        }
      }
#pragma unroll
      for (int i = 0; i < kRows; ++i)
#pragma unroll
        for (int h = 0; h < kGper; ++h) {
          int u, v;
          if (pair_of(i, h, &u, &v)) {
            const float ru = lr[u], rv = lr[v];
            // pm[centre][token]
            float d = __fsub_rn(1.0f, __fmul_rn(__fmul_rn(g[i][h], rv), ru)), dt = d;
            if constexpr (EX) dt = __fsub_rn(1.0f, __fmul_rn(__fmul_rn(g[i][h], ru), rv));
            else if (!tri_in_range(ru) || !tri_in_range(rv)) d = dt = __int_as_float(0x7fffffff);
            pm[u * kGpairLd + v] = d;
            pm[v * kGpairLd + u] = dt;
          }
        }
      if constexpr (EX) __syncthreads();
      else csync();
      // 4. replay the greedy on the list (warp 0; lane u holds members u, u + 32, ..).
      // A member's delta is at most hi, and exact until an accepted centre's distance
      // reaches below hi + eps; such centres are kept in `pend` and evaluated only when
      // the member's place in the order depends on it.
      if (warp == 0) {
        uint32_t kh[kGper], id[kGper];   // upper key (high word), token
        float e[kGper], hi[kGper], wv[kGper];
        unsigned long long pend[kGper];
#pragma unroll
        for (int h = 0; h < kGper; ++h) {
          const int u = lane + 32 * h;
          kh[h] = 0u;
          id[h] = 0u;
          e[h] = wv[h] = 0.f;
          if (u < nL) {
            const float4 v = res[u];
            kh[h] = __float_as_uint(v.x);
            e[h] = v.y;
            wv[h] = v.z;
            id[h] = (uint32_t)lidx[u];
          }
          hi[h] = e[h];
          pend[h] = 0ull;
        }
        const uint32_t up_hi = (uint32_t)(Up >> 32);
        int nA = 0;
        const int most = min(K - taken, kGmaxAccept);
        // picks [j0, j0 + n) as centres for the workers (n < kGbatch ends the round)
        auto post = [&](int j0, int n) {
          if (lane < n) {
            const int u = acc_s[j0 + lane], t = lidx[u];
            cen[j0 + lane] = make_float2(__int_as_float(t), lr[u]);
            crow[j0 + lane] = (uint32_t)t * (uint32_t)ld;   // N^2 < 2^32 (the matrix is at most 12 GiB)
          }
          __syncwarp();
          if (lane == 0) {
            cnt[4 + j0 / kGbatch] = n;
            mbar_arrive(&bars[j0 / kGbatch]);
          }
        };
        while (nA < most) {
          // the member with the largest upper key (equal values: the lowest token)
          uint32_t lk = kh[0];
#pragma unroll
          for (int h = 1; h < kGper; ++h) lk = max(lk, kh[h]);
          const uint32_t mx = __reduce_max_sync(0xffffffffu, lk);
          unsigned win[kGper];
          int leads = 0, bl = 0;
          bool inexact = false;
#pragma unroll
          for (int h = kGper - 1; h >= 0; --h) {
            win[h] = __ballot_sync(0xffffffffu, kh[h] == mx);
            leads += __popc(win[h]);
            const unsigned open = EX ? 0u : __ballot_sync(0xffffffffu, kh[h] == mx && pend[h] != 0ull);
            bl = win[h] ? __ffs(win[h]) - 1 + 32 * h : bl;
            inexact = win[h] ? open != 0u : inexact;
          }
          if (mx <= up_hi || leads > 1) {
            if (mx < up_hi || mx == 0u) break;   // also the end of the list
            uint32_t lid = 0xffffffffu;
#pragma unroll
            for (int h = 0; h < kGper; ++h) lid = kh[h] == mx ? min(lid, id[h]) : lid;
            const uint32_t low = __reduce_min_sync(0xffffffffu, lid);
            if (gram_key(mx, low) <= Up) break;
#pragma unroll
            for (int h = 0; h < kGper; ++h) {
              const unsigned w = __ballot_sync(0xffffffffu, kh[h] == mx && id[h] == low);
              const unsigned open =
                  EX ? 0u : __ballot_sync(0xffffffffu, kh[h] == mx && id[h] == low && pend[h] != 0ull);
              if (w) {
                bl = __ffs(w) - 1 + 32 * h;
                inexact = open != 0u;
              }
            }
          }
          if (!EX && inexact) {
            // accepted as it is only if its lower key leads every other upper key
            const int src = bl & 31;
            unsigned long long bp = 0ull;
            uint32_t second = 0u;   // best other upper key (high word)
            float bhi = 0.f, be = 0.f;
#pragma unroll
            for (int h = 0; h < kGper; ++h) {
              if (lane + 32 * h == bl) {
                bp = pend[h];
                bhi = hi[h];
                be = e[h];
              } else {
                second = max(second, kh[h]);
              }
            }
            bp = shfl_u64(bp, src);
            be = __shfl_sync(0xffffffffu, be, src);
            second = __reduce_max_sync(0xffffffffu, second);
            // the lower end: e or the nearest pending centre less eps (NaN: none)
            const float bw = res[bl].z;
            uint32_t low = key_high(bw, be);
#pragma unroll
            for (int h = 0; h < kGmaxAccept / 32; ++h) {
              const int j = lane + 32 * h;
              if ((bp >> j) & 1ull) {
                const float d = __fsub_rd(pm[acc_s[j] * kGpairLd + bl], eps);
                low = min(low, d == d ? key_high(bw, d) : 0u);
              }
            }
            low = __reduce_min_sync(0xffffffffu, low);
            if (!(low > up_hi && low > second)) {
              bhi = __shfl_sync(0xffffffffu, bhi, src);
              U4 xv[NCH], xc[NCH];
              load_row(lidx[bl], xv);
              while (bp) {
                const int j = __ffsll((long long)bp) - 1;
                bp &= bp - 1;
                const int cj = acc_s[j];
                if (__fsub_rd(pm[cj * kGpairLd + bl], eps) >= bhi) continue;   // excluded since
                load_row(lidx[cj], xc);
                be = fminf(be, distance(xv, xc, res[bl].w, res[cj].w));
              }
#pragma unroll
              for (int h = 0; h < kGper; ++h)
                if (lane + 32 * h == bl) {
                  pend[h] = 0ull;
                  e[h] = hi[h] = be;
                  kh[h] = key_high(wv[h], be);
                }
              continue;
            }
          }
          const unsigned long long bit = 1ull << nA;
#pragma unroll
          for (int h = 0; h < kGper; ++h) {
            const int u = lane + 32 * h;
            const float d = pm[bl * kGpairLd + u];
            if (EX) {
              // w min(delta, d) = min(w delta, w d) (NaN has the largest key), or for a weight
              // below zero their maximum
              const uint32_t kd = key_high(wv[h], d);
              const uint32_t to = wv[h] < 0.f ? (d == d ? max(kh[h], kd) : kh[h]) : min(kh[h], kd);
              kh[h] = kh[h] == 0u || u == bl ? 0u : to;
              continue;
            } else {
              if (!(__fsub_rd(d, eps) >= hi[h])) pend[h] |= bit;   // NaN too
              hi[h] = fminf(hi[h], __fadd_ru(d, eps));             // (above hi unless pending; NaN keeps it)
            }
            kh[h] = kh[h] == 0u || u == bl ? 0u : key_high(wv[h], hi[h]);
          }
          if (lane == 0) acc_s[nA] = bl;
          __syncwarp();
          ++nA;
          if (nA % kGbatch == 0) post(nA - kGbatch, kGbatch);
        }
        if (lane == 0) cnt[2] = nA;
        if (nA < kGmaxAccept) {
          post(nA / kGbatch * kGbatch, nA % kGbatch);
          // the batches that this round does not reach complete too: one phase a round
          if (lane > nA / kGbatch && lane < kGmaxAccept / kGbatch) mbar_arrive(&bars[lane]);
        }
      } else if (widx >= 0) {
        // 5. meanwhile the workers fold the accepted centres into their tokens
        for (int i = 0; i < kGmaxAccept / kGbatch; ++i) {
          // an expired wait (the call is reported as failed): nothing that the replay may
          // not have posted is read, cen and crow would be offsets into the matrix.  The
          // rounds go on, in step with the cluster, and end after at most K picks.
          const bool posted = mbar_wait_bounded(&bars[i], par, a.err, kErrTimeout);
          if (!__all_sync(0xffffffffu, posted)) break;
          const int n = cnt[4 + i];
          if (n > 0) update(i * kGbatch, n);
          if (n < kGbatch) break;
        }
      }
      __syncthreads();
      const int nA = cnt[2];
      if (tid < nA) {
        const int gi = lidx[acc_s[tid]], k = gi >> 5;
        atomicOr(&sel[k], 1u << (gi & 31));
        if (owned(k)) ks[slot_of(gi)] = 0u;
      }
      taken += nA;
      __syncthreads();
    }
  }
  __syncthreads();

  // ---- Eq. 12: ascending positions from the request's selected bits; every CTA
  // writes the indices and rows of its own blocks ----
  int2 *out = reinterpret_cast<int2 *>(smem + S.e);   // (token, position) of the kept tokens, over e and hi
  int *wsum = reinterpret_cast<int *>(misc);
  if (tid == 0) cnt[0] = 0;
  int run = 0;
  for (int v0 = 0; v0 < nblk; v0 += kGthreads) {
    const int v = v0 + tid;
    uint32_t bits = v < nblk ? sel[v] : 0u;
    if (v == nblk - 1 && (N & 31)) bits &= (1u << (N & 31)) - 1u;
    const int c = __popc(bits);
    int inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += n;
    }
    __syncthreads();
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    int before = run, tot = 0;
#pragma unroll
    for (int q = 0; q < kGwarps; ++q) {
      before += q < warp ? wsum[q] : 0;
      tot += wsum[q];
    }
    run += tot;
    if (v < nblk && v % C == rank && c > 0) {
      int pos = before + inc - c, at = atomicAdd(&cnt[0], c);
      while (bits) {
        const int t = 32 * v + __ffs(bits) - 1;
        bits &= bits - 1;
        a.idx_out[koff + pos] = t;
        out[at++] = make_int2(t, pos++);
      }
    }
  }
  if (a.x_out != nullptr) {
    __syncthreads();
    const int nvec = rb / 16, n = cnt[0];
    for (int r = warp; r < n; r += kGwarps) {
      const int2 tp = out[r];
      const char *src = xreq + (long long)tp.x * rb;
      char *dst = a.x_out + (long long)(koff + tp.y) * rb;
      for (int v = lane; v < nvec; v += 32)
        *reinterpret_cast<U4 *>(dst + 16 * v) = ldg_stream(src + 16 * v);
    }
  }
}

namespace {

template <typename T, int NCH>
void pick_nch(int nch, void **sel, void **norm) {
  if (nch == NCH) {
    if constexpr (sizeof(T) == 2) *sel = (void *)select_gram_kernel<NCH, false>;
    *norm = (void *)norms_kernel<T, NCH>;
  } else if constexpr (NCH > 1) {
    pick_nch<T, NCH - 1>(nch, sel, norm);
  }
}

struct SelShape {
  int C = 0, mc = 0, slots = 0, words = 0;
  size_t smem = 0;
};
// The shape of one request's cluster for clusters of c CTAs.
SelShape shape_for(int c, int max_vis, int optin) {
  SelShape s;
  s.C = c;
  s.mc = c == 1 ? 8 : c == 2 ? 6 : c <= 4 ? 4 : 3;
  const int nblk = (max_vis + 31) / 32;
  s.slots = (nblk + c * kGwork - 1) / (c * kGwork);
  s.words = nblk;
  s.smem = gram_sel_smem(s.slots, s.words, c, s.mc).total;
  if (s.smem > (size_t)optin || s.slots * kGtok > 0xffff) return SelShape();
  return s;
}

}  // namespace

bool gram_select_fits(int max_vis) {
  if (max_vis > 0xffff) return false;   // (token ids of 16 bits)
  for (int c = kMaxCluster; c >= 1; --c)
    if (shape_for(c, max_vis, kSmemOptinSm100).C != 0) return true;
  return false;
}

cudaError_t launch_select_gram(const Plan &pl, const float *w, const void *x, int32_t *idx_out,
                               void *x_out, char *ws, cudaStream_t s, bool *done) {
  *done = false;
  int dev = 0, optin = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int rb = pl.dv * pl.elem;
  void *sel_fn = nullptr, *norm_fn = nullptr;
  const bool f32 = pl.dtype == LAST_DTYPE_F32;
  if (f32) pick_nch<float, 8>((pl.dv + 255) / 256, &sel_fn, &norm_fn);
  else pick_nch<__nv_bfloat16, 8>((pl.dv + 255) / 256, &sel_fn, &norm_fn);
  if (pl.gram_exact) sel_fn = (void *)select_gram_kernel<1, true>;

  // The cluster size with the shortest schedule (about k / 16 + 2 rounds a request).
  // Clusters of two instead of one: 2.88 -> 2.52 ms on 128 requests of 256..4096.
  const int32_t *meta = pl.host_blob.data() + pl.off_meta / 4;
  const int32_t *order = pl.host_blob.data() + pl.off_order / 4;
  Schedule sched;
  schedule_begin(&sched, pl.B, [&](int i) {
    const int32_t *m = meta + order[i] * kMetaFields;
    return SchedRequest{(m[kNumVis] + 31) / 32, m[kNumKeep] / 16.0 + 2.0};
  });
  SelShape sh;
  double best = 0.0;
  for (int c = 1; c <= kMaxCluster; ++c) {
    const SelShape t = shape_for(c, pl.max_vis, optin);
    if (t.C == 0) continue;
    const int active = active_clusters(sel_fn, c, t.smem, kGthreads);
    if (active <= 0) continue;
    const double end = schedule_end(&sched, c, active, kGwork, sh.C == 0 ? INFINITY : best);
    if (sh.C == 0 || end < best) {
      sh = t;
      best = end;
    }
  }
  if (sh.C == 0 || !gram_select_fits(pl.max_vis)) return cudaSuccess;   // the caller's other paths

  GramArgs g;
  std::memset(&g, 0, sizeof g);
  if (!pl.gram_exact && !encode_x_map(&g.tmap, x, pl.total_vis, pl.dv)) return cudaSuccess;
  g.gram = reinterpret_cast<float *>(ws + pl.off_gram);
  g.meta = reinterpret_cast<const int32_t *>(ws + pl.off_meta);
  g.tile0 = reinterpret_cast<const int32_t *>(ws + pl.off_tile0);
  g.B = pl.B;
  g.dv = pl.dv;
  g.total_tiles = pl.gram_tiles;
  const bool pair = gram_long(pl.max_vis);
  const int chunk = gram_chunk(pl.max_vis);
  g.chunk_kb = chunk / kGK;
  g.err = reinterpret_cast<unsigned *>(ws + pl.off_err);
  float *rn = reinterpret_cast<float *>(ws + pl.off_rn);
  cudaError_t e = cudaSuccess;
  if (pl.gram_tiles > 0) {
    const char *xc = static_cast<const char *>(x);
    int dv = pl.dv, row = rb;
    long long total = pl.total_vis;
    void *nargs[] = {&xc, &rn, &dv, &row, &total};
    const int ngrid = (int)std::min<long long>((pl.total_vis + 7) / 8, (long long)sms * 8);
    if ((e = cudaLaunchKernel(norm_fn, dim3(ngrid), dim3(256), nargs, 0, s)) != cudaSuccess) return e;
    if (pl.gram_exact) {
      GramExactArgs x1 = {};
      x1.x = static_cast<const char *>(x);
      x1.gram = g.gram; x1.meta = g.meta; x1.tile0 = g.tile0;
      x1.B = pl.B; x1.dv = pl.dv; x1.row_bytes = rb;
      void *fn = f32 ? (void *)gram_exact_kernel<float> : (void *)gram_exact_kernel<__nv_bfloat16>;
      const int cols = f32 ? kExCols<float> : kExCols<__nv_bfloat16>;
      const size_t smem = (size_t)kExBufs * (kExRows + cols) * 256 * pl.elem;
      e = allow_smem(fn, smem);
      if (e != cudaSuccess) return e;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(pl.gram_tiles);
      cfg.blockDim = dim3(16 * cols);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = s;
      cudaLaunchAttribute attr[1];   // beside the norms' kernel, as below
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      void *args[] = {&x1};
      if ((e = cudaLaunchKernelExC(&cfg, fn, args)) != cudaSuccess) return e;
    } else {
      // the matrix needs no norms: its kernel starts beside the norms' and ends after them
      void *fn = pair ? (void *)gram_pair_kernel : (void *)gram_kernel;
      const size_t smem = 192 * 1024 + 1024;
      static_assert(kGramStages * kGramStageBytes == 192 * 1024 && kPairStages * kPairStageBytes == 192 * 1024,
                    "the ring of either kernel");
      e = allow_smem(fn, smem);
      if (e != cudaSuccess) return e;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(pair ? 2 * std::min(sms / 2, pl.gram_tiles) : std::min(sms, pl.gram_tiles));
      cfg.blockDim = dim3(kGramThreads);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = s;
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = pair ? 2 : 1;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[1].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 2;
      void *args[] = {&g};
      if ((e = cudaLaunchKernelExC(&cfg, fn, args)) != cudaSuccess) return e;
    }
  }
  GramSelArgs a;
  std::memset(&a, 0, sizeof a);
  a.x = static_cast<const char *>(x);
  a.w = w; a.rn = rn; a.gram = g.gram;
  a.idx_out = idx_out; a.x_out = static_cast<char *>(x_out);
  a.meta = g.meta;
  a.order = reinterpret_cast<const int32_t *>(ws + pl.off_order);
  a.dv = pl.dv; a.row_bytes = rb; a.csize = sh.C; a.mc = sh.mc; a.slots = sh.slots; a.words = sh.words;
  a.eps = pl.gram_exact ? 0.f : gram_distance_eps(pl.dv, chunk);
  a.err = g.err;
  e = cudaFuncSetAttribute(sel_fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = allow_smem(sel_fn, sh.smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sh.C * pl.B);
  cfg.blockDim = dim3(kGthreads);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = sh.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  // (behind the tensor-core kernels an early start cost 1% on long requests)
  cfg.numAttrs = pl.gram_exact ? 2 : 1;
  void *args[] = {&a};
  *done = true;
  return cudaLaunchKernelExC(&cfg, sel_fn, args);
}

}  // namespace last
