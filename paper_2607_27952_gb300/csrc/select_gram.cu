// Eq. 9-12 (Sec. 3.4): the greedy selection of bf16 features from a Gram matrix.
//
// Three launches.  norms_kernel: 1/|x_i| of every token (canonical order).
// gram_kernel: every request's dot products x_i . x_j on the tensor cores, fp32, to
// the workspace (lower triangle computed, mirrored on the way out).
// select_gram_kernel: the greedy, one thread-block cluster of C CTAs per request,
// in rounds that accept a batch of consecutive picks at once and give exactly the
// sequential Eq. 10-11 sequence:
//   1. every warp publishes its `mc` best live keys (w~_i delta_i, index) and its
//      (mc+1)-th key to every CTA of the cluster (DSMEM; one cluster barrier);
//   2. the published entries above U = the largest (mc+1)-th key form the candidate
//      list (at most kGlist; U rises to the first key cut off).  No token outside
//      the list has a key above U, and keys never increase;
//   3. the list's pairwise distances come from the Gram matrix, certified: a pair
//      whose tensor-core distance is at least eps above both members' delta cannot
//      matter; the others are evaluated in the canonical order;
//   4. the greedy is replayed on the list alone while its best key is above U;
//   5. the accepted centres' Gram rows are folded into the delta of the CTA's
//      tokens: a centre with d~ - eps >= delta_i cannot lower delta_i, every other
//      (token, centre) pair is evaluated in the canonical order.
// Every CTA of a cluster does steps 2-4 alike, so a round has one cluster barrier.
//
// Against the rounds that stream X (select_impl.cuh) a round reads 4 bytes per token
// and centre instead of a whole row per token, so its cost no longer grows with
// d_v, and the N^2 d_v contraction runs once, at tensor-core rates, on every SM.
//
// Measured against them (GB300, whole last_prune call): 64 requests of 576 x 2048,
// k 64/128/192: 1.71 -> 0.84 ms; 32 of 2880, k = 360: 5.27 -> 2.49; 128 of 256..4096 x
// 1536, k = N/8: 10.3 -> 6.0; 8 of 16384 x 2048, k = 2048: 16.9 -> 8.6.
//
// Tokens are dealt to the cluster in blocks of 32: block k belongs to CTA k % C,
// warp (k / C) % 16, so neighbouring tokens (tiles, frames, near-duplicates) spread
// over all warps and both the ranking and the exact pairs stay balanced.
//
// Arithmetic of every decision is the canonical fp32 of the public header: the kept
// indices are bit-identical to the sequential definition.
#include "select_impl.cuh"

#include <algorithm>
#include <cstring>

namespace last {

namespace {

constexpr int kGwarps = 16;
constexpr int kGthreads = kGwarps * 32;
constexpr int kGlist = 64;                 // candidate list: two members per lane of the replay
constexpr int kGper = kGlist / 32;
constexpr int kGmaxAccept = 64;            // one bit per accepted centre
constexpr int kGpairLd = kGlist + 1;
constexpr int kGcand = 1024;               // published entries above U kept before the cut

// ---- Gram tiles: 128 rows x 256 columns, the lower triangle of each request ----
constexpr int kGM = 128, kGN = 256, kGK = 64;
constexpr int kGramStages = 4;
constexpr int kGramStageBytes = (kGM + kGN) * kGK * 2;   // 48 KB
constexpr int kGramThreads = 192;          // 4 epilogue warps, TMA producer, MMA issuer
constexpr int kGroupRows = 16;             // row blocks per tile group (L2 reuse of both operands)

}  // namespace

// Tiles of a request with R row blocks, in groups of 16 row blocks: group g has 16
// rows of 8g full column blocks and a triangular part of 8 more.
__host__ __device__ inline int gram_group_tiles(int g, int h) {
  int n = h * 8 * g;
  for (int c = 0; 2 * c < h; ++c) n += h - 2 * c;
  return n;
}
int gram_tiles(int n_tokens) {
  const int R = (n_tokens + kGM - 1) / kGM;
  int n = 0;
  for (int g = 0; 16 * g < R; ++g) n += gram_group_tiles(g, std::min(kGroupRows, R - 16 * g));
  return n;
}

struct GramArgs {
  CUtensorMap tmap;        // X as [total_vis][dv] bf16, box 64 x 128, 128-byte swizzle
  float *gram;
  const int32_t *meta;
  const int32_t *tile0;    // [B + 1] first tile of each request
  int B, dv, total_tiles;
  unsigned *err;
};

__global__ void __launch_bounds__(kGramThreads, 1) gram_kernel(const __grid_constant__ GramArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  __shared__ unsigned long long full[kGramStages], empty[kGramStages], afull[2], aempty[2];
  __shared__ uint32_t tslot[2];   // TMEM base, abort word
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkb = tc_kblocks(a.dv);
  if (threadIdx.x == 0) {
    for (int i = 0; i < kGramStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&afull[i], 1);
      mbar_init(&aempty[i], 4);
    }
    tslot[1] = 0;
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc(&tslot[0], 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot[0];
  // after one expired wait every later wait returns at once and the call reports it
  auto twait = [&](unsigned long long *bar, uint32_t par) -> bool {
    volatile uint32_t *abort_w = &tslot[1];
    if (*abort_w) return false;
    if (mbar_wait_bounded(bar, par, a.err, kErrTimeout)) return true;
    *abort_w = 1u;
    return false;
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

  if (warp == 4) {
    if (lane == 0) {
      uint32_t it = 0;
      for (int tile = blockIdx.x; tile < a.total_tiles; tile += gridDim.x) {
        int b, ti, tj;
        decode(tile, &b, &ti, &tj);
        const int row0 = a.meta[b * kMetaFields + kVisOff];
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int st = it % kGramStages;
          if (it >= kGramStages && !twait(&empty[st], ((it / kGramStages) - 1) & 1)) continue;
          unsigned char *dst = smem + st * kGramStageBytes;
          mbar_expect_tx(&full[st], kGramStageBytes);
          tma_load_2d(dst, &a.tmap, kb * kGK, row0 + ti * kGM, &full[st]);
          tma_load_2d(dst + kGM * kGK * 2, &a.tmap, kb * kGK, row0 + tj * kGN, &full[st]);
          tma_load_2d(dst + 2 * kGM * kGK * 2, &a.tmap, kb * kGK, row0 + tj * kGN + 128, &full[st]);
        }
      }
      // an aborted call: the last copies still land before the CTA may exit
      if (*reinterpret_cast<volatile uint32_t *>(&tslot[1]))
        for (uint32_t k = it > kGramStages ? it - kGramStages : 0; k < it; ++k)
          mbar_wait_bounded(&full[k % kGramStages], (k / kGramStages) & 1, a.err, kErrTimeout);
    }
  } else if (warp == 5) {
    if (lane == 0) {
      const uint32_t idesc = umma_idesc_bf16(kGM, kGN);
      uint32_t it = 0, nt = 0;
      for (int tile = blockIdx.x; tile < a.total_tiles; tile += gridDim.x, ++nt) {
        const int ab = nt & 1;
        if (nt >= 2) twait(&aempty[ab], ((nt >> 1) - 1) & 1);
        tc_fence_after();
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int st = it % kGramStages;
          const bool ok = twait(&full[st], (it / kGramStages) & 1);
          tc_fence_after();
          if (ok) {
            const uint32_t sa = smem_addr(smem + st * kGramStageBytes);
#pragma unroll
            for (int k = 0; k < kGK / 16; ++k)
              umma_bf16(tmem + ab * kGN, umma_desc_sw128(sa + k * 32),
                        umma_desc_sw128(sa + kGM * kGK * 2 + k * 32), idesc, (kb | k) != 0 ? 1u : 0u);
          }
          umma_commit(&empty[st]);
        }
        umma_commit(&afull[ab]);
      }
    }
  } else {
    uint32_t nt = 0;
    for (int tile = blockIdx.x; tile < a.total_tiles; tile += gridDim.x, ++nt) {
      const int ab = nt & 1;
      int b, ti, tj;
      decode(tile, &b, &ti, &tj);
      const int32_t *m = a.meta + b * kMetaFields;
      const int N = m[kNumVis], ld = gram_ld(N);
      float *G = a.gram + (long long)m[kGramOff] * 32;
      twait(&afull[ab], (nt >> 1) & 1);
      __syncwarp();
      tc_fence_after();
      const int i = ti * kGM + 32 * warp + lane;
      const uint32_t tb = tmem + ab * kGN + ((uint32_t)(32 * warp) << 16);
      for (int c0 = 0; c0 < kGN; c0 += 32) {
        const int j0 = tj * kGN + c0;
        if (j0 >= N) break;
        uint32_t v[32];
        tmem_ld32(tb + c0, v);
        if (i < N) {
          float *row = G + (long long)i * ld + j0;
#pragma unroll
          for (int q = 0; q < 32; q += 8) st_global_v8(row + q, v + q);
        }
        // the transposed 128 x 128 block, unless a tile of its own computes it
        if (j0 / kGM < 2 * (ti / 2) && i < ld) {
          float *col = G + (long long)j0 * ld + i;
#pragma unroll
          for (int q = 0; q < 32; ++q)
            if (j0 + q < N) col[(long long)q * ld] = __uint_as_float(v[q]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&aempty[ab]);
    }
  }
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// 1/|x_i| in the canonical order, one warp per token.
template <typename T, int NCH>
__global__ void __launch_bounds__(256) norms_kernel(const char *x, float *rn, int dv, int row_bytes,
                                                    long long total) {
  const int lane = threadIdx.x & 31;
  const long long nw = (long long)gridDim.x * 8;
  for (long long t = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); t < total; t += nw) {
    const char *row = x + t * row_bytes;
    const float ss = dot_rows<T, NCH>(row, false, row, false, dv, lane);
    if (lane == 0) rn[t] = ss > 0.f ? __fdiv_rn(1.0f, __fsqrt_rn(ss)) : 0.f;
  }
}

struct GramSelArgs {
  const char *x;
  const float *w, *rn, *gram;
  int32_t *idx_out;
  char *x_out;             // nullable
  const int32_t *meta, *order;
  int dv, row_bytes, csize, mc, slots, words, accept;
  float eps;
  unsigned *err;
};

// Shared memory of select_gram_kernel (host sizing and device carve-up alike).
struct GramSelSmem {
  size_t rows, w, r, dl, fmask, fidx, sel, pub, cand, pm, plist, key, lidx, ld, lw, lr, acc, misc, bar, total;
};
__host__ __device__ inline GramSelSmem gram_sel_smem(int accept, int row_bytes, int slots, int words,
                                                     int csize, int mc) {
  GramSelSmem s;
  size_t o = 0;
  const size_t cap = (size_t)slots * kGthreads;   // token slots of a CTA
  s.rows = o; o += (size_t)accept * row_bytes;    // the round's accepted centres
  s.w = o; o += 4 * cap;
  s.r = o; o += 4 * cap;
  s.dl = o; o += 4 * cap;
  s.fmask = o; o += 8 * cap;                      // flagged tokens: centres to evaluate
  s.fidx = o; o += align16(2 * cap);
  s.sel = o; o += align16(4 * (size_t)words);     // selected bits of the whole request
  s.pub = o; o += (size_t)2 * kGwarps * csize * (mc + 1) * 16;
  s.cand = o; o += 2 * kGcand;
  s.pm = o; o += align16(4 * kGlist * kGpairLd);  // pair dots of the list
  s.plist = o; o += 2 * kGlist * kGlist / 2;
  s.key = o; o += 8 * kGlist;
  s.lidx = o; o += 4 * kGlist;
  s.ld = o; o += 4 * kGlist;
  s.lw = o; o += 4 * kGlist;
  s.lr = o; o += 4 * kGlist;
  s.acc = o; o += 4 * kGmaxAccept;
  s.misc = o; o += 8 * 40;
  s.bar = o; o += 16;
  s.total = align16(o);
  return s;
}

template <int NCH>
__global__ void __launch_bounds__(kGthreads, 1)
select_gram_kernel(const __grid_constant__ GramSelArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int C = a.csize, rank = (int)cluster_ctarank();
  const int b = a.order[cluster_id_x()];
  const int32_t *m = a.meta + b * kMetaFields;
  const int voff = m[kVisOff], N = m[kNumVis], koff = m[kKeepOff], K = m[kNumKeep];
  if (K == 0) return;   // the whole cluster leaves together
  const GramSelSmem S = gram_sel_smem(a.accept, a.row_bytes, a.slots, a.words, C, a.mc);
  {
    uint32_t dyn;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
    if (S.total > dyn) {   // host and device plans disagree: every CTA leaves before any barrier
      if (tid == 0) atomicOr(a.err, kErrConfig);
      return;
    }
  }
  char *rows = reinterpret_cast<char *>(smem + S.rows);
  float *w_s = reinterpret_cast<float *>(smem + S.w);
  float *r_s = reinterpret_cast<float *>(smem + S.r);
  float *dl_s = reinterpret_cast<float *>(smem + S.dl);
  unsigned long long *fmask = reinterpret_cast<unsigned long long *>(smem + S.fmask);
  uint16_t *fidx = reinterpret_cast<uint16_t *>(smem + S.fidx);
  uint32_t *sel = reinterpret_cast<uint32_t *>(smem + S.sel);
  uint4 *pub = reinterpret_cast<uint4 *>(smem + S.pub);
  uint16_t *cand = reinterpret_cast<uint16_t *>(smem + S.cand);
  float *pm = reinterpret_cast<float *>(smem + S.pm);
  uint16_t *plist = reinterpret_cast<uint16_t *>(smem + S.plist);
  unsigned long long *lkey = reinterpret_cast<unsigned long long *>(smem + S.key);
  int *lidx = reinterpret_cast<int *>(smem + S.lidx);
  float *ldl = reinterpret_cast<float *>(smem + S.ld);
  float *lw = reinterpret_cast<float *>(smem + S.lw);
  float *lr = reinterpret_cast<float *>(smem + S.lr);
  int *acc_s = reinterpret_cast<int *>(smem + S.acc);
  unsigned long long *misc = reinterpret_cast<unsigned long long *>(smem + S.misc);
  int *cnt = reinterpret_cast<int *>(misc + 32);   // [0] flagged tokens, [1] candidates, [2] pairs, [3] list, [4] picks
  unsigned long long *bar = reinterpret_cast<unsigned long long *>(smem + S.bar);

  const int rb = a.row_bytes, dv = a.dv, ld = gram_ld(N);
  const int nblk = (N + 31) >> 5;
  const char *xreq = a.x + (long long)voff * rb;
  const float *rreq = a.rn + voff, *wreq = a.w + voff;
  const float *G = a.gram + (long long)m[kGramOff] * 32;
  const int P = kGwarps * C;                          // publishing warps of the cluster
  const int step = C * kGwarps;                       // blocks between a warp's slots
  const int blk0 = rank + C * warp;                   // this warp's first block

  if (tid == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  for (int v = tid; v < nblk; v += kGthreads) sel[v] = K == N ? 0xffffffffu : 0u;
  for (int s = 0, k = blk0; k < nblk; ++s, k += step) {
    const int t = 32 * k + lane, li = s * kGthreads + tid;
    const bool in = t < N;
    w_s[li] = in ? wreq[t] : 0.f;
    r_s[li] = in ? rreq[t] : 0.f;
    dl_s[li] = INFINITY;
  }
  uint32_t phase = 0;

  if (K < N) {
    auto csync = [&]() {
      if (C == 1) __syncthreads();
      else cluster_sync();
    };
    // 8 coordinates per lane of chunk g of a row
    auto load_row = [&](const char *row, U4 *v) {
#pragma unroll
      for (int g = 0; g < NCH; ++g) {
        const int col = 256 * g + 8 * lane;
        v[g] = col < dv ? ldg_nc(row + col * 2) : U4{0, 0, 0, 0};
      }
    };
    auto fma8 = [&](const U4 &x, const U4 &c, float acc) {
      const uint32_t xw[4] = {x.x, x.y, x.z, x.w}, cw[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        acc = fma_bf16_lo(xw[h], cw[h], acc);
        acc = fma_bf16_hi(xw[h], cw[h], acc);
      }
      return acc;
    };
    const uint32_t rows_sa = smem_addr(rows);

    // Fold the nA accepted centres lidx[acc_s[j]] into the tokens' delta.
    auto update = [&](int nA, bool seed) {
      // the centres' rows into shared memory (one bulk copy each)
      if (warp == 0) {
        if (lane == 0) mbar_expect_tx(bar, (uint32_t)(nA * rb));
        __syncwarp();
        for (int j = lane; j < nA; j += 32)
          bulk_g2s(rows + (long long)j * rb, xreq + (long long)lidx[acc_s[j]] * rb, (uint32_t)rb, bar);
      }
      if (tid == 0) cnt[0] = 0;
      __syncthreads();
      for (int s = 0, k = blk0; k < nblk; ++s, k += step) {
        const int t = 32 * k + lane, li = s * kGthreads + tid;
        const bool live = t < N && !((sel[k] >> lane) & 1u);
        unsigned long long msk = 0ull;
        const float ri = r_s[li], dl = dl_s[li];
        const bool in_range = tri_in_range(ri);
        if (seed) {
          msk = 1ull;
        } else {
          for (int j0 = 0; j0 < nA; j0 += 8) {
            float g[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int c = lidx[acc_s[min(j0 + j, nA - 1)]];
              g[j] = live ? ldg_f32_stream(G + (long long)c * ld + t) : 0.f;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if (j0 + j < nA) {
                const float rc = lr[acc_s[j0 + j]];
                const float d = __fsub_rn(1.0f, __fmul_rn(__fmul_rn(g[j], ri), rc));
                // NaN and rows outside the certificate's norm range go to the exact path
                if (!(__fsub_rn(d, a.eps) >= dl) || !in_range || !tri_in_range(rc)) msk |= 1ull << (j0 + j);
              }
            }
          }
        }
        if (!live) msk = 0ull;
        const unsigned bal = __ballot_sync(0xffffffffu, msk != 0ull);
        if (bal) {
          int base = 0;
          if (lane == 0) base = atomicAdd(&cnt[0], __popc(bal));
          base = __shfl_sync(0xffffffffu, base, 0);
          if (msk) {
            const int pos = base + __popc(bal & ((1u << lane) - 1u));
            fidx[pos] = (uint16_t)li;
            fmask[pos] = msk;
          }
        }
      }
      mbar_wait_bounded(bar, phase, a.err, kErrTimeout);
      phase ^= 1u;
      __syncthreads();
      // exact canonical distances of the flagged pairs, a warp per token; the next
      // token's row is in flight while the current one is evaluated
      const int nf = cnt[0];
      auto row_of = [&](int f) {
        const int li = fidx[f];
        const int k = rank + C * ((li >> 5) % kGwarps) + (li / kGthreads) * step;
        return xreq + (long long)(32 * k + (li & 31)) * rb;
      };
      auto exact_token = [&](int f, const U4 *xv) {
        const int li = fidx[f];
        unsigned long long msk = fmask[f];
        const float ri = r_s[li];
        float dl = dl_s[li];
        while (msk) {
          const int j = __ffsll(msk) - 1;
          msk &= msk - 1;
          const uint32_t cr = rows_sa + (uint32_t)(j * rb);
          float acc = 0.f;
#pragma unroll
          for (int g = 0; g < NCH; ++g) {
            const int col = 256 * g + 8 * lane;
            if (col < dv) acc = fma8(xv[g], lds32(cr + col * 2), acc);
          }
          const float dot = butterfly_sum(acc);
          dl = fminf(dl, __fsub_rn(1.0f, __fmul_rn(__fmul_rn(dot, ri), lr[acc_s[j]])));
        }
        if (lane == 0) dl_s[li] = dl;
      };
      {
        U4 xa[NCH], xb[NCH];
        int f = warp;
        if (f < nf) load_row(row_of(f), xa);
        while (f < nf) {
          if (f + kGwarps < nf) load_row(row_of(f + kGwarps), xb);
          exact_token(f, xa);
          f += kGwarps;
          if (f >= nf) break;
          if (f + kGwarps < nf) load_row(row_of(f + kGwarps), xa);
          exact_token(f, xb);
          f += kGwarps;
        }
      }
      __syncthreads();
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
        lidx[0] = seed;
        lr[0] = rreq[seed];
        acc_s[0] = 0;
        sel[seed >> 5] |= 1u << (seed & 31);
      }
      __syncthreads();
    }
    int taken = 1;
    if (taken < K) update(1, true);

    csync();   // every CTA of the cluster runs before the first remote write
    // ---- rounds (Eq. 10-11) ----
    const int ent = a.mc + 1;
    for (int round = 0; taken < K; ++round) {
      const int par = round & 1;
      uint4 *pubp = pub + (size_t)par * P * ent;
      // 1. this warp's best live keys, best first: {index, delta, w~, 1/|x|}
      {
        unsigned long long limit = ~0ull, mine;
        int ms = 0;
        auto best_below = [&]() {
          unsigned long long bk = 0ull;
          for (int s = 0, k = blk0; k < nblk; ++s, k += step) {
            const int t = 32 * k + lane, li = s * kGthreads + tid;
            if (t < N && !((sel[k] >> lane) & 1u)) {
              const unsigned long long kk = argmax_key(__fmul_rn(w_s[li], dl_s[li]), t);
              if (kk < limit && kk > bk) {
                bk = kk;
                ms = s;
              }
            }
          }
          return bk;
        };
        mine = best_below();
        for (int e = 0; e < ent; ++e) {
          const unsigned long long best = warp_max_u64(mine);
          uint4 v = make_uint4(0xffffffffu, 0u, 0u, 0u);   // no token left
          if (best != 0ull) {
            const int src = __ffs(__ballot_sync(0xffffffffu, mine == best)) - 1;
            const int li = __shfl_sync(0xffffffffu, ms, src) * kGthreads + warp * 32 + src;
            v = make_uint4((uint32_t)key_index(best), __float_as_uint(dl_s[li]), __float_as_uint(w_s[li]),
                           __float_as_uint(r_s[li]));
            if (lane == src) {
              limit = best;
              mine = best_below();
            }
          }
          if (lane < C)
            st_cluster_v4u(map_shared(&pubp[(rank * kGwarps + warp) * ent + e], lane), v);
        }
      }
      if (tid == 0) {
        cnt[1] = 0;
        cnt[2] = 0;
        cnt[3] = 0;
      }
      csync();
      // 2. the list: published entries above U
      auto entry_key = [&](const uint4 &v) {
        return v.x == 0xffffffffu
                   ? 0ull
                   : argmax_key(__fmul_rn(__uint_as_float(v.z), __uint_as_float(v.y)), (int)v.x);
      };
      unsigned long long U = 0ull;
      for (int q = lane; q < P; q += 32) U = max(U, entry_key(pubp[q * ent + a.mc]));
      U = warp_max_u64(U);
      for (int e0 = warp * 32; e0 < P * ent; e0 += kGthreads) {
        const int e = e0 + lane;
        const bool up = e < P * ent && entry_key(pubp[e]) > U;
        const unsigned bal = __ballot_sync(0xffffffffu, up);
        if (bal) {
          int base = 0;
          if (lane == 0) base = atomicAdd(&cnt[1], __popc(bal));
          base = __shfl_sync(0xffffffffu, base, 0);
          if (up) cand[base + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)e;
        }
      }
      __syncthreads();
      const int nc = cnt[1];
      // the best kGlist of them; U' = the first key cut off
      if (warp * 32 < nc) {
        for (int c0 = warp * 32; c0 < nc; c0 += kGthreads) {
          const int c = c0 + lane;
          const uint4 v = c < nc ? pubp[cand[c]] : make_uint4(0xffffffffu, 0u, 0u, 0u);
          const unsigned long long kk = entry_key(v);
          int pos = c;
          if (nc > kGlist) {
            pos = 0;
            for (int q = 0; q < nc; ++q) pos += entry_key(pubp[cand[q]]) > kk ? 1 : 0;
          }
          if (c < nc) {
            if (pos < kGlist) {
              lkey[pos] = kk;
              lidx[pos] = (int)v.x;
              ldl[pos] = __uint_as_float(v.y);
              lw[pos] = __uint_as_float(v.z);
              lr[pos] = __uint_as_float(v.w);
            } else if (pos == kGlist) {
              misc[20] = kk;
            }
          }
        }
      }
      __syncthreads();
      const int nL = min(nc, kGlist);
      const unsigned long long Up = nc > kGlist ? misc[20] : U;
      // the list's Gram rows for this CTA's tokens start towards L2
      for (int k = blk0; k < nblk; k += step)
        for (int u = lane; u < nL; u += 32) prefetch_l2(G + (long long)lidx[u] * ld + 32 * k);
      // 3. pair dots: -inf (distance +inf) where the certificate excludes the pair
      for (int u = warp; u < nL; u += kGwarps) {
        const int iu = lidx[u];
        const float ru = lr[u], du = ldl[u];
        const bool cu = tri_in_range(ru);
#pragma unroll
        for (int h = 0; h < kGper; ++h) {
          const int v = lane + 32 * h;
          bool need = false;
          if (v > u && v < nL) {
            const float g = ldg_f32_stream(G + (long long)iu * ld + lidx[v]);
            const float rv = lr[v];
            const float d = __fsub_rn(1.0f, __fmul_rn(__fmul_rn(g, ru), rv));
            need = !cu || !tri_in_range(rv) || !(__fsub_rn(d, a.eps) >= fmaxf(du, ldl[v]));
            if (!need) pm[u * kGpairLd + v] = pm[v * kGpairLd + u] = -INFINITY;
          }
          const unsigned bal = __ballot_sync(0xffffffffu, need);
          if (bal) {
            int base = 0;
            if (lane == 0) base = atomicAdd(&cnt[2], __popc(bal));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (need) plist[base + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(u * kGlist + v);
          }
        }
      }
      __syncthreads();
      const int np = cnt[2];
      for (int p = warp; p < np; p += kGwarps) {
        const int u = plist[p] / kGlist, v = plist[p] % kGlist;
        U4 xu[NCH], xv[NCH];
        load_row(xreq + (long long)lidx[u] * rb, xu);
        load_row(xreq + (long long)lidx[v] * rb, xv);
        float acc = 0.f;
#pragma unroll
        for (int g = 0; g < NCH; ++g)
          if (256 * g + 8 * lane < dv) acc = fma8(xu[g], xv[g], acc);
        const float dot = butterfly_sum(acc);
        if (lane == 0) pm[u * kGpairLd + v] = pm[v * kGpairLd + u] = dot;
      }
      __syncthreads();
      // 4. replay the greedy on the list (warp 0; lane u holds members u, u + 32)
      if (warp == 0) {
        unsigned long long key[kGper];
        float cd[kGper], wv[kGper], rv[kGper];
        int gi[kGper];
#pragma unroll
        for (int h = 0; h < kGper; ++h) {
          const int u = lane + 32 * h;
          const bool in = u < nL;
          key[h] = in ? lkey[u] : 0ull;
          cd[h] = in ? ldl[u] : 0.f;
          wv[h] = in ? lw[u] : 0.f;
          rv[h] = in ? lr[u] : 0.f;
          gi[h] = in ? lidx[u] : 0;
        }
        int nA = 0;
        while (taken + nA < K && nA < a.accept) {
          unsigned long long lk = key[0];
          int lh = 0;
#pragma unroll
          for (int h = 1; h < kGper; ++h)
            if (key[h] > lk) {
              lk = key[h];
              lh = h;
            }
          const unsigned long long bk = warp_max_u64(lk);
          if (bk <= Up) break;   // also the end of the list (key 0)
          const int src = __ffs(__ballot_sync(0xffffffffu, lk == bk)) - 1;
          const int bl = src + 32 * __shfl_sync(0xffffffffu, lh, src);
          if (lane == 0) acc_s[nA] = bl;
          ++nA;
          const float rbv = lr[bl];
#pragma unroll
          for (int h = 0; h < kGper; ++h) {
            const int u = lane + 32 * h;
            if (u == bl) key[h] = 0ull;
            if (key[h] != 0ull) {
              cd[h] = fminf(cd[h], __fsub_rn(1.0f, __fmul_rn(__fmul_rn(pm[bl * kGpairLd + u], rv[h]), rbv)));
              key[h] = argmax_key(__fmul_rn(wv[h], cd[h]), gi[h]);
            }
          }
        }
        if (lane == 0) cnt[4] = nA;
      }
      __syncthreads();
      const int nA = cnt[4];
      if (nA == 0) {   // cannot happen (the best live key is above U): leave rather than loop
        if (tid == 0) atomicOr(a.err, kErrConfig);
        break;
      }
      if (tid < nA) {
        const int gi = lidx[acc_s[tid]];
        atomicOr(&sel[gi >> 5], 1u << (gi & 31));
      }
      taken += nA;
      __syncthreads();
      // 5. update
      if (taken < K) update(nA, false);
    }
  }
  __syncthreads();

  // ---- Eq. 12: ascending positions from the request's selected bits; every CTA
  // writes the indices and rows of its own blocks ----
  int2 *out = reinterpret_cast<int2 *>(smem + S.fmask);   // (token, position) of the kept tokens
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

template <int NCH>
void pick_nch(int nch, void **sel, void **norm) {
  if (nch == NCH) {
    *sel = (void *)select_gram_kernel<NCH>;
    *norm = (void *)norms_kernel<__nv_bfloat16, NCH>;
  } else if constexpr (NCH > 1) {
    pick_nch<NCH - 1>(nch, sel, norm);
  }
}

struct SelShape {
  int C = 0, mc = 0, slots = 0, words = 0, accept = 0;
  size_t smem = 0;
};
// The shape of one request's cluster for clusters of c CTAs.
SelShape shape_for(int c, int max_vis, int rb, int optin) {
  SelShape s;
  s.C = c;
  s.mc = c == 1 ? 8 : c == 2 ? 6 : c <= 4 ? 4 : 3;
  const int nblk = (max_vis + 31) / 32;
  s.slots = (nblk + c * kGwarps - 1) / (c * kGwarps);
  s.words = nblk;
  const size_t fixed = gram_sel_smem(0, rb, s.slots, s.words, c, s.mc).total;
  if (fixed + 8 * (size_t)rb > (size_t)optin || s.slots * kGthreads > 65536) return SelShape();
  s.accept = (int)std::min<size_t>(kGmaxAccept, (optin - fixed) / rb);
  s.smem = gram_sel_smem(s.accept, rb, s.slots, s.words, c, s.mc).total;
  return s;
}

}  // namespace

cudaError_t launch_select_gram(const Plan &pl, const float *w, const void *x, int32_t *idx_out,
                               void *x_out, char *ws, cudaStream_t s, bool *done) {
  *done = false;
  int dev = 0, optin = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int rb = pl.dv * pl.elem;
  void *sel_fn = nullptr, *norm_fn = nullptr;
  pick_nch<8>((pl.dv + 255) / 256, &sel_fn, &norm_fn);

  // The largest clusters that still run every request at once, but no more CTAs than
  // give each warp a block of tokens; when none does, the smallest that fits.
  SelShape sh;
  const int cmax = std::min(kMaxCluster, std::max(1, (pl.max_vis + kGthreads - 1) / kGthreads));
  for (int c = cmax; c >= 1; --c) {
    const SelShape t = shape_for(c, pl.max_vis, rb, optin);
    if (t.C == 0) continue;
    const int active = active_clusters(sel_fn, c, t.smem, kGthreads);
    if (active <= 0) continue;
    sh = t;
    if (active >= pl.B) break;
  }
  if (sh.C == 0) return cudaSuccess;   // too long for a cluster: the caller's other paths

  GramArgs g;
  std::memset(&g, 0, sizeof g);
  if (!encode_x_map(&g.tmap, x, pl.total_vis, pl.dv)) return cudaSuccess;
  g.gram = reinterpret_cast<float *>(ws + pl.off_gram);
  g.meta = reinterpret_cast<const int32_t *>(ws + pl.off_meta);
  g.tile0 = reinterpret_cast<const int32_t *>(ws + pl.off_tile0);
  g.B = pl.B;
  g.dv = pl.dv;
  g.total_tiles = pl.gram_tiles;
  g.err = reinterpret_cast<unsigned *>(ws + pl.off_err);
  float *rn = reinterpret_cast<float *>(ws + pl.off_rn);
  cudaError_t e;
  {
    const char *xc = static_cast<const char *>(x);
    int dv = pl.dv, row = rb;
    long long total = pl.total_vis;
    void *args[] = {&xc, &rn, &dv, &row, &total};
    const int grid = (int)std::min<long long>((pl.total_vis + 7) / 8, (long long)sms * 8);
    if ((e = cudaLaunchKernel(norm_fn, dim3(grid), dim3(256), args, 0, s)) != cudaSuccess) return e;
  }
  if (pl.gram_tiles > 0) {
    const size_t smem = (size_t)kGramStages * kGramStageBytes + 1024;
    e = cudaFuncSetAttribute(gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    gram_kernel<<<std::min(sms, pl.gram_tiles), kGramThreads, smem, s>>>(g);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  GramSelArgs a;
  std::memset(&a, 0, sizeof a);
  a.x = static_cast<const char *>(x);
  a.w = w; a.rn = rn; a.gram = g.gram;
  a.idx_out = idx_out; a.x_out = static_cast<char *>(x_out);
  a.meta = g.meta;
  a.order = reinterpret_cast<const int32_t *>(ws + pl.off_order);
  a.dv = pl.dv; a.row_bytes = rb; a.csize = sh.C; a.mc = sh.mc; a.slots = sh.slots; a.words = sh.words;
  a.accept = sh.accept;
  a.eps = tc_distance_eps(pl.dv);
  a.err = g.err;
  e = cudaFuncSetAttribute(sel_fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(sel_fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh.smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sh.C * pl.B);
  cfg.blockDim = dim3(kGthreads);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = sh.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void *args[] = {&a};
  *done = true;
  return cudaLaunchKernelExC(&cfg, sel_fn, args);
}

}  // namespace last
