// Table 4 (attention sources): the importance of Eq. 7 from the attention rows of
// several query positions per request (First, Middle, All Mean), bf16 q and K.
//
// Request b has M_b query rows at positions row_pos (after its visual span); row m
// sees the keys 0 .. row_pos[m] (causal softmax, Eq. 6).  Scores are summed over
// rows, layers and q-heads at the visual positions and normalised (Eq. 8).  A
// "column" is one (row, q-head of kv-head g) pair: G = Hq / Hkv columns per row.
//
// Four launches, all deterministic (fixed reduction orders, no float atomics).  The two
// passes over K are one persistent kernel each (rows_pass_kernel): a TMA thread streams
// (request, 128-key chunk, layer, kv-head) items, the keys' and the query columns' tiles
// together, through a ring of stages; one thread issues tcgen05.mma with the keys as M
// and the columns as N (bf16, fp32 accumulators in TMEM, one buffer per epilogue group);
// groups of four warps take the finished items in turn, thread = key.
// pass 1: per column the chunk's masked max of the logits (log2 domain) and the sums of
//   2^(z - max) over all and over the visual keys (Eq. 6's softmax statistics), reduced
//   over a warp's 32 keys for 32 columns at once (31 exchanges instead of 160) and over
//   the group's four warps through shared memory;
// rows_merge_kernel (request, 32 columns): the chunk statistics of each column into
//   (max, 1/Z) and the columns' visual probability mass;
// pass 2 (visual chunks): per key the probabilities 2^(z - max) / Z summed over the
//   columns (every column sees every visual key);
// rows_final_kernel (request, 256 visual tokens): adds the (layer, kv-head)
//   partial sums and divides by the visual mass (Eq. 7-8).
// Every chunk's sums are formed against the chunk's maximum and scaled once, against the
// column's maximum over all chunks, in the merge: rescaling the warps' sums and a running
// sum cost a quarter of the precision (64 bits: 9.2e-8 against 7.4e-8 on 8 of 16384) and
// time (140 and 162 us against the 121 and 130 below).
// The passes are bound by K's bytes and by the exponentials and exchanges of pass 1.
// One CTA per item, staging by its own loads, spent 19 us of latency on each: 64 requests
// of 576 tokens and 32 rows 369 us, 8 of 16384 456 us for the whole call; now 121 us (K
// read twice at the copy rate is 52) and 130 us.
#include "last_device.cuh"
#include "last_internal.h"
#include "tensor_map.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

namespace last {

namespace {

// Per-request metadata (int32 slots; the 64-bit statistics offset takes two slots
// and sits 8-byte aligned since a row is 12 slots).
enum RowsField : int {
  kRSeqStart = 0, kRSeqLen, kRVisStart, kRVisOff, kRNumVis, kRRowOff, kRNumRows,
  kRNumChunks, kRStatBase = 8, kRCoefBase = 10, kRowsFields = 12
};

constexpr int kRowsChunk = 128;     // keys per item
constexpr int kRowsMaxN = 256;      // columns (rows x G) per request
constexpr int kRowsMaxRH = 6144;    // (row, layer, q-head) triples per request

constexpr int kRowsGroups = 4;      // epilogue groups of four warps (two when npad > 128)
constexpr int kPassThreads = 32 * (4 * kRowsGroups + 2);
constexpr int kRowsMaxStages = 8;

struct RowsArgs {
  CUtensorMap kmap;      // K as [L * total_keys][Hkv * D], box 64 x 128, 128-byte swizzle
  CUtensorMap qmap;      // q as [rows][L * Hq][D], box 64 x G x qbox
  const int32_t *meta;
  const int2 *items1, *items2;
  const int32_t *row_pos;
  float4 *stats;         // per request [chunk][row, layer, head]: max, sum, visual sum
  float2 *coef;          // per (row, layer, head): max, 1 / Z
  float *mass;           // per request and block of 32 such triples: visual mass
  float *partial;        // [L][Hkv][total_vis] probability sums
  float *w;
  long long total_keys, total_vis;
  int L, Hq, Hkv, D, G, npad, qbox, n_items, nstage, ngroup, mass_blocks;
  uint32_t tmem_cols;    // TMEM columns of one group's accumulator
  float qscale;          // softmax scale * log2(e)
  unsigned *err;
};

__device__ __forceinline__ long long stat_base(const int32_t *m) {
  return *reinterpret_cast<const long long *>(m + kRStatBase);
}

// 32 values per lane, one per column, reduced over the warp's lanes: lane c ends with
// column c.  At each step a lane keeps the half of the columns its bit selects.
template <typename F>
__device__ __forceinline__ float warp_columns(float *v, int lane, F op) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int q = 0; q < o; ++q) {
      const float send = (lane & o) ? v[q] : v[q + o];
      const float keep = (lane & o) ? v[q + o] : v[q];
      v[q] = op(keep, __shfl_xor_sync(0xffffffffu, send, o));
    }
  return v[0];
}

}  // namespace

template <bool STATS>
__global__ void __launch_bounds__(kPassThreads, 1) rows_pass_kernel(const __grid_constant__ RowsArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  __shared__ unsigned long long full[kRowsMaxStages], empty[kRowsMaxStages];
  __shared__ unsigned long long afull[kRowsGroups], aempty[kRowsGroups], never;
  __shared__ uint32_t tslot;
  __shared__ volatile int gave_up;   // a role's wait has expired
  __shared__ float2 part[kRowsGroups][4][32];   // pass 1: the warps' sums of 32 columns
  __shared__ float2 cf[kRowsGroups][kRowsMaxN]; // pass 2: the item's (max, 1 / Z)
  // pass 1: the warps' column maxima, and the chunk's as each warp uses them
  __shared__ float wmax[kRowsGroups * 4][32], cmax[kRowsGroups * 4][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkb = a.D / 64, ngroup = a.ngroup;
  const int kbytes = nkb * kRowsChunk * 128, qbytes = nkb * a.npad * 128, stage_bytes = kbytes + qbytes;
  if (threadIdx.x == 0) {
    for (int i = 0; i < a.nstage; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < ngroup; ++i) {
      mbar_init(&afull[i], 1);
      mbar_init(&aempty[i], 4);
    }
    mbar_init(&never, 1);
    fence_mbar_init();
    gave_up = 0;
  }
  const uint32_t tmem_total = a.tmem_cols * (uint32_t)ngroup;
  if (warp == 0) tmem_alloc(&tslot, tmem_total);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot;
  bool dead = false;   // after one expired wait a role's others return at once
  auto twait = [&](unsigned long long *bar, uint32_t par) -> bool {
    if (!dead && !mbar_wait_bounded(bar, par, a.err, kErrTimeout)) {
      dead = true;
      gave_up = 1;
    }
    return !dead;
  };
  const int2 *items = STATS ? a.items1 : a.items2;
  // item -> (request, chunk), layer, kv-head; heads fastest, so that CTAs running side by
  // side read neighbouring bytes of the same keys
  auto decode = [&](int item, int *b, int *c, int *l, int *g) {
    const int hl = a.Hkv * a.L, it = item / hl, r = item - it * hl;
    const int2 v = items[it];
    *b = v.x;
    *c = v.y;
    *l = r / a.Hkv;
    *g = r - *l * a.Hkv;
  };

  if (warp == 4 * kRowsGroups) {
    if (lane == 0) {
      int st = 0;
      uint32_t ph = 1;
      for (int item = blockIdx.x; item < a.n_items; item += gridDim.x) {
        int b, c, l, g;
        decode(item, &b, &c, &l, &g);
        const int32_t *m = a.meta + b * kRowsFields;
        const int key0 = (int)((long long)l * a.total_keys) + m[kRSeqStart] + c * kRowsChunk;
        if (!twait(&empty[st], ph)) break;
        unsigned char *dst = smem + (size_t)st * stage_bytes;
        mbar_expect_tx(&full[st], (uint32_t)(kbytes + nkb * a.G * a.qbox * 128));
        for (int kb = 0; kb < nkb; ++kb) {
          tma_load_2d(dst + kb * kRowsChunk * 128, &a.kmap, g * a.D + 64 * kb, key0, &full[st]);
          tma_load_3d(dst + kbytes + kb * a.npad * 128, &a.qmap, 64 * kb, l * a.Hq + g * a.G, m[kRRowOff],
                      &full[st]);
        }
        if (++st == a.nstage) {
          st = 0;
          ph ^= 1u;
        }
      }
    }
  } else if (warp == 4 * kRowsGroups + 1) {
    if (lane == 0) {
      const uint32_t idesc = umma_idesc_bf16(kRowsChunk, a.npad);
      int st = 0, gr = 0;
      uint32_t ph = 0, gph = 1;
      for (int item = blockIdx.x; item < a.n_items; item += gridDim.x) {
        twait(&aempty[gr], gph);
        const bool ok = twait(&full[st], ph);
        tc_fence_after();
        if (ok) {
          const uint32_t sk = smem_addr(smem + (size_t)st * stage_bytes), sq = sk + kbytes;
          for (int kb = 0; kb < nkb; ++kb)
#pragma unroll
            for (int k = 0; k < 4; ++k)
              umma_bf16(tmem + gr * a.tmem_cols, umma_desc_sw128(sk + kb * kRowsChunk * 128 + k * 32),
                        umma_desc_sw128(sq + kb * a.npad * 128 + k * 32), idesc, (kb | k) != 0 ? 1u : 0u);
        }
        umma_commit(&empty[st]);
        umma_commit(&afull[gr]);
        if (++st == a.nstage) {
          st = 0;
          ph ^= 1u;
        }
        if (++gr == ngroup) {
          gr = 0;
          gph ^= 1u;
        }
      }
    }
  } else if (warp < 4 * ngroup) {
    const int gr = warp >> 2, quad = warp & 3, gt = threadIdx.x & 127;   // group, its warp, its thread
    uint32_t ph = 0;
    for (int item = blockIdx.x + gr * gridDim.x; item < a.n_items; item += ngroup * gridDim.x, ph ^= 1u) {
      int b, c, l, g;
      decode(item, &b, &c, &l, &g);
      const int32_t *m = a.meta + b * kRowsFields;
      const int P = m[kRSeqLen], v0 = m[kRVisStart], v1 = v0 + m[kRNumVis], row0 = m[kRRowOff];
      const int ncol = m[kRNumRows] * a.G, p0 = c * kRowsChunk, p = p0 + gt;
      // rows sit after the visual span: keys up to its end are seen by every row
      const bool seen = p0 + kRowsChunk <= v1, in_vis = p >= v0 && p < v1;
      const uint32_t acc = tmem + gr * a.tmem_cols + ((uint32_t)(32 * quad) << 16);
      const long long rh0 = (long long)l * a.Hq + g * a.G;   // triple of (row 0, l, first head of g)
      if (!STATS) {
        for (int n = gt; n < ncol; n += 128) {
          const int r = n / a.G;
          cf[gr][n] = a.coef[m[kRCoefBase] + (long long)r * a.L * a.Hq + rh0 + (n - r * a.G)];
        }
        asm volatile("bar.sync %0, 128;" :: "r"(1 + gr) : "memory");
      }
      twait(&afull[gr], ph);
      __syncwarp();
      tc_fence_after();
      if constexpr (STATS) {
        float4 *st = a.stats + stat_base(m) + (long long)c * m[kRNumRows] * a.L * a.Hq;
        for (int n0 = 0; n0 < ncol; n0 += 32) {
          float z[32], t[32];
          {
            uint32_t raw[32];
            tmem_ld16(acc + n0, raw);
            if (n0 + 16 < a.npad) tmem_ld16(acc + n0 + 16, raw + 16);
#pragma unroll
            for (int q = 0; q < 32; ++q) z[q] = __uint_as_float(raw[q]) * a.qscale;
          }
          if (!seen) {   // causal mask of the text rows, keys past the request
#pragma unroll
            for (int q = 0; q < 32; ++q) {
              const int pos = n0 + q < ncol ? a.row_pos[row0 + (n0 + q) / a.G] : -1;
              if (p >= P || p > pos) z[q] = -INFINITY;
            }
          }
#pragma unroll
          for (int q = 0; q < 32; ++q) t[q] = z[q];
          // the chunk's maximum, so that no sum is rescaled before the merge
          const float wmx = warp_columns(t, lane, [](float x, float y) { return fmaxf(x, y); });
          wmax[warp][lane] = wmx;
          asm volatile("bar.sync %0, 128;" :: "r"(1 + gr) : "memory");
          const float mx = fmaxf(fmaxf(wmax[4 * gr][lane], wmax[4 * gr + 1][lane]),
                                 fmaxf(wmax[4 * gr + 2][lane], wmax[4 * gr + 3][lane]));
          // (a column without a finite logit here is left at zero, not at 2^(-inf + inf))
          cmax[warp][lane] = mx == -INFINITY ? 0.f : mx;
          __syncwarp();
#pragma unroll
          for (int q = 0; q < 32; ++q) {
            z[q] = exp2f(z[q] - cmax[warp][q]);
            t[q] = z[q];
          }
          __syncwarp();
          const float sum = warp_columns(t, lane, [](float x, float y) { return x + y; });
          float vis;
          const int wp0 = p0 + 32 * quad;   // the warp's keys
          if (wp0 >= v0 && wp0 + 32 <= v1) {
            vis = sum;
          } else if (wp0 + 32 <= v0 || wp0 >= v1) {
            vis = 0.f;
          } else {
#pragma unroll
            for (int q = 0; q < 32; ++q) t[q] = in_vis ? z[q] : 0.f;
            vis = warp_columns(t, lane, [](float x, float y) { return x + y; });
          }
          // (the first warp reads these before it reaches the next barrier for the maxima)
          part[gr][quad][lane] = make_float2(sum, vis);
          asm volatile("bar.sync %0, 128;" :: "r"(1 + gr) : "memory");
          if (quad == 0 && n0 + lane < ncol) {   // the four warps in order
            float s4 = 0.f, vv = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float2 x = part[gr][q][lane];
              s4 += x.x;
              vv += x.y;
            }
            const int n = n0 + lane, r = n / a.G;
            st[(long long)r * a.L * a.Hq + rh0 + (n - r * a.G)] = make_float4(mx, s4, vv, 0.f);
          }
        }
      } else {
        float s0 = 0.f, s1 = 0.f;
        for (int n0 = 0; n0 < ncol; n0 += 16) {
          uint32_t raw[16];
          tmem_ld16(acc + n0, raw);
          if (n0 + 16 <= ncol) {
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
              const float2 c0 = cf[gr][n0 + j], c1 = cf[gr][n0 + j + 1];
              s0 += exp2f(__uint_as_float(raw[j]) * a.qscale - c0.x) * c0.y;
              s1 += exp2f(__uint_as_float(raw[j + 1]) * a.qscale - c1.x) * c1.y;
            }
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (n0 + j < ncol) s0 += exp2f(__uint_as_float(raw[j]) * a.qscale - cf[gr][n0 + j].x) * cf[gr][n0 + j].y;
          }
        }
        if (in_vis) a.partial[((long long)l * a.Hkv + g) * a.total_vis + m[kRVisOff] + (p - v0)] = s0 + s1;
        asm volatile("bar.sync %0, 128;" :: "r"(1 + gr) : "memory");   // cf is rewritten next
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&aempty[gr]);
    }
  }
  __syncthreads();
  if (gave_up) {   // an aborted call: time for copies and MMAs in flight before the CTA may exit
    if (threadIdx.x == 0) wait_out(&never);
    __syncthreads();
  }
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, tmem_total);
}

// One CTA per (32 (row, layer, head) triples, request): 8 warps take the chunks in turn,
// lane = triple.  The maximum over all chunks first, then the sums, each chunk's scaled
// once, and the warps' sums in order.
__global__ void __launch_bounds__(256) rows_merge_kernel(const RowsArgs a) {
  __shared__ float wmax[8][32];
  __shared__ float2 part[8][32];
  const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t *m = a.meta + b * kRowsFields;
  const int RH = m[kRNumRows] * a.L * a.Hq, nch = m[kRNumChunks];
  if ((int)blockIdx.x * 32 >= RH) return;
  const int rh = blockIdx.x * 32 + lane;
  const float4 *st = a.stats + stat_base(m) + min(rh, RH - 1);
  float mx = -INFINITY;
#pragma unroll 4
  for (int c = warp; c < nch; c += 8) mx = fmaxf(mx, st[(long long)c * RH].x);
  wmax[warp][lane] = mx;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) mx = fmaxf(mx, wmax[q][lane]);
  float z = 0.f, vz = 0.f;
#pragma unroll 4
  for (int c = warp; c < nch; c += 8) {
    const float4 v = st[(long long)c * RH];
    const float f = v.x == -INFINITY ? 0.f : exp2f(v.x - mx);   // chunks past the row
    z += v.y * f;
    vz += v.z * f;
  }
  part[warp][lane] = make_float2(z, vz);
  __syncthreads();
  if (warp != 0) return;
  z = vz = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    z += part[q][lane].x;
    vz += part[q][lane].y;
  }
  float mass = 0.f;
  if (rh < RH) {
    a.coef[m[kRCoefBase] + rh] = make_float2(mx, 1.0f / z);
    mass = vz / z;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mass += __shfl_xor_sync(0xffffffffu, mass, o);
  if (lane == 0) a.mass[(long long)b * a.mass_blocks + blockIdx.x] = mass;
}

__global__ void __launch_bounds__(kScoreThreads)
rows_final_kernel(const RowsArgs a) {
  __shared__ float inv_s;
  const int b = blockIdx.y;
  const int32_t *m = a.meta + b * kRowsFields;
  if ((int)blockIdx.x * kScoreThreads >= m[kRNumVis]) return;
  if (threadIdx.x < 32) {   // the request's visual mass: the blocks over the lanes, a fixed tree
    const int nb = (m[kRNumRows] * a.L * a.Hq + 31) / 32;
    float t = 0.f;
    for (int q = threadIdx.x; q < nb; q += 32) t += a.mass[(long long)b * a.mass_blocks + q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) inv_s = 1.0f / t;
  }
  __syncthreads();
  const int i = blockIdx.x * kScoreThreads + threadIdx.x;
  if (i >= m[kRNumVis]) return;
  const long long tok = m[kRVisOff] + i;
  float s = 0.f;
  for (int lg = 0; lg < a.L * a.Hkv; ++lg) s += a.partial[(long long)lg * a.total_vis + tok];
  a.w[tok] = s * inv_s;
}

namespace {

struct RowsPlan {
  int B = 0, L = 0, Hq = 0, Hkv = 0, D = 0, G = 0, npad = 0, max_vis = 0, mass_blocks = 0;
  long long total_keys = 0, total_vis = 0, total_rows = 0, n_items1 = 0, n_items2 = 0;
  size_t off_meta = 0, off_items1 = 0, off_items2 = 0, off_pos = 0, blob_bytes = 0;
  size_t off_stats = 0, off_coef = 0, off_mass = 0, off_partial = 0, total_bytes = 0;
  std::vector<int32_t> blob;
  float scale = 0.f;
};

constexpr size_t kAlignR = 256;
size_t alignr(size_t v) { return (v + kAlignR - 1) / kAlignR * kAlignR; }

last_status rows_fail(last_status st, const std::string &msg) {
  set_error(msg);
  return st;
}

last_status make_rows_plan(const last_problem *p, const int32_t *cu_rows, const int32_t *row_pos,
                           RowsPlan *pl) {
  if (p == nullptr) return rows_fail(LAST_ERR_INVALID_ARG, "problem is NULL");
  if (cu_rows == nullptr || row_pos == nullptr)
    return rows_fail(LAST_ERR_INVALID_ARG, "cu_rows and row_pos are required");
  if (p->dtype != LAST_DTYPE_BF16)
    return rows_fail(LAST_ERR_UNSUPPORTED, "multi-row scoring takes bf16 q and K");
  if (p->batch < 0 || p->cu_seqlens == nullptr || p->vis_start == nullptr || p->cu_vis == nullptr)
    return rows_fail(LAST_ERR_INVALID_ARG, "batch, cu_seqlens, vis_start and cu_vis are required");
  if (p->num_layers < 1 || p->num_q_heads < 1 || p->num_kv_heads < 1 ||
      p->num_q_heads % p->num_kv_heads != 0)
    return rows_fail(LAST_ERR_INVALID_ARG, "layers and heads must be >= 1, Hq a multiple of Hkv");
  if (p->head_dim < 64 || p->head_dim % 64 != 0 || p->head_dim > 256)
    return rows_fail(LAST_ERR_UNSUPPORTED, "multi-row scoring takes head_dim 64, 128, 192 or 256");
  if (!std::isfinite(p->softmax_scale))
    return rows_fail(LAST_ERR_INVALID_ARG, "softmax_scale must be finite");
  if (p->cu_seqlens[0] != 0 || p->cu_vis[0] != 0 || cu_rows[0] != 0)
    return rows_fail(LAST_ERR_INVALID_ARG, "cu_seqlens[0], cu_vis[0] and cu_rows[0] must be 0");
  const int B = p->batch;
  pl->B = B; pl->L = p->num_layers; pl->Hq = p->num_q_heads; pl->Hkv = p->num_kv_heads;
  pl->D = p->head_dim; pl->G = pl->Hq / pl->Hkv;
  pl->scale = p->softmax_scale > 0.f ? p->softmax_scale : (float)(1.0 / std::sqrt((double)p->head_dim));
  int max_cols = 0;
  long long stats = 0, rh_total = 0;
  for (int b = 0; b < B; ++b) {
    const int P = p->cu_seqlens[b + 1] - p->cu_seqlens[b];
    const int N = p->cu_vis[b + 1] - p->cu_vis[b];
    const int M = cu_rows[b + 1] - cu_rows[b];
    if (P < 1 || N < 0 || p->vis_start[b] < 0 || (long long)p->vis_start[b] + N > (long long)P - 1)
      return rows_fail(LAST_ERR_INVALID_ARG, "request " + std::to_string(b) +
                                                 ": visual span must end before the last position");
    if (M < 1) return rows_fail(LAST_ERR_INVALID_ARG, "request " + std::to_string(b) + ": no query row");
    for (int r = cu_rows[b]; r < cu_rows[b + 1]; ++r)
      if (row_pos[r] < p->vis_start[b] + N || row_pos[r] > P - 1)
        return rows_fail(LAST_ERR_INVALID_ARG,
                         "request " + std::to_string(b) + ": a query row must sit after the visual "
                         "span and before P_b");
    max_cols = std::max(max_cols, M * pl->G);
    const long long rh = (long long)M * pl->L * pl->Hq;
    if (rh > kRowsMaxRH)
      return rows_fail(LAST_ERR_UNSUPPORTED, "rows x layers x q-heads must be <= 6144 per request");
    const int nch = (P + kRowsChunk - 1) / kRowsChunk;
    stats += rh * nch;
    rh_total += rh;
    pl->mass_blocks = std::max(pl->mass_blocks, (int)((rh + 31) / 32));
    pl->n_items1 += nch;
    if (N > 0)
      pl->n_items2 += (p->vis_start[b] + N - 1) / kRowsChunk - p->vis_start[b] / kRowsChunk + 1;
    pl->max_vis = std::max(pl->max_vis, N);
  }
  if (max_cols > kRowsMaxN)
    return rows_fail(LAST_ERR_UNSUPPORTED, "query rows x (num_q_heads / num_kv_heads) must be <= 256");
  if (rh_total > 0x7fffffffLL) return rows_fail(LAST_ERR_UNSUPPORTED, "too many query rows in all");
  pl->npad = std::max(16, (max_cols + 15) / 16 * 16);
  pl->total_keys = p->cu_seqlens[B];
  pl->total_vis = p->cu_vis[B];
  pl->total_rows = cu_rows[B];
  size_t o = alignr(64);                     // error word first
  pl->off_meta = o;
  o = alignr(o + sizeof(int32_t) * kRowsFields * std::max(B, 1));
  pl->off_items1 = o;
  o = alignr(o + sizeof(int32_t) * 2 * std::max<long long>(pl->n_items1, 1));
  pl->off_items2 = o;
  o = alignr(o + sizeof(int32_t) * 2 * std::max<long long>(pl->n_items2, 1));
  pl->off_pos = o;
  o = alignr(o + sizeof(int32_t) * std::max<long long>(pl->total_rows, 1));
  pl->blob_bytes = o;
  pl->off_stats = o;
  o = alignr(o + sizeof(float) * 4 * (size_t)std::max<long long>(stats, 1));
  pl->off_coef = o;
  o = alignr(o + sizeof(float) * 2 * (size_t)std::max<long long>(rh_total, 1));
  pl->off_mass = o;
  o = alignr(o + sizeof(float) * (size_t)std::max(B, 1) * pl->mass_blocks);
  pl->off_partial = o;
  o = alignr(o + sizeof(float) * (size_t)pl->L * pl->Hkv * (size_t)std::max<long long>(pl->total_vis, 1));
  pl->total_bytes = o;
  // staging blob: [error word][meta][items of every chunk][items of visual chunks][positions]
  pl->blob.assign(pl->blob_bytes / sizeof(int32_t), 0);
  int32_t *meta = pl->blob.data() + pl->off_meta / 4;
  int32_t *it1 = pl->blob.data() + pl->off_items1 / 4;
  int32_t *it2 = pl->blob.data() + pl->off_items2 / 4;
  int32_t *pos = pl->blob.data() + pl->off_pos / 4;
  long long sb = 0, i1 = 0, i2 = 0;
  int cb = 0;
  for (int b = 0; b < B; ++b) {
    int32_t *mm = meta + b * kRowsFields;
    const int P = p->cu_seqlens[b + 1] - p->cu_seqlens[b];
    const int N = p->cu_vis[b + 1] - p->cu_vis[b];
    const int M = cu_rows[b + 1] - cu_rows[b];
    const int nch = (P + kRowsChunk - 1) / kRowsChunk;
    mm[kRSeqStart] = p->cu_seqlens[b];
    mm[kRSeqLen] = P;
    mm[kRVisStart] = p->vis_start[b];
    mm[kRVisOff] = p->cu_vis[b];
    mm[kRNumVis] = N;
    mm[kRRowOff] = cu_rows[b];
    mm[kRNumRows] = M;
    mm[kRNumChunks] = nch;
    std::memcpy(mm + kRStatBase, &sb, sizeof sb);   // 64-bit offset in two int32 slots
    mm[kRCoefBase] = cb;
    const int rh = M * pl->L * pl->Hq;
    sb += (long long)rh * nch;
    cb += rh;
    for (int c = 0; c < nch; ++c, ++i1) {
      it1[2 * i1] = b;
      it1[2 * i1 + 1] = c;
    }
    if (N > 0)
      for (int c = p->vis_start[b] / kRowsChunk; c <= (p->vis_start[b] + N - 1) / kRowsChunk; ++c, ++i2) {
        it2[2 * i2] = b;
        it2[2 * i2 + 1] = c;
      }
  }
  for (long long r = 0; r < pl->total_rows; ++r) pos[r] = row_pos[r];
  return LAST_OK;
}

// One query row per request: the row at position pos attends keys 0 .. pos, which
// is the last-row computation of Eq. 6-8 on the request cut after pos, so the
// last-row scoring kernels take it (the last_scores plan with P'_b = pos + 1).
// Returns LAST_OK only when that plan applies.
last_status single_row_plan(const last_problem *p, const int32_t *cu_rows, const int32_t *row_pos,
                            Plan *lp) {
  if (p->batch < 1 || cu_rows[p->batch] != p->batch) return LAST_ERR_UNSUPPORTED;
  std::vector<int32_t> len(p->batch);
  for (int b = 0; b < p->batch; ++b) len[b] = row_pos[b] + 1;
  last_problem pc = *p;
  if (pc.cu_keep == nullptr) pc.cu_keep = pc.cu_vis;   // scoring needs no budgets
  // a probe: when the plan does not apply, the multi-row kernels run instead and the
  // call's error message must not report the probe's rejection
  const std::string saved = get_error();
  const last_status st = make_plan(&pc, true, false, lp, len.data());
  if (st != LAST_OK) set_error(saved);
  return st;
}

}  // namespace
}  // namespace last

using namespace last;

extern "C" last_status last_scores_rows_workspace_size(const last_problem *p, const int32_t *cu_rows,
                                                       const int32_t *row_pos, size_t *bytes) {
  if (bytes == nullptr) return rows_fail(LAST_ERR_INVALID_ARG, "bytes is NULL");
  RowsPlan pl;
  last_status st = make_rows_plan(p, cu_rows, row_pos, &pl);
  if (st != LAST_OK) return st;
  Plan lp;
  *bytes = pl.total_bytes;
  if (single_row_plan(p, cu_rows, row_pos, &lp) == LAST_OK) *bytes = std::max(*bytes, lp.score_bytes);
  return LAST_OK;
}

extern "C" last_status last_scores_rows(const last_problem *p, const int32_t *cu_rows,
                                        const int32_t *row_pos, const void *q_rows, const void *k,
                                        float *w_out, void *ws, size_t ws_bytes, void *stream) {
  RowsPlan pl;
  last_status st = make_rows_plan(p, cu_rows, row_pos, &pl);
  if (st != LAST_OK) return st;
  Plan lp;
  const bool single = single_row_plan(p, cu_rows, row_pos, &lp) == LAST_OK;
  const size_t need = single ? std::max(pl.total_bytes, lp.score_bytes) : pl.total_bytes;
  if (ws == nullptr) return rows_fail(LAST_ERR_INVALID_ARG, "workspace is NULL");
  if ((reinterpret_cast<uintptr_t>(ws) & (kAlignR - 1)) != 0)
    return rows_fail(LAST_ERR_INVALID_ARG, "workspace must be 256-byte aligned");
  if (ws_bytes < need)
    return rows_fail(LAST_ERR_WORKSPACE_TOO_SMALL, "workspace needs " + std::to_string(need) + " bytes");
  if (pl.total_vis > 0 && (q_rows == nullptr || k == nullptr || w_out == nullptr))
    return rows_fail(LAST_ERR_INVALID_ARG, "q_rows, k and w_out are required");
  if ((reinterpret_cast<uintptr_t>(q_rows) & 15u) || (reinterpret_cast<uintptr_t>(k) & 15u))
    return rows_fail(LAST_ERR_INVALID_ARG, "q_rows and k must be 16-byte aligned");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char *wsc = static_cast<char *>(ws);
  if (single) {
    cudaError_t e = cudaMemcpyAsync(wsc, lp.host_blob.data(), lp.blob_bytes, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = launch_scores(lp, q_rows, k, w_out, wsc, s);
    if (e != cudaSuccess) return rows_fail(LAST_ERR_CUDA, std::string("single-row scoring: ") +
                                                            cudaGetErrorString(e));
    return LAST_OK;
  }
  cudaError_t e = cudaMemcpyAsync(wsc, pl.blob.data(), pl.blob_bytes, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return rows_fail(LAST_ERR_CUDA, std::string("plan copy: ") + cudaGetErrorString(e));
  if (pl.total_vis == 0 || pl.B == 0) return LAST_OK;

  RowsArgs a;
  std::memset(&a, 0, sizeof a);
  a.meta = reinterpret_cast<const int32_t *>(wsc + pl.off_meta);
  a.items1 = reinterpret_cast<const int2 *>(wsc + pl.off_items1);
  a.items2 = reinterpret_cast<const int2 *>(wsc + pl.off_items2);
  a.row_pos = reinterpret_cast<const int32_t *>(wsc + pl.off_pos);
  a.stats = reinterpret_cast<float4 *>(wsc + pl.off_stats);
  a.coef = reinterpret_cast<float2 *>(wsc + pl.off_coef);
  a.mass = reinterpret_cast<float *>(wsc + pl.off_mass);
  a.partial = reinterpret_cast<float *>(wsc + pl.off_partial);
  a.w = w_out;
  a.total_keys = pl.total_keys;
  a.total_vis = pl.total_vis;
  a.L = pl.L; a.Hq = pl.Hq; a.Hkv = pl.Hkv; a.D = pl.D; a.G = pl.G; a.npad = pl.npad;
  a.mass_blocks = pl.mass_blocks;
  uint32_t cols = 32;
  while ((int)cols < pl.npad) cols *= 2;
  a.tmem_cols = cols;
  a.ngroup = (int)std::min<uint32_t>(kRowsGroups, 512 / cols);
  a.qbox = std::min(pl.npad / pl.G, 256);
  a.qscale = pl.scale * 1.4426950408889634f;
  a.err = reinterpret_cast<unsigned *>(wsc);
  auto fail_launch = [](cudaError_t err, const char *what) {
    return rows_fail(LAST_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(err));
  };
  {
    const uint64_t kd[2] = {(uint64_t)pl.Hkv * pl.D, (uint64_t)pl.L * pl.total_keys};
    const uint64_t ks[1] = {(uint64_t)pl.Hkv * pl.D * 2};
    const uint32_t kb[2] = {64, kRowsChunk};
    const uint64_t qd[3] = {(uint64_t)pl.D, (uint64_t)pl.L * pl.Hq, (uint64_t)pl.total_rows};
    const uint64_t qs[2] = {(uint64_t)pl.D * 2, (uint64_t)pl.L * pl.Hq * pl.D * 2};
    const uint32_t qb[3] = {64, (uint32_t)pl.G, (uint32_t)a.qbox};
    if (!encode_bf16_map(&a.kmap, k, 2, kd, ks, kb) || !encode_bf16_map(&a.qmap, q_rows, 3, qd, qs, qb))
      return rows_fail(LAST_ERR_CUDA, "multi-row scoring: the tensor maps cannot be encoded");
  }
  int dev = 0, sms = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  // as many stages as fit; more than half of an SM in all cases, so that one CTA holds
  // an SM's tensor memory
  const size_t stage = (size_t)(pl.D / 64) * (kRowsChunk + pl.npad) * 128;
  const size_t fixed = 16 * 1024 + 1024;   // the kernel's own arrays (15 KB) and the alignment
  a.nstage = (int)std::min<size_t>(kRowsMaxStages, ((size_t)optin - fixed) / stage);
  const size_t smem = std::max<size_t>(a.nstage * stage + 1024, 116 * 1024);
  for (int pass = 0; pass < 2; ++pass) {
    void *fn = pass == 0 ? (void *)rows_pass_kernel<true> : (void *)rows_pass_kernel<false>;
    const long long n = (pass == 0 ? pl.n_items1 : pl.n_items2) * pl.L * pl.Hkv;
    if (n > 0x7fffffffLL) return rows_fail(LAST_ERR_UNSUPPORTED, "too many key chunks in all");
    if (n > 0) {
      a.n_items = (int)n;
      if ((e = allow_smem(fn, smem)) != cudaSuccess) return fail_launch(e, "rows pass");
      void *args[] = {&a};
      e = cudaLaunchKernel(fn, dim3((unsigned)std::min<long long>(n, sms)), dim3(kPassThreads), args, smem, s);
      if (e != cudaSuccess) return fail_launch(e, "rows pass launch");
    }
    if (pass == 0) {
      rows_merge_kernel<<<dim3(pl.mass_blocks, pl.B), 256, 0, s>>>(a);
      if ((e = cudaGetLastError()) != cudaSuccess) return fail_launch(e, "rows merge launch");
    }
  }
  const int tiles = (pl.max_vis + kScoreThreads - 1) / kScoreThreads;
  rows_final_kernel<<<dim3(tiles, pl.B), kScoreThreads, 0, s>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return fail_launch(e, "rows final launch");
  return LAST_OK;
}
