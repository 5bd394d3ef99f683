// Table 5 ("LAST (Top-k)"): the selection variant that keeps the k_b tokens of
// highest importance score w~ per request, ties to the lower index, returned in
// ascending index order (Eq. 12's sort(S)).
//
// topk_kernel: one CTA per request; a request of up to kTopkCacheTokens scores keeps
// them in shared memory for every pass.  The scores' order-preserving 32-bit keys are
// narrowed by an MSB-first radix select over 11-bit digits that starts at the first bit
// in which the request's keys differ (scores of one request share their leading bits),
// to the k-th largest key T and the number of keys equal to T that are kept, lowest
// indices first.  Each warp owns a contiguous part of the tokens, so the ordered
// compaction takes one count and one write pass without a barrier per 1024 tokens.
// Integer histograms: exact and deterministic.  Latency-bound (one CTA): 56 us with
// 8-bit digits of 64-bit keys and warp-aggregated adds on 16384 tokens, k = 2048; now
// 16 us.
#include "last_device.cuh"
#include "last_internal.h"

#include <algorithm>

namespace last {

constexpr int kTopkThreads = 1024;
constexpr int kTopkBits = 11, kTopkBins = 1 << kTopkBits;
constexpr int kTopkCacheTokens = 48 * 1024;   // 192 KB of scores

// order-preserving bits of a score (-0 folded into +0); larger = kept first
__device__ __forceinline__ uint32_t topk_key(float w) { return (uint32_t)(argmax_key(w, 0) >> 32); }

__global__ void __launch_bounds__(kTopkThreads)
topk_kernel(const float *__restrict__ w, const int32_t *__restrict__ meta,
            int32_t *__restrict__ idx_out, int cache_tokens) {
  extern __shared__ uint32_t kcache[];
  constexpr int kWarps = kTopkThreads / 32;
  __shared__ unsigned hist[kTopkBins];
  __shared__ unsigned red[2][kWarps];
  __shared__ uint32_t s_prefix;
  __shared__ unsigned s_need;
  __shared__ int s_done;
  const int32_t *m = meta + blockIdx.x * kMetaFields;
  const int N = m[kNumVis], k = m[kNumKeep];
  if (k <= 0) return;
  const float *wg = w + m[kVisOff];
  int32_t *out = idx_out + m[kKeepOff];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool cached = N <= cache_tokens;
  auto key_at = [&](int i) { return cached ? kcache[i] : topk_key(wg[i]); };

  // the keys' range (and their cached copies)
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  for (int i = tid; i < N; i += kTopkThreads) {
    const uint32_t key = topk_key(wg[i]);
    if (cached) kcache[i] = key;
    kmin = min(kmin, key);
    kmax = max(kmax, key);
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) {
    red[0][warp] = kmin;
    red[1][warp] = kmax;
  }
  __syncthreads();
  kmin = __reduce_min_sync(0xffffffffu, red[0][lane]);
  kmax = __reduce_max_sync(0xffffffffu, red[1][lane]);

  uint32_t thr = 0u;                          // keys above it are kept
  unsigned need = 0u;                         // and this many equal to it
  if (k < N) {
    need = static_cast<unsigned>(k);
    // bits above `top` are common to all keys
    int top = kmin == kmax ? 0 : 32 - __clz(kmin ^ kmax);
    uint32_t prefix = top < 32 ? kmax >> top << top : 0u;
    uint32_t mask = top < 32 ? ~0u << top : 0u;
    thr = prefix;
    while (top > 0) {
      const int shift = max(0, top - kTopkBits), bins = 1 << (top - shift);
      for (int i = tid; i < bins; i += kTopkThreads) hist[i] = 0;
      __syncthreads();
      for (int i = tid; i < N; i += kTopkThreads) {
        const uint32_t key = key_at(i);
        if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & (bins - 1)], 1u);
      }
      __syncthreads();
      // thread t owns the bins bins - 1 - 2t and below: keys in higher bins than its own
      unsigned c0 = 0, c1 = 0;
      const int b0 = bins - 1 - 2 * tid;
      if (b0 >= 0) c0 = hist[b0];
      if (b0 >= 1) c1 = hist[b0 - 1];
      unsigned incl = c0 + c1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      if (lane == 31) red[0][warp] = incl;
      __syncthreads();
      unsigned before = lane < warp ? red[0][lane] : 0u;
      before = __reduce_add_sync(0xffffffffu, before);
      const unsigned above = before + incl - c0 - c1;   // keys in higher bins
      if (above < need && need <= above + c0 + c1) {    // exactly one thread
        const bool first = need <= above + c0;
        const unsigned up = first ? above : above + c0, in = first ? c0 : c1;
        s_prefix = prefix | (uint32_t)(first ? b0 : b0 - 1) << shift;
        s_need = need - up;
        s_done = in == need - up;   // every key of this bin is kept
      }
      __syncthreads();
      prefix = thr = s_prefix;
      need = s_need;
      mask |= (uint32_t)(bins - 1) << shift;
      top = shift;
      if (s_done) {   // keep the whole bin: everything above its lower end minus one
        thr = prefix - 1u;
        need = 0u;
        break;
      }
      __syncthreads();   // the shared words are rewritten by the next pass
    }
  }

  // warp q owns tokens [q seg, (q + 1) seg): count, prefix over the warps, write
  const int seg = ((N + kWarps - 1) / kWarps + 31) / 32 * 32;
  const int lo = min(N, warp * seg), hi = min(N, lo + seg);
  const bool all = k >= N;
  unsigned gt = 0, eq = 0;
  for (int i0 = lo; i0 < hi; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t key = i < hi ? key_at(i) : 0u;
    gt += __popc(__ballot_sync(0xffffffffu, i < hi && (all || key > thr)));
    eq += __popc(__ballot_sync(0xffffffffu, i < hi && !all && key == thr));
  }
  __syncthreads();
  if (lane == 0) {
    red[0][warp] = gt;
    red[1][warp] = eq;
  }
  __syncthreads();
  const unsigned g0 = __reduce_add_sync(0xffffffffu, lane < warp ? red[0][lane] : 0u);
  const unsigned e0 = __reduce_add_sync(0xffffffffu, lane < warp ? red[1][lane] : 0u);
  unsigned ebase = e0;                       // equal keys before the warp's part
  unsigned pos = g0 + min(e0, need);         // kept tokens before it
  for (int i0 = lo; i0 < hi; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t key = i < hi ? key_at(i) : 0u;
    const bool is_eq = i < hi && !all && key == thr;
    const unsigned eb = __ballot_sync(0xffffffffu, is_eq);
    const bool sel = (i < hi && (all || key > thr)) ||
                     (is_eq && ebase + __popc(eb & ((1u << lane) - 1u)) < need);
    const unsigned sb = __ballot_sync(0xffffffffu, sel);
    if (sel) out[pos + __popc(sb & ((1u << lane) - 1u))] = i;
    pos += __popc(sb);
    ebase += __popc(eb);
  }
}

cudaError_t launch_topk(const Plan &pl, const float *w, int32_t *idx_out, char *ws,
                        cudaStream_t s) {
  if (pl.total_keep == 0 || pl.B == 0) return cudaSuccess;
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  // cache every request's scores when they fit beside the kernel's own arrays (8.3 KB)
  const int cache = std::min<int>(std::min(kTopkCacheTokens, pl.max_vis),
                                  std::max(0, (optin - 12 * 1024) / 4));
  const size_t smem = sizeof(float) * (size_t)cache;
  cudaError_t e = allow_smem((const void *)topk_kernel, smem);
  if (e != cudaSuccess) return e;
  topk_kernel<<<pl.B, kTopkThreads, smem, s>>>(
      w, reinterpret_cast<const int32_t *>(ws + pl.off_meta), idx_out, cache);
  return cudaGetLastError();
}

}  // namespace last
