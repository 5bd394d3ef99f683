// C-ABI entry points of liblast: argument validation, workspace layout, the
// small host->device plan copy, and the kernel launch sequence.
#include "last_internal.h"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <numeric>

namespace last {

namespace {
thread_local std::string g_error;

constexpr size_t kAlign = 256;
size_t align_up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }

last_status fail(last_status st, const std::string &msg) {
  g_error = msg;
  return st;
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
}  // namespace

void set_error(const std::string &msg) { g_error = msg; }
std::string get_error() { return g_error; }

last_status make_plan(const last_problem *p, bool need_scores, bool need_select, Plan *pl,
                      const int32_t *seq_len) {
  if (p == nullptr) return fail(LAST_ERR_INVALID_ARG, "problem is NULL");
  if (p->batch < 0) return fail(LAST_ERR_INVALID_ARG, "batch < 0");
  if (p->dtype != LAST_DTYPE_F32 && p->dtype != LAST_DTYPE_BF16)
    return fail(LAST_ERR_INVALID_ARG, "dtype must be LAST_DTYPE_F32 or LAST_DTYPE_BF16");
  const int B = p->batch;
  pl->B = B;
  pl->L = p->num_layers;
  pl->Hq = p->num_q_heads;
  pl->Hkv = p->num_kv_heads;
  pl->D = p->head_dim;
  pl->dv = p->feat_dim;
  pl->dtype = p->dtype;
  pl->elem = p->dtype == LAST_DTYPE_F32 ? 4 : 2;

  if (p->cu_vis == nullptr || p->cu_keep == nullptr)
    return fail(LAST_ERR_INVALID_ARG, "cu_vis and cu_keep are required");
  if (p->cu_vis[0] != 0 || p->cu_keep[0] != 0)
    return fail(LAST_ERR_INVALID_ARG, "cu_vis[0] and cu_keep[0] must be 0");
  for (int b = 0; b < B; ++b) {
    const int n = p->cu_vis[b + 1] - p->cu_vis[b];
    const int kb = p->cu_keep[b + 1] - p->cu_keep[b];
    if (n < 0) return fail(LAST_ERR_INVALID_ARG, "cu_vis must be non-decreasing");
    if (kb < 0 || kb > n)
      return fail(LAST_ERR_INVALID_ARG, "request " + std::to_string(b) + ": need 0 <= k_b <= N_b");
    pl->max_vis = std::max(pl->max_vis, n);
    pl->max_keep = std::max(pl->max_keep, kb);
  }
  pl->total_vis = p->cu_vis[B];
  pl->total_keep = p->cu_keep[B];

  if (need_select) {
    if (p->feat_dim < 8 || p->feat_dim % 8 != 0)
      return fail(LAST_ERR_INVALID_ARG, "feat_dim must be a positive multiple of 8");
    std::string why;
    if (!select_supported(*pl, &why)) return fail(LAST_ERR_UNSUPPORTED, why);
  }

  pl->total_chunks = 0;
  const bool have_seq = p->cu_seqlens != nullptr && p->vis_start != nullptr;
  if (need_scores && !have_seq)
    return fail(LAST_ERR_INVALID_ARG, "cu_seqlens and vis_start are required for scoring");
  if (have_seq && p->num_layers > 0) {
    if (p->num_layers < 1 || p->num_q_heads < 1 || p->num_kv_heads < 1 || p->head_dim < 1)
      return fail(LAST_ERR_INVALID_ARG, "layers, heads and head_dim must be >= 1");
    if (p->num_q_heads % p->num_kv_heads != 0)
      return fail(LAST_ERR_INVALID_ARG, "num_q_heads must be a multiple of num_kv_heads");
    if (!std::isfinite(p->softmax_scale))
      return fail(LAST_ERR_INVALID_ARG, "softmax_scale must be finite");
    if ((long long)p->num_layers * p->num_q_heads > 6144)
      return fail(LAST_ERR_UNSUPPORTED, "num_layers * num_q_heads must be <= 6144");
    if (p->cu_seqlens[0] != 0) return fail(LAST_ERR_INVALID_ARG, "cu_seqlens[0] must be 0");
    pl->G = p->num_q_heads / p->num_kv_heads;
    pl->chunk = score_chunk_keys(p->num_kv_heads);
    pl->scale = p->softmax_scale > 0.f ? p->softmax_scale
                                       : (float)(1.0 / std::sqrt((double)p->head_dim));
    for (int b = 0; b < B; ++b) {
      const int P_full = p->cu_seqlens[b + 1] - p->cu_seqlens[b];
      const int P = seq_len != nullptr ? seq_len[b] : P_full;
      const int n = p->cu_vis[b + 1] - p->cu_vis[b];
      if (P > P_full)
        return fail(LAST_ERR_INVALID_ARG, "request " + std::to_string(b) + ": cut beyond P_b");
      if (P < 1)
        return fail(LAST_ERR_INVALID_ARG, "request " + std::to_string(b) +
                                              ": P_b must be >= 1 (the query position)");
      if (p->vis_start[b] < 0 || (long long)p->vis_start[b] + n > (long long)P - 1)
        return fail(LAST_ERR_INVALID_ARG, "request " + std::to_string(b) +
                                              ": visual span must end before the query position");
      pl->max_seq = std::max(pl->max_seq, P);
      pl->total_chunks += (P + pl->chunk - 1) / pl->chunk;
    }
    pl->total_keys = p->cu_seqlens[B];
    if (need_scores) {
      std::string why;
      if (!scores_supported(*pl, &why)) return fail(LAST_ERR_UNSUPPORTED, why);
    }
  } else if (need_scores) {
    return fail(LAST_ERR_INVALID_ARG, "num_layers must be >= 1 for scoring");
  }

  // ---- workspace layout ----
  size_t o = 0;
  pl->off_err = o;
  o = align_up(o + 64);
  pl->off_meta = o;
  o = align_up(o + sizeof(int32_t) * kMetaFields * std::max(B, 1));
  pl->off_items = o;
  o = align_up(o + sizeof(int32_t) * 2 * std::max(pl->total_chunks, 1));
  pl->off_order = o;
  o = align_up(o + sizeof(int32_t) * std::max(B, 1));
  pl->off_gbar = o;   // abort word and one barrier counter per request slot
  o = align_up(o + sizeof(uint32_t) * (1 + kGridMaxReq));
  pl->off_tile0 = o;
  o = align_up(o + sizeof(int32_t) * (B + 1));
  const size_t blob_end = o;
  pl->off_stats = o;
  o = align_up(o + sizeof(float) * 4 * (size_t)std::max(pl->L, 0) * std::max(pl->Hq, 0) *
                       pl->total_chunks);
  pl->off_zlog = o;
  o = align_up(o + sizeof(float) * (size_t)std::max(pl->L, 0) * std::max(pl->Hq, 0) *
                       (size_t)pl->total_vis);
  pl->off_w = o;
  o = align_up(o + sizeof(float) * (size_t)pl->total_vis);
  pl->score_bytes = o;
  // The bf16 greedy's row skipping keeps up to kRootsPerRequest feature rows per
  // request (min(k_b, kRootsPerRequest) rounded up to whole groups of 16, each row
  // padded to whole 64-element blocks) and a table of bounds per root.
  pl->root_rows = 0;
  const bool sel_scratch = p->dtype == LAST_DTYPE_BF16 && p->feat_dim >= 8 &&
                           p->feat_dim % 8 == 0 && p->feat_dim <= kMaxFeatDim;
  auto root_cap = [&](int b) {
    return (std::min(p->cu_keep[b + 1] - p->cu_keep[b], kRootsPerRequest) + 15) / 16 * 16;
  };
  if (sel_scratch)
    for (int b = 0; b < B; ++b) pl->root_rows += root_cap(b);
  pl->off_roots = o;
  o = align_up(o + (size_t)pl->root_rows * (size_t)((std::max(p->feat_dim, 0) + 63) / 64) * 128);
  pl->off_rtab = o;
  o = align_up(o + (size_t)pl->root_rows * kRootTableCols * sizeof(float));
  // the whole-GPU selection's published keys, where launches of few requests may take it
  // (room for them whatever the batch: what a call needs grows with its problem)
  pl->off_gpub = o;
  if (pl->max_vis >= kGridMinTokens) o = align_up(o + grid_pub_bytes());
  pl->base_bytes = o;
  // The greedy from a Gram matrix: N_b rows of gram_ld(N_b) floats for every request
  // that has a choice to make (1 < k_b < N_b).
  auto gram_units = [&](int b) -> long long {
    const int n = p->cu_vis[b + 1] - p->cu_vis[b], kb = p->cu_keep[b + 1] - p->cu_keep[b];
    return kb > 1 && kb < n ? (long long)n * (gram_ld(n) / 32) : 0;
  };
  long long units = 0, tokens = 0;
  int choices = 0, keep = 2;   // requests with a choice, their tokens and largest budget
  const bool gram_ok = p->feat_dim >= 8 && p->feat_dim % 8 == 0 && p->feat_dim <= kMaxFeatDim;
  if (gram_ok)
    for (int b = 0; b < B; ++b)
      if (gram_units(b) > 0) {
        units += gram_units(b);
        tokens += p->cu_vis[b + 1] - p->cu_vis[b];
        keep = std::max(keep, p->cu_keep[b + 1] - p->cu_keep[b]);
        ++choices;
      }
  const bool f32 = p->dtype == LAST_DTYPE_F32;
  const double pairs = 0.5 * (double)units * 32.0;
  const double exact_s = pairs * p->feat_dim / 20e12;   // canonical order, 20 T fma/s
  // ... whose kernel takes whole groups of 256 coordinates and one more for its butterfly
  const double exact_all_s = pairs * 256.0 * ((std::max(p->feat_dim, 0) + 255) / 256 + 1) / 20e12;
  // bf16 batches take the canonical matrix where it costs little; measured against the tensor
  // cores' (us, whole selection, k = N/8): one request of 576 x 2048 85 / 110, four 138 / 122;
  // of 1100 x 512 126 / 142, of 2000 x 512 210 / 194; narrow rows, 16 of 576 x 64 140 / 111.
  pl->gram_exact = f32 || (exact_s <= kGramExactSeconds && exact_all_s <= 55e-6);
  // A matrix is used where it costs less than the rounds over X that it replaces: its bytes
  // at 5.2 TB/s beside its products (1.1 PFLOP/s, 1.7 in the long chains of requests of
  // 8192 tokens), and 50 us + 0.9 us a request for what surrounds it.  The rounds cost a
  // pass that grows with the width and the tokens per CTA and recurs a little with every
  // doubling of the budget.  Both sides measured, matrix / rounds, us: 8 requests of 16384
  // x 64 at k = 2 1723 / 303, 256 1864 / 1628; x 2048 at 32 3169 / 2580, 64 3203 / 3378, 256
  // 3323 / 6006; one of 50000 x 64 at 2 1971 / 564, 32 2096 / 1550, 128 2236 / 2570; two of
  // 16384 x 256 at 2 489 / 266, 16 528 / 574; 64 of 2048 x 256 at 2 327 / 263, 4 337 / 360; 32
  // of 2880 x 2048 at 2 630 / 652.  Of 361 shapes so measured, fp32 ones included, four take
  // the slower side by more than 6% (8 to 26%).  The second line, in products alone, keeps
  // wide features at tiny budgets on the rounds, which is where it was measured.
  // fp32, canonical order: 576 x 1024 at k = 2 39 / 30, 4 43 / 46; two of 2048 at 32 350 / 319,
  // 64 378 / 598; four of 4096 at 128 2456 / 1585; 10000 at 128 3551 / 3313; 12000 x 8 at 8 1834
  // / 455; 8 of 1200 x 64 at 8 203 / 141, 32 220 / 276 (rows narrower than 32 lanes' worth of
  // coordinates make the rounds slower: 1200 x 8 at 8 207 / 235).
  bool faster;
  if (f32) {
    const double pick = (2.3e-6 + 2.4e-9 * std::min(pl->max_vis, 4096)) * std::max(1.0, 32.0 / std::max(p->feat_dim, 1));
    faster = exact_all_s <= keep * pick && exact_s <= 6e-6 * keep;
  } else {
    const double flops = 2.0 * pairs * ((std::max(p->feat_dim, 0) + 63) / 64 * 64);
    const double matrix_s = (pl->gram_exact ? exact_all_s
                                            : std::hypot(8.0 * pairs / 5.2e12, flops / (pl->max_vis >= 8192 ? 1.7e15 : 1.1e15))) +
                            50e-6 + 0.9e-6 * std::min(choices, 152);
    const double per_cta = (double)tokens / std::min(152, 16 * std::max(choices, 1));
    const double rounds_s = (0.20e-3 + 0.28e-3 * p->feat_dim / 1024) * (0.5 + 0.7e-3 * per_cta) *
                            (1.0 + 0.34 * std::log2(0.5 * keep) + 0.006 * std::max(0, keep - 64));
    faster = matrix_s <= rounds_s && flops / 1.1e15 <= std::max(0.8e-3, 1.2e-4 * keep);
  }
  pl->gram = units > 0 && units * 128 <= kGramMaxBytes && faster && gram_select_fits(pl->max_vis);
  if (pl->gram) {
    pl->off_rn = o;
    o = align_up(o + sizeof(float) * (size_t)pl->total_vis);
    pl->off_gram = o;
    o = align_up(o + (size_t)units * 128);
  }
  pl->min_bytes = pl->base_bytes + (gram_ok && pl->total_keep > 0 ? kGramSmallBytes : 0);
  pl->total_bytes = std::max(o, pl->min_bytes);

  // ---- host staging: [err words][meta][items][order], one copy ----
  pl->blob_bytes = blob_end;
  pl->host_blob.assign(blob_end / sizeof(int32_t), 0);
  int32_t *meta = pl->host_blob.data() + pl->off_meta / 4;
  int32_t *items = pl->host_blob.data() + pl->off_items / 4;
  int32_t *order = pl->host_blob.data() + pl->off_order / 4;
  int32_t *tile0 = pl->host_blob.data() + pl->off_tile0 / 4;
  int chunk = 0;
  long long root_off = 0, gram_off = 0;
  for (int b = 0; b < B; ++b) {
    int32_t *m = meta + b * kMetaFields;
    tile0[b] = pl->gram_tiles;
    if (pl->gram) {
      m[kGramOff] = (int32_t)gram_off;
      gram_off += gram_units(b);
      if (gram_units(b) > 0) {
        const int n = p->cu_vis[b + 1] - p->cu_vis[b];
        pl->gram_tiles += pl->gram_exact ? gram_exact_tiles(n, p->dtype == LAST_DTYPE_F32) : gram_tiles(n, gram_long(pl->max_vis));
      }
    }
    m[kRootOff] = (int32_t)root_off;
    if (sel_scratch) root_off += root_cap(b);
    m[kVisOff] = p->cu_vis[b];
    m[kNumVis] = p->cu_vis[b + 1] - p->cu_vis[b];
    m[kKeepOff] = p->cu_keep[b];
    m[kNumKeep] = p->cu_keep[b + 1] - p->cu_keep[b];
    if (have_seq && p->num_layers > 0) {
      m[kSeqStart] = p->cu_seqlens[b];
      m[kSeqLen] = seq_len != nullptr ? seq_len[b] : p->cu_seqlens[b + 1] - p->cu_seqlens[b];
      m[kVisStart] = p->vis_start[b];
      m[kChunkBase] = chunk;
      const int nch = (m[kSeqLen] + pl->chunk - 1) / pl->chunk;
      for (int c = 0; c < nch; ++c) {
        items[2 * (chunk + c)] = b;
        items[2 * (chunk + c) + 1] = c;
      }
      chunk += nch;
    }
  }
  tile0[B] = pl->gram_tiles;
  // selection clusters take the most expensive requests (k_b * N_b) first
  std::vector<int> ord(B);
  std::iota(ord.begin(), ord.end(), 0);
  std::stable_sort(ord.begin(), ord.end(), [&](int a, int c) {
    const long long wa = (long long)meta[a * kMetaFields + kNumKeep] * meta[a * kMetaFields + kNumVis];
    const long long wc = (long long)meta[c * kMetaFields + kNumKeep] * meta[c * kMetaFields + kNumVis];
    return wa > wc;
  });
  for (int b = 0; b < B; ++b) order[b] = ord[b];
  return LAST_OK;
}

namespace {

last_status check_ws(const void *ws, size_t ws_bytes, size_t need) {
  if (ws == nullptr) return fail(LAST_ERR_INVALID_ARG, "workspace is NULL");
  if ((reinterpret_cast<uintptr_t>(ws) & (kAlign - 1)) != 0)
    return fail(LAST_ERR_INVALID_ARG, "workspace must be 256-byte aligned");
  if (ws_bytes < need)
    return fail(LAST_ERR_WORKSPACE_TOO_SMALL, "workspace needs " + std::to_string(need) + " bytes");
  return LAST_OK;
}

// The selection's workspace: without room for the matrices its rounds read X.
last_status check_select_ws(Plan *pl, const void *ws, size_t ws_bytes) {
  if (ws_bytes < pl->total_bytes) pl->gram = false;
  return check_ws(ws, ws_bytes, pl->min_bytes);
}

last_status cuda_fail(cudaError_t e, const char *what) {
  return fail(LAST_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// Device copies of last_prune_host's tensors after the plan workspace (of `plan_bytes`),
// each 256-byte aligned.
struct HostLayout {
  size_t q, k, x, w, idx, xo, total;
  size_t q_bytes, k_bytes, x_bytes, w_bytes, idx_bytes, xo_bytes;
};
HostLayout host_layout(const Plan &pl, size_t plan_bytes) {
  auto al = [](size_t v) { return (v + kAlign - 1) & ~(size_t)(kAlign - 1); };
  HostLayout h;
  h.q_bytes = (size_t)pl.B * pl.L * pl.Hq * pl.D * pl.elem;
  h.k_bytes = (size_t)pl.L * pl.total_keys * pl.Hkv * pl.D * pl.elem;
  h.x_bytes = (size_t)pl.total_vis * pl.dv * pl.elem;
  h.w_bytes = (size_t)pl.total_vis * sizeof(float);
  h.idx_bytes = (size_t)pl.total_keep * sizeof(int32_t);
  h.xo_bytes = (size_t)pl.total_keep * pl.dv * pl.elem;
  size_t o = al(plan_bytes);
  h.q = o; o += al(h.q_bytes);
  h.k = o; o += al(h.k_bytes);
  h.x = o; o += al(h.x_bytes);
  h.w = o; o += al(h.w_bytes);
  h.idx = o; o += al(h.idx_bytes);
  h.xo = o; o += al(h.xo_bytes);
  h.total = o;
  return h;
}

last_status stage(const Plan &pl, void *ws, cudaStream_t s) {
  cudaError_t e = cudaMemcpyAsync(ws, pl.host_blob.data(), pl.blob_bytes, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return cuda_fail(e, "plan copy");
  return LAST_OK;
}

}  // namespace
}  // namespace last

using namespace last;

extern "C" {

last_status last_workspace_size(const last_problem *p, size_t *bytes) {
  if (bytes == nullptr) return fail(LAST_ERR_INVALID_ARG, "bytes is NULL");
  Plan pl;
  const bool have_seq = p != nullptr && p->cu_seqlens != nullptr && p->vis_start != nullptr &&
                        p->num_layers > 0;
  last_status st = make_plan(p, have_seq, false, &pl);
  if (st != LAST_OK) return st;
  *bytes = pl.total_bytes;
  return LAST_OK;
}

last_status last_scores(const last_problem *p, const void *q, const void *k, float *w_out,
                        void *ws, size_t ws_bytes, void *stream) {
  Plan pl;
  last_status st = make_plan(p, true, false, &pl);
  if (st != LAST_OK) return st;
  if ((st = check_ws(ws, ws_bytes, pl.score_bytes)) != LAST_OK) return st;
  if (pl.total_vis > 0 && (q == nullptr || k == nullptr || w_out == nullptr))
    return fail(LAST_ERR_INVALID_ARG, "q, k and w_out are required");
  if (!aligned16(q) || !aligned16(k)) return fail(LAST_ERR_INVALID_ARG, "q and k must be 16-byte aligned");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if ((st = stage(pl, ws, s)) != LAST_OK) return st;
  cudaError_t e = launch_scores(pl, q, k, w_out, static_cast<char *>(ws), s);
  if (e != cudaSuccess) return cuda_fail(e, "scoring launch");
  return LAST_OK;
}

namespace {
last_status check_select_fits(const last::Plan &pl) {
  std::string why;
  return last::select_fits(pl, &why) ? LAST_OK : fail(LAST_ERR_UNSUPPORTED, why);
}
}  // namespace

last_status last_select(const last_problem *p, const float *w, const void *x, int32_t *idx_out,
                        void *x_out, void *ws, size_t ws_bytes, void *stream) {
  Plan pl;
  last_status st = make_plan(p, false, true, &pl);
  if (st != LAST_OK) return st;
  if ((st = check_select_fits(pl)) != LAST_OK) return st;
  if ((st = check_select_ws(&pl, ws, ws_bytes)) != LAST_OK) return st;
  if (pl.total_keep > 0 && (w == nullptr || x == nullptr || idx_out == nullptr))
    return fail(LAST_ERR_INVALID_ARG, "w, x and idx_out are required");
  if (!aligned16(x) || !aligned16(x_out))
    return fail(LAST_ERR_INVALID_ARG, "x and x_out must be 16-byte aligned");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if ((st = stage(pl, ws, s)) != LAST_OK) return st;
  cudaError_t e = launch_select(pl, w, x, idx_out, x_out, static_cast<char *>(ws), s);
  if (e != cudaSuccess) return cuda_fail(e, "selection launch");
  return LAST_OK;
}

last_status last_select_topk(const last_problem *p, const float *w, const void *x,
                             int32_t *idx_out, void *x_out, void *ws, size_t ws_bytes,
                             void *stream) {
  Plan pl;
  last_status st = make_plan(p, false, false, &pl);
  if (st != LAST_OK) return st;
  if ((st = check_ws(ws, ws_bytes, pl.base_bytes)) != LAST_OK) return st;
  if (pl.total_keep > 0 && (w == nullptr || idx_out == nullptr))
    return fail(LAST_ERR_INVALID_ARG, "w and idx_out are required");
  if (x_out != nullptr) {
    if (p->feat_dim < 8 || p->feat_dim % 8 != 0)
      return fail(LAST_ERR_INVALID_ARG, "feat_dim must be a positive multiple of 8");
    if (pl.total_keep > 0 && x == nullptr)
      return fail(LAST_ERR_INVALID_ARG, "x is required when x_out is given");
    if (!aligned16(x) || !aligned16(x_out))
      return fail(LAST_ERR_INVALID_ARG, "x and x_out must be 16-byte aligned");
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if ((st = stage(pl, ws, s)) != LAST_OK) return st;
  char *wsc = static_cast<char *>(ws);
  cudaError_t e = launch_topk(pl, w, idx_out, wsc, s);
  if (e != cudaSuccess) return cuda_fail(e, "top-k launch");
  if (x_out != nullptr) {
    e = launch_gather(pl, x, idx_out, x_out, wsc, s);
    if (e != cudaSuccess) return cuda_fail(e, "gather launch");
  }
  return LAST_OK;
}

last_status last_gather(const last_problem *p, const void *x, const int32_t *idx, void *x_out,
                        void *ws, size_t ws_bytes, void *stream) {
  Plan pl;
  // Eq. 12 is a row copy: only the row width must suit the kernel's 16-byte copies
  // (the selection's own feature-width limit does not apply)
  last_status st = make_plan(p, false, false, &pl);
  if (st != LAST_OK) return st;
  if (p->feat_dim < 8 || p->feat_dim % 8 != 0)
    return fail(LAST_ERR_INVALID_ARG, "feat_dim must be a positive multiple of 8");
  if ((st = check_ws(ws, ws_bytes, pl.base_bytes)) != LAST_OK) return st;
  if (pl.total_keep > 0 && (x == nullptr || idx == nullptr || x_out == nullptr))
    return fail(LAST_ERR_INVALID_ARG, "x, idx and x_out are required");
  if (!aligned16(x) || !aligned16(x_out))
    return fail(LAST_ERR_INVALID_ARG, "x and x_out must be 16-byte aligned");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if ((st = stage(pl, ws, s)) != LAST_OK) return st;
  cudaError_t e = launch_gather(pl, x, idx, x_out, static_cast<char *>(ws), s);
  if (e != cudaSuccess) return cuda_fail(e, "gather launch");
  return LAST_OK;
}

last_status last_prune(const last_problem *p, const void *q, const void *k, const void *x,
                       float *w_out, int32_t *idx_out, void *x_out, void *ws, size_t ws_bytes,
                       void *stream) {
  Plan pl;
  last_status st = make_plan(p, true, true, &pl);
  if (st != LAST_OK) return st;
  if ((st = check_select_fits(pl)) != LAST_OK) return st;
  if ((st = check_select_ws(&pl, ws, ws_bytes)) != LAST_OK) return st;
  if (pl.total_vis > 0 && (q == nullptr || k == nullptr || x == nullptr))
    return fail(LAST_ERR_INVALID_ARG, "q, k and x are required");
  if (pl.total_keep > 0 && idx_out == nullptr)
    return fail(LAST_ERR_INVALID_ARG, "idx_out is required");
  if (!aligned16(q) || !aligned16(k) || !aligned16(x) || !aligned16(x_out))
    return fail(LAST_ERR_INVALID_ARG, "q, k, x and x_out must be 16-byte aligned");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char *wsc = static_cast<char *>(ws);
  float *w = w_out != nullptr ? w_out : reinterpret_cast<float *>(wsc + pl.off_w);
  if ((st = stage(pl, ws, s)) != LAST_OK) return st;
  cudaError_t e = launch_scores(pl, q, k, w, wsc, s);
  if (e != cudaSuccess) return cuda_fail(e, "scoring launch");
  e = launch_select(pl, w, x, idx_out, x_out, wsc, s);
  if (e != cudaSuccess) return cuda_fail(e, "selection launch");
  return LAST_OK;
}

last_status last_host_workspace_size(const last_problem *p, size_t *bytes) {
  if (bytes == nullptr) return fail(LAST_ERR_INVALID_ARG, "bytes is NULL");
  Plan pl;
  last_status st = make_plan(p, true, true, &pl);
  if (st != LAST_OK) return st;
  *bytes = host_layout(pl, pl.total_bytes).total;
  return LAST_OK;
}

last_status last_prune_host(const last_problem *p, const void *q, const void *k, const void *x,
                            float *w_out, int32_t *idx_out, void *x_out, void *ws, size_t ws_bytes,
                            void *stream) {
  Plan pl;
  last_status st = make_plan(p, true, true, &pl);
  if (st != LAST_OK) return st;
  if ((st = check_select_fits(pl)) != LAST_OK) return st;
  HostLayout h = host_layout(pl, pl.total_bytes);
  if (ws_bytes < h.total) {   // no room for the matrices: the rounds read X
    h = host_layout(pl, pl.min_bytes);
    pl.gram = false;
  }
  if (ws == nullptr) return fail(LAST_ERR_INVALID_ARG, "workspace is NULL");
  if ((reinterpret_cast<uintptr_t>(ws) & (kAlign - 1)) != 0)
    return fail(LAST_ERR_INVALID_ARG, "workspace must be 256-byte aligned");
  if (ws_bytes < h.total)
    return fail(LAST_ERR_WORKSPACE_TOO_SMALL,
                "last_prune_host's workspace needs " + std::to_string(h.total) + " bytes");
  if (pl.total_vis > 0 && (q == nullptr || k == nullptr || x == nullptr))
    return fail(LAST_ERR_INVALID_ARG, "q, k and x are required");
  if (pl.total_keep > 0 && idx_out == nullptr)
    return fail(LAST_ERR_INVALID_ARG, "idx_out is required");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char *wsc = static_cast<char *>(ws);
  void *qd = wsc + h.q, *kd = wsc + h.k, *xd = wsc + h.x, *xod = wsc + h.xo;
  float *wd = reinterpret_cast<float *>(wsc + h.w);
  int32_t *idd = reinterpret_cast<int32_t *>(wsc + h.idx);
  cudaError_t e = cudaSuccess;
  // one copy per tensor
  if (h.q_bytes && e == cudaSuccess) e = cudaMemcpyAsync(qd, q, h.q_bytes, cudaMemcpyHostToDevice, s);
  if (h.k_bytes && e == cudaSuccess) e = cudaMemcpyAsync(kd, k, h.k_bytes, cudaMemcpyHostToDevice, s);
  if (h.x_bytes && e == cudaSuccess) e = cudaMemcpyAsync(xd, x, h.x_bytes, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return cuda_fail(e, "host-to-device copy");
  if ((st = stage(pl, ws, s)) != LAST_OK) return st;
  e = launch_scores(pl, qd, kd, wd, wsc, s);
  if (e != cudaSuccess) return cuda_fail(e, "scoring launch");
  e = launch_select(pl, wd, xd, idd, x_out != nullptr ? xod : nullptr, wsc, s);
  if (e != cudaSuccess) return cuda_fail(e, "selection launch");
  if (h.idx_bytes && e == cudaSuccess)
    e = cudaMemcpyAsync(idx_out, idd, h.idx_bytes, cudaMemcpyDeviceToHost, s);
  if (x_out != nullptr && h.xo_bytes && e == cudaSuccess)
    e = cudaMemcpyAsync(x_out, xod, h.xo_bytes, cudaMemcpyDeviceToHost, s);
  if (w_out != nullptr && h.w_bytes && e == cudaSuccess)
    e = cudaMemcpyAsync(w_out, wd, h.w_bytes, cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return cuda_fail(e, "device-to-host copy");
  return LAST_OK;
}

last_status last_poll(const void *ws, void *stream) {
  if (ws == nullptr) return fail(LAST_ERR_INVALID_ARG, "workspace is NULL");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  unsigned flag = 0;
  cudaError_t e = cudaMemcpyAsync(&flag, ws, sizeof flag, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "poll");
  if (flag & kErrConfig)
    return fail(LAST_ERR_CUDA, "internal error: a kernel's shared-memory plan exceeded its launch; "
                               "outputs of that call are invalid");
  if (flag & kErrTimeout)
    return fail(LAST_ERR_TIMEOUT, "a bounded device wait expired; outputs of that call are invalid");
  if (flag & kErrGatherIndex)
    return fail(LAST_ERR_DEVICE_INDEX, "a gather index was outside [0, N_b)");
  return LAST_OK;
}

int32_t last_budget(int32_t n_vis, int32_t num, int32_t den) {
  if (n_vis < 0 || num < 0 || den <= 0) return -1;
  const long long prod = (long long)num * n_vis;
  long long kq = prod / den;
  if (kq * den < prod) ++kq;
  return kq > 0x7fffffffLL ? -1 : (int32_t)kq;
}

const char *last_status_string(last_status s) {
  switch (s) {
    case LAST_OK: return "LAST_OK";
    case LAST_ERR_INVALID_ARG: return "LAST_ERR_INVALID_ARG";
    case LAST_ERR_UNSUPPORTED: return "LAST_ERR_UNSUPPORTED";
    case LAST_ERR_WORKSPACE_TOO_SMALL: return "LAST_ERR_WORKSPACE_TOO_SMALL";
    case LAST_ERR_CUDA: return "LAST_ERR_CUDA";
    case LAST_ERR_DEVICE_INDEX: return "LAST_ERR_DEVICE_INDEX";
    case LAST_ERR_TIMEOUT: return "LAST_ERR_TIMEOUT";
  }
  return "LAST_ERR_UNKNOWN";
}

const char *last_error_message(void) { return g_error.c_str(); }

}  // extern "C"
