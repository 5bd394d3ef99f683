"""The greedy from a Gram matrix (select_gram.cu; on tensor cores, or in the canonical
order for fp32 and small batches) at the sizes where it can go wrong: around the
128-row and 256-column tiles (of one CTA and of pairs) and the 32-token blocks, one token
more than the cluster's warps hold, feature widths that end inside a K block, every budget from
one pick to all but one, exact ties, zero rows and rows outside the certificate's norm
range.  Indices and rows are exact against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2607_27952_gb300 as last
from gpu_util import (DeviceWorkload, assert_gather_equal, assert_selection_equal, least_workspace,
                      oracle_selection, problem_of, to_dev, to_host_bits)
from workloads import bf16_bits_to_f32, custom, f32_to_bf16_bits

pytestmark = pytest.mark.gpu


def _wl(n_vis, keep, d_v, seed=5, dtype="bf16", **kw):
    return custom(name="gram", seed=seed, batch=len(n_vis), n_vis=n_vis, n_text=4, num_layers=1,
                  num_q_heads=4, num_kv_heads=2, head_dim=64, feat_dim=d_v, dtype=dtype, keep=keep,
                  n_clusters=kw.pop("n_clusters", 12), n_planted=3, **kw)


def _run(wl, x=None, w=None):
    import torch
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(3)
    n = int(wl.cu_vis[-1])
    w = (rng.random(n) + 0.5).astype(np.float32) if w is None else w
    prob = problem_of(wl)
    ws = last.workspace(prob, dev)
    xd = to_dev(wl.x if x is None else x, dev)
    idx = torch.full((int(wl.cu_keep[-1]),), -7, dtype=torch.int32, device=dev)
    xs = torch.zeros((int(wl.cu_keep[-1]), wl.feat_dim), dtype=xd.dtype, device=dev)
    last.last_select(prob, torch.from_numpy(w).to(dev), xd, idx, ws, x_out=xs)
    last.last_poll(ws)
    return w, idx.cpu().numpy(), to_host_bits(xs)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("d_v", [8, 72, 520, 1536, 2048])
@pytest.mark.parametrize("n_vis,keep", [
    ([1, 31, 33, 127, 129], [1, 30, 2, 64, 40]),
    ([255, 256, 257, 513], [254, 1, 100, 60]),
    ([545, 640, 2049], [100, 0, 130]),
    ([8200, 90, 257], [60, 20, 60]),       # CTA pairs
    # enough for the tensor cores at any width, one CTA a tile
    ([1900, 255, 256, 257, 513, 127, 129, 33, 700, 96], [90, 200, 3, 100, 60, 64, 20, 2, 50, 95]),
])
def test_selection_equals_the_oracle(n_vis, keep, d_v, dtype):
    wl = _wl(n_vis, keep, d_v, dtype=dtype)
    w, idx, xs = _run(wl)
    assert_selection_equal(wl, w, idx, range(wl.batch))
    assert_gather_equal(wl, idx, xs, range(wl.batch))


@pytest.mark.parametrize("dtype,n", [("bf16", 300), ("bf16", 1900), ("f32", 300)])
def test_ties_zero_rows_and_extreme_norms(dtype, n):
    d = 512   # 300 tokens: canonical matrix, 1900: tensor cores
    wl = _wl([n], [150], d, dtype=dtype)
    x = (bf16_bits_to_f32(wl.x) if dtype == "bf16" else wl.x).copy()
    x[10:60] = x[9]                      # exact duplicates
    x[60:70] = 0.0
    x[70:110] *= np.float32(2.0) ** -70   # outside the certificate's norm range
    x[110:150] *= np.float32(2.0) ** 55
    wl.x = f32_to_bf16_bits(x) if dtype == "bf16" else x
    w = np.full(n, 1.0 / n, dtype=np.float32)
    w[:5] = 0.0
    w, idx, _ = _run(wl, w=w)
    assert np.array_equal(idx, np.sort(oracle_selection(wl, w, 0)))


@pytest.mark.parametrize("batch,k", [(13, 200), (8, 20)])
def test_batches_past_the_matrix_keep_the_rounds_over_x(batch, k):
    """13 requests of 16384 tokens are past the matrices' 12 GiB, 8 with 20 picks are
    cheaper without them: the clustered kernel that streams X (and skips rows) takes both.
    One request's features repeated, other weights per request."""
    import torch
    n, d = 16384, 2048
    rng = np.random.default_rng(8)
    x = rng.standard_normal((n // 512, 512, d), dtype=np.float32)
    x[1:] *= 0.05
    x = f32_to_bf16_bits(np.cumsum(x, 0).reshape(n, d))
    w = (1.0 + 0.01 * rng.random((batch, n))).astype(np.float32)
    prob = last.Problem(batch=batch, num_layers=0, num_q_heads=0, num_kv_heads=0, head_dim=0, feat_dim=d,
                        dtype="bf16", cu_seqlens=None, vis_start=None, cu_vis=np.arange(batch + 1) * n,
                        cu_keep=np.arange(batch + 1) * k)
    ws = last.workspace(prob, "cuda:0")
    idx = torch.full((batch * k,), -7, dtype=torch.int32, device="cuda:0")
    last.last_select(prob, torch.from_numpy(w).cuda(), to_dev(x, torch.device("cuda:0")).repeat(batch, 1), idx, ws)
    last.last_poll(ws)
    got = idx.cpu().numpy().reshape(batch, k)
    for b in (0, batch - 1):
        assert np.array_equal(got[b], np.sort(oracle.select_fp32(x, w[b], k)))


def test_best_tokens_on_one_lane_of_every_warp():
    """A lane queues its three best tokens, the third of them taken bounds the rest.  Every
    token of weight sits on the same lane (tokens are dealt in blocks of 32), and so many
    requests run on one CTA each, whose warps hold four or five blocks."""
    import torch
    batch, n, d, k = 150, 2100, 512, 40
    rng = np.random.default_rng(9)
    x = f32_to_bf16_bits(rng.standard_normal((n, d), dtype=np.float32))
    at = np.arange(n)
    w = np.where(at % 32 == 5, 1.0 + rng.random((batch, n)), 1e-3 * rng.random((batch, n))).astype(np.float32)
    prob = last.Problem(batch=batch, num_layers=0, num_q_heads=0, num_kv_heads=0, head_dim=0, feat_dim=d,
                        dtype="bf16", cu_seqlens=None, vis_start=None, cu_vis=np.arange(batch + 1) * n,
                        cu_keep=np.arange(batch + 1) * k)
    ws = last.workspace(prob, "cuda:0")
    idx = torch.full((batch * k,), -7, dtype=torch.int32, device="cuda:0")
    last.last_select(prob, torch.from_numpy(w).cuda(), to_dev(x, torch.device("cuda:0")).repeat(batch, 1), idx, ws)
    last.last_poll(ws)
    got = idx.cpu().numpy().reshape(batch, k)
    for b in (0, 70, batch - 1):
        assert np.array_equal(got[b], np.sort(oracle.select_fp32(x, w[b], k)))


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_without_room_for_the_matrices(dtype):
    """last_select, last_prune and last_prune_host with the least workspace they take, and with
    one byte less than the matrices need: the rounds over X give the same picks."""
    import torch
    wl = _wl([900, 40, 1300], [130, 40, 70], 256, dtype=dtype)
    dw, prob, rng = DeviceWorkload(wl), problem_of(wl), np.random.default_rng(3)
    w = (rng.random(int(wl.cu_vis[-1])) + 0.5).astype(np.float32)
    want = dw.select(w, path="matrix")
    assert np.array_equal(dw.select(w, path="rounds"), want)
    assert_selection_equal(wl, w, want, range(wl.batch))
    least, full = least_workspace(prob), last.last_workspace_size(prob)
    w_full, idx_full, xs_full = dw.prune()
    for n in (least, full - 1):
        w_out, idx, xs = dw.outputs()
        ws = torch.empty(n, dtype=torch.uint8, device=dw.dev)
        last.last_prune(prob, dw.q, dw.k, dw.x, w_out, idx, xs, ws)
        last.last_poll(ws)
        assert np.array_equal(idx.cpu().numpy(), idx_full)
        assert np.array_equal(to_host_bits(xs), xs_full) and np.array_equal(w_out.cpu().numpy(), w_full)
    host = [t.cpu().pin_memory() for t in (dw.q, dw.k, dw.x)]
    out = torch.empty(int(wl.cu_keep[-1]), dtype=torch.int32).pin_memory()
    ws = torch.empty(last.last_host_workspace_size(prob) - full + least, dtype=torch.uint8, device=dw.dev)
    last.last_prune_host(prob, *host, None, out, None, ws)
    last.last_poll(ws)
    assert np.array_equal(out.numpy(), idx_full)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_weights_below_zero_once_all_tokens_are_candidates(dtype):
    """Scores are never negative and the rounds rely on keys that only fall; weights below zero
    are still taken in their order when the tokens left fit the candidate list (canonical
    matrix: the replay follows w times the smaller distance, whatever w's sign)."""
    rng = np.random.default_rng(5)
    n, d = 400, 512
    x = (rng.standard_normal((60, d))[rng.integers(0, 60, n)] + 0.05 * rng.standard_normal((n, d))).astype(np.float32)
    x[20:60] = x[19]
    w = (rng.random(n).astype(np.float32) - np.float32(0.3))
    wl = _wl([n], [n - 3], d, dtype=dtype)
    w, idx, _ = _run(wl, w=w, x=_put(wl, x))
    assert np.array_equal(idx, np.sort(oracle_selection(wl, w, 0)))


def _put(wl, x):
    wl.x = f32_to_bf16_bits(x) if wl.dtype == "bf16" else x
    return wl.x
