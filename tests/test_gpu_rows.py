"""GPU parity of the multi-row attention sources (Table 4: First, Middle, All Mean)
against the oracle, through the C ABI: scores within rtol 1e-3."""
import numpy as np
import pytest

import oracle
from workloads import bf16_bits_to_f32, config, custom, f32_to_bf16_bits, query_rows

from gpu_util import SCORE_ATOL, SCORE_RTOL, problem_of, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2607_27952_gb300.build import build
    import paper_2607_27952_gb300 as last
    build()
    last.load_library()
    oracle.build()


def make_rows(wl, source, rng, m_rows=8):
    """Query rows of the given source (First, Middle, Last or All Mean over up to
    m_rows text rows), seeded from rng."""
    return query_rows(wl, source, m_rows=m_rows, seed=int(rng.integers(1 << 30)))


def run_rows(wl, cu, pos, q):
    import torch
    import paper_2607_27952_gb300 as last
    dev = torch.device("cuda:0")
    prob = problem_of(wl)
    rows = last.QueryRows(cu, pos)
    w = torch.full((int(wl.cu_vis[-1]),), float("nan"), dtype=torch.float32, device=dev)
    ws = last.rows_workspace(prob, rows, dev)
    last.last_scores_rows(prob, rows, to_dev(q, dev), to_dev(wl.k, dev), w, ws)
    last.last_poll(ws)
    return w.cpu().numpy()


def check(wl, cu, pos, q):
    w_gpu = run_rows(wl, cu, pos, q)
    w_ref = oracle.scores_rows(q, wl.k, wl.cu_seqlens, wl.vis_start, wl.cu_vis, cu, pos,
                               num_kv_heads=wl.num_kv_heads, scale=wl.scale)
    assert np.isfinite(w_gpu).all()
    err = np.abs(w_gpu.astype(np.float64) - w_ref)
    bad = err > SCORE_RTOL * np.abs(w_ref) + SCORE_ATOL
    assert not bad.any(), f"{bad.sum()} scores outside rtol; worst {(err / w_ref).max():.2e}"
    return w_gpu


CASES = {
    "c2": lambda: config("c2", batch=4, budget="mixed"),
    "c3": lambda: config("c3", batch=2, n_vis=1152),
    "c5": lambda: config("c5", batch=2, n_vis=1024, budget=12.5),
    "gqa8_d64": lambda: custom(name="g8d64", seed=61, batch=3, n_vis=[200, 77, 300],
                               n_text=[40, 12, 3], n_before=[5, 0, 17], num_layers=2,
                               num_q_heads=16, num_kv_heads=2, head_dim=64, feat_dim=64,
                               dtype="bf16"),
    "mha_d256": lambda: custom(name="d256", seed=62, batch=2, n_vis=[130, 260], n_text=[9, 70],
                               num_layers=1, num_q_heads=4, num_kv_heads=4, head_dim=256,
                               feat_dim=64, dtype="bf16"),
}


@pytest.mark.parametrize("source", ["first", "middle", "last", "all"])
@pytest.mark.parametrize("name", list(CASES))
def test_rows_match_oracle(name, source):
    wl = CASES[name]()
    cu, pos, q = make_rows(wl, source, np.random.default_rng(7))
    check(wl, cu, pos, q)


def test_last_row_equals_single_row_scoring():
    """The Last source is the method's own Eq. 6-8: one row per request runs the
    last-row scoring kernels (cut after the row), so it equals last_scores bit for
    bit."""
    from gpu_util import DeviceWorkload
    wl = CASES["c3"]()
    cu, pos, q = make_rows(wl, "last", np.random.default_rng(8))
    w_rows = check(wl, cu, pos, q)
    w_one = DeviceWorkload(wl).scores()
    assert np.array_equal(w_rows.view(np.uint32), w_one.view(np.uint32))


def test_single_row_beyond_the_last_row_kernels():
    """G = 16 q-heads per kv-head is past the last-row kernels (G <= 8): one row per
    request then runs on the multi-row kernels, still within tolerance."""
    wl = custom(name="g16", seed=64, batch=3, n_vis=[120, 40, 260], n_text=[30, 5, 64],
                num_layers=1, num_q_heads=32, num_kv_heads=2, head_dim=64, feat_dim=64,
                dtype="bf16")
    for source in ("first", "middle"):
        cu, pos, q = make_rows(wl, source, np.random.default_rng(10))
        check(wl, cu, pos, q)


def test_many_rows_full_width():
    """64 rows x G = 4 = 256 MMA columns (the limit), ragged row counts."""
    wl = custom(name="wide", seed=63, batch=3, n_vis=[300, 500, 64], n_text=[80, 64, 200],
                num_layers=1, num_q_heads=8, num_kv_heads=2, head_dim=128, feat_dim=64,
                dtype="bf16")
    cu, pos, q = make_rows(wl, "all", np.random.default_rng(9), m_rows=64)
    assert int(np.diff(cu).max()) == 64
    check(wl, cu, pos, q)


@pytest.mark.parametrize("hq,hkv,D,m_rows,n_vis,n_text,n_before", [
    (9, 3, 64, 43, [129, 255, 257], [60, 47, 50], [0, 127, 128]),   # 129 columns: two epilogue groups
    (8, 1, 256, 32, [128, 1], [40, 34], [1, 5]),                    # 256 columns, one stage
    (4, 4, 128, 5, [2000, 31, 640], [7, 129, 8], [128, 0, 63]),     # more items than stages and CTAs
])
def test_chunk_edges_and_column_counts(hq, hkv, D, m_rows, n_vis, n_text, n_before):
    wl = custom(name="edges", seed=71, batch=len(n_vis), n_vis=n_vis, n_text=n_text, n_before=n_before,
                num_layers=2, num_q_heads=hq, num_kv_heads=hkv, head_dim=D, feat_dim=64, dtype="bf16",
                keep=[1] * len(n_vis), n_planted=1)
    check(wl, *make_rows(wl, "all", np.random.default_rng(3), m_rows=m_rows))


@pytest.mark.parametrize("masked", [(32, 64), (128, 256), (32, 256)])
def test_keys_whose_logits_are_minus_infinity(masked):
    """Visual keys whose products overflow to -inf take no part in the softmax, also where they
    fill a warp's 32 keys or a whole 128-key chunk that every row sees."""
    wl = custom(name="inf", seed=72, batch=1, n_vis=[400], n_text=[8], num_layers=1, num_q_heads=4,
                num_kv_heads=2, head_dim=64, feat_dim=64, dtype="bf16", keep=[1], n_planted=1)
    cu, pos, q = make_rows(wl, "all", np.random.default_rng(4), m_rows=6)
    big, low = f32_to_bf16_bits(np.float32([3e38, -3e38]))
    v0 = int(wl.vis_start[0])
    wl.k[..., 0] = 0
    wl.k[:, v0 + masked[0]:v0 + masked[1], :, 0] = low
    q[..., 0] = big
    w = check(wl, cu, pos, q)
    assert (w[masked[0]:masked[1]] == 0).all() and (np.delete(w, np.arange(*masked)) > 0).all()


def test_sums_over_many_chunks_keep_their_precision():
    """32 requests of 16384 keys, two rows of one head with near-uniform attention: the error of
    w~ against 64 bits is that of sums of about 130 chunks.  Every chunk's sum is scaled once,
    against the row's maximum, so the root mean square over the requests stays below one
    unit in the last place of 1 (2^-23); rescaling a running sum gives 1.5 of them."""
    import torch
    import paper_2607_27952_gb300 as last
    B, n, P, D = 32, 16384, 16400, 64
    rng = np.random.default_rng(73)
    k = f32_to_bf16_bits(rng.standard_normal((1, B * P, 1, D), dtype=np.float32))
    q = f32_to_bf16_bits(np.float32(0.3) * rng.standard_normal((2 * B, 1, 1, D), dtype=np.float32))
    cu, pos = np.arange(B + 1), np.tile([P - 9, P - 1], B)
    prob = last.Problem(batch=B, num_layers=1, num_q_heads=1, num_kv_heads=1, head_dim=D, feat_dim=8,
                        dtype="bf16", cu_seqlens=cu * P, vis_start=[0] * B, cu_vis=cu * n, cu_keep=cu * 0)
    rows, dev = last.QueryRows(cu * 2, pos), torch.device("cuda:0")
    w = torch.empty(B * n, dtype=torch.float32, device=dev)
    ws = last.rows_workspace(prob, rows, dev)
    last.last_scores_rows(prob, rows, to_dev(q, dev), to_dev(k, dev), w, ws)
    last.last_poll(ws)
    got = w.cpu().numpy().astype(np.float64).reshape(B, n)
    kd = bf16_bits_to_f32(k).astype(np.float64).reshape(B, P, D)
    qd = bf16_bits_to_f32(q).astype(np.float64).reshape(B, 2, D)
    z = np.einsum("brd,bpd->brp", qd, kd) / 8.0
    z[:, 0, P - 8:] = -np.inf
    a = np.exp(z - z.max(2, keepdims=True))
    a = (a / a.sum(2, keepdims=True)).sum(1)[:, :n]
    want = a / a.sum(1, keepdims=True)
    err = np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)
    assert np.sqrt((err ** 2).mean()) < 2.0 ** -23
