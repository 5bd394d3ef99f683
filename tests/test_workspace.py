"""Sizes of the caller's workspace: what a call takes at least grows with its problem, also
where the reported size does not because it holds Gram matrices.  Host checks only (the
calls stop at a misaligned pointer, after the size has been accepted)."""
import numpy as np
import pytest

import paper_2607_27952_gb300 as last
from gpu_util import least_workspace


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2607_27952_gb300.build import build
    build()
    return last.load_library()


def _problem(batch, n, k, dtype="bf16", dv=2048, text=4):
    cu = np.arange(batch + 1)
    return last.Problem(batch=batch, num_layers=1, num_q_heads=4, num_kv_heads=4, head_dim=64, feat_dim=dv,
                        dtype=dtype, cu_seqlens=cu * (n + text), vis_start=[0] * batch, cu_vis=cu * n,
                        cu_keep=cu * k)


def _accepts(call, *args):
    """Whether a call gets past its workspace check, to the one for aligned pointers."""
    with pytest.raises(last.LastError) as e:
        call(*args)
    if e.value.status == last.LAST_ERR_WORKSPACE_TOO_SMALL:
        return False
    assert e.value.status == last.LAST_ERR_INVALID_ARG and "align" in str(e.value)
    return True


def _select(prob, n):
    return _accepts(lambda: last.last_select(prob, 256, 24, 256, (256, n), stream=0))


def _prune(prob, n):
    return _accepts(lambda: last.last_prune(prob, 256, 256, 24, None, 256, None, (256, n), stream=0))


def test_a_larger_batchs_workspace_serves_a_smaller_one():
    """13 requests of 16384 tokens are past the matrices' 12 GiB and report 57 MB; 12 of them
    report 12.9 GB and run in the 57 MB all the same, as do other budgets."""
    large = last.last_workspace_size(_problem(13, 16384, 2048))
    assert large < 1 << 27 < 1 << 33 < last.last_workspace_size(_problem(12, 16384, 2048))
    for batch, k in [(12, 2048), (8, 2048), (8, 64), (1, 1000), (13, 24)]:
        assert _select(_problem(batch, 16384, k), large) and _prune(_problem(batch, 16384, k), large)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("batch,n", [(1, 6), (3, 40), (1, 576), (64, 576), (8, 16384), (2, 9000)])
def test_the_size_for_keeping_all_is_enough_for_every_budget(batch, n, dtype):
    all_of_them = last.last_workspace_size(_problem(batch, n, n, dtype, dv=512))
    for k in sorted({1, 2, min(n, 32), n // 2, n - 1, n}):
        prob = _problem(batch, n, k, dtype, dv=512)
        least = least_workspace(prob)
        assert least <= min(all_of_them, last.last_workspace_size(prob))
        for call in (_select, _prune):
            assert call(prob, least) and call(prob, all_of_them) and not call(prob, least - 1)


def test_the_least_size_grows_with_the_problem():
    sizes = [least_workspace(_problem(b, n, k)) for b, n, k in
             [(1, 30, 5), (1, 200, 5), (1, 1000, 5), (1, 1000, 300), (8, 1000, 300), (12, 16384, 300),
              (12, 16384, 2048), (13, 16384, 2048), (13, 16384, 16384)]]
    assert sizes == sorted(sizes)
    for dtype in ("bf16", "f32"):   # up to four long requests may run on the whole GPU
        sizes = [least_workspace(_problem(b, 5000, 5, dtype, dv=64)) for b in (1, 4, 5, 9)]
        assert sizes == sorted(sizes)


def test_small_matrices_always_have_their_room():
    """A few requests of some tens of tokens report what they need at least: one byte less is
    refused."""
    prob = _problem(2, 60, 9, dv=256)
    assert last.last_workspace_size(prob) == least_workspace(prob)


def test_prune_host_takes_less_than_the_matrices():
    prob = _problem(8, 16384, 2048)
    full = last.last_host_workspace_size(prob)
    least = least_workspace(prob) + full - last.last_workspace_size(prob)
    assert full - least > 8 << 30

    def call(n):   # (all arguments are checked before the first copy: a missing idx_out ends it)
        with pytest.raises(last.LastError) as e:
            last.last_prune_host(prob, 16, 16, 16, None, None, None, (256, n), stream=0)
        return e.value.status
    assert call(full) == call(least) == last.LAST_ERR_INVALID_ARG
    assert call(least - 1) == last.LAST_ERR_WORKSPACE_TOO_SMALL


def test_python_workspaces_do_without_the_matrices_when_memory_is_short(monkeypatch):
    import torch
    real = torch.empty

    def empty(n, **kw):
        if n > 2 << 30:
            raise torch.OutOfMemoryError("as on a device with 2 GiB free")
        return real(n, **kw)
    monkeypatch.setattr(torch, "empty", empty)
    prob = _problem(8, 16384, 2048)
    assert _select(prob, last.workspace(prob, "meta").numel())
    assert last.host_workspace(prob, "meta").numel() < 2 << 30
    with pytest.raises(torch.OutOfMemoryError):   # no smaller one to fall back on
        last.workspace(_problem(1000, 16384, 16384), "meta")


@pytest.mark.parametrize("dtype,batch,n,dv,k,matrix_us,rounds_us", [
    ("bf16", 8, 16384, 64, 2, 1723, 303), ("bf16", 8, 16384, 256, 64, 1925, 943),
    ("bf16", 8, 16384, 1024, 32, 2247, 1411), ("bf16", 8, 16384, 1024, 256, 2372, 3241),
    ("bf16", 8, 16384, 2048, 256, 3323, 6006), ("bf16", 1, 50000, 64, 2, 1971, 564),
    ("bf16", 1, 50000, 256, 32, 2153, 1575), ("bf16", 1, 50000, 64, 256, 2338, 3214),
    ("bf16", 2, 16384, 64, 4, 491, 390), ("bf16", 2, 16384, 512, 64, 603, 1044),
    ("bf16", 64, 2048, 64, 2, 317, 254), ("bf16", 64, 2048, 64, 32, 365, 604),
    ("bf16", 64, 2048, 2048, 64, 720, 2512), ("bf16", 128, 2048, 64, 2, 556, 400),
    ("bf16", 16, 4096, 256, 2, 278, 208), ("bf16", 16, 4096, 1024, 32, 393, 734),
    ("bf16", 32, 2880, 512, 2, 331, 273), ("bf16", 32, 2880, 2048, 8, 648, 978),
    ("bf16", 256, 576, 64, 2, 216, 322), ("bf16", 16, 576, 64, 2, 98, 110),
    ("f32", 1, 4096, 8, 2, 245, 120), ("f32", 8, 1200, 64, 8, 203, 141), ("f32", 8, 1200, 64, 32, 220, 276),
    ("f32", 1, 12000, 8, 8, 1834, 455), ("f32", 1, 4096, 256, 32, 268, 308), ("f32", 8, 1200, 512, 32, 298, 228),
    ("f32", 1, 576, 1024, 2, 39, 30), ("f32", 1, 4096, 8, 32, 284, 877),
])
def test_a_matrix_is_used_where_it_was_measured_faster(dtype, batch, n, dv, k, matrix_us, rounds_us):
    """The matrix's bytes count as well as its products: narrow features at small budgets are
    cheaper in rounds over X.  Both sides as measured on a GB300; a matrix shows in the
    reported size."""
    prob = _problem(batch, n, k, dtype, dv=dv)
    assert (last.last_workspace_size(prob) > least_workspace(prob)) == (matrix_us < rounds_us)


def test_only_requests_with_a_choice_count():
    """A request that keeps all its tokens needs no matrix and says nothing about the budgets
    of those that do."""
    cu = np.array([0, 16384, 32768, 33768])

    def size(keep_all):
        prob = last.Problem(batch=3, num_layers=0, num_q_heads=0, num_kv_heads=0, head_dim=0, feat_dim=64,
                            dtype="bf16", cu_seqlens=None, vis_start=None, cu_vis=cu,
                            cu_keep=[0, 2, 4, 4 + keep_all])
        return last.last_workspace_size(prob) - least_workspace(prob)
    assert size(0) == size(1000) == 0


def test_no_matrix_is_reserved_for_requests_too_long_for_a_cluster():
    """Past about 53 800 tokens no cluster holds a request's per-token state: its matrix (11 to
    12 GiB) would never be used."""
    for n in (53000, 54000, 56000, 56700):
        prob = _problem(1, n, n // 8)
        used = last.last_workspace_size(prob) - least_workspace(prob) >= 4 * n * n
        assert used == (n < 53800), n
    prob = _problem(1, 56700, 56700 // 8)
    assert last.last_workspace_size(prob) == least_workspace(prob)
