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
