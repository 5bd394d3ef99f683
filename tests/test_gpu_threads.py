"""Host threads that run one kernel at different sizes, each on its own stream and workspace.
How much shared memory a kernel may be launched with is a property of the process: a thread
with a small problem must not lower it under one with a large problem."""
import threading

import numpy as np
import pytest

import paper_2607_27952_gb300 as last

pytestmark = pytest.mark.gpu


def _problem(n, k, dtype="f32", batch=1, layers=1, heads=4, kv=4, d=64):
    cu = np.arange(batch + 1)
    return last.Problem(batch=batch, num_layers=layers, num_q_heads=heads, num_kv_heads=kv, head_dim=d,
                        feat_dim=64, dtype=dtype, cu_seqlens=cu * (n + 40), vis_start=[0] * batch,
                        cu_vis=cu * n, cu_keep=cu * k)


def _rand(shape, dtype, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda").to(torch.float32 if dtype == "f32" else torch.bfloat16)


def _call(kind, big, seed):
    """A closure that runs one call and returns its (device) result."""
    import torch
    n = 1400 if big else 130
    dtype = "f32" if kind == "select_f32" else "bf16"
    w = torch.rand(n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))
    if kind.startswith("select"):
        p = _problem(n, n // 20, dtype)
        x, idx, ws = _rand((n, 64), dtype, seed), torch.empty(n // 20, dtype=torch.int32, device="cuda"), last.workspace(p)

        def run(s):
            last.last_select(p, w, x, idx, ws, stream=s)
            return idx
    elif kind == "topk":
        n = 40000 if big else 11000
        p = _problem(n, 500, dtype)
        w = torch.rand(n, device="cuda")
        idx, ws = torch.empty(500, dtype=torch.int32, device="cuda"), last.workspace(p)

        def run(s):
            last.last_select_topk(p, w, idx, ws, stream=s)
            return idx
    elif kind == "rows":   # 256 or 128 query columns
        m = 32 if big else 16
        p = _problem(n, 0, dtype, heads=8, kv=1)
        rows = last.QueryRows([0, m], np.arange(n + 1, n + 1 + m))
        q, k = _rand((m, 1, 8, 64), dtype, seed), _rand((1, n + 40, 1, 64), dtype, seed + 1)
        out, ws = torch.empty(n, device="cuda"), last.rows_workspace(p, rows, torch.device("cuda"))

        def run(s):
            last.last_scores_rows(p, rows, q, k, out, ws, stream=s)
            return out
    else:                  # scores: 5000 or 4500 (layer, head) pairs in one token tile
        layers = 50 if big else 45
        p = _problem(130, 0, dtype, layers=layers, heads=100, kv=100, d=8)
        q, k = _rand((1, layers, 100, 8), dtype, seed), _rand((layers, 170, 100, 8), dtype, seed + 1)
        out, ws = torch.empty(130, device="cuda"), last.workspace(p)

        def run(s):
            last.last_scores(p, q, k, out, ws, stream=s)
            return out
    return run


@pytest.mark.parametrize("kind", ["select_f32", "select_bf16", "topk", "rows", "scores"])
def test_threads_with_different_sizes(kind):
    import torch
    calls = [_call(kind, i % 2 == 0, 10 + i) for i in range(6)]
    torch.cuda.synchronize()
    want = [run(torch.cuda.current_stream()).clone() for run in calls]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in calls]
    errors, start = [], threading.Barrier(len(calls))

    def work(i):
        start.wait()
        try:
            for r in range(400):
                calls[i](streams[i])
                if r % 50 == 49:
                    streams[i].synchronize()
        except Exception as e:   # reported by the main thread
            errors.append(f"thread {i}: {e}")

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for i, run in enumerate(calls):
        assert torch.equal(run(torch.cuda.current_stream()), want[i])
