"""The calls that a user of this library makes, as measurable cases.

A case is one call of a public entry point on one ragged batch: the whole path
(`last_prune`, `last_prune_host`), the scores alone (`last_scores`), the
multi-row attention sources (`last_scores_rows`) and the Top-k variant with its
gather (`last_select_topk`).  Sizes are those of the benchmark presets (one image
in fp32, a batch of LLaVA-1.5-shaped images, tiled images, dynamic resolution,
video) plus the smallest call and an odd-sized fp32 batch like the tests' ones.

Inputs are drawn on the GPU with the value models of `workloads/`: q and K are
N(0, 1)/sqrt(D), ten keys per request are planted three standard deviations up,
features are unit-norm cluster centres plus noise of norm 0.1 (optionally with
near-duplicate tokens) or a per-frame random walk (video).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2607_27952_gb300 as last

# Work of the largest listed selection (8 video requests, 16384 tokens, k = 2048):
# a drawn case stays at or below it.
_MAX_PAIRS = 8 * 16384 * 2048
_MAX_TOKENS = 8 * 16384


def _case(name, call, batch, n_lo, n_hi, t_lo, t_hi, layers, hq, hkv, d, dv, dtype, keep,
          clusters=64, dup=0.0, frame=0, rows=0):
    """keep: "num/den" of the visual tokens, or budgets "a,b,c" taken round-robin.
    n_lo..n_hi / t_lo..t_hi: visual and text tokens per request.  frame > 0: video
    features of that many tokens per frame.  rows: query rows per request."""
    c = dict(call=call, batch=batch, n_lo=n_lo, n_hi=n_hi, t_lo=t_lo, t_hi=t_hi, layers=layers,
             hq=hq, hkv=hkv, d=d, dv=dv, dtype=dtype, keep=keep, clusters=clusters, dup=dup,
             frame=frame, rows=rows)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one image on the edge device, fp32 features: the smallest call, latency
        _case("image-f32", "prune", 1, 576, 576, 32, 32, 1, 16, 16, 64, 1024, "f32", "72", 24),
        # one image whose q, K and features arrive in pinned host memory
        _case("image-host", "prune_host", 1, 576, 576, 48, 48, 1, 16, 16, 128, 2048, "bf16", "64"),
        # fp32 features, ragged and odd sizes (feature width 1000, head width 80, GQA 8)
        _case("odd-f32", "prune", 6, 257, 1201, 5, 77, 2, 16, 2, 80, 1000, "f32", "1/8", 40),
        # a server's batch of 576-token images with three budgets
        _case("images", "prune", 64, 576, 576, 16, 128, 1, 16, 16, 128, 2048, "bf16", "64,128,192"),
        # tiled high-resolution images, four layers summed, near-duplicate tokens
        _case("tiles", "prune", 32, 2880, 2880, 64, 64, 4, 16, 4, 128, 2048, "bf16", "360", 128, 0.3),
        # dynamic resolution: ragged 256..4096 tokens per request
        _case("ragged", "prune", 128, 256, 4096, 8, 256, 1, 12, 2, 128, 1536, "bf16", "1/8"),
        # one video request at a small budget
        _case("video-one", "prune", 1, 16384, 16384, 128, 128, 1, 16, 4, 128, 2048, "bf16", "1/20",
              0, 0.0, 512),
        # the largest: a batch of video requests
        _case("video", "prune", 8, 16384, 16384, 128, 128, 1, 16, 4, 128, 2048, "bf16", "1/8",
              0, 0.0, 512),
        # the scores alone, four layers (a caller with its own selection)
        _case("scores-tiles", "scores", 32, 2880, 2880, 64, 64, 4, 16, 4, 128, 2048, "bf16", "1/8"),
        # attention source "All Mean": 32 query rows per request
        _case("rows-images", "rows", 64, 576, 576, 40, 128, 1, 16, 16, 128, 2048, "bf16", "1/8",
              rows=32),
        _case("rows-video", "rows", 8, 16384, 16384, 128, 128, 1, 16, 4, 128, 2048, "bf16", "1/8",
              rows=32),
        # Top-k variant with the gather of the kept rows
        _case("topk-video", "topk", 8, 16384, 16384, 128, 128, 1, 16, 4, 128, 2048, "bf16", "1/8",
              0, 0.0, 512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["prune", "prune", "prune", "prune", "prune_host", "scores", "rows", "topk"])
    dtype = "f32" if call in ("prune", "scores") and rng.random() < 0.2 else "bf16"
    hq, hkv = rng.choice([(16, 16), (16, 4), (12, 2), (14, 2), (16, 2), (8, 8)])
    if dtype == "f32":   # one image or a small batch
        n = _log_int(rng, 64, 1400)
        batch = _log_int(rng, 1, max(1, min(8, 6000 // n)))
        dv, d = rng.choice([512, 768, 1000, 1024]), rng.choice([64, 80])
    else:
        n = _log_int(rng, 64, 16384)
        most = 128 if call != "prune_host" else 8
        batch = _log_int(rng, 1, max(1, min(most, _MAX_TOKENS // n)))
        dv = rng.choice([768, 1024, 1152, 1536, 2048, 8 * rng.randint(64, 256)])
        d = rng.choice([64, 128])
    ragged = rng.random() < 0.5
    n_lo = max(16, n // rng.randint(2, 8)) if ragged else n
    den = rng.choice([4, 5, 8, 8, 10, 20])
    while den < 20 and batch * n * (n // den) > _MAX_PAIRS:
        den += 1
    layers = rng.choice([1, 1, 1, 2, 4]) if batch * n <= 100000 else 1
    video = dtype == "bf16" and n >= 1024 and rng.random() < 0.3
    rows = 0
    if call == "rows":
        rows = rng.randint(2, 32)
        layers = 1
    t_lo = max(8, rows + 1)
    return _case(None, call, batch, n_lo, n, t_lo, t_lo + rng.randint(1, 120), layers, hq, hkv, d,
                 dv, dtype, f"1/{den}", 0 if video else rng.choice([24, 64, 128]),
                 rng.choice([0.0, 0.0, 0.3]), rng.choice([196, 256, 512]) if video else 0, rows)


# ---- shapes: host arithmetic shared by prepare, work and exact ----

def _sizes(case, seed=0):
    """Per-request visual and text token counts; a ragged range is spread evenly over
    its ends (the same sizes for every seed, in a seeded order)."""
    B = case["batch"]
    g = np.random.default_rng([seed, 7])
    spread = np.linspace(0.0, 1.0, B) if B > 1 else np.array([1.0])
    n = np.rint(case["n_lo"] + (case["n_hi"] - case["n_lo"]) * spread).astype(np.int64)
    t = np.rint(case["t_lo"] + (case["t_hi"] - case["t_lo"]) * spread).astype(np.int64)
    return n[g.permutation(B)], t[g.permutation(B)]


def _keeps(case, n):
    if "/" in case["keep"]:
        num, den = (int(v) for v in case["keep"].split("/"))
        return np.array([-(-num * int(v) // den) for v in n], dtype=np.int64)
    ks = [int(v) for v in case["keep"].split(",")]
    return np.array([min(ks[b % len(ks)], int(v)) for b, v in enumerate(n)], dtype=np.int64)


def _cu(v):
    return np.concatenate([[0], np.cumsum(v)]).astype(np.int32)


# ---- inputs ----

def _planted_keys(k, q, cu_p, vis0, n, case, gen):
    """Ten visual keys per request moved by 3/sqrt(D) along each kv-head's mean query."""
    B, hq, hkv, d = case["batch"], case["hq"], case["hkv"], case["d"]
    for b in range(B):
        dirs = q[b].view(case["layers"], hkv, hq // hkv, d).float().mean(2)
        dirs = dirs / dirs.norm(dim=-1, keepdim=True)
        m = min(10, int(n[b]))
        pos = torch.randperm(int(n[b]), generator=gen, device="cuda")[:m] + int(cu_p[b] + vis0[b])
        k[:, pos] += (dirs * (3.0 / math.sqrt(d))).unsqueeze(1).to(k.dtype)


def _features(case, n, gen, dt):
    dv, out = case["dv"], []
    for nb in (int(v) for v in n):
        if case["frame"]:
            frames = -(-nb // case["frame"])
            x = torch.randn((frames, case["frame"], dv), generator=gen, device="cuda")
            x[1:] *= 0.05
            x = torch.cumsum(x, 0).view(-1, dv)[:nb]
        else:
            c = torch.randn((case["clusters"], dv), generator=gen, device="cuda")
            c /= c.norm(dim=1, keepdim=True)
            at = torch.randint(case["clusters"], (nb,), generator=gen, device="cuda")
            x = c[at] + torch.randn((nb, dv), generator=gen, device="cuda") * (0.1 / math.sqrt(dv))
            if case["dup"] > 0:   # copies of a first-half token, perturbed by a tenth of its norm
                half = max(1, nb // 2)
                m = int(case["dup"] * nb)
                dst = half + torch.randperm(nb - half, generator=gen, device="cuda")[:m]
                src = torch.randint(half, (len(dst),), generator=gen, device="cuda")
                e = torch.randn((len(dst), dv), generator=gen, device="cuda")
                x[dst] = x[src] + e * (0.1 / math.sqrt(dv)) * x[src].norm(dim=1, keepdim=True)
        out.append(x.to(dt))
    return torch.cat(out)


def _inputs(case, seed):
    """The tensors and offsets of one batch, from the seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * seed + 17)
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    n, t = _sizes(case, seed)
    B, L, hq, hkv, d = (case[k] for k in ("batch", "layers", "hq", "hkv", "d"))
    p = n + t
    host = np.random.default_rng([seed, 8])
    # the visual span starts somewhere in the first half of the text
    vis0 = np.array([int(host.integers(0, max(1, (int(v) - case["rows"]) // 2))) for v in t])
    cu_p = _cu(p)
    s = dict(n=n, p=p, vis0=vis0, cu_p=cu_p, cu_v=_cu(n), cu_k=_cu(_keeps(case, n)))
    scale = 1.0 / math.sqrt(d)
    if case["rows"]:   # query rows spread over the text after the visual span, the last one at the end
        pos = [np.unique(np.rint(np.linspace(v0 + nb, pb - 1, case["rows"])).astype(np.int64))
               for v0, nb, pb in zip(vis0, n, p)]
        s["cu_r"], s["row_pos"] = _cu([len(v) for v in pos]), np.concatenate(pos).astype(np.int32)
        nq = int(s["cu_r"][-1])
    else:
        nq = B
    q = torch.randn((nq, L, hq, d), generator=gen, device="cuda") * scale
    k = torch.empty((L, int(cu_p[-1]), hkv, d), dtype=dt, device="cuda")
    for l in range(L):
        k[l] = (torch.randn(k.shape[1:], generator=gen, device="cuda") * scale).to(dt)
    s["q"] = q.to(dt)
    lead = s["q"] if not case["rows"] else s["q"][torch.as_tensor(s["cu_r"][1:] - 1, device="cuda").long()]
    _planted_keys(k, lead, cu_p, vis0, n, case, gen)
    s["k"] = k
    if case["call"] in ("prune", "prune_host", "topk"):
        s["x"] = _features(case, n, gen, dt)
    return s


def _row_scores(case, s):
    """Eq. 6-8 in 64 bits, plain torch: softmax rows over all their keys, summed over
    rows, layers and heads at the visual positions and normalised per request."""
    out, g = [], case["hq"] // case["hkv"]
    for b in range(case["batch"]):
        k = s["k"][:, int(s["cu_p"][b]):int(s["cu_p"][b + 1])].double()        # [L][P][Hkv][D]
        k = k.repeat_interleave(g, dim=2)
        if case["rows"]:
            r = slice(int(s["cu_r"][b]), int(s["cu_r"][b + 1]))
            q, pos = s["q"][r].double(), torch.as_tensor(s["row_pos"][r], device="cuda")
        else:
            q, pos = s["q"][b:b + 1].double(), torch.tensor([int(s["p"][b]) - 1], device="cuda")
        acc = 0.0
        for l in range(case["layers"]):
            z = torch.einsum("rhd,phd->rhp", q[:, l], k[l]) / math.sqrt(case["d"])
            seen = torch.arange(z.shape[-1], device="cuda")[None, None, :] <= pos[:, None, None]
            acc = acc + torch.softmax(z.masked_fill(~seen, -math.inf), -1).sum((0, 1))
        v = acc[int(s["vis0"][b]):int(s["vis0"][b] + s["n"][b])]
        out.append(v / v.sum())
    return torch.cat(out)


# ---- the interface ----

def prepare(case, seed):
    s = _inputs(case, seed)
    dev = torch.device("cuda")
    prob = last.Problem(batch=case["batch"], num_layers=case["layers"], num_q_heads=case["hq"],
                        num_kv_heads=case["hkv"], head_dim=case["d"], feat_dim=case["dv"],
                        dtype=case["dtype"], cu_seqlens=s["cu_p"], vis_start=s["vis0"],
                        cu_vis=s["cu_v"], cu_keep=s["cu_k"])
    st = dict(call=case["call"], prob=prob, q=s["q"], k=s["k"], x=s.get("x"))
    host = case["call"] == "prune_host"
    place = dict(device="cpu", pin_memory=True) if host else dict(device=dev)
    st["w"] = torch.empty(prob.total_vis, dtype=torch.float32, **place)
    st["idx"] = torch.empty(prob.total_keep, dtype=torch.int32, **place)
    if st["x"] is not None:
        st["x_out"] = torch.empty((prob.total_keep, case["dv"]), dtype=s["x"].dtype, **place)
    if host:
        for name in ("q", "k", "x"):
            st[name] = st[name].cpu().pin_memory()
        st["ws"] = last.host_workspace(prob, dev)
    elif case["rows"]:
        st["rows"] = last.QueryRows(s["cu_r"], s["row_pos"])
        st["ws"] = last.rows_workspace(prob, st["rows"], dev)
    else:
        st["ws"] = last.workspace(prob, dev)
    if case["call"] == "topk":   # scores in hand from an earlier call
        st["w"].copy_(_row_scores(case, s).float())
        st["q"] = st["k"] = None
    return st


def run(st):
    call, p = st["call"], st["prob"]
    if call in ("prune", "prune_host"):
        fn = last.last_prune if call == "prune" else last.last_prune_host
        fn(p, st["q"], st["k"], st["x"], st["w"], st["idx"], st["x_out"], st["ws"])
        return {"w": st["w"], "idx": st["idx"], "x_out": st["x_out"]}
    if call == "scores":
        last.last_scores(p, st["q"], st["k"], st["w"], st["ws"])
        return {"w": st["w"]}
    if call == "rows":
        last.last_scores_rows(p, st["rows"], st["q"], st["k"], st["w"], st["ws"])
        return {"w": st["w"]}
    last.last_select_topk(p, st["w"], st["idx"], st["ws"], x=st["x"], x_out=st["x_out"])
    return {"idx": st["idx"], "x_out": st["x_out"]}


def work(case):
    """Bytes: q, K and X read once, w~, the indices and the kept rows written once.
    Flops: the logits, and the greedy's distances as Sec. 3.4 counts them (k N d_v)."""
    e = 4 if case["dtype"] == "f32" else 2
    n, t = _sizes(case)
    kb = _keeps(case, n)
    dv, call = case["dv"], case["call"]
    nbytes = flops = 0
    if call != "topk":
        keys = int((n + t).sum()) * case["layers"]
        rows = max(1, case["rows"])
        nbytes += (keys * case["hkv"] + case["batch"] * rows * case["layers"] * case["hq"]) * case["d"] * e
        nbytes += 4 * int(n.sum())
        flops += 2 * keys * case["hq"] * case["d"] * rows
    if call in ("prune", "prune_host"):
        nbytes += int(n.sum()) * dv * e + int(kb.sum()) * (4 + dv * e)
        flops += 2 * int((kb * n).sum()) * dv
    if call == "topk":
        nbytes += 4 * int(n.sum()) + int(kb.sum()) * (4 + 2 * dv * e)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # The kept indices and rows are exact: the selection's arithmetic is fixed by the
    # public header.  The scores are 32-bit sums of 2^z terms in any order: 7e-8 from
    # 64 bits as measured, two orders up to twice that apart.
    if case["call"] == "topk":
        return "exact"
    return {"rel": 6e-7, "max": 6e-6}


def exact(case, seed):
    s = _inputs(case, seed)
    if case["call"] == "topk":
        w = _row_scores(case, s).float()
        idx, rows = [], []
        for b in range(case["batch"]):
            v0, v1 = int(s["cu_v"][b]), int(s["cu_v"][b + 1])
            kb = int(s["cu_k"][b + 1] - s["cu_k"][b])
            keep = torch.sort(torch.sort(w[v0:v1], descending=True, stable=True).indices[:kb]).values
            idx.append(keep.int())
            rows.append(s["x"][v0:v1][keep].double())
        return {"idx": torch.cat(idx), "x_out": torch.cat(rows)}
    w = _row_scores(case, s)
    if case["call"] in ("prune", "prune_host"):
        # the greedy's picks are defined in 32 bits (public header): no 64-bit value
        return {"w": w, "idx": None, "x_out": None}
    return {"w": w}
