"""Workloads of the decode-step library as a serving program runs them: decode steps on sessions of 4 thousand to a
million tokens, the offloaded multi-session step, opening a session's store (raw and KLT-rotated) and appending to it.

A case names a `kind` and its sizes:

    decode   alloc_depth -> scan -> topk -> sparse_attend on a store in device memory; with rotated=True the query first
             goes through rotate_query.  fused=True takes scan_topk in place of scan and topk, so no scores exist.
    offload  several sessions with plane words, scales and K/V rows in pinned host memory: alloc_depth per session, one
             scan_batch over all of them, then topk -> gather_union -> sparse_attend over the staged rows per session.
    open     channel_variance and build_planes of a session's keys (once per prefill).
    append   new keys arrive: the tail of every KV head's store is rebuilt from a block index that is a multiple of 8.
    calib    calibrate and klt_basis of a session's keys (once per prefill, KLT store).
    rotate   the rotated store from a known basis: rotate_keys then build_planes, or build_planes_rotated (one_call=True).

Keys follow the synthetic layer recipe of the tests: per-channel spread log-uniform in [0.1, 4], four outlier channels
at 16 per KV head, eight needle keys aligned with a query; values and queries are N(0, 1).  No keys are read while a
decode pass runs: the store and the rows are what a session holds.
"""
import math

import torch

from paper_2609_17652_b200 import binding as fb

D = 128
BUDGETS = (32, 40, 48, 64, 80, 136)


def listed():
    return [
        # One short head: nothing but latency, launches and the host path of the four calls.
        dict(name="decode_4k_one_head", kind="decode", n=4096, kv=1, heads=1, plan=1, mode="waterfill", budget=48, k=64,
             sink=0, local=0, rows="bf16", fused=False, rotated=False, tight=False),
        # A chat-length session with attention sinks and a local window, odd length, densest-packed strides.
        dict(name="decode_33k_sinks", kind="decode", n=33001, kv=8, heads=32, plan=4, mode="waterfill", budget=64, k=512,
             sink=4, local=32, rows="bf16", fused=False, rotated=False, tight=True),
        # The 131k-token layer, the middle of the range.
        dict(name="decode_131k", kind="decode", n=131072, kv=8, heads=32, plan=4, mode="waterfill", budget=48, k=2048,
             sink=0, local=0, rows="bf16", fused=False, rotated=False, tight=False),
        # Half a million tokens, odd, at the budget of 32 whole channels, KLT-rotated store.
        dict(name="decode_500k_b136", kind="decode", n=500003, kv=8, heads=32, plan=4, mode="waterfill", budget=136, k=2048,
             sink=0, local=0, rows="bf16", fused=False, rotated=True, tight=False),
        # The million-token session, one layer: the flagship decode step.
        dict(name="decode_1m", kind="decode", n=1048576, kv=8, heads=32, plan=4, mode="waterfill", budget=48, k=4096,
             sink=0, local=0, rows="bf16", fused=False, rotated=False, tight=False),
        # The same session for a program that does not keep scores, at the larger budget.
        dict(name="decode_1m_fused_b80", kind="decode", n=1048576, kv=8, heads=32, plan=4, mode="waterfill", budget=80, k=4096,
             sink=4, local=32, rows="bf16", fused=True, rotated=False, tight=False),
        # Four agent sessions whose store and rows live in host memory: the offloaded step.
        dict(name="offload_4_sessions", kind="offload", lengths="98304,65537,30011,20480", kv=8, heads=32, plan=4, budget=48,
             k=512),
        # Prefill of the million-token session: statistics and planes from fp32 keys.
        dict(name="open_1m", kind="open", n=1048576, kv=8, keys="f32"),
        # One decoded token is appended to a session: eight small rebuilds of the last blocks.
        dict(name="append_1", kind="append", n=33001, new=1, kv=8, keys="f32"),
        # Calibration of a KLT session.
        dict(name="calib_131k", kind="calib", n=131072, kv=8, keys="f32"),
        # Rotated stores: from bf16 keys with room for the rotated copy, and from fp32 keys without.
        dict(name="rotate_200k_bf16", kind="rotate", n=200001, kv=8, keys="bf16", one_call=False),
        dict(name="rotate_one_call_262k", kind="rotate", n=262144, kv=8, keys="f32", one_call=True),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode"] * 6 + ["offload", "open", "append", "calib", "rotate", "rotate"])
    if kind == "decode":
        kv, heads = rng.choice([(1, 1), (2, 8), (8, 32), (8, 32), (8, 32), (4, 32)])
        n = _log_uniform(rng, 4096, 1048576)
        mode, budget = rng.choice([("waterfill", b) for b in BUDGETS] * 3 + [("top_r", 16), ("top_r", 32), ("uniform", 2)])
        sink, local = rng.choice([(0, 0), (4, 32)])
        return dict(kind=kind, n=n, kv=kv, heads=heads, plan=rng.choice([heads // kv, heads // kv, 1]), mode=mode,
                    budget=budget, k=max(64, min(4096, n // 16, _log_uniform(rng, 64, 4096))), sink=sink, local=local,
                    rows=rng.choice(["bf16", "bf16", "bf16", "f32"]), fused=rng.random() < 0.3, rotated=rng.random() < 0.25,
                    tight=rng.random() < 0.3)
    if kind == "offload":
        lengths = [_log_uniform(rng, 16384, 98304) for _ in range(rng.randint(2, 4))]
        return dict(kind=kind, lengths=",".join(str(n) for n in lengths), kv=8, heads=32, plan=4,
                    budget=rng.choice(BUDGETS[:5]), k=rng.choice([256, 512]))
    if kind == "append":
        n = _log_uniform(rng, 4096, 65536)
        return dict(kind=kind, n=n, new=min(n // 2, _log_uniform(rng, 1, 1024)), kv=8, keys=rng.choice(["f32", "bf16"]))
    keys = rng.choice(["f32", "bf16"])
    if kind == "open":
        return dict(kind=kind, n=_log_uniform(rng, 4096, 1048576), kv=8, keys=keys)
    if kind == "calib":
        return dict(kind=kind, n=_log_uniform(rng, 8192, 131072), kv=rng.choice([2, 8]), keys=keys)
    return dict(kind=kind, n=_log_uniform(rng, 8192, 262144), kv=8, keys=keys, one_call=rng.random() < 0.4)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _keys(g, n, kv, heads):
    """(K [kv][n][D], q [heads][D]), fp32."""
    dev = "cuda"
    sigma = torch.exp(math.log(0.1) + torch.rand(kv, D, generator=g, device=dev) * math.log(40.0))
    sigma.scatter_(1, torch.rand(kv, D, generator=g, device=dev).argsort(1)[:, :4], 16.0)
    q = torch.randn(heads, D, generator=g, device=dev)
    K = torch.empty(kv, n, D, device=dev)
    for h in range(kv):                                    # a head at a time keeps the transient small
        K[h].normal_(generator=g).mul_(sigma[h])
    needles = torch.rand(kv, n, generator=g, device=dev).topk(8, dim=1).indices
    qhat = torch.nn.functional.normalize(q.view(kv, heads // kv, D), dim=2)
    qhat = qhat[:, (torch.arange(8, device=dev) * (heads // kv)) // 8]
    z = torch.randn(kv, 8, D, generator=g, device=dev)
    z = torch.nn.functional.normalize(z - (z * qhat).sum(2, keepdim=True) * qhat, dim=2)
    K.scatter_(1, needles.unsqueeze(2).expand(-1, -1, D),
               sigma.norm(dim=1).view(kv, 1, 1) * (0.9 * qhat + math.sqrt(0.19) * z))
    return K, q


def _values(g, kv, n, dtype):
    V = torch.empty(kv, n, D, device="cuda", dtype=dtype)
    for h in range(kv):
        V[h] = torch.randn(n, D, generator=g, device="cuda")
    return V


def _basis(g, kv):
    """Orthonormal bases near the channel axes and means, as the keys of a model without QK-norm would give."""
    A = torch.eye(D, device="cuda") + 0.05 * torch.randn(kv, D, D, generator=g, device="cuda")
    return torch.linalg.qr(A.double())[0].float().contiguous(), torch.randn(kv, D, generator=g, device="cuda")


def _variance(K):
    return torch.stack([x.var(dim=0) for x in K])


def _store(lay, device="cuda"):
    planes = torch.zeros(lay.n_kv_heads, D, 4, lay.plane_stride_words, dtype=torch.int64, device=device)
    scales = torch.zeros(lay.n_kv_heads, D, lay.scale_stride, dtype=torch.int16, device=device)
    return planes, scales


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def _dtype(name):
    return torch.float32 if name == "f32" else torch.bfloat16


def _prepare_decode(c, g):
    n, kv, heads, k = c["n"], c["kv"], c["heads"], c["k"]
    K, q = _keys(g, n, kv, heads)
    lay = fb.make_layout(kv, heads, n, D, 16 if c["tight"] else 128)
    ctx = fb.Context(torch.cuda.current_device(), fb.fathom_scratch_bytes(lay, k))
    planes, scales = _store(lay)
    basis = _basis(g, kv)[0] if c["rotated"] else None
    stored = torch.stack([K[h] @ basis[h] for h in range(kv)]) if c["rotated"] else K
    ctx.fathom_build_planes(lay, stored, planes, scales)
    s = dict(lay=lay, ctx=ctx, planes=planes, scales=scales, q=q, var=_variance(stored), plan=c["plan"], k=k, sink=c["sink"],
             local=c["local"], budget=c["budget"], fused=c["fused"],
             mode=dict(waterfill=fb.DEPTH_WATERFILL, top_r=fb.DEPTH_FIXED_TOP_R, uniform=fb.DEPTH_UNIFORM)[c["mode"]])
    s["Krows"] = K if c["rows"] == "f32" else K.to(torch.bfloat16)
    s["Vrows"] = _values(g, kv, n, _dtype(c["rows"]))
    s["basis"] = basis
    s["q_scan"] = torch.zeros_like(q) if c["rotated"] else q
    s["depth"] = torch.zeros(heads // c["plan"], D, dtype=torch.uint8, device="cuda")
    s["idx"] = torch.zeros(heads, k, dtype=torch.int32, device="cuda")
    s["attended"] = torch.zeros(heads, D, device="cuda")
    s["result"] = dict(depth=s["depth"], idx=s["idx"], out=s["attended"])
    if not c["fused"]:
        s["scores"] = torch.zeros(heads, lay.score_stride, device="cuda")
        s["result"]["scores"] = s["scores"][:, :n]
    if c["rotated"]:
        s["result"]["q_rot"] = s["q_scan"]
    return s


def _run_decode(s):
    ctx, lay, k = s["ctx"], s["lay"], s["k"]
    if s["basis"] is not None:
        ctx.fathom_rotate_query(lay, s["q"], s["basis"], s["q_scan"])
    ctx.fathom_alloc_depth(lay, s["q_scan"], s["var"], s["mode"], s["budget"], s["plan"], s["depth"])
    if s["fused"]:
        ctx.fathom_scan_topk(lay, s["planes"], s["scales"], s["q_scan"], s["depth"], s["plan"], k, s["sink"], s["local"],
                             s["idx"])
    else:
        ctx.fathom_scan(lay, s["planes"], s["scales"], s["q_scan"], s["depth"], s["plan"], s["scores"])
        ctx.fathom_topk(lay, s["scores"], k, s["sink"], s["local"], s["idx"])
    ctx.fathom_sparse_attend(lay, s["q"], s["Krows"], s["Vrows"], s["idx"], k, 1.0 / math.sqrt(D), s["attended"])
    return s["result"]


def _prepare_offload(c, g):
    kv, heads, k = c["kv"], c["heads"], c["k"]
    lengths = [int(x) for x in c["lengths"].split(",")]
    group = heads // kv
    staged = fb.make_layout(kv, heads, group * k, D)
    lays = [fb.make_layout(kv, heads, n, D) for n in lengths]
    scratch = max(fb.fathom_scratch_bytes(x, k) for x in lays + [staged])
    ctx = fb.Context(torch.cuda.current_device(), scratch)
    sessions = []
    for n, lay in zip(lengths, lays):
        K, q = _keys(g, n, kv, heads)
        planes, scales = _store(lay)
        ctx.fathom_build_planes(lay, K, planes, scales)
        x = dict(lay=lay, q=q, var=_variance(K), planes=_pinned(planes), scales=_pinned(scales),
                 Krows=_pinned(K.to(torch.bfloat16)), Vrows=_pinned(_values(g, kv, n, torch.bfloat16)))
        x["depth"] = torch.zeros(heads // c["plan"], D, dtype=torch.uint8, device="cuda")
        x["scores"] = torch.zeros(heads, lay.score_stride, device="cuda")
        x["idx"] = torch.zeros(heads, k, dtype=torch.int32, device="cuda")
        x["picked"] = torch.zeros(heads, k, dtype=torch.int32, device="cuda")
        x["count"] = torch.zeros(kv, dtype=torch.int32, device="cuda")
        x["out"] = torch.zeros(heads, D, device="cuda")
        sessions.append(x)
    Kst = torch.zeros(kv, group * k, D, dtype=torch.bfloat16, device="cuda")
    return dict(ctx=ctx, staged=staged, sessions=sessions, Kst=Kst, Vst=torch.zeros_like(Kst), plan=c["plan"], k=k,
                budget=c["budget"],
                items=[(x["lay"], x["planes"], x["scales"], x["q"], x["depth"], x["scores"]) for x in sessions],
                result=[dict(depth=x["depth"], scores=x["scores"][:, :n], idx=x["idx"], picked=x["picked"], count=x["count"],
                             out=x["out"]) for n, x in zip(lengths, sessions)])


def _run_offload(s):
    ctx, k = s["ctx"], s["k"]
    for x in s["sessions"]:
        ctx.fathom_alloc_depth(x["lay"], x["q"], x["var"], fb.DEPTH_WATERFILL, s["budget"], s["plan"], x["depth"])
    ctx.fathom_scan_batch(s["items"], s["plan"])
    for x in s["sessions"]:
        ctx.fathom_topk(x["lay"], x["scores"], k, 0, 0, x["idx"])
        ctx.fathom_gather_union(x["lay"], x["idx"], k, x["Krows"], x["Vrows"], s["Kst"], s["Vst"], x["picked"], x["count"])
        ctx.fathom_sparse_attend(s["staged"], x["q"], s["Kst"], s["Vst"], x["picked"], k, 1.0 / math.sqrt(D), x["out"])
    return s["result"]


def _prepare_keys(c, g):
    """What the session-opening kinds share: keys, a layout (one query head per KV head), a context, an empty store."""
    K, _ = _keys(g, c["n"], c["kv"], c["kv"])
    K = K.to(_dtype(c["keys"]))
    lay = fb.make_layout(c["kv"], c["kv"], c["n"], D)
    ctx = fb.Context(torch.cuda.current_device(), fb.fathom_scratch_bytes(lay, 64))
    planes, scales = _store(lay)
    return dict(lay=lay, ctx=ctx, K=K, planes=planes, scales=scales)


def _floats(*shape):
    return torch.zeros(*shape, device="cuda")


def prepare(case, seed):
    c, g = case, _generator(seed)
    kind, kv = c["kind"], c["kv"]
    if kind in ("decode", "offload"):
        s = _prepare_decode(c, g) if kind == "decode" else _prepare_offload(c, g)
    else:
        s = _prepare_keys(c, g)
        if kind == "open":
            s["result"] = dict(mean=_floats(kv, D), var=_floats(kv, D), planes=s["planes"], scales=s["scales"])
        elif kind == "append":
            lay, n, old = s["lay"], c["n"], c["n"] - c["new"]
            b0 = 8 * (old // 64 // 8)                      # from a multiple of 8 blocks on: every pointer stays aligned
            s["ctx"].fathom_build_planes(lay, s["K"], s["planes"], s["scales"])
            s["tail"] = fb.Layout(1, 1, D, 0, n - 64 * b0, lay.plane_stride_words, lay.scale_stride, lay.score_stride)
            s["heads"] = [(s["K"][h, 64 * b0:], s["planes"][h, :, :, b0:], s["scales"][h, :, b0:]) for h in range(kv)]
            s["planes"][..., b0:] = 0
            s["scales"][..., b0:] = 0
            s["result"] = dict(planes=s["planes"], scales=s["scales"])
        elif kind == "calib":
            s["result"] = dict(mean=_floats(kv, D), cov=_floats(kv, D, D), basis=_floats(kv, D, D), eig=_floats(kv, D))
        else:
            s["basis"], s["mean"] = _basis(g, kv)
            s["result"] = dict(planes=s["planes"], scales=s["scales"])
            s["K_rot"] = None if c["one_call"] else _floats(kv, c["n"], D)
            if not c["one_call"]:
                s["result"]["K_rot"] = s["K_rot"]
    s["kind"] = kind
    return s


def run(state):
    s, kind = state, state["kind"]
    if kind == "decode":
        return _run_decode(s)
    if kind == "offload":
        return _run_offload(s)
    ctx, lay, r = s["ctx"], s["lay"], s["result"]
    if kind == "open":
        ctx.fathom_channel_variance(lay, s["K"], r["mean"], r["var"])
        ctx.fathom_build_planes(lay, s["K"], s["planes"], s["scales"])
    elif kind == "append":
        for K, planes, scales in s["heads"]:
            ctx.fathom_build_planes(s["tail"], K, planes, scales)
    elif kind == "calib":
        ctx.fathom_calibrate(lay, s["K"], r["mean"], r["cov"])
        ctx.fathom_klt_basis(lay, r["cov"], r["basis"], r["eig"])
    elif s["K_rot"] is None:
        ctx.fathom_build_planes_rotated(lay, s["K"], s["mean"], s["basis"], s["planes"], s["scales"])
    else:
        ctx.fathom_rotate_keys(lay, s["K"], s["mean"], s["basis"], s["K_rot"])
        ctx.fathom_build_planes(lay, s["K_rot"], s["planes"], s["scales"])
    return r


def _scan_rows(c):
    """(planes, channels) that a plan reads per token; water-filled plans touch at least budget / 4 channels."""
    mode, b = c.get("mode", "waterfill"), c["budget"]
    return (4 * b, b) if mode == "top_r" else (D * b, D) if mode == "uniform" else (b, -(-b // 4))


def _step_work(c, n):
    kv, heads, k = c["kv"], c["heads"], c["k"]
    rows, channels = _scan_rows(c)
    plans_per_kv = heads // kv // c["plan"]
    reads = kv * plans_per_kv * n * (rows / 8 + channels / 32)
    reads = min(reads, kv * n * D * (4 / 8 + 1 / 32))              # plans of one KV head can share what they read
    row = D * (4 if c.get("rows") == "f32" else 2)
    nbytes = reads + 2 * heads * k * row + heads * (4 * k + 8 * D) + 4 * kv * D + heads // c["plan"] * D
    if not c.get("fused"):
        nbytes += 4 * heads * n
    return nbytes, 2.0 * heads * n * rows + 4.0 * heads * k * D


def work(case):
    c, kind = case, case["kind"]
    if kind == "decode":
        b, f = _step_work(c, c["n"])
    elif kind == "offload":
        b, f = (sum(x) for x in zip(*(_step_work(c, int(n)) for n in c["lengths"].split(","))))
    else:
        kv, n = c["kv"], c["n"]
        key = D * (4 if c["keys"] == "f32" else 2)
        keys, store, product = kv * n * key, kv * n * 68, 2.0 * kv * n * D * D
        if kind == "open":
            b, f = keys + store, 3.0 * kv * n * D
        elif kind == "append":
            m = n - 512 * ((n - c["new"]) // 512)
            b, f = kv * m * (key + 68), kv * m * D
        elif kind == "calib":
            b, f = keys + kv * 4 * (2 * D * D + 2 * D), product + kv * 9.0 * D ** 3
        else:
            b, f = keys + store + (0 if c["one_call"] else kv * n * D * 4), product
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    kind = case["kind"]
    if kind in ("decode", "offload"):
        # Scores are fp32 sums of up to 512 products, attention exponentiates logits of a few tens; tokens whose scores lie
        # within a rounding of the k-th may be chosen the other way, and one such token shifts part of an ascending list.
        return {"rel": 3e-5, "max": 1e-3, "differ": 0.01}
    if kind == "open":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}           # statistics in fp32; planes and scales are exact
    if kind == "append":
        return "exact"
    if kind == "calib":
        # Eigenvectors of neighbouring eigenvalues turn by rounding / relative gap; gaps are a few thousandths.
        return {"rel": 1e-4, "max": 1e-2}
    # Rotated keys in fp32: a key within a rounding of a code's edge may take the other code; a word holds 64 codes.
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
