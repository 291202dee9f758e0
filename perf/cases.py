"""The work that a user of this library has it do, as cases that can be timed and checked.

A case is one block of a model with token-level local/global attention, run through the public
entry points (``logo.py``, ``layer.py``), or the whole attention layer:

  route    the routing loop of a training step: threshold selection with the threshold on the
           device, and the budget controller's update of it
  prefill  ``LogoAttention.forward``: selection, both branches, the fusion (inference over a prompt)
  local    the sliding-window branch of a training step, forward and backward
  global   the query-sparse branch of a training step, forward and backward
  fuse     ContextNorm and fusion of a training step, forward and backward with gain gradients
  lift     what surrounds the attention in a training step: the gate with its selection, and the
           transforms that make the global branch's Q, K, V, forward and backward
  decode   one decoding step over a batch of sequences, captured once in a CUDA graph as a serving
           program does and replayed per token

Sizes of the listed cases are those of the repository's workloads (``workloads.py``, ``bench.py``)
and of its tests' kinds: ragged lengths, grouped-query heads, both head dimensions.  ``exact``
states each block in 64-bit torch arithmetic.
"""
from __future__ import annotations

import math

import torch

from paper_2608_29539_gb300 import logo as L
from paper_2608_29539_gb300.layer import LayerConfig, LogoAttention

EPS = 1e-6


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # routing decisions of one step for a batch of 4K-token sequences: smallest call, all latency
        dict(name="route_4x4k", kind="route", B=4, T=4096, rho=0.125),
        # a short prompt through the whole layer with small heads: launches and the host count
        dict(name="prefill_512_d64", kind="prefill", B=1, T=512, Hq=4, Hkv=4, D=64, W=64, mode="threshold", ratio=0.25,
             gates="normal"),
        # a long grouped-query prompt through the whole layer: the largest prefill
        dict(name="prefill_64k_gqa", kind="prefill", B=1, T=65536, Hq=32, Hkv=8, D=128, W=2048, mode="ratio",
             ratio=0.0625, gates="normal"),
        # window attention of a training step at two sequence lengths
        dict(name="local_4k", kind="local", B=2, T=4096, Hq=16, Hkv=16, D=128, W=512),
        dict(name="local_16k", kind="local", B=1, T=16384, Hq=32, Hkv=32, D=128, W=1024),
        # ... of a smaller model: 64-wide heads, grouped queries, lengths that divide nothing
        dict(name="local_ragged_d64", kind="local", B=3, T=2987, Hq=12, Hkv=4, D=64, W=300),
        # the query-sparse branch of a training step: few rows, the long clustered workload, 64-wide heads
        dict(name="global_4k", kind="global", B=2, T=4096, Hq=16, Hkv=16, D=128, ratio=0.125, gates="normal"),
        dict(name="global_16k", kind="global", B=1, T=16384, Hq=32, Hkv=32, D=128, ratio=0.125, gates="clustered"),
        dict(name="global_8k_d64", kind="global", B=2, T=8192, Hq=16, Hkv=16, D=64, ratio=0.125, gates="normal"),
        # normalisation and fusion with trained gains at the long training length
        dict(name="fuse_16k", kind="fuse", B=1, T=16384, Hq=32, D=128, ratio=0.125, gates="clustered"),
        # gate and matrix transforms of a grouped-query layer
        dict(name="lift_8k", kind="lift", B=1, T=8192, Hq=32, Hkv=8, D=128, d_model=4096, form="lp", ratio=0.125),
        # one token for each of 32 sequences with long caches
        dict(name="decode_32x16k", kind="decode", B=32, L=16384, Hq=32, Hkv=8, D=128, W=1024, selected=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(("route", "prefill", "prefill", "local", "local", "global", "global", "fuse", "lift", "decode"))
        D = rng.choice((64, 128, 128))
        Hkv = rng.choice((1, 2, 4, 8, 16, 32))
        Hq = Hkv * rng.choice((1, 1, 2, 4, 8))
        B = rng.choice((1, 1, 2, 3, 4, 8))
        T = _log(rng, 100, 65536)
        if rng.random() < 0.5:
            T = max(128, T // 128 * 128)
        W = _log(rng, 16, 4096)
        ratio = rng.choice((1.0 / 32, 0.0625, 0.125, 0.125, 0.25, 0.5))
        gates = rng.choice(("normal", "clustered"))
        if kind == "route":
            c = dict(kind=kind, B=B, T=T, rho=ratio)
        elif kind == "prefill":
            c = dict(kind=kind, B=B, T=T, Hq=Hq, Hkv=Hkv, D=D, W=W, mode=rng.choice(("ratio", "threshold")), ratio=ratio,
                     gates=gates)
        elif kind == "local":
            c = dict(kind=kind, B=B, T=T, Hq=Hq, Hkv=Hkv, D=D, W=W)
        elif kind == "global":
            c = dict(kind=kind, B=B, T=T, Hq=Hq, Hkv=Hkv, D=D, ratio=ratio, gates=gates)
        elif kind == "fuse":
            c = dict(kind=kind, B=B, T=T, Hq=Hq, D=D, ratio=ratio, gates=gates)
        elif kind == "lift":
            c = dict(kind=kind, B=B, T=T, Hq=Hq, Hkv=Hkv, D=D, d_model=rng.choice((512, 1024, 2048, 4096)),
                     form=rng.choice(("lp", "lp", "so")), ratio=ratio)
        else:
            B = rng.choice((1, 2, 5, 8, 16, 32))
            c = dict(kind=kind, B=B, L=_log(rng, 512, 32768), Hq=Hq, Hkv=Hkv, D=D, W=min(W, 2048),
                     selected=rng.randint(0, max(1, B // 4)))
            c["W"] = max(64, min(c["W"], c["L"]))
        if Hq > 32 or (Hq * D > 4096) or (kind == "decode" and Hq // Hkv > 16):
            continue
        if kind not in ("route", "decode") and B * T > 65536:
            continue
        w = work(c)
        if w["flops"] <= 1.5e12 and w["bytes"] <= 3e9:
            return c


# ------------------------------------------------------------------ inputs
def _gen(seed, dev="cuda"):
    return torch.Generator(device=dev).manual_seed(int(seed) * 7919 + 11)


def _bf(g, *shape, std=1.0):
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
    return (x.mul_(std) if std != 1.0 else x).to(torch.bfloat16)


def _gate_logits(g, B, T, gates):
    """Normal logits, or runs of high ones (on-runs of mean 16, an eighth of the tokens)."""
    x = torch.randn((B, T), generator=g, device="cuda")
    if gates == "clustered":
        n = T // 64 + 64  # pairs of an off- and an on-run, mean 128 tokens a pair
        u = torch.rand((B, n, 2), generator=g, device="cuda", dtype=torch.float64).clamp_min_(1e-12)
        p = torch.tensor([1 / 112.0, 1 / 16.0], device="cuda", dtype=torch.float64)
        ends = (torch.log(u) / torch.log1p(-p)).ceil().clamp_min_(1).reshape(B, 2 * n).cumsum(1)
        t = torch.arange(T, device="cuda", dtype=torch.float64).expand(B, T).contiguous()
        run = torch.searchsorted(ends, t, right=True)
        x = x + 4.0 * (run & 1).to(x.dtype)
    return x


def _threshold(p, ratio):
    """A threshold that about ratio * T of the first sequence's gates exceed, halfway between two gates."""
    s = torch.sort(p[0].double()).values
    k = min(max(int(ratio * p.shape[1]), 1), p.shape[1] - 1)
    return float(((s[-k - 1] + s[-k]) / 2).float())


def _ring(c):
    """Slots of a ring cache that serves windows of W: allocated in blocks of 64."""
    return -(-c["W"] // 64) * 64


def _inputs(c, seed):
    """Everything of a case that is drawn; the same for prepare() and exact()."""
    g = _gen(seed)
    kind = c["kind"]
    x = {}
    if kind == "route":
        x["p"] = torch.sigmoid(torch.randn((c["B"], c["T"]), generator=g, device="cuda"))
        x["b_th"], x["gamma"] = _threshold(x["p"], c["rho"]), 5e-4
        return x
    Hq, D = c["Hq"], c["D"]
    if kind == "decode":
        B, Hkv = c["B"], c["Hkv"]
        for n in ("qL", "qG"):
            x[n] = _bf(g, B, Hq, D)
        for n, r in (("kR", _ring(c)), ("vR", _ring(c)), ("kG", c["L"]), ("vG", c["L"])):
            x[n] = _bf(g, B, r, Hkv, D)
        x["len"] = torch.randint(max(1, c["L"] // 2), c["L"] + 1, (B,), generator=g, device="cuda", dtype=torch.int32)
        x["p"] = torch.rand((B, 1), generator=g, device="cuda") * 0.98 + 0.01
        s, n = torch.sort(x["p"].flatten()).values.tolist(), c["selected"]
        x["b_th"] = 0.995 if n == 0 else (0.005 if n >= B else float(torch.tensor((s[B - n - 1] + s[B - n]) / 2)))
        return x
    B, T = c["B"], c["T"]
    if kind == "local":
        x["q"], x["k"], x["v"] = _bf(g, B, T, Hq, D), _bf(g, B, T, c["Hkv"], D), _bf(g, B, T, c["Hkv"], D)
        x["dO"] = _bf(g, B, T, Hq, D)
    elif kind == "global":
        x["q"], x["k"], x["v"] = _bf(g, B, T, Hq, D), _bf(g, B, T, c["Hkv"], D), _bf(g, B, T, c["Hkv"], D)
        x["p"] = torch.sigmoid(_gate_logits(g, B, T, c["gates"]))
        x["dO_c"] = _bf(g, B * T, Hq, D)
    elif kind == "prefill":
        for s in "LG":
            x["q" + s], x["k" + s], x["v" + s] = (_bf(g, B, T, h, D) for h in (Hq, c["Hkv"], c["Hkv"]))
        x["p"] = torch.sigmoid(_gate_logits(g, B, T, c["gates"]))
        x["b_th"] = _threshold(x["p"], c["ratio"])
    elif kind == "fuse":
        x["o_l"], x["o_c"], x["dO"] = (_bf(g, *s, Hq, D, std=t) for s, t in (((B, T), 0.3), ((B * T,), 0.1), ((B, T), 1.0)))
        x["p"] = torch.sigmoid(_gate_logits(g, B, T, c["gates"]))
        for n in ("gain_l", "gain_g"):
            x[n] = 1.0 + 0.1 * torch.randn((Hq, D), generator=g, device="cuda")
    else:  # lift
        dm = c["d_model"]
        x["x"], x["w_g"] = _bf(g, B, T, dm), torch.randn((dm,), generator=g, device="cuda") * dm ** -0.5
        x["dgate"] = torch.randn((B, T), generator=g, device="cuda")
        for n, h in (("q", Hq), ("k", c["Hkv"]), ("v", c["Hkv"])):
            x[n], x["g" + n], x["d" + n] = (_bf(g, B, T, h, D) for _ in range(3))
            if c["form"] == "lp":  # near the identity that it starts from
                eye = torch.eye(D, device="cuda").expand(h, D, D)
                x["t" + n] = dict(a=(eye + 0.05 * torch.randn((h, D, D), generator=g, device="cuda")).to(torch.bfloat16))
            else:
                x["t" + n] = dict(s=1.0 + 0.1 * torch.randn((h, D), generator=g, device="cuda"),
                                  b=0.1 * torch.randn((h, D), generator=g, device="cuda"))
    return x


def _zeros(*shape, dtype=torch.bfloat16):
    return torch.zeros(shape, dtype=dtype, device="cuda")


def _ws(fn, *args):
    return torch.empty(max(16, int(getattr(L.lib(), fn)(*args))), dtype=torch.uint8, device="cuda")


def _selection(B, T):
    """Buffers that logo_select fills; packed entries past the selected count stay zero."""
    i32 = torch.int32
    return dict(z=_zeros(B, T, dtype=torch.uint8), pos=_zeros(B * T, dtype=i32), cu_q=_zeros(B + 1, dtype=i32),
                row_of=_zeros(B, T, dtype=i32), n_sel_total=_zeros(1, dtype=i32))


def prepare(case, seed):
    c, x = case, _inputs(case, seed)
    kind, s = c["kind"], dict(case=case, x=x)
    if kind == "route":
        B, T = c["B"], c["T"]
        s["sel"] = _selection(B, T)
        s["ws"] = _ws("logo_select_workspace_size", L.Dims(B, T, 1, 1, 64))
        s["b_th"] = torch.full((1,), x["b_th"], device="cuda")
        s["f"] = _zeros(1, dtype=torch.float32)
        return s
    Hq, D = c["Hq"], c["D"]
    if kind == "decode":
        B, Hkv, W, Lc = c["B"], c["Hkv"], _ring(c), c["L"]
        s["sel"] = _selection(B, 1)
        s["ws_s"] = _ws("logo_select_workspace_size", L.Dims(B, 1, 1, 1, 64))
        s["ws_l"] = _ws("logo_decode_workspace_size", L.Dims(B, W, Hq, Hkv, D))
        s["ws_g"] = _ws("logo_decode_workspace_size", L.Dims(B, Lc, Hq, Hkv, D))
        s["o_l"], s["o_c"], s["o"] = _zeros(B, Hq, D), _zeros(B, Hq, D), _zeros(B, 1, Hq, D)
        s["rl"], s["rg"] = _zeros(B, 1, Hq, dtype=torch.float32), _zeros(B, Hq, dtype=torch.float32)
        s["side"] = torch.cuda.Stream()
        warm = torch.cuda.Stream()
        warm.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(warm):
            _decode_step(s)
        torch.cuda.current_stream().wait_stream(warm)
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _decode_step(s)
        return s
    B, T = c["B"], c["T"]
    if kind == "prefill":
        mode = L.LOGO_SELECT_RATIO if c["mode"] == "ratio" else L.LOGO_SELECT_THRESHOLD
        s["layer"] = LogoAttention(LayerConfig(B, T, Hq, c["Hkv"], D, c["W"], mode=mode, b_th=x["b_th"], ratio=c["ratio"],
                                               eps=EPS))
    elif kind == "local":
        d = L.Dims(B, T, Hq, c["Hkv"], D)
        s["o"], s["lse"] = _zeros(B, T, Hq, D), _zeros(B, Hq, T, dtype=torch.float32)
        s["dq"], s["dk"], s["dv"] = (torch.zeros_like(x[n]) for n in "qkv")
        s["ws"] = _ws("logo_local_attn_bwd_workspace_size", d)
    elif kind == "global":
        d, cap = L.Dims(B, T, Hq, c["Hkv"], D), B * T
        s["sel"] = L.logo_select(x["p"], L.LOGO_SELECT_RATIO, ratio=c["ratio"], **_selection(B, T))[1:]
        s["o_c"], s["lse_c"] = _zeros(cap, Hq, D), _zeros(Hq, cap, dtype=torch.float32)
        s["dq"], s["dk"], s["dv"] = (torch.zeros_like(x[n]) for n in "qkv")
        s["ws"] = _ws("logo_global_attn_fwd_workspace_size", d)
        s["ws_b"] = _ws("logo_global_attn_bwd_workspace_size", d)
    elif kind == "fuse":
        f32 = torch.float32
        s["z"], _, _, s["row_of"], _ = L.logo_select(x["p"], L.LOGO_SELECT_RATIO, ratio=c["ratio"], **_selection(B, T))
        s["o"], s["rstd_l"], s["rstd_g"] = _zeros(B, T, Hq, D), _zeros(B, T, Hq, dtype=f32), _zeros(B * T, Hq, dtype=f32)
        s["dO_l"], s["dO_c"], s["dgate"] = _zeros(B, T, Hq, D), _zeros(B * T, Hq, D), _zeros(B, T, dtype=f32)
        s["dgl"], s["dgg"] = _zeros(Hq, D, dtype=f32), _zeros(Hq, D, dtype=f32)
        s["ws"] = _ws("logo_combine_bwd_workspace_size", L.Dims(B, T, Hq, Hq, D))
    else:  # lift
        s["sel"] = _selection(B, T)
        s["gate_p"], s["dx"] = _zeros(B, T, dtype=torch.float32), torch.zeros_like(x["x"])
        s["dw"] = torch.zeros_like(x["w_g"])
        s["ws"] = _ws("logo_select_workspace_size", L.Dims(B, T, 1, 1, 64))
        s["ws_g"] = _ws("logo_gate_bwd_workspace_size", L.Dims(B, T, 1, 1, 64), c["d_model"])
        for n in "qkv":
            h = x[n].shape[2]
            s["u" + n] = torch.zeros_like(x[n])
            s["d" + n] = x["d" + n].clone()  # the local branch's gradient, added to
            s["ws_" + n] = _ws("logo_branch_transform_bwd_workspace_size", L.Dims(B, T, h, h, D))
    return s


# ------------------------------------------------------------------ one pass
def _decode_step(s):
    c, x = s["case"], s["x"]
    B, Hq, D = c["B"], c["Hq"], c["D"]
    z, _, cu_q, row_of, n = L.logo_select(x["p"], L.LOGO_SELECT_THRESHOLD, b_th=x["b_th"], workspace=s["ws_s"], **s["sel"])
    main = torch.cuda.current_stream()
    s["side"].wait_stream(main)
    with torch.cuda.stream(s["side"]):  # the two branches are independent
        L.logo_decode_local_attn(x["qL"], x["kR"], x["vR"], x["len"], c["W"], o=s["o_l"], workspace=s["ws_l"])
    L.logo_decode_global_sparse_attn(x["qG"], x["kG"], x["vG"], x["len"], cu_q, n, o_c=s["o_c"], workspace=s["ws_g"])
    main.wait_stream(s["side"])
    L.logo_combine(s["o_l"].view(B, 1, Hq, D), s["o_c"], x["p"], z, row_of, None, None, EPS, s["o"], s["rl"], s["rg"])


def run(state):
    s, c, x = state, state["case"], state["x"]
    kind = c["kind"]
    if kind == "route":
        z, pos, cu_q, row_of, n = L.logo_select_device_threshold(x["p"], s["b_th"], workspace=s["ws"], **s["sel"])
        L.logo_budget_update(n, c["B"], c["T"], c["rho"], x["gamma"], s["b_th"], s["f"])
        return dict(z=z, pos=pos, cu_q=cu_q, row_of=row_of, n=n, b_th=s["b_th"], f=s["f"])
    if kind == "decode":
        s["graph"].replay()
        return dict(o=s["o"], o_l=s["o_l"], o_c=s["o_c"], z=s["sel"]["z"])
    if kind == "prefill":
        return dict(o=s["layer"].forward(x["qL"], x["kL"], x["vL"], x["qG"], x["kG"], x["vG"], x["p"]))
    if kind == "local":
        o, lse = L.logo_local_attn_fwd(x["q"], x["k"], x["v"], c["W"], o=s["o"], lse=s["lse"])
        dq, dk, dv = L.logo_local_attn_bwd(x["q"], x["k"], x["v"], o, lse, x["dO"], c["W"], dq=s["dq"], dk=s["dk"],
                                           dv=s["dv"], workspace=s["ws"])
        return dict(o=o, lse=lse, dq=dq, dk=dk, dv=dv)
    if kind == "global":
        pos, cu_q, _, n = s["sel"]
        o, lse = L.logo_global_sparse_attn_fwd(x["q"], x["k"], x["v"], pos, cu_q, n, o_c=s["o_c"], lse_c=s["lse_c"],
                                               workspace=s["ws"])
        dq, dk, dv = L.logo_global_sparse_attn_bwd(x["q"], x["k"], x["v"], pos, cu_q, n, o, lse, x["dO_c"], dq=s["dq"],
                                                   dk=s["dk"], dv=s["dv"], workspace=s["ws_b"])
        return dict(o=o, lse=lse, dq=dq, dk=dk, dv=dv)
    if kind == "fuse":
        g = (x["gain_l"], x["gain_g"], EPS)
        o, rl, rg = L.logo_combine(x["o_l"], x["o_c"], x["p"], s["z"], s["row_of"], *g, s["o"], s["rstd_l"], s["rstd_g"])
        dl, dc, dp, dgl, dgg = L.logo_combine_bwd_gains(x["dO"], x["o_l"], x["o_c"], x["p"], s["z"], s["row_of"], *g,
                                                        s["dO_l"], s["dO_c"], s["dgate"], s["dgl"], s["dgg"], s["ws"])
        return dict(o=o, rstd_l=rl, rstd_g=rg, dO_l=dl, dO_c=dc, dgate=dp, dgain_l=dgl, dgain_g=dgg)
    # lift
    p, z, pos, cu_q, row_of, n = L.logo_gate_select(x["x"], x["w_g"], L.LOGO_SELECT_RATIO, ratio=c["ratio"],
                                                    gate_p=s["gate_p"], workspace=s["ws"], **s["sel"])
    rows = dict(q=(pos, cu_q, n), k=None, v=None)  # Q on the selected rows only
    out = dict(p=p, z=z, pos=pos)
    for m in "qkv":
        out["u" + m] = L.logo_branch_transform(x[m], rows=rows[m], u_g=s["u" + m], **x["t" + m])
    for m in "qkv":
        t = {k: v for k, v in x["t" + m].items() if k != "b"}
        got = L.logo_branch_transform_bwd(x[m], x["g" + m], rows=rows[m], du_l=s["d" + m], accumulate=True,
                                          workspace=s["ws_" + m], **t)
        out["d" + m], out["dt" + m] = got[0], list(got[1:])
    out["dx"], out["dw"] = L.logo_gate_bwd(x["x"], x["w_g"], p, x["dgate"], dx=s["dx"], dw_g=s["dw"], workspace=s["ws_g"])
    return out


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    c, kind = case, case["kind"]
    if kind == "route":
        n = c["B"] * c["T"]
        return dict(bytes=n * (4 + 1 + 4) + 4 * n * c["rho"], flops=n)
    Hq, D, B = c["Hq"], c["D"], c["B"]
    if kind == "decode":
        rows = B * min(c["W"], 0.75 * c["L"]) + c["selected"] * 0.75 * c["L"]
        return dict(bytes=rows * c["Hkv"] * D * 4 + 6 * B * Hq * D, flops=rows * Hq * D * 4)
    T = c["T"]
    n, sel = B * T, B * T * c.get("ratio", 1.0)
    if kind == "fuse":
        return dict(bytes=(4 * n + 2 * sel) * Hq * D * 2, flops=n * Hq * D * 20)
    if kind == "lift":
        q, kv, dm = Hq * D * 2, c["Hkv"] * D * 2 * 2, c["d_model"]
        f = 6 * D if c["form"] == "lp" else 8
        return dict(bytes=n * dm * 2 * 2 + (sel * q + n * kv) * 5, flops=(sel * Hq + 2 * n * c["Hkv"]) * D * f + n * dm * 6)
    q, kv = n * Hq * D * 2, n * c["Hkv"] * D * 2
    W = min(c.get("W", T), T)
    loc = B * (W * (W + 1) / 2 + (T - W) * W)
    glob = sel * (T + 1) / 2
    if kind == "prefill":
        return dict(bytes=q * 2 + q * c["ratio"] + 4 * kv + 4 * n, flops=(loc + glob) * Hq * D * 4)
    if kind == "local":
        return dict(bytes=q * 4 + kv * 4 + n * Hq * 4, flops=loc * Hq * D * 14)
    return dict(bytes=q * c["ratio"] * 3 + q + kv * 4 + sel * Hq * 4, flops=glob * Hq * D * 14)


# ------------------------------------------------------------------ the same in 64 bits
def _topk(p, ratio):
    """The k = floor(ratio * T) largest gates of each sequence, ties to the lower position."""
    B, T = p.shape
    k = int(math.floor(float(torch.tensor(ratio, dtype=torch.float32)) * T))
    order = torch.sort(p.double(), dim=1, descending=True, stable=True).indices[:, :k]
    return torch.zeros((B, T), dtype=torch.bool, device="cuda").scatter_(1, order, True)


def _attn(q, k, v, pos, W, dO=None):
    """Rows q [n, Hq, D] at ascending positions pos against one sequence's k, v [T, Hkv, D]: (o, lse [Hq, n]),
    and with dO also (dq, dk, dv)."""
    n, Hq, D = q.shape
    G, scale = Hq // k.shape[1], D ** -0.5
    o, lse = torch.zeros((n, Hq, D), dtype=torch.float64, device="cuda"), torch.zeros((Hq, n), dtype=torch.float64, device="cuda")
    dq, dk, dv = (torch.zeros(t.shape, dtype=torch.float64, device="cuda") for t in (q, k, v))
    at, R = pos.tolist(), min(2048, max(512, W)) if W < (1 << 29) else 512
    for r0 in range(0, n, R):
        r1 = min(n, r0 + R)
        lo, hi = max(0, at[r0] - W + 1), at[r1 - 1] + 1
        key, row = torch.arange(lo, hi, device="cuda"), pos[r0:r1, None]
        hidden = (key > row) | (key <= row - W)
        for h in range(Hq):
            kk, vv, qq = k[lo:hi, h // G].double(), v[lo:hi, h // G].double(), q[r0:r1, h].double()
            s = (qq @ kk.T).mul_(scale).masked_fill_(hidden, -math.inf)
            m = torch.logsumexp(s, 1)
            s.sub_(m[:, None]).exp_()
            o[r0:r1, h], lse[h, r0:r1] = s @ vv, m
            if dO is not None:
                g = dO[r0:r1, h].double()
                dv[lo:hi, h // G] += s.T @ g
                ds = (g @ vv.T).sub_((g * o[r0:r1, h]).sum(1)[:, None]).mul_(s).mul_(scale)
                dq[r0:r1, h] = ds @ kk
                dk[lo:hi, h // G] += ds.T @ qq
    return (o, lse) if dO is None else (o, lse, dq, dk, dv)


def _rms(o):
    return (o.square().mean(-1, keepdim=True) + EPS).rsqrt()


def _norm_back(dy, o, r, gain):
    """Gradient of o * r(o) * gain with respect to o, r = 1 / sqrt(mean o^2 + eps)."""
    t = dy * gain
    return r * t - o * r ** 3 * (t * o).mean(-1, keepdim=True)


def _fused(o_l, o_g, p, z, gl, gg):
    y = o_l * _rms(o_l) * gl
    w = (p * z)[..., None, None]
    return (1 - w) * y + w * (o_g * _rms(o_g) * gg)


def exact(case, seed):
    c, kind, x = case, case["kind"], _inputs(case, seed)
    if kind == "route":
        F = float((x["p"] > x["b_th"]).double().mean())
        step = x["gamma"] * ((F > c["rho"]) - (F < c["rho"]))
        one = lambda v: torch.full((1,), v, dtype=torch.float64)  # noqa: E731
        return dict(z=None, pos=None, cu_q=None, row_of=None, n=None, b_th=one(x["b_th"] + step), f=one(F))
    B, Hq, D = c["B"], c["Hq"], c["D"]
    inf = 1 << 30
    if kind == "decode":
        z = (x["p"] > x["b_th"]).double()
        ol, og = (torch.zeros((B, 1, Hq, D), dtype=torch.float64, device="cuda") for _ in range(2))
        for b, n in enumerate(x["len"].tolist()):
            s = torch.arange(max(0, n - c["W"]), n, device="cuda") % _ring(c)
            last = torch.tensor([len(s) - 1], device="cuda")
            ol[b] = _attn(x["qL"][b:b + 1], x["kR"][b, s], x["vR"][b, s], last, inf)[0]
            if z[b, 0] > 0:
                og[b] = _attn(x["qG"][b:b + 1], x["kG"][b], x["vG"][b], torch.tensor([n - 1], device="cuda"), inf)[0]
        on = z[:, 0] > 0  # packed rows: the selected sequences in order
        return dict(o=_fused(ol, og, x["p"].double(), z, 1.0, 1.0), o_l=ol[:, 0], o_c=torch.cat([og[on, 0], og[~on, 0]]),
                    z=None)
    T = c["T"]
    every = torch.arange(T, device="cuda")
    if kind == "local":
        out = [_attn(x["q"][b], x["k"][b], x["v"][b], every, c["W"], x["dO"][b]) for b in range(B)]
        return {n: torch.stack([o[i] for o in out]) for i, n in enumerate(("o", "lse", "dq", "dk", "dv"))}
    if kind == "lift":
        p = torch.sigmoid(x["x"].double() @ x["w_g"].double())
        z = _topk(p, c["ratio"])
        out, dl = dict(p=p, z=None, pos=None), x["dgate"].double() * p * (1 - p)
        for n in "qkv":
            u, g, live = x[n].double(), x["g" + n].double(), z if n == "q" else torch.ones_like(z)
            live = live[..., None, None]
            g = g * live
            if c["form"] == "lp":
                a = x["t" + n]["a"].double()
                y, du = torch.einsum("bthi,hij->bthj", u, a), torch.einsum("bthj,hij->bthi", g, a)
                dt = [torch.einsum("bthi,bthj->hij", u, g)]
            else:
                a, b = x["t" + n]["s"].double(), x["t" + n]["b"].double()
                y, du, dt = u * a + b, g * a, [(u * g).sum((0, 1)), g.sum((0, 1))]
            out["u" + n], out["d" + n], out["dt" + n] = y * live, x["d" + n].double() + du, dt
        out["dx"], out["dw"] = dl[..., None] * x["w_g"].double(), torch.einsum("bt,btd->d", dl, x["x"].double())
        return out
    p = x["p"].double()
    z = _topk(x["p"], c["ratio"]) if c.get("mode") != "threshold" else x["p"] > x["b_th"]
    at = [torch.nonzero(z[b]).flatten() for b in range(B)]
    n = sum(len(a) for a in at)
    pad = lambda t, dim=0: torch.cat([t, torch.zeros([B * T - n if i == dim else m for i, m in enumerate(t.shape)],  # noqa: E731
                                                     dtype=t.dtype, device="cuda")], dim)
    if kind == "global":
        first, out = 0, []
        for b, a in enumerate(at):
            out.append(_attn(x["q"][b, a], x["k"][b], x["v"][b], a, inf, x["dO_c"][first:first + len(a)]))
            first += len(a)
        dq = torch.zeros((B, T, Hq, D), dtype=torch.float64, device="cuda")
        for b, a in enumerate(at):
            dq[b, a] = out[b][2]
        return dict(o=pad(torch.cat([o[0] for o in out])), lse=pad(torch.cat([o[1] for o in out], 1), 1), dq=dq,
                    dk=torch.stack([o[3] for o in out]), dv=torch.stack([o[4] for o in out]))
    if kind == "prefill":
        ol, og = (torch.zeros((B, T, Hq, D), dtype=torch.float64, device="cuda") for _ in range(2))
        for b, a in enumerate(at):
            ol[b] = _attn(x["qL"][b], x["kL"][b], x["vL"][b], every, c["W"])[0]
            og[b, a] = _attn(x["qG"][b, a], x["kG"][b], x["vG"][b], a, inf)[0]
        return dict(o=_fused(ol, og, p, z.double(), 1.0, 1.0))
    # fuse
    gl, gg, ol, oc, dO = (x[m].double() for m in ("gain_l", "gain_g", "o_l", "o_c", "dO"))
    oc = oc[:n]
    rl, rg, g, pz = _rms(ol), _rms(oc), dO[z], p[z][:, None, None]
    yl, yg = ol * rl * gl, oc * rg * gg
    o, keep = yl.clone(), (1 - p * z)[..., None, None]
    o[z] = (1 - pz) * yl[z] + pz * yg
    dp = torch.zeros_like(p)
    dp[z] = (g * (yg - yl[z])).sum((1, 2))
    return dict(o=o, rstd_l=rl[..., 0], rstd_g=pad(rg[..., 0]), dO_l=_norm_back(dO * keep, ol, rl, gl),
                dO_c=pad(_norm_back(g * pz, oc, rg, gg)), dgate=dp, dgain_l=(dO * keep * ol * rl).sum((0, 1)),
                dgain_g=(g * pz * oc * rg).sum(0))
