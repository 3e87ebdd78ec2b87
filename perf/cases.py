"""The work that a program built on this library has it do, as measurable cases.

A case is one call (or one graph replay) through the Python binding of the C
ABI.  Four kinds:

  layer   one MoE-layer forward over a decode or verify batch, on packed or
          plain expert weights, in one of the five selection modes
  route   selection, refinement and permutation on scores the caller holds
          (an engine that runs its own expert FFN)
  static  the same without a workspace (a plugin that may not allocate)
  stack   a CUDA graph of L residual layers under one global budget

Shapes are those of workloads.py (olmoe, qwen3, dsr1) and generic ones.
Inputs follow its distributions: router weights N(0, 1/sqrt(d)), expert
weights N(0, 0.02), tokens independent, sharing a request-level part, or drawn
from a few domains; scores handed to `route` are softmaxes of such logits.
"""
import math

import torch

from paper_2602_07265_gb300 import xshare as X

MODES = {"topk": 0, "batch": 1, "group": 2, "hier": 3, "thresh": 4}

# Layer shapes: experts, top-k, model width, expert width, token correlation.
SHAPES = {
    "olmoe": dict(N=64, k=8, d=2048, F=1024, x="iid"),
    "qwen3": dict(N=128, k=8, d=2048, F=768, x="request"),
    "dsr1": dict(N=256, k=8, d=7168, F=2048, x="domains"),
}

# Fields a case leaves out.
DEFAULTS = dict(budget=0, k0=0, m_r=0, T=1, G=1, m_g=0, tau=0.0, sparse=0, shared=0, packed=True,
                L=1, P=1)


def _layer(name, shape, **kw):
    return {"name": name, "kind": "layer", **SHAPES[shape], **kw}


def listed():
    return [
        # One user, one token: the latency of a decode step.
        _layer("olmoe_b1", "olmoe", B=1, mode="batch", budget=24),
        # A decode batch on a small layer, budget m = 24.
        _layer("olmoe_b32", "olmoe", B=32, mode="batch", budget=24),
        # A very large batch (the most tokens a call takes): hundreds of tokens per expert.
        _layer("olmoe_b8192", "olmoe", B=8192, mode="batch", budget=48),
        # Speculative verify, 25 requests of 1 + 4 tokens, weights as the checkpoint holds them.
        _layer("qwen3_b125_t5_plain", "qwen3", B=125, mode="hier", T=5, k0=1, m_r=4, packed=False),
        # Speculative verify, 64 requests of 1 + 3 tokens.
        _layer("qwen3_b256_hier", "qwen3", B=256, mode="hier", T=4, k0=1, m_r=4),
        # Plain top-k routing of a large batch: the baseline every selection is compared with.
        _layer("qwen3_b2048_topk", "qwen3", B=2048, mode="topk"),
        # A few users on a large layer that also has a shared expert.
        _layer("dsr1_b7_shared", "dsr1", B=7, mode="batch", budget=24, k0=1, shared=1),
        # The decode batch the paper's figures are quoted on.
        _layer("dsr1_b32", "dsr1", B=32, mode="batch", budget=24, k0=1),
        # Expert groups (as over 8 devices) on a verify batch of 64 requests of 4 tokens.
        _layer("dsr1_b256_group", "dsr1", B=256, mode="group", T=4, k0=1, G=8, m_g=5),
        # Routing only, for an engine with an FFN of its own, grouped experts.
        dict(name="route_b2048_group", kind="route", B=2048, N=256, k=8, mode="group", k0=1, G=8, m_g=5),
        # Routing only, from a plugin without memory of its own; many experts, odd sizes.
        dict(name="static_b100_n1000", kind="static", B=100, N=1000, k=8, mode="batch", budget=64, k0=1),
        # Sixteen layers of a small model as one graph, budget 24 per layer.
        dict(name="olmoe_stack16", kind="stack", **SHAPES["olmoe"], B=32, mode="batch", budget=384, L=16, P=4),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _selection(rng, c, mode):
    """A mode and its options, over what the paper sweeps; B follows the request length."""
    N = c["N"]
    c["mode"] = mode
    if mode in ("batch", "group", "thresh"):
        c["k0"] = rng.choice([0, 1, 1, 2])
    if mode == "batch":
        c["budget"] = rng.randint(min(N, 8), min(N, 64))
    elif mode == "thresh":
        c["tau"] = round(rng.uniform(0.3, 0.9), 2)
    elif mode == "group":
        c["G"] = rng.choice([g for g in (1, 2, 4, 8, 16) if N % g == 0])
        c["m_g"] = max(1, rng.randint(16, 64) // c["G"])
    elif mode == "hier":
        c["k0"], c["m_r"], c["budget"] = rng.choice([(1, 4, 0), (1, 5, 0), (2, 4, 0), (0, 4, 16)])
        c["T"] = rng.randint(2, 8)
        c["B"] = max(1, c["B"] // c["T"]) * c["T"]
    if mode != "topk" and c["kind"] != "static" and rng.random() < 0.2:
        c["sparse"] = 1
    return c


def draw(rng):
    kind = rng.choices(["layer", "generic", "route", "static", "stack"], [10, 4, 3, 1, 1])[0]
    modes = ["batch", "batch", "hier", "group", "thresh", "topk"]
    if kind == "layer":
        shape = rng.choice(["olmoe", "qwen3", "dsr1"])
        c = dict(kind="layer", **SHAPES[shape])
        # The widest layer streams gigabytes at any batch: it is run in decode and verify batches.
        c["B"] = _log_int(rng, 1, 300 if shape == "dsr1" else 8192)
        if shape == "dsr1":
            modes = ["batch", "batch", "hier", "group"] if c["B"] <= 64 else ["batch", "group"]
        _selection(rng, c, rng.choice(modes))
        if shape == "dsr1" and c["mode"] == "batch":
            c["budget"] = min(c["budget"], 40)
            c["k0"] = min(c["k0"], 1)
        c["packed"] = rng.random() < 0.75
        if rng.random() < 0.25:
            c["shared"] = rng.randint(1, 2)
            c["B"] = min(c["B"], 6000 // c.get("T", 1) * c.get("T", 1))
        return c
    if kind == "generic":
        c = dict(kind="layer", N=_log_int(rng, 8, 512), x=rng.choice(["iid", "request", "domains"]),
                 d=128 * _log_int(rng, 2, 40), F=128 * _log_int(rng, 1, 16))
        c["k"] = rng.randint(1, min(12, c["N"]))
        c["N"] = max(c["k"], min(c["N"], int(4e9 / (6 * c["d"] * c["F"]))))
        c["B"] = min(_log_int(rng, 1, 8192), max(1, int(7e11 / (c["k"] * 6 * c["d"] * c["F"]))))
        _selection(rng, c, rng.choice(modes))
        c["packed"] = rng.random() < 0.75
        return c
    if kind == "stack":
        c = dict(kind="stack", **SHAPES[rng.choice(["olmoe", "qwen3"])], B=_log_int(rng, 1, 64),
                 L=rng.randint(3, 12), P=2, mode="batch", k0=rng.choice([0, 1]))
        c["budget"] = c["L"] * rng.randint(16, 32)
        return c
    c = dict(kind=kind, N=_log_int(rng, 32, 1024), B=_log_int(rng, 1, 8192 if kind == "route" else 1024))
    c["k"] = rng.choice([1, 2, 4, 6, 8, 8, 8, 10, 16])
    return _selection(rng, c, rng.choice(modes))


# ---------------------------------------------------------------- inputs


def _full(case):
    return {**DEFAULTS, **case}


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1_000_003 + stream)
    return g


def _tokens(c, seed):
    """x [B, d] bf16 and the routers W_g [P][N, d] fp32."""
    g = _gen(seed, 1)
    B, d, T = c["B"], c["d"], max(1, c["T"])
    Wg = [torch.randn(c["N"], d, generator=g, device="cuda") / math.sqrt(d) for _ in range(c["P"])]
    z = torch.randn(B, d, generator=g, device="cuda")
    req = torch.arange(B, device="cuda") // T
    n_req = (B + T - 1) // T
    if c["x"] == "request":
        z = torch.randn(n_req, d, generator=g, device="cuda")[req] + 0.5 * z
    elif c["x"] == "domains":
        u = 1.5 * torch.randn(4, d, generator=g, device="cuda")
        z = u[torch.randint(0, 4, (n_req,), generator=g, device="cuda")[req]] + z
    return z.to(torch.bfloat16), Wg


def _experts(c, seed, n, stream):
    """W_gate, W_up [n, F, d] and W_down [n, d, F], bf16.  In a stack W_down is
    ten times smaller, so that the residual stream stays near 1."""
    g = _gen(seed, stream)
    d, F = c["d"], c["F"]
    out = []
    for shape, std in (((n, F, d), 0.02), ((n, F, d), 0.02),
                       ((n, d, F), 0.002 if c["kind"] == "stack" else 0.02)):
        out.append(torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=g))
    return tuple(out)


def _scores(c, seed):
    """[B, N] softmax scores of logits with a batch-wide, a request and a token part."""
    g = _gen(seed, 1)
    B, N, T = c["B"], c["N"], max(1, c["T"])
    req = torch.arange(B, device="cuda") // T
    h = 1.5 * torch.randn(4, N, generator=g, device="cuda")[req % 4]
    h = h + 0.5 * torch.randn((B + T - 1) // T, N, generator=g, device="cuda")[req]
    h = h + torch.randn(B, N, generator=g, device="cuda")
    return torch.softmax(h, dim=1)


def _params(c):
    return X.route_params(k0=c["k0"], m_r=c["m_r"], tokens_per_request=c["T"], n_groups=c["G"],
                          m_g=c["m_g"], tau=c["tau"], sparse_scores=c["sparse"])


def prepare(case, seed):
    c = _full(case)
    B, N, k = c["B"], c["N"], c["k"]
    mode, prm = MODES[c["mode"]], _params(c)
    dev = torch.device("cuda")
    st = dict(c=c, mode=mode, prm=prm)
    out = dict(mask=torch.empty(N, dtype=torch.uint8, device=dev),
               ids=torch.empty(B, k, dtype=torch.int32, device=dev),
               w=torch.empty(B, k, dtype=torch.float32, device=dev),
               stats=torch.zeros(X.STATS_WORDS, dtype=torch.int32, device=dev))
    if c["kind"] in ("route", "static"):
        st["scores"] = _scores(c, seed)
        out.update(counts=torch.empty(N, dtype=torch.int32, device=dev),
                   offsets=torch.empty(N + 1, dtype=torch.int32, device=dev),
                   perm=torch.zeros(B * k, dtype=torch.int32, device=dev))
        if c["kind"] == "route":
            st["ws"] = torch.empty(X.xshare_workspace_size(B, N, k, 0, 0, mode, prm),
                                   dtype=torch.uint8, device=dev)
        st["out"] = out
        return st
    x, Wg = _tokens(c, seed)
    st["x"] = x
    st["ws"] = torch.empty(X.xshare_workspace_size(B, N, k, c["d"], c["F"], mode, prm, c["shared"]),
                           dtype=torch.uint8, device=dev)
    if c["kind"] == "stack":
        packs = [X.Packed(*_experts(c, seed, N, 10 + p)) for p in range(c["P"])]
        layers = [(Wg[i % c["P"]], packs[i % c["P"]]) for i in range(c["L"])]
        h = torch.empty(c["L"], B, c["d"], dtype=torch.bfloat16, device=dev)
        st["out"] = dict(h=h)
        st["layers"] = layers
        torch.cuda.synchronize()
        st["graph"] = X.StackGraph(x, layers, k, c["budget"], mode, prm, h, st["ws"])
        return st
    st["W_g"] = Wg[0]
    raw = _experts(c, seed, N, 10)
    sh = _experts(c, seed, c["shared"], 9) if c["shared"] else None
    if c["packed"]:
        st["experts"] = X.Packed(*raw)
        st["shared"] = X.Packed(*sh) if sh else None
    else:
        st["experts"], st["shared"] = raw, sh
    out["y"] = torch.empty(B, c["d"], dtype=torch.bfloat16, device=dev)
    st["out"] = out
    return st


def run(st):
    c, o = st["c"], st["out"]
    if c["kind"] == "stack":
        st["graph"].launch()
        return o
    if c["kind"] == "route":
        X.xshare_route(st["scores"], c["k"], c["budget"], st["mode"], st["prm"], o["mask"], o["ids"],
                       o["w"], st["ws"], stats=o["stats"], expert_counts=o["counts"],
                       expert_offsets=o["offsets"], perm=o["perm"])
        return o
    if c["kind"] == "static":
        X.xshare_route_static(st["scores"], c["k"], c["budget"], st["mode"], st["prm"], o["mask"],
                              o["ids"], o["w"], stats=o["stats"], expert_counts=o["counts"],
                              expert_offsets=o["offsets"], perm=o["perm"])
        return o
    kw = dict(shared=st["shared"], sel_mask=o["mask"], topk_ids=o["ids"], topk_w=o["w"], stats=o["stats"])
    if c["packed"]:
        X.xshare_moe_forward_packed(st["x"], st["W_g"], st["experts"], c["k"], c["budget"], st["mode"],
                                    st["prm"], o["y"], st["ws"], **kw)
    else:
        X.xshare_moe_forward(st["x"], st["W_g"], *st["experts"], c["k"], c["budget"], st["mode"],
                             st["prm"], o["y"], st["ws"], **kw)
    return o


# ---------------------------------------------------------------- 64-bit reference


def _best(values, count, live):
    """Mask of the `count` largest live values (equal ones: lower index first)."""
    v = torch.where(live, values, torch.full_like(values, -math.inf))
    order = torch.sort(v, descending=True, stable=True).indices
    mask = torch.zeros_like(live)
    mask[order[:count]] = True
    return mask & live


def _route64(c, p):
    """Selected set, ids [B, k'], weights [B, k'] from 64-bit scores p [B, N]."""
    B, N, k, k0, mode = c["B"], c["N"], c["k"], c["k0"], c["mode"]
    order = torch.sort(p, dim=1, descending=True, stable=True).indices
    warm = torch.zeros(B, N, dtype=torch.bool, device=p.device)
    if mode != "topk" and k0:
        warm.scatter_(1, order[:, :k0], True)
    g = p
    if c["sparse"] and mode != "topk":
        top = p.gather(1, order[:, :k])
        g = torch.zeros_like(p).scatter_(1, order[:, :k], top / top.sum(1, keepdim=True))
    s = g.sum(0)
    sel = warm.any(0)
    gain = s > 0 if c["sparse"] else torch.ones(N, dtype=torch.bool, device=p.device)
    if mode == "topk":
        sel = torch.ones(N, dtype=torch.bool, device=p.device)
    elif mode == "group":
        G = c["G"]
        live = ((~sel) & gain).view(G, N // G)
        avail, base = live.sum(1), int(sel.sum())
        R = 0
        while base + int(torch.clamp(avail, max=R).sum()) < min(c["m_g"], N) * G and R < int(avail.max()):
            R += 1
        add = torch.stack([_best(s.view(G, -1)[j], R, live[j]) for j in range(G)])
        sel = sel | add.reshape(-1)
    elif mode == "thresh":
        cand = torch.sort(torch.where((~sel) & gain, s, torch.full_like(s, -math.inf)), descending=True, stable=True)
        f, target, n = float(s[sel].sum()), c["tau"] * float(s.sum()), int(((~sel) & gain).sum())
        vals, idx, i = cand.values.tolist(), cand.indices.tolist(), 0
        sel = sel.clone()
        while f < target and i < n:
            sel[idx[i]] = True
            f += vals[i]
            i += 1
    else:
        if mode == "hier":
            T = c["T"]
            sr, wr = g.view(-1, T, N).sum(1), warm.view(-1, T, N).any(1)
            live = (~wr) & (sr > 0 if c["sparse"] else True)
            v = torch.where(live, sr, torch.full_like(sr, -math.inf))
            o = torch.sort(v, dim=1, descending=True, stable=True).indices[:, :c["m_r"]]
            add = torch.zeros_like(wr).scatter_(1, o, True) & live
            sel = (wr | add).any(0)
        sel = sel | _best(s, c["budget"], (~sel) & gain)
    kp = min(k, int(sel.sum()))
    v = torch.where(sel, p, torch.full_like(p, -1.0))
    ids = torch.sort(v, dim=1, descending=True, stable=True).indices[:, :kp]
    top = p.gather(1, ids)
    return sel, ids, top / top.sum(1, keepdim=True)


def _ffn64(x, Wg, Wu, Wd, e):
    a = x @ Wg[e].double().T
    return (a * torch.sigmoid(a) * (x @ Wu[e].double().T)) @ Wd[e].double().T


def _layer64(c, x, W_g, experts, shared):
    x = x.double()
    p = torch.softmax(x @ W_g.double().T, dim=1)
    sel, ids, w = _route64(c, p)
    y = torch.zeros_like(x)
    for e in torch.unique(ids).tolist():
        t, slot = torch.nonzero(ids == e, as_tuple=True)
        y.index_add_(0, t, w[t, slot, None] * _ffn64(x[t], *experts, e))
    for j in range(c["shared"]):
        y += _ffn64(x, *shared, j)
    return y, w


def _pad(w, k):
    return torch.nn.functional.pad(w, (0, k - w.shape[1]))


def exact(case, seed):
    c = _full(case)
    none = dict.fromkeys(["mask", "ids", "stats"])
    if c["kind"] in ("route", "static"):
        w = _route64(c, _scores(c, seed).double())[2]
        return dict(none, w=_pad(w, c["k"]), counts=None, offsets=None, perm=None)
    x, Wg = _tokens(c, seed)
    if c["kind"] == "stack":
        sets = [_experts(c, seed, c["N"], 10 + p) for p in range(c["P"])]
        hs = []
        for i in range(c["L"]):
            # The interface hands bf16 from layer to layer.
            b = dict(c, budget=c["budget"] // c["L"] + (1 if i < c["budget"] % c["L"] else 0))
            h = x.double() + _layer64(b, x, Wg[i % c["P"]], sets[i % c["P"]], None)[0]
            hs.append(h)
            x = h.to(torch.bfloat16)
        return dict(h=torch.stack(hs))
    y, w = _layer64(c, x, Wg[0], _experts(c, seed, c["N"], 10),
                    _experts(c, seed, c["shared"], 9) if c["shared"] else None)
    return dict(none, y=y, w=_pad(w, c["k"]))


def tolerance(case):
    c = _full(case)
    if c["kind"] in ("route", "static"):
        return "exact"  # the interface fixes every sum's order: all results are defined to the bit
    # bf16 outputs of 32-bit sums over bf16 activations: y is 2.4e-3 off 64 bits.
    # `differ`: routing decides on 32-bit scores, whose last bits depend on the
    # order of the router's sums; equal-looking scores may swap.
    return {"rel": 1e-2, "max": 0.1, "differ": 2e-3}


def work(case):
    c = _full(case)
    B, N, k = c["B"], c["N"], c["k"]
    out = B * k * 8 + N
    if c["kind"] in ("route", "static"):
        return {"bytes": B * N * 4 + out + B * k * 4 + 8 * N, "flops": 2 * B * N}
    d, F = c["d"], c["F"]
    x, Wg = _tokens(c, 0)
    per = dict(c, budget=c["budget"] // c["L"])
    ids = _route64(per, torch.softmax(x.double() @ Wg[0].double().T, dim=1))[1]
    used = int(torch.unique(ids).numel())
    rows = ids.numel() + c["shared"] * B
    # Weights of the used experts, router, tokens in and out; two flops a weight and row.
    one = {"bytes": (used + c["shared"]) * 6 * d * F + N * d * 4 + 4 * B * d + (out if c["kind"] == "layer" else 0),
           "flops": rows * 6 * d * F + 2 * B * N * d}
    return {m: float(v) * c["L"] for m, v in one.items()}
