"""Performance cases of the LoRA linear library, each one pass through its
public entry points (paper_2606_19528_gb300.lora).

Kinds of case:
  linear   one adapted projection: forward and backward as two calls, as an
           autograd function makes them (`calls` "two"), as one stack call
           ("step"), the forward alone ("fwd"), or the forward without a
           workspace ("noalloc")
  layer    the seven projections of a decoder layer in one stack call, with
           bf16 or 4-bit base weights, adapters on every projection or on q
           and v only
  ckpt     a stack of decoder layers under the checkpointed schedule
  ce       the LM head's reduced-vocabulary cross entropy
  topk     the top-k similarity table of an embedding

Sizes are those of the Llama-3.2-3B- and Qwen-2.5-3B-shaped layers and LM head
of paper_2606_19528_gb300/workloads.py and of the tests, or generic.
"""
from __future__ import annotations

import math

import torch

from paper_2606_19528_gb300 import lora, workloads

LLAMA = {"h": 3072, "kv": 1024, "f": 8192}
QWEN = {"h": 2048, "kv": 256, "f": 11008}
FULL, FWD = "fwd_bwd", "fwd"


def _layer(name, T, rank, dims, mode=FULL, q4=False, qv_only=False):
    return dict(kind="layer", name=name, T=T, rank=rank, q4=q4, qv_only=qv_only, mode=mode, **dims)


def listed():
    return [
        # the smallest adapted linear of the configurations: bound by launches and latency
        dict(kind="linear", name="linear_T128_256x256_r8", T=128, K=256, N=256, rank=8, q4=False, calls="two"),
        # one attention projection at a short sequence: forward and backward of one module in one call
        dict(kind="linear", name="llama_q_T512_r16", T=512, K=3072, N=3072, rank=16, q4=False, calls="step"),
        # sizes that are multiples of 8 and of nothing larger, a rank that is padded: forward, then backward
        dict(kind="linear", name="ragged_T1000_3080x4104_r12", T=1000, K=3080, N=4104, rank=12, q4=False,
             calls="two"),
        # evaluating a 32-token prompt: the no-grad forward of a layer, bound by reading the weights
        _layer("llama_layer_T32_fwd", 32, 16, LLAMA, mode=FWD),
        # a training step on a short sample with 4-bit weights, adapters on q and v as the method places them
        _layer("llama_layer_T64_q4_qv", 64, 16, LLAMA, q4=True, qv_only=True),
        # a training step on a short sequence, bf16 weights, every projection adapted
        _layer("llama_layer_T256_r16", 256, 16, LLAMA),
        # the ordinary training step
        _layer("llama_layer_T2048_r16", 2048, 16, LLAMA),
        # the same step with 4-bit weights
        _layer("llama_layer_T2048_q4", 2048, 16, LLAMA, q4=True),
        # a long sequence, the other model's narrow k and v, a large rank
        _layer("qwen_layer_T4096_r64", 4096, 64, QWEN),
        # the checkpointed schedule, adapters on q and v, 4-bit weights
        dict(kind="ckpt", name="llama_ckpt3_T1024_q4_qv", layers=3, T=1024, rank=16, q4=True, qv_only=True, **LLAMA),
        # the LM head over a top-500 vocabulary, 30 % of the positions trainable
        dict(kind="ce", name="lm_head_ce_T2048_top500", T=2048, d=3072, V=128256, k=500, trainable=0.3),
        # the one-time table of an embedding
        dict(kind="topk", name="topk_table_V40000_k500", V=40000, d=3072, k=500),
    ]


# ---------------------------------------------------------------- drawn cases
def _log8(rng, lo, hi, step=8):
    """A multiple of `step` in [lo, hi], spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi + step - 1)))
    return max(lo, min(hi, int(v) // step * step))


def draw(rng):
    while True:
        kind = rng.choice(["linear", "linear", "linear", "layer", "layer", "layer", "ckpt", "ce", "topk"])
        if kind == "linear":
            q4 = rng.random() < 0.25
            c = dict(kind=kind, T=_log8(rng, 8, 8192), K=_log8(rng, 256, 11008, 256 if q4 else 8),
                     N=_log8(rng, 64, 11008), rank=rng.choice([1, 4, 8, 8, 12, 16, 16, 20, 32, 64, 128]), q4=q4,
                     calls=rng.choice(["two", "two", "step", "fwd", "fwd" if q4 else "noalloc"]))
            if c["calls"] == "noalloc" and c["T"] * c["K"] * c["rank"] > 1 << 27:
                continue
        elif kind == "layer":
            dims = rng.choice([LLAMA, QWEN, {"h": _log8(rng, 1024, 4096, 256), "kv": _log8(rng, 256, 1024, 128),
                                             "f": _log8(rng, 2048, 11008, 256)}])
            c = dict(kind=kind, T=_log8(rng, 32, 4096), rank=rng.choice([4, 8, 16, 16, 32, 64]),
                     q4=rng.random() < 0.35, qv_only=rng.random() < 0.35, mode=rng.choice([FULL, FULL, FWD]), **dims)
        elif kind == "ckpt":
            qv = rng.random() < 0.5
            c = dict(kind=kind, layers=rng.randint(2, 3) if qv else 2, T=_log8(rng, 128, 1024),
                     rank=rng.choice([8, 16, 32]), q4=rng.random() < 0.5, qv_only=qv, **rng.choice([LLAMA, QWEN]))
        elif kind == "ce":
            V = _log8(rng, 2000, 128256, 1)
            c = dict(kind=kind, T=_log8(rng, 32, 4096, 1), d=_log8(rng, 256, 4096), V=V,
                     k=rng.choice([0, 50, 100, 200, 500]), trainable=round(rng.uniform(0.1, 1.0), 2))
        else:
            V = _log8(rng, 2000, 39999, 1)
            c = dict(kind=kind, V=V, d=_log8(rng, 256, 3072), k=_log8(rng, 16, 1024, 1))
        # none costs more than the largest ordinary step (the table's draws stay below the listed table)
        if kind == "topk" or work(c)["flops"] <= 1.4e12:
            return c


# ---------------------------------------------------------------- shapes
def _projs(case):
    """(K, N, rank, input buffer) of each projection of one layer, or of the one linear."""
    if case["kind"] == "linear":
        return [(case["K"], case["N"], case["rank"], 0)]
    h, kv, f = case["h"], case["kv"], case["f"]
    r = case["rank"]
    o = 0 if case["qv_only"] else r
    return [(h, h, r, 0), (h, kv, o, 0), (h, kv, r, 0), (h, h, o, 1), (h, f, o, 2), (h, f, o, 2), (f, h, o, 3)]


def _parts(case):
    """Which of forward and backward a case runs, and whether the forward saves su."""
    if case["kind"] == "linear":
        bwd = case["calls"] in ("two", "step")
        return True, bwd, True
    bwd = case["kind"] == "ckpt" or case["mode"] == FULL
    return True, bwd, bwd and case["kind"] != "ckpt"


def work(case):
    if case["kind"] == "ce":
        T, d, V = case["T"], case["d"], case["V"]
        nT = max(1, round(T * case["trainable"]))
        nJ = min(V, _expected_vocab(case))
        return {"bytes": 2 * nT * d + 2 * nJ * d + 2 * T * d + 9 * T + (4 * nT * case["k"] if case["k"] else 0),
                "flops": 4 * nT * nJ * d}
    if case["kind"] == "topk":
        V, d = case["V"], case["d"]
        return {"bytes": 2 * V * d + 4 * V * case["k"], "flops": V * (V + 1) * d}  # the matrix is symmetric
    fwd, bwd, save = _parts(case)
    T, layers = case["T"], case.get("layers", 1)
    flops = nbytes = 0
    for K, N, r, g in _projs(case):
        w = N * K // 2 + N * K // 16 if case["q4"] else 2 * N * K
        nbytes += w + 2 * r * (K + N) + 2 * T * N
        flops += 2 * T * K * N + 2 * T * r * (K + N)
        if save:
            nbytes += 2 * T * r
        if bwd:
            nbytes += 2 * T * N + 2 * T * K + 4 * r * (K + N)
            flops += 2 * T * K * N + 4 * T * r * (K + N)
    nbytes += sum(2 * T * K for K in {g: K for K, N, r, g in _projs(case)}.values())
    return {"bytes": nbytes * layers, "flops": flops * layers}


def _cluster(V):
    return min(512, V)


def _expected_vocab(case):
    """Tokens of the reduced vocabulary J, from the distribution of the targets (exactly V without a table)."""
    V, k = case["V"], case["k"]
    if not k:
        return V
    nT = max(1, round(case["T"] * case["trainable"]))
    c = _cluster(V)
    n_cl = -(-V // c)
    w = [(i + 1) ** -2.5 for i in range(n_cl)]
    s = sum(w)
    kk = min(k, c)
    return max(1, int(sum(c * (1 - (1 - kk / c) ** (nT * x / s)) for x in w)))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(g, shape, std):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).mul_(std).to(torch.bfloat16)


def _projections(case, g):
    """One layer's inputs: activations and gradients N(0, 1), W of variance 1 / K, A uniform, B with std 0.02,
    4-bit weights of about the same variance."""
    T, xs, out = case["T"], {}, []
    bwd = _parts(case)[1]
    for K, N, r, grp in _projs(case):
        if grp not in xs:
            xs[grp] = _normal(g, (T, K), 1.0)
        p = {"K": K, "N": N, "r": r, "x": xs[grp]}
        if case["q4"]:
            p["codes"] = torch.randint(0, 256, (N, K // 2), generator=g, device="cuda", dtype=torch.uint8)
            u = torch.rand((N, K // 64, 2), generator=g, device="cuda")
            s = ((0.5 + u[:, :, 0]) * (2 * math.sqrt(3) / (15 * math.sqrt(K)))).to(torch.bfloat16)
            b = (-(7.5 + 2 * u[:, :, 1] - 1) * s.float()).to(torch.bfloat16)
            p["params"] = torch.stack([s, b], dim=-1).contiguous()
        else:
            p["W"] = _normal(g, (N, K), 1 / math.sqrt(K))
        if r:
            p["A"] = ((torch.rand((r, K), generator=g, device="cuda") * 2 - 1) / math.sqrt(K)).to(torch.bfloat16)
            p["B"] = _normal(g, (N, r), 0.02)
        if bwd:
            p["dy"] = _normal(g, (T, N), 1.0)
        out.append(p)
    return out


def _outputs(case, p):
    T, bf = case["T"], dict(dtype=torch.bfloat16, device="cuda")
    fwd, bwd, save = _parts(case)
    p["y"] = torch.empty((T, p["N"]), **bf)
    if save and p["r"]:
        p["su"] = torch.empty((T, p["r"]), **bf)
    if bwd:
        p["dx"] = torch.empty((T, p["K"]), **bf)
        if p["r"]:
            p["dA"] = torch.empty((p["r"], p["K"]), dtype=torch.float32, device="cuda")
            p["dB"] = torch.empty((p["N"], p["r"]), dtype=torch.float32, device="cuda")


def _scale(case):
    return 2.0  # alpha = 2 r


def _ws(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def _proj(case, p):
    shape = lora.make_shape(case["T"], p["K"], p["N"], p["r"], _scale(case))
    q = lora.make_q4(p["codes"], p["params"]) if case["q4"] else None
    return lora.make_proj(shape, x=p["x"], W=p.get("W"), A=p.get("A"), B=p.get("B"), dy=p.get("dy"), y=p["y"],
                          su=p.get("su"), dx=p.get("dx"), dA=p.get("dA"), dB=p.get("dB"), Wq=q)


def _ce_inputs(case, g):
    T, d, V, k = case["T"], case["d"], case["V"], case["k"]
    st = {"h": _normal(g, (T, d), 1.0), "E": _normal(g, (V, d), 1 / math.sqrt(d))}
    c = _cluster(V)
    n_cl = -(-V // c)
    w = torch.arange(1, n_cl + 1, device="cuda", dtype=torch.float64) ** -2.5
    cdf = torch.cumsum(w, 0) / w.sum()
    u = torch.rand((2, T), generator=g, device="cuda", dtype=torch.float64)
    cl = torch.searchsorted(cdf, u[0]).clamp_(max=n_cl - 1)
    base = (cl * c).clamp_(max=V - c)
    st["targets"] = (base + (u[1] * c).long().clamp_(max=c - 1)).to(torch.int32)
    n = max(1, round(T * case["trainable"]))
    st["mask"] = torch.zeros(T, dtype=torch.uint8, device="cuda")
    st["mask"][T - n:] = 1  # a prompt, then its trainable response
    if k:
        kk = min(k, c)
        i = torch.arange(V, device="cuda")
        base = (i // c * c).clamp_(max=V - c)
        table = torch.empty((V, kk), dtype=torch.int32, device="cuda")
        for a in range(0, V, 16384):
            e = min(V, a + 16384)
            off = torch.rand((e - a, c - 1), generator=g, device="cuda").argsort(dim=1)[:, :kk - 1] + 1
            table[a:e, 0] = i[a:e].to(torch.int32)
            table[a:e, 1:] = (base[a:e, None] + (i[a:e, None] - base[a:e, None] + off) % c).to(torch.int32)
        st["topk"] = table
    return st


def prepare(case, seed):
    g = _gen(seed)
    if case["kind"] == "ce":
        st = _ce_inputs(case, g)
        T, d, V = case["T"], case["d"], case["V"]
        st["loss"] = torch.empty(1, dtype=torch.float32, device="cuda")
        st["token_loss"] = torch.empty(T, dtype=torch.float32, device="cuda")
        st["dh"] = torch.empty((T, d), dtype=torch.bfloat16, device="cuda")
        st["vocab"] = torch.zeros(V, dtype=torch.int32, device="cuda")  # J, then zeros
        t = st.get("topk")
        st["args"] = lora.make_ce_args(T, d, V, st["h"], st["E"], st["targets"], st["loss"], mask=st["mask"], topk=t,
                                       ld_topk=t.shape[1] if t is not None else 0,
                                       k=t.shape[1] if t is not None else 0, token_loss=st["token_loss"],
                                       dh=st["dh"], vocab=st["vocab"])
        st["ws"] = _ws(lora.lora_ce_workspace_size(st["args"]))
    elif case["kind"] == "topk":
        V, d, k = case["V"], case["d"], min(case["k"], case["V"])
        st = {"E": _normal(g, (V, d), 1 / math.sqrt(d)), "table": torch.empty((V, k), dtype=torch.int32, device="cuda"),
              "ws": _ws(lora.lora_topk_workspace_size(V, d, k))}
    else:
        layers = []
        for _ in range(case.get("layers", 1)):
            L = _projections(case, g)
            for p in L:
                _outputs(case, p)
            layers.append(L)
        st = {"layers": layers, "projs": [[_proj(case, p) for p in L] for L in layers]}
        if case["kind"] == "ckpt":
            st["ws"] = _ws(lora.lora_stack_ckpt_workspace_size(st["projs"]))
        elif case["kind"] == "layer":
            st["mode"] = lora.LORA_FWD_BWD if case["mode"] == FULL else lora.LORA_FWD
            st["ws"] = _ws(lora.lora_stack_workspace_size(st["projs"][0], st["mode"]))
        else:
            p = layers[0][0]
            st["shape"] = lora.make_shape(case["T"], p["K"], p["N"], p["r"], _scale(case))
            if case["q4"]:
                st["Wq"] = lora.make_q4(p["codes"], p["params"])
            if case["calls"] != "noalloc":
                mode = lora.LORA_FWD if case["calls"] == "fwd" else lora.LORA_FWD_BWD
                st["ws"] = _ws(lora.lora_workspace_size(st["shape"], mode))
    st["case"] = case
    return st


# ---------------------------------------------------------------- one pass
def _results(case, layers):
    return [{k: p[k] for k in ("y", "su", "dx", "dA", "dB") if k in p} for L in layers for p in L]


def run(st):
    case = st["case"]
    if case["kind"] == "ce":
        nT, nJ = lora.lora_ce_fwd_bwd(st["args"], st["ws"], st["ws"].numel())
        return {"trainable": nT, "loss": st["loss"], "token_loss": st["token_loss"], "dh": st["dh"],
                "vocab": st["vocab"], "tokens": nJ}
    if case["kind"] == "topk":
        V, k = st["table"].shape
        lora.lora_topk_table(st["E"], V, case["d"], k, st["table"], st["ws"], st["ws"].numel())
        return st["table"]
    if case["kind"] == "ckpt":
        lora.lora_stack_ckpt(st["projs"], st["ws"], st["ws"].numel())
    elif case["kind"] == "layer":
        lora.lora_stack_step(st["projs"][0], st["mode"], st["ws"], st["ws"].numel())
    else:
        p, shape, ws = st["layers"][0][0], st["shape"], st.get("ws")
        n = ws.numel() if ws is not None else 0
        if case["calls"] == "step":
            lora.lora_stack_step(st["projs"][0], lora.LORA_FWD_BWD, ws, n)
        elif case["calls"] == "noalloc":
            lora.lora_linear_fwd_noalloc(shape, p["x"], p["W"], p["A"], p["B"], p["y"], p["su"])
        else:
            fwd = lora.lora_linear_fwd_q4 if case["q4"] else lora.lora_linear_fwd
            bwd = lora.lora_linear_bwd_q4 if case["q4"] else lora.lora_linear_bwd
            W = st["Wq"] if case["q4"] else p["W"]
            fwd(shape, p["x"], W, p["A"], p["B"], p["y"], p["su"], ws, n)
            if case["calls"] == "two":
                bwd(shape, p["dy"], p["x"], W, p["A"], p["B"], p["su"], p["dx"], p["dA"], p["dB"], ws, n)
    return _results(case, st["layers"])


# ---------------------------------------------------------------- what is right
def tolerance(case):
    if case["kind"] == "topk":
        # the order of similarities that differ by less than fp32 sums in another order
        return {"rel": 0.0, "differ": 4e-3}
    # y, dx, su and dh are rounded to bf16 once; dA and dB inherit the rounding of su and sv, dh that of
    # softmax - onehot: 1.7e-3 against 64-bit arithmetic, the largest single difference about one rounding
    # step of the largest values
    return {"rel": 7e-3, "max": 0.06}


def _f64(t):
    return t.to(torch.float64)


def _dense_weight(p):
    if "W" in p:
        return _f64(p["W"])
    words = p["codes"].view(torch.int32).to(torch.int64)  # [N, K / 8]
    q = torch.stack([(words >> (4 * (i // 2) + 16 * (i % 2))) & 15 for i in range(8)], dim=-1)
    q = _f64(q.reshape(p["N"], p["K"] // 64, 64))
    s, b = _f64(p["params"][:, :, 0:1]), _f64(p["params"][:, :, 1:2])
    return _f64((s * q + b).to(torch.float32).to(torch.bfloat16)).reshape(p["N"], p["K"])


def _exact_proj(case, p):
    """The layer's definition: y = x W^T + s (x A^T) B^T and its gradients, W rounded to bf16 as its format says."""
    s, r = _scale(case), p["r"]
    fwd, bwd, save = _parts(case)
    W, x = _dense_weight(p), _f64(p["x"])
    o = {"y": x @ W.T}
    if r:
        A, B = _f64(p["A"]), _f64(p["B"])
        su = s * (x @ A.T)
        o["y"] += su @ B.T
        if save:
            o["su"] = su
    if bwd:
        dy = _f64(p["dy"])
        o["dx"] = dy @ W
        if r:
            sv = s * (dy @ B)
            o["dx"] += sv @ A
            o["dA"] = sv.T @ x
            o["dB"] = dy.T @ su
    return o


def _exact_ce(case, st):
    T, V, k = case["T"], case["V"], case["k"]
    t = st["mask"].nonzero().flatten()
    y = st["targets"].long()[t]
    J = torch.unique(st["topk"].long()[y].flatten()) if k else torch.arange(V, device="cuda")
    H, EJ = _f64(st["h"])[t], _f64(st["E"])[J]
    z = H @ EJ.T
    lse = torch.logsumexp(z, dim=1)
    col = torch.searchsorted(J, y)
    i = torch.arange(len(t), device="cuda")
    row = lse - z[i, col]
    G = torch.exp(z - lse[:, None])
    G[i, col] -= 1.0
    tl = torch.zeros(T, dtype=torch.float64, device="cuda")
    tl[t] = row
    dh = torch.zeros((T, case["d"]), dtype=torch.float64, device="cuda")
    dh[t] = G @ EJ
    vocab = torch.zeros(V, dtype=torch.int32, device="cuda")
    vocab[:len(J)] = J.to(torch.int32)
    return {"trainable": len(t), "loss": row.sum().reshape(1), "token_loss": tl, "dh": dh, "vocab": vocab,
            "tokens": len(J)}


def exact(case, seed):
    g = _gen(seed)
    if case["kind"] == "ce":
        return _exact_ce(case, _ce_inputs(case, g))
    if case["kind"] == "topk":
        V, d, k = case["V"], case["d"], min(case["k"], case["V"])
        if V * V * d > 1.3e12:
            return None  # many seconds at the 64-bit rate
        E = _f64(_normal(g, (V, d), 1 / math.sqrt(d)))
        E = _f64((E / E.norm(dim=1, keepdim=True)).to(torch.float32).to(torch.bfloat16))
        out = torch.empty((V, k), dtype=torch.int32, device="cuda")
        for a in range(0, V, 2048):
            out[a:a + 2048] = torch.sort(E[a:a + 2048] @ E.T, dim=1, descending=True, stable=True)[1][:, :k].to(
                torch.int32)
        return out
    res = []
    for _ in range(case.get("layers", 1)):
        L = _projections(case, g)
        for p in L:
            res.append(_exact_proj(case, p))
    return res
