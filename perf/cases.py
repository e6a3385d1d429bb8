"""The workloads this library is timed on, and a generator of more of the same kind.

A case is a dict of plain values.  ``kind`` says which public entry point it goes through:

    linear       Context.linear: one weight tensor applied to ``rows`` activation rows
    head         Context.lm_head: final norm and vocabulary projection
    decode       Context.layer_decode: one token through a decoder layer with attention and a dense FFN
    prefill      Context.layer_prefill: ``tokens`` prompt tokens at cache position ``pos`` through such a layer
    moe_decode   Context.layer_decode on a layer with routed experts (``heads`` = 0: the FFN half alone)
    moe_prefill  Context.layer_prefill on the FFN half of a layer with routed experts

``fmt`` is the weight format: q4 (integer codes), mx (microscaling 4-bit floats) or w16 (unquantized fp16).  ``budget`` is
the share of the weight bytes that may be resident on the GPU, in percent: below 100 the static placement decides which
tensors stay in host memory and are streamed for every pass.  ``odd_on_host`` places the experts with odd index there.

Everything a pass reads is made from the seed: weights, norm gains, router, activations and the filled part of the KV
cache, with the distributions of the library's synthetic workloads (uniform codes, scales |N(0, 0.02)|, activations and
cache N(0, 1)).  A state owns its weights, so passes over several states find none of them in the L2 cache.
"""
import math

import numpy as np
import torch

from paper_2607_10183_b200 import binding as B

BLOCK = 32
DENSE_GAIN, MOE_GAIN = 0.25, 1.0  # standard deviation of the norm gains
MIB = 1 << 20

# The dense layer of the decode and prefill configurations and the expert block of the mixture configuration.
DENSE = {"hidden": 4096, "heads": 32, "kv_heads": 8, "head_dim": 128, "ffn": 14336}
MOE = {"hidden": 2048, "experts": 128, "top_k": 8, "ffn": 768}
MOE_ATTN = {"heads": 32, "kv_heads": 4, "head_dim": 128}


def listed():
    return [
        # One projection, one token (the down projection of a dense layer): the smallest call; what a launch costs matters as
        # much as the kernel.
        {"name": "linear_q4_1row", "kind": "linear", "fmt": "q4", "n": 4096, "k": 14336, "rows": 1},
        # A wide projection for a handful of sequences decoded together.
        {"name": "linear_mx_5rows", "kind": "linear", "fmt": "mx", "n": 14336, "k": 4096, "rows": 5},
        # The end of every decoded token: final norm and a large vocabulary.
        {"name": "head_q4", "kind": "head", "fmt": "q4", "n": 128256, "k": 4096, "rows": 1},
        # One token through one dense layer after a prompt of a thousand tokens: the headline decode step.
        {"name": "decode_q4", "kind": "decode", "fmt": "q4", **DENSE, "pos": 1024, "budget": 100},
        # The same step in the microscaling format late in a long conversation, where the cache is read too.
        {"name": "decode_mx_long", "kind": "decode", "fmt": "mx", **DENSE, "pos": 4090, "budget": 100},
        # The hybrid placement the library exists for: 60 % of the bytes resident, the rest streamed for every token.
        {"name": "decode_q4_hybrid", "kind": "decode", "fmt": "q4", **DENSE, "pos": 600, "budget": 60},
        # One token through a layer with attention and routed experts.
        {"name": "decode_moe", "kind": "moe_decode", "fmt": "q4", **MOE, **MOE_ATTN, "rows": 1, "pos": 700, "odd_on_host": False},
        # Eight sequences through a routed-expert block.
        {"name": "decode_moe_8rows", "kind": "moe_decode", "fmt": "q4", **MOE, "heads": 0, "kv_heads": 0, "head_dim": 0, "rows": 8,
         "pos": 0, "odd_on_host": False},
        # A short prompt of odd length.
        {"name": "prefill_mx_77", "kind": "prefill", "fmt": "mx", **DENSE, "tokens": 77, "pos": 0, "budget": 100},
        # The usual prompt chunk.
        {"name": "prefill_q4_512", "kind": "prefill", "fmt": "q4", **DENSE, "tokens": 512, "pos": 0, "budget": 100},
        # The second large chunk of a long prompt, unquantized weights: the most work of all.
        {"name": "prefill_w16_2048", "kind": "prefill", "fmt": "w16", **DENSE, "tokens": 2048, "pos": 2048, "budget": 100},
        # A prompt chunk through a routed-expert block.
        {"name": "prefill_moe_512", "kind": "moe_prefill", "fmt": "q4", **MOE, "tokens": 512},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dense_shape(rng):
    head_dim = rng.choice([64, 128, 128])
    kv_heads = rng.choice([2, 4, 8])
    hidden = rng.choice([1024, 1536, 2048, 2560, 2880, 3072, 4096, 5120])
    group = max(1, min(8, hidden // (head_dim * kv_heads)))
    ffn = int(hidden * rng.uniform(2.0, 3.5)) // BLOCK * BLOCK
    if rng.random() < 0.5:
        ffn = max(256, ffn // 256 * 256)
    return {"hidden": hidden, "heads": kv_heads * group, "kv_heads": kv_heads, "head_dim": head_dim, "ffn": ffn}


def _moe_shape(rng):
    experts = rng.choice([16, 32, 64, 128])
    return {"hidden": rng.choice([1024, 1536, 2048, 2880]), "experts": experts, "top_k": rng.choice([2, 4, 8]),
            "ffn": rng.choice([512, 768, 1024, 1408])}


def draw(rng):
    kind = rng.choice(["linear", "linear", "linear", "head", "decode", "decode", "prefill", "prefill", "moe_decode", "moe_prefill"])
    fmt = rng.choice(["q4", "q4", "mx", "w16"])
    if kind == "linear":
        n, k = _log_int(rng, 500, 16384), _log_int(rng, 16, 512) * BLOCK
        if rng.random() < 0.5:
            n, k = (n + 255) // 256 * 256, (k + 255) // 256 * 256
        rows = rng.choice([1, _log_int(rng, 2, 8), _log_int(rng, 9, 64), _log_int(rng, 65, 4096)])
        return {"kind": kind, "fmt": fmt, "n": n, "k": k, "rows": max(1, min(rows, int(4.4e11 / (n * k))))}
    if kind == "head":
        return {"kind": kind, "fmt": "q4" if fmt == "w16" else fmt, "n": _log_int(rng, 30000, 128256) // 16 * 16,
                "k": rng.choice([1024, 2048, 2560, 3072, 4096]), "rows": rng.choice([1, 1, _log_int(rng, 2, 8)])}
    if kind in ("decode", "prefill"):
        s = _dense_shape(rng)
        budget = rng.choice([100, 100, 100, rng.randrange(50, 91)])
        if kind == "decode":
            return {"kind": kind, "fmt": fmt, **s, "pos": _log_int(rng, 16, 4200), "budget": budget}
        tokens = rng.choice([_log_int(rng, 9, 128), _log_int(rng, 129, 2048)])
        c = {"kind": kind, "fmt": fmt, **s, "tokens": tokens, "pos": rng.choice([0, 0, rng.randrange(0, 2049)]), "budget": budget}
        while work(c)["flops"] > 9e11:  # at most what the largest listed case takes
            c["tokens"] = c["tokens"] * 4 // 5
        return c
    s = _moe_shape(rng)
    fmt = "q4" if fmt == "w16" else fmt
    if kind == "moe_decode":
        attn = rng.random() < 0.5
        heads = {"heads": s["hidden"] // 128 // 4 * 4, "kv_heads": 4, "head_dim": 128} if attn else {"heads": 0, "kv_heads": 0, "head_dim": 0}
        return {"kind": kind, "fmt": fmt, **s, **heads, "rows": 1 if attn else _log_int(rng, 1, 32),
                "pos": _log_int(rng, 16, 4200) if attn else 0, "odd_on_host": rng.random() < 0.25}
    return {"kind": kind, "fmt": fmt, **s, "tokens": _log_int(rng, 16, 2048)}


# ----------------------------------------------------------------------------------------------------- inputs
class _Draws:
    """Random values of one seed, drawn on the GPU (where that is quick)."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def bytes(self, shape, lo=0, hi=256):
        return torch.randint(lo, hi, shape, dtype=torch.uint8, device="cuda", generator=self.g)

    def normal(self, shape, std=1.0):
        return (torch.randn(shape, device="cuda", generator=self.g) * std).half()

    def weight(self, fmt, n, k, experts=0):
        """(codes, scales) of a block format, or (matrix,), as host arrays in the library's interchange layout."""
        lead = (experts,) if experts else ()
        if fmt == "w16":
            return (self.normal((n, k), 0.09).cpu().numpy(),)
        codes = self.bytes(lead + (n, k // 2))
        if fmt == "mx":
            scales = self.bytes(lead + (n, k // BLOCK), 119, 124)
        else:
            scales = self.normal(lead + (n, k // BLOCK), 0.02).abs()
        return codes.cpu().numpy(), scales.cpu().numpy()


def _matrices(c):
    """(name, n_out, k_in) of the weight matrices of a case in execution order."""
    if c["kind"] in ("linear", "head"):
        return [("w", c["n"], c["k"])]
    h, f = c["hidden"], c["ffn"]
    out = []
    if c.get("heads"):
        qd, kvd = c["heads"] * c["head_dim"], c["kv_heads"] * c["head_dim"]
        out += [("wq", qd, h), ("wk", kvd, h), ("wv", kvd, h), ("wo", h, qd)]
    return out + [("w_gate", f, h), ("w_up", f, h), ("w_down", h, f)]


def tensors(c, seed):
    """Host arrays of everything a case's model holds: {name: array or tuple of arrays}, in registration order."""
    d = _Draws(seed)
    out = {}
    if c["kind"] == "linear":
        out["w"] = d.weight(c["fmt"], c["n"], c["k"])
        return out
    if c["kind"] == "head":
        out["norm"] = d.normal((c["k"],), DENSE_GAIN).cpu().numpy()
        out["w"] = d.weight(c["fmt"], c["n"], c["k"])
        return out
    moe = "experts" in c
    gain = MOE_GAIN if moe and not c.get("heads") else DENSE_GAIN
    for name, n, k in _matrices(c):
        if name == "wq":
            out["attn_norm"] = d.normal((c["hidden"],), gain).cpu().numpy()
        if name == "w_gate":
            out["ffn_norm"] = d.normal((c["hidden"],), gain).cpu().numpy()
            if moe:
                out["router"] = d.normal((c["hidden"], c["experts"]), 0.02).cpu().numpy()
        stacked = moe and name in ("w_gate", "w_up", "w_down")
        out[name] = d.weight(c["fmt"], n, k, c["experts"] if stacked else 0)
    return out


def activations(c, seed):
    """Device tensors a pass reads: the input rows, and the key and value caches with the past positions filled."""
    d = _Draws(seed + 1_000_003)
    rows = c.get("tokens", c.get("rows", 1))
    out = {"x": d.normal((rows, c["k"] if "k" in c else c["hidden"]))}
    if c.get("heads"):
        cap = (c["pos"] + c.get("tokens", 1) + 127) // 128 * 128
        for name in ("k_cache", "v_cache"):
            cache = torch.zeros((c["kv_heads"], cap, c["head_dim"]), dtype=torch.float16, device="cuda")
            cache[:, :c["pos"]] = d.normal((c["kv_heads"], c["pos"], c["head_dim"]))
            out[name] = cache
    return out


_stream = None


def _compute_stream():
    """All states run on one compute stream, like the layers of one model: a high-priority one, which never is one of the
    streams that contexts take for their transfers."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream(priority=-1)
    return _stream


def _slice_bytes(c, n, k):
    return n * k * 2 if c["fmt"] == "w16" else n * k // 2 + n * (k // BLOCK) * 2


def _weight_bytes(c):
    copies = lambda name: c["experts"] if "experts" in c and name in ("w_gate", "w_up", "w_down") else 1  # noqa: E731
    return sum(copies(name) * _slice_bytes(c, n, k) for name, n, k in _matrices(c))


def prepare(case, seed):
    c = case
    rows = c.get("tokens", c.get("rows", 1))
    mats = _matrices(c)
    largest = max(_slice_bytes(c, n, k) for _, n, k in mats)
    hybrid = c.get("budget", 100) < 100 or c.get("odd_on_host", False)
    if c["kind"] in ("linear", "head"):
        # scratch of the split-K GEMM: up to eight fp32 partial results
        workspace = 64 * 1024 + (32 * c["n"] * rows if rows > 8 else 0)
        desc = None
    else:
        kw = {k: c[k] for k in ("hidden", "ffn")}
        if c.get("heads"):
            kw.update(n_q_heads=c["heads"], n_kv_heads=c["kv_heads"], head_dim=c["head_dim"], wq=0)
        if "experts" in c:
            kw.update(n_experts=c["experts"], top_k=c["top_k"])
    act = activations(c, seed)
    if c["kind"] not in ("linear", "head"):
        if c.get("heads"):
            kw["kv_capacity"] = act["k_cache"].shape[1]
        workspace = B.workspace_bytes(B.layer_desc(**kw), rows)
        if c.get("odd_on_host"):  # room for the experts a call gathers
            workspace += _weight_bytes(c) // 2 + 4 * MIB
    slots = 8 if hybrid else 0
    n_slices = sum(c["experts"] if "experts" in c else 1 for _ in mats) + 8
    arena = workspace + slots * (largest + 512) + _weight_bytes(c) + n_slices * 512 + 4 * MIB
    ctx = B.Context(arena, workspace_bytes=workspace, ring_slots=slots, slot_bytes=largest if slots else 0,
                    compute_stream=_compute_stream())
    ids = {}
    for name, t in tensors(c, seed).items():
        if not isinstance(t, tuple):
            ids[name] = ctx.register_f16(t)
        elif len(t) == 1:
            ids[name] = ctx.register_w16(t[0])
        else:
            ids[name] = ctx.register_q4(*t)
    weights = [ids[name] for name, _, _ in mats]
    if c.get("budget", 100) < 100:
        ctx.plan_placement(_weight_bytes(c) * c["budget"] // 100, len(weights))
    elif c.get("odd_on_host"):
        stacked = [ids[name] for name in ("w_gate", "w_up", "w_down")]
        ctx.set_placement([(w, -1, B.ATS_GPU) for w in weights if w not in stacked] +
                          [(w, e, B.ATS_HOST if e % 2 else B.ATS_GPU) for w in stacked for e in range(c["experts"])])
    else:
        ctx.set_placement([(w, -1, B.ATS_GPU) for w in weights])
    state = {"case": c, "ctx": ctx, "ids": ids, **act}
    if c["kind"] in ("linear", "head"):
        state["y"] = torch.empty((rows, c["n"]), dtype=torch.float16, device="cuda")
        state["scratch"] = torch.empty((rows, c["k"]), dtype=torch.float16, device="cuda")
    else:
        kw.update(ids)
        state["desc"] = B.layer_desc(**kw)
        state["y"] = torch.empty_like(act["x"])
    torch.cuda.synchronize()
    return state


def run(state):
    c, ctx = state["case"], state["ctx"]
    kind, x, y = c["kind"], state["x"], state["y"]
    if kind == "linear":
        ctx.linear(state["ids"]["w"], x, y, c["rows"])
        return y
    if kind == "head":
        ctx.lm_head(state["ids"]["norm"], state["ids"]["w"], 1e-5, x, y, c["rows"], state["scratch"])
        return y
    kc, vc = state.get("k_cache"), state.get("v_cache")
    if kind in ("decode", "moe_decode"):
        ctx.layer_decode(state["desc"], x, y, kc, vc, c["pos"], c.get("rows", 1))
    else:
        ctx.layer_prefill(state["desc"], x, y, kc, vc, c.get("pos", 0), c["tokens"])
    return y if kc is None else (y, kc, vc)


# ----------------------------------------------------------------------------------------------------- what a pass costs
def work(case):
    """Every weight that takes part read once (of stacked experts, those that the rows are expected to select), inputs
    read and outputs written once, the attended part of the cache read once."""
    c = case
    rows = c.get("tokens", c.get("rows", 1))
    if c["kind"] in ("linear", "head"):
        n, k = c["n"], c["k"]
        return {"bytes": _slice_bytes(c, n, k) + rows * 2 * (k + n), "flops": 2 * rows * n * k}
    h, f = c["hidden"], c["ffn"]
    nbytes, flops = 4 * rows * h, 0
    if c.get("heads"):
        qd, kvd, pos = c["heads"] * c["head_dim"], c["kv_heads"] * c["head_dim"], c["pos"]
        nbytes += sum(_slice_bytes(c, n, k) for name, n, k in _matrices(c) if name in ("wq", "wk", "wv", "wo"))
        nbytes += 4 * kvd * (pos + 2 * rows)
        flops += 2 * rows * h * (2 * qd + 2 * kvd)
        flops += 4 * qd * sum(pos + t + 1 for t in range(rows))
    ffn_bytes = 2 * _slice_bytes(c, f, h) + _slice_bytes(c, h, f)
    if "experts" in c:
        e, k = c["experts"], c["top_k"]
        nbytes += ffn_bytes * e * (1 - (1 - k / e) ** rows) + 2 * h * e
        flops += 2 * rows * h * e + 6 * rows * k * h * f
    else:
        nbytes += ffn_bytes
        flops += 6 * rows * h * f
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Outputs are fp16 (relative spacing 2^-11).  Against the same pass in 64 bits one operator is off by 2 to 3e-4 (its
    rounding and the order of its fp32 sums), a decode step by up to 5.4e-4, a prefill layer, whose intermediates are all
    stored as fp16, by up to 1.5e-3 and an expert block by 4 to 6e-4: four times that is what is allowed."""
    return {"linear": {"rel": 1e-3}, "head": {"rel": 1e-3}, "decode": {"rel": 2e-3}, "moe_decode": {"rel": 2e-3},
            "prefill": {"rel": 6e-3}, "moe_prefill": {"rel": 2.5e-3}}[case["kind"]]
