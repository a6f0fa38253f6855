"""Performance cases of the test-time-learning library: what a program that uses it calls.

Every case goes through the public binding.  A case has a "kind":

  context    a new context on every chain: reset the fast weights to W_0, learn the context
             (mone_ttl_context, its _metrics or its _host form), read the memory for a query
             (mone_mem_generate_kv), and copy the learned state out (what a server keeps of a
             context).  Outputs: K, V, W1, W2 (and the momentum in paper mode, the per-segment
             loss and step norms with metrics).
  segment    streaming: a backbone that runs layer by layer hands one segment per layer to
             mone_ttl_segment, with a loss, and the state is copied out.
  read       the memory read alone (mone_mem_generate_kv): prompts of 1 to 4096 query tokens.
  attention  the consumer attention (mone_attention) over [memory || own tokens]: prefill of a
             prompt, and decode steps over a growing cache.

Sizes are those of the repository's workloads (16 layers of 2048 -> 1024 -> 1024, 28 layers of
3072 -> 2048 -> 2048, 8 contexts x 16 layers, 24 layers of per-head SwiGLU with d = 896, the
fp32 256 -> 512 -> 256 chain), with shorter and ragged contexts, and generic ones around them.
Activations, targets, weights and meta-parameters follow the same distributions as the
workloads': X ~ r_l N(0, 1), targets a random linear map of X plus 1% noise.
"""
import math

import torch

import paper_2608_17616_gb300 as mone

DEV = "cuda"

L16 = dict(n_ctx=1, n_layers=16, d_in=2048, d_hid=1024, d_out=1024, hd=64)
L28 = dict(n_ctx=1, n_layers=28, d_in=3072, d_hid=2048, d_out=2048, hd=128)
SWIGLU = dict(n_ctx=1, n_layers=24, d_in=896, d_hid=224, d_out=896, hd=64, memory="swiglu", heads=4)

LEARN = dict(memory="mlp", heads=1, dtype="bf16", mode="paper", loss="dot", renorm="rows", metrics=False, host=False)


def _ctx(name, shape, **kw):
    return {"name": name, "kind": "context", **LEARN, **shape, **kw}


def listed():
    return [
        # one fp32 chain over a whole 4K context: the smallest learning call, a chain of 32 short
        # segments in which latency counts
        _ctx("f32_chain_4k", dict(n_ctx=1, n_layers=1, d_in=256, d_hid=512, d_out=256, hd=64), dtype="f32",
             mode="plain", T=128, N=4096, Q=32),
        # a model's layers in fp32 (a run that checks numerics): widths beyond the on-chip chain
        _ctx("f32_l4_d1024_2k", dict(n_ctx=1, n_layers=4, d_in=1024, d_hid=1024, d_out=1024, hd=64), dtype="f32",
             T=256, N=2000, Q=32),
        # a 1B-class backbone learning a 32K document: the ordinary long context
        _ctx("l16_32k", L16, T=512, N=32768, Q=64),
        # a 3B-class backbone, an 8K prompt with a ragged last segment
        _ctx("l28_8k_ragged", L28, T=1024, N=7777, Q=64),
        # batched serving: 8 contexts x 16 layers, short segments, per-segment metrics on
        _ctx("ctx8_l16_T256_2k", dict(L16, n_ctx=8), T=256, N=2048, Q=64, metrics=True),
        # the paper's own per-head SwiGLU memory
        _ctx("swiglu_l24_8k", SWIGLU, T=512, N=8192, Q=64),
        # the context arrives in pinned host memory
        _ctx("l16_host_4k", L16, T=512, N=4096, Q=64, host=True),
        # streaming: one segment through every layer, layer by layer
        dict(L16, name="segment_l16", kind="segment", T=512, n_tok=512),
        # the memory read of a short query on every layer (time to first token)
        dict(L16, name="read_l16_q64", kind="read", memory="mlp", heads=1, Q=64),
        # the read of a long prompt, a ragged number of query tokens
        dict(L28, name="read_l28_q1000", kind="read", memory="mlp", heads=1, Q=1000),
        # decode: one token over 64 memory tokens and 1023 earlier ones, 32 query heads on 8
        dict(name="attn_decode_1k", kind="attention", n_ctx=1, n_layers=16, n_kv=8, n_q=32, hd=64, Lq=1, n_mem=1087),
        # prefill: a 2K prompt over 64 memory tokens
        dict(name="attn_prefill_2k", kind="attention", n_ctx=1, n_layers=16, n_kv=8, n_q=32, hd=64, Lq=2048, n_mem=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MAX_FLOPS = 6.0e12     # below the largest listed case
MAX_BYTES = 5.5e9
MAX_STATE = 4.0e8      # parameters over all chains


def draw(rng):
    kind = rng.choice(["mlp", "mlp", "mlp", "swiglu", "f32", "f32", "segment", "read", "read", "prefill", "decode"])
    if kind == "prefill":
        hd, n_kv = rng.choice([64, 128]), rng.choice([1, 2, 4, 8])
        c = dict(kind="attention", n_ctx=rng.choice([1, 1, 2, 4]), n_layers=rng.choice([1, 4, 8, 16]), n_kv=n_kv,
                 n_q=n_kv * rng.choice([1, 2, 3, 4, 7, 8]), hd=hd, Lq=_log(rng, 16, 3000), n_mem=_log(rng, 1, 2000))
        while work(c)["flops"] > 6e11:
            c["Lq"] //= 2
        return c
    if kind == "decode":
        n_kv = rng.choice([1, 2, 4, 8])
        c = dict(kind="attention", n_ctx=rng.choice([1, 2, 8]), n_layers=rng.choice([1, 4, 16, 28]), n_kv=n_kv,
                 n_q=n_kv * rng.choice([1, 2, 4, 7, 8]), hd=rng.choice([64, 128]), Lq=rng.choice([1, 1, 1, 2, 5]),
                 n_mem=_log(rng, 16, 16000))
        while work(c)["bytes"] > 2e9:
            c["n_mem"] //= 2
        return c
    if kind == "f32":
        if rng.random() < 0.5:  # chains that fit on chip
            shape = dict(d_in=64 * rng.randint(1, 4), d_hid=64 * rng.randint(1, 12), d_out=128 * rng.randint(1, 2))
        else:
            shape = dict(d_in=64 * rng.randint(4, 24), d_hid=64 * rng.randint(4, 24), d_out=128 * rng.randint(3, 12))
        c = {"kind": "context", **LEARN, **shape, "n_ctx": 1, "n_layers": rng.choice([1, 1, 2, 4, 8]), "hd": 64,
             "dtype": "f32", "mode": rng.choice(["plain", "paper"]), "T": 64 * rng.randint(1, 8),
             "N": _log(rng, 100, 4000), "Q": _log(rng, 1, 100)}
        while work(c)["flops"] > 1.2e11:
            c["N"] = c["N"] // 2 + 1
        return c
    if kind == "swiglu":
        heads = rng.choice([2, 4])
        dh = 32 * rng.choice([4, 6, 8] if heads == 2 else [4, 6, 7, 8])
        c = {"kind": "context", **LEARN, "n_ctx": rng.choice([1, 1, 2]), "n_layers": rng.choice([2, 8, 24]),
             "d_in": heads * dh, "d_out": heads * dh, "d_hid": 32 * rng.randint(3, 8), "hd": 64, "memory": "swiglu",
             "heads": heads, "T": 128 * rng.randint(1, 8), "N": _log(rng, 500, 16000), "Q": _log(rng, 1, 300)}
        return c
    wide = dict(d_in=128 * rng.randint(4, 24), d_hid=256 * rng.randint(2, 8), d_out=256 * rng.randint(2, 8))
    wide = rng.choice([wide, wide, dict(d_in=2048, d_hid=1024, d_out=1024), dict(d_in=3072, d_hid=2048, d_out=2048)])
    wide["hd"] = rng.choice([64, 128])
    if kind == "segment":
        T = 128 * rng.randint(1, 8)
        return dict(wide, kind="segment", n_ctx=1, n_layers=rng.choice([1, 4, 16]), T=T,
                    n_tok=T if rng.random() < 0.5 else rng.randint(1, T))
    if kind == "read":
        if rng.random() < 0.25:
            return dict(SWIGLU, kind="read", n_layers=rng.choice([4, 24]), Q=_log(rng, 1, 1000))
        return dict(wide, kind="read", memory="mlp", heads=1, n_ctx=rng.choice([1, 1, 4]),
                    n_layers=rng.choice([1, 8, 16, 28]), Q=_log(rng, 1, 2000))
    host = rng.random() < 0.15
    c = {"kind": "context", **LEARN, **wide, "n_ctx": rng.choice([1, 1, 1, 2, 8]), "n_layers": rng.choice([1, 4, 16, 28]),
         "loss": "mse" if rng.random() < 0.15 else "dot", "renorm": "out" if rng.random() < 0.1 else "rows",
         "metrics": not host and rng.random() < 0.3, "host": host, "T": 128 * rng.choice([1, 2, 3, 4, 4, 8, 16]),
         "N": _log(rng, 500, 4000 if host else 32768), "Q": _log(rng, 1, 300)}
    while _chains(c) * _params(c) > MAX_STATE:
        c["n_ctx"], c["n_layers"] = max(1, c["n_ctx"] // 2), max(1, c["n_layers"] // 2)
    while work(c)["flops"] > MAX_FLOPS or work(c)["bytes"] > MAX_BYTES:
        c["N"] = c["N"] // 2 + 1
    return c


# ------------------------------------------------------------------ sizes and work

def _chains(c):
    return c["n_ctx"] * c["n_layers"]


def _params(c):
    """Fast weights of a chain."""
    if c.get("memory") == "swiglu":
        return 3 * c["d_hid"] * c["d_in"]
    return c["d_hid"] * (c["d_in"] + c["d_out"])


def work(c):
    """Inputs read once, outputs written once; the contractions of the method."""
    if c["kind"] == "attention":
        el, C, Lq, n = 2, _chains(c), c["Lq"], c["n_mem"]
        pairs = Lq * n + Lq * (Lq + 1) // 2
        return {"bytes": el * C * c["hd"] * (2 * c["n_q"] * Lq + 2 * c["n_kv"] * (n + Lq)),
                "flops": 4 * c["hd"] * pairs * c["n_q"] * C}
    C, p = _chains(c), _params(c)
    if c["kind"] == "read":
        return {"bytes": 2 * C * (p + c["Q"] * (c["d_in"] + c["d_out"])), "flops": 2 * p * c["Q"] * C}
    if c["kind"] == "segment":
        n = c["n_tok"]
        return {"bytes": C * (2 * n * (c["d_in"] + c["d_out"]) + 16 * p), "flops": 4 * p * n * C}
    el = 4 if c["dtype"] == "f32" else 2
    state = 12 if c["mode"] == "paper" else 8  # W_0 in, W (and the momentum) out
    learn = 4 * p + (2 * c["d_hid"] * c["d_out"] if c["loss"] == "mse" else 0)
    return {"bytes": C * (el * (c["N"] + c["Q"]) * (c["d_in"] + c["d_out"]) + state * p),
            "flops": C * (learn * c["N"] + 2 * p * c["Q"])}


def tolerance(c):
    """About four times the distance from exact() that the library shows: fp32 8e-7 (32-bit sums
    through the chain and the read), bf16 3.7e-3 (K, V and the momentum carry the 8-bit mantissa
    of their operands), attention 2.2e-3 (bf16 probabilities and outputs)."""
    if c.get("dtype") == "f32":
        return {"rel": 4e-6, "max": 4e-4}
    if c["kind"] == "attention":
        return {"rel": 9e-3, "max": 0.06}
    return {"rel": 1.6e-2, "max": 0.12}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _layer_scale(c, chain):
    """Activation scale of a layer: 0.5 at the first to 2 at the last (1 for one layer)."""
    L = c["n_layers"]
    return 1.0 if L == 1 else 0.5 + 1.5 * (chain % L) / (L - 1)


def _dtype(c):
    return torch.float32 if c.get("dtype") == "f32" else torch.bfloat16


def _weights(c, g):
    C, F = _chains(c), c["d_hid"]
    if c.get("memory") == "swiglu":
        H, dh = c["heads"], c["d_in"] // c["heads"]
        return (torch.randn(C, H, 2 * F, dh, generator=g, device=DEV) / math.sqrt(dh),
                torch.randn(C, H, F, dh, generator=g, device=DEV) / math.sqrt(F))
    return (torch.randn(C, F, c["d_in"], generator=g, device=DEV) / math.sqrt(c["d_in"]),
            torch.randn(C, F, c["d_out"], generator=g, device=DEV) / math.sqrt(F))


def _meta(c, g, lr=1e-2):
    C, d, H = _chains(c), c["d_in"], c["d_out"] // c["hd"]
    rn = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    return {"alpha": 1 + 0.1 * rn(C, d), "gamma": 0.1 * rn(C, d), "w_eta": 0.5 * rn(C, d) / math.sqrt(d),
            "w_beta": rn(C, d) / math.sqrt(d), "b_eta": torch.full((C,), math.log(math.expm1(lr)), device=DEV),
            "b_beta": torch.zeros(C, device=DEV), "gate": 1 + 0.1 * rn(C, H)}


def _tokens(c, g, n):
    """X [chains, n, d_in] and targets K, V [chains, n, d_out / 2] in the case's type."""
    C, dt, half = _chains(c), _dtype(c), c["d_out"] // 2
    X = torch.empty(C, n, c["d_in"], dtype=dt, device=DEV)
    K = torch.empty(C, n, half, dtype=dt, device=DEV)
    V = torch.empty_like(K)
    for i in range(C):
        r = _layer_scale(c, i)
        x = torch.randn(n, c["d_in"], generator=g, device=DEV) * r
        X[i] = x
        wt = torch.randn(c["d_in"], c["d_out"], generator=g, device=DEV) / (r * math.sqrt(c["d_in"]))
        y = X[i].float() @ wt + 0.01 * torch.randn(n, c["d_out"], generator=g, device=DEV)
        K[i], V[i] = y[:, :half], y[:, half:]
    return X, K, V


def _queries(c, g, Q):
    Xq = torch.randn(_chains(c), Q, c["d_in"], generator=g, device=DEV)
    for i in range(_chains(c)):
        Xq[i] *= _layer_scale(c, i)
    return Xq.to(_dtype(c))


def _inputs(c, seed):
    g = _gen(seed)
    if c["kind"] == "attention":
        C, n = _chains(c), c["n_mem"] + c["Lq"]
        rn = lambda h, t: torch.randn(C, h, t, c["hd"], generator=g, device=DEV).bfloat16()  # noqa: E731
        return {"q": rn(c["n_q"], c["Lq"]), "k": rn(c["n_kv"], n), "v": rn(c["n_kv"], n)}
    d = dict(zip(("W1", "W2"), _weights(c, g)))
    d["meta"] = None if c.get("mode") == "plain" else _meta(c, g)
    if c["kind"] == "context":
        d["X"], d["K"], d["V"] = _tokens(c, g, c["N"])
    elif c["kind"] == "segment":
        d["X"], d["K"], d["V"] = _tokens(c, g, c["n_tok"])
    if "Q" in c:
        d["Xq"] = _queries(c, g, c["Q"])
    return d


# ------------------------------------------------------------------ a program's handle and buffers

class Program:
    """What a program keeps: the memory's handle, its inputs and its output buffers."""

    def __init__(self, c, seed):
        self.c, self.h = c, None
        d = self.d = _inputs(c, seed)
        if c["kind"] == "attention":  # the memory's widths play no part in the attention
            d_out, C = 2 * c["n_kv"] * c["hd"], _chains(c)
            if d_out >= 256:
                cfg = mone.make_config(c["n_ctx"], c["n_layers"], 256, 256, d_out, c["n_kv"], c["hd"], 128, mone.MONE_BF16,
                                       mone.MONE_PLAIN, 1e-2)
                W = torch.zeros(C, 256, 256, device=DEV), torch.zeros(C, 256, d_out, device=DEV)
            else:  # one head of 64: narrower than the MLP memory's tiles, so a two-head SwiGLU memory's handle
                cfg = mone.make_config(c["n_ctx"], c["n_layers"], d_out, 64, d_out, c["n_kv"], c["hd"], 128, mone.MONE_BF16,
                                       mone.MONE_PLAIN, 1e-2, memory=mone.MONE_MEM_SWIGLU, mem_heads=2)
                W = torch.zeros(C, 2, 128, 64, device=DEV), torch.zeros(C, 2, 64, 64, device=DEV)
            self.h = mone.mone_mem_init(cfg, *W)
            self.out = torch.empty_like(d["q"])
            n = c["n_mem"] + c["Lq"]
            self.strides = mone.kv_strides(c["n_layers"], c["n_kv"], n, c["hd"])
            return
        memory, n_kv = c.get("memory", "mlp"), c["d_out"] // (2 * c["hd"])
        cfg = mone.make_config(c["n_ctx"], c["n_layers"], c["d_in"], c["d_hid"], c["d_out"], n_kv, c["hd"],
                               c.get("T", 512), mone.MONE_FP32 if c.get("dtype") == "f32" else mone.MONE_BF16,
                               mone.MONE_PLAIN if c.get("mode") == "plain" else mone.MONE_PAPER, 1e-2,
                               loss=mone.MONE_LOSS_MSE if c.get("loss") == "mse" else mone.MONE_LOSS_DOT,
                               memory=mone.MONE_MEM_SWIGLU if memory == "swiglu" else mone.MONE_MEM_MLP,
                               mem_heads=c.get("heads", 1),
                               renorm_axis=mone.MONE_RENORM_OUT if c.get("renorm") == "out" else mone.MONE_RENORM_ROWS)
        self.h = mone.mone_mem_init(cfg, d["W1"], d["W2"], d["meta"])
        if c.get("host"):
            for k in ("X", "K", "V"):
                d[k] = d[k].cpu().pin_memory()
        out = self.out = {}
        if "Q" in c:
            out["Kq"] = torch.empty(_chains(c), n_kv, c["Q"], c["hd"], dtype=_dtype(c), device=DEV)
            out["Vq"] = torch.empty_like(out["Kq"])
            self.strides = mone.kv_strides(c["n_layers"], n_kv, c["Q"], c["hd"])
        if c["kind"] != "read":
            out["W1"], out["W2"] = torch.empty_like(d["W1"]), torch.empty_like(d["W2"])
            if c.get("mode") != "plain":
                self.zero = torch.zeros_like(d["W1"]), torch.zeros_like(d["W2"])
                out["mu1"], out["mu2"] = torch.empty_like(d["W1"]), torch.empty_like(d["W2"])
        if c["kind"] == "segment":
            out["loss"] = torch.empty(c["n_layers"], device=DEV)
        if c.get("metrics"):
            S = -(-c["N"] // c["T"])
            out["loss"], out["step"] = (torch.empty(S, _chains(c), device=DEV) for _ in range(2))

    def __del__(self):
        if self.h:
            mone.mone_mem_free(self.h)


def prepare(c, seed):
    return Program(c, seed)


def run(p):
    c, d, out, h = p.c, p.d, p.out, p.h
    if c["kind"] == "attention":
        mone.mone_attention(h, d["q"], c["n_q"], c["Lq"], d["k"], d["v"], p.strides, c["n_mem"], out)
        return {"out": out}
    if c["kind"] == "segment":
        for layer in range(c["n_layers"]):
            mone.mone_ttl_segment(h, 0, layer, d["X"][layer], d["K"][layer], d["V"][layer], c["n_tok"],
                                  loss_out=out["loss"][layer:])
    elif c["kind"] == "context":
        if c["mode"] == "paper":
            mone.mone_mem_write_state(h, d["W1"], d["W2"], *p.zero)
        else:
            mone.mone_mem_write_state(h, d["W1"], d["W2"])
        if c["metrics"]:
            mone.mone_ttl_context_metrics(h, d["X"], d["K"], d["V"], c["N"], out["loss"], out["step"])
        elif c["host"]:
            mone.mone_ttl_context_host(h, d["X"], d["K"], d["V"], c["N"])
        else:
            mone.mone_ttl_context(h, d["X"], d["K"], d["V"], c["N"])
    if "Q" in c:
        mone.mone_mem_generate_kv(h, d["Xq"], c["Q"], out["Kq"], out["Vq"], p.strides)
    if c["kind"] != "read":
        mone.mone_mem_read_state(h, out["W1"], out["W2"], out.get("mu1"), out.get("mu2"))
    return out


# ------------------------------------------------------------------ the same in 64 bits

def _exact_attention(c, seed):
    d = _inputs(c, seed)
    group, Lq, n = c["n_q"] // c["n_kv"], c["Lq"], c["n_mem"]
    out = torch.empty(d["q"].shape, dtype=torch.float64, device=DEV)
    hidden = torch.arange(n + Lq, device=DEV)[None, :] > n + torch.arange(Lq, device=DEV)[:, None]
    for i in range(_chains(c)):
        for kv in range(c["n_kv"]):
            q = d["q"][i, kv * group:(kv + 1) * group].double()
            k, v = d["k"][i, kv].double(), d["v"][i, kv].double()
            z = (q @ k.T / math.sqrt(c["hd"])).masked_fill(hidden, -math.inf)
            out[i, kv * group:(kv + 1) * group] = torch.softmax(z, dim=-1) @ v
    return {"out": out}


def _transform(x, m):
    if m is None:
        return x
    z = torch.nn.functional.silu(m["alpha"][:, None] * x + m["gamma"][:, None])
    return z / torch.sqrt((z * z).sum(-1, keepdim=True) + 1e-12)


def _heads(c, x):
    """[chains, n, d] -> [chains, heads, n, d / heads]."""
    return x.unflatten(-1, (c.get("heads", 1), -1)).transpose(1, 2)


def _forward(c, u, W1, W2):
    """The memory's output and what its gradient needs; weights [chains, heads, hidden, width]."""
    h = u @ W1.transpose(-1, -2)
    if c.get("memory") == "swiglu":
        P, G = h.split(c["d_hid"], dim=-1)
        return torch.nn.functional.silu(P) * G, (P, G)
    return torch.nn.functional.silu(h), (h, None)


def _silu_prime(h):
    s = torch.sigmoid(h)
    return s * (1 + h * (1 - s))


def exact(c, seed):
    if c["kind"] == "attention":
        return _exact_attention(c, seed) if work(c)["flops"] < 4e12 else None
    if work(c)["flops"] > 1.0e13:
        return None
    d = _inputs(c, seed)
    m = None if d["meta"] is None else {k: v.double() for k, v in d["meta"].items()}
    swiglu, C = c.get("memory") == "swiglu", _chains(c)
    W = [d["W1"].double(), d["W2"].double()]
    if not swiglu:
        W = [w[:, None] for w in W]                       # one head
    out = {}
    if c["kind"] != "read":
        mu = [torch.zeros_like(w) for w in W]
        axes = [-1, -2 if c.get("renorm") == "out" else -1]
        norms = [w.norm(dim=a, keepdim=True) for w, a in zip(W, axes)]
        n, T = c.get("N", c.get("n_tok")), c["T"]
        losses, steps = [], []
        for s in range(0, n, T):
            x = d["X"][:, s:s + T].double()
            y = torch.cat([d["K"][:, s:s + T], d["V"][:, s:s + T]], -1).double()
            u, y, t = _heads(c, _transform(x, m)), _heads(c, y), x.shape[1]
            A, (P, G) = _forward(c, u, *W)
            eta, beta = torch.full((C, t), 1e-2, dtype=torch.float64, device=DEV), None
            if m is not None:
                eta = torch.nn.functional.softplus(torch.einsum("ctd,cd->ct", x, m["w_eta"]) + m["b_eta"][:, None])
                beta = torch.sigmoid(torch.einsum("cd,cd->c", x.mean(1), m["w_beta"]) + m["b_beta"])
            o = A @ W[1]
            if c.get("loss") == "mse":
                losses.append(0.5 * ((o - y) ** 2).sum((1, 2, 3)) / t)
                dO = (o - y) * (eta / t)[:, None, :, None]
            else:
                losses.append(-(o * y).sum((1, 2, 3)) / t)
                dO = -y * (eta / t)[:, None, :, None]
            dA = dO @ W[1].transpose(-1, -2)
            if swiglu:
                dh = torch.cat([dA * G * _silu_prime(P), dA * torch.nn.functional.silu(P)], -1)
            else:
                dh = dA * _silu_prime(P)
            for i, g in enumerate((dh.transpose(-1, -2) @ u, A.transpose(-1, -2) @ dO)):
                mu[i] = g if beta is None else beta[:, None, None, None] * mu[i] + g
                W[i] = W[i] - mu[i]
                if m is not None:
                    W[i] = W[i] * (norms[i] / W[i].norm(dim=axes[i], keepdim=True))
            steps.append(sum((g * g).sum((1, 2, 3)) for g in mu))
        for k, w in (("W1", W[0]), ("W2", W[1]), ("mu1", mu[0]), ("mu2", mu[1])):
            if k[0] == "W" or m is not None:
                out[k] = w if swiglu else w[:, 0]
        if c["kind"] == "segment":
            out["loss"] = losses[0]
        if c.get("metrics"):
            out["loss"], out["step"] = torch.stack(losses), torch.stack(steps)
    if "Q" in c:
        o = _forward(c, _heads(c, _transform(d["Xq"].double(), m)), *W)[0] @ W[1]
        o = o.transpose(1, 2).flatten(2).unflatten(-1, (-1, c["hd"])).transpose(1, 2)   # [chains, out heads, Q, hd]
        o = o / torch.sqrt((o * o).mean(-1, keepdim=True) + 1e-6)
        if m is not None:
            o = o * m["gate"][:, :, None, None]
        n_kv = c["d_out"] // (2 * c["hd"])
        out["Kq"], out["Vq"] = o[:, :n_kv].contiguous(), o[:, n_kv:].contiguous()
    return out
