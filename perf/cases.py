"""The workloads whose speed this framework is judged by: one transformer layer's calls as a serving program issues them.

A case names a kind of work, a model shape and a batch; `prepare` makes what a program has in hand (weights as loaded,
activations of this pass), `run` makes the library calls of one layer through the Python binding.  Shapes are the ones
the benchmark measures: a 2B-class and an 8B-class dense layer in 8-bit weights, a 3B-class dense layer in 4-bit weights
and a routed layer of 128 experts, eight per token, in 4-bit weights.
"""
import math

import torch

from paper_2607_19438_b200 import binding as qg

# Dense layers: weight format, hidden size, feed-forward size, query heads, key/value heads, head dimension.  The QKV
# projection has (Hq + 2 Hkv) d rows.
DENSE = {
    "2b-q8": dict(qbits=8, K=2048, F=8192, Hq=32, Hkv=4, d=64),
    "3b-q4": dict(qbits=4, K=3072, F=8192, Hq=24, Hkv=8, d=128),
    "8b-q8": dict(qbits=8, K=4096, F=14336, Hq=32, Hkv=8, d=128),
}
# Routed layer: hidden size, experts, experts per token, expert feed-forward size, 4-bit weights.
MOE = dict(H=2048, E=128, k=8, F=768)
HOT_BIAS = 0.80        # added to a quarter of the experts' logits in a skewed case: they get about 60 % of the rows


def listed():
    return [
        # One sequence being generated: every projection reads its weights for a single token, latency counts.
        dict(name="decode 2b-q8 1", kind="decode", model="2b-q8", M=1),
        # A handful of sequences generated together, 4-bit weights.
        dict(name="decode 3b-q4 6", kind="decode", model="3b-q4", M=6),
        # The largest batch of the small-batch call: sixteen sequences, or one with a block of drafted tokens to verify.
        dict(name="decode 8b-q8 16", kind="decode", model="8b-q8", M=16),
        # The routed layer while generating for four sequences: a few rows, each for another expert.
        dict(name="moe 4", kind="moe", M=4, skewed=False, shared=False),
        # A short prompt through the routed layer: every expert is needed, each for a few rows.
        dict(name="moe 128", kind="moe", M=128, skewed=False, shared=False),
        # The ordinary prompt through the routed layer, with the shared expert that some of these models add.
        dict(name="moe 2048 shared", kind="moe", M=2048, skewed=False, shared=True),
        # A long, odd-sized prompt whose routing prefers a quarter of the experts.
        dict(name="moe 5001 skewed", kind="moe", M=5001, skewed=True, shared=False),
        # A short prompt of odd length (a chat turn) through a dense layer in 4-bit weights.
        dict(name="prefill 3b-q4 333", kind="prefill", model="3b-q4", M=333),
        # The ordinary prompt length through a small dense layer in 8-bit weights.
        dict(name="prefill 2b-q8 2048", kind="prefill", model="2b-q8", M=2048),
        # The longest prompt: a document through the largest dense layer.
        dict(name="prefill 8b-q8 8192", kind="prefill", model="8b-q8", M=8192),
        # Attention without a mask over an odd length (an embedding or encoder pass).
        dict(name="attention 3b 1500 full", kind="attention", model="3b-q4", M=1500, causal=False),
        # The dense projections with both operands re-encoded to block-scaled FP8, for callers who accept that format.
        dict(name="fp8 8b 2048", kind="fp8", model="8b-q8", M=2048),
    ]


def _log_size(rng, lo, hi):
    """A size between lo and hi, spread over the logarithm; odd sizes as often as even ones."""
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "moe", "moe", "moe", "prefill", "prefill", "prefill", "attention", "fp8"])
    if kind == "decode":
        return dict(kind=kind, model=rng.choice(sorted(DENSE)), M=rng.randint(1, 16))
    if kind == "moe":
        return dict(kind=kind, M=_log_size(rng, 1, 8192), skewed=rng.random() < 0.3, shared=rng.random() < 0.3)
    if kind == "prefill":
        return dict(kind=kind, model=rng.choice(sorted(DENSE)), M=_log_size(rng, 17, 8000))
    if kind == "attention":
        return dict(kind=kind, model=rng.choice(sorted(DENSE)), M=_log_size(rng, 64, 8000), causal=rng.random() < 0.5)
    return dict(kind=kind, model=rng.choice(sorted(DENSE)), M=_log_size(rng, 17, 8000))


# ------------------------------------------------------------------------------------------------ inputs
class _Source:
    """Seeded tensors on the GPU with the value distributions of the path."""

    def __init__(self, seed):
        self.dev = torch.device("cuda", torch.cuda.current_device())
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(seed)

    def activations(self, rows, cols):
        return torch.randn((rows, cols), device=self.dev, generator=self.g).to(torch.bfloat16)

    def weights(self, qbits, N, K, E=None):
        """(codes, scales): uniform codes, fp16 scales |N(0, 0.02)| / largest code, one per 32 consecutive k."""
        lead = (N,) if E is None else (E, N)
        if qbits == 8:
            q = torch.randint(-127, 128, lead + (K,), dtype=torch.int8, device=self.dev, generator=self.g)
        else:
            q = torch.randint(0, 256, lead + (K // 2,), dtype=torch.uint8, device=self.dev, generator=self.g)
        s = torch.randn(lead + (K // 32,), device=self.dev, generator=self.g).abs_() * (0.02 / (127 if qbits == 8 else 7))
        return q, s.to(torch.float16)


def _projections(m):
    """(name, N, K) of a dense layer's four projections."""
    return [("qkv", (m["Hq"] + 2 * m["Hkv"]) * m["d"], m["K"]), ("o", m["K"], m["Hq"] * m["d"]),
            ("gate_up", 2 * m["F"], m["K"]), ("down", m["K"], m["F"])]


def prepare(case, seed):
    src, kind, M = _Source(seed), case["kind"], case["M"]
    st = dict(kind=kind)
    if kind == "moe":
        H, E, F = MOE["H"], MOE["E"], MOE["F"]
        x, wr = src.activations(M, H), torch.randn((E, H), device=src.dev, generator=src.g) / math.sqrt(H)
        if case["skewed"]:        # hidden states share a component, and a quarter of the experts is tuned to it
            x = x + 0.25
            wr[::4] += HOT_BIAS / (0.25 * H)
        st.update(x=x, router=wr.to(torch.bfloat16), w1=src.weights(4, 2 * F, H, E), w2=src.weights(4, H, F, E))
        if case["shared"]:
            st.update(shared1=src.weights(4, 2 * F, H), shared2=src.weights(4, H, F))
        return st
    m = DENSE[case["model"]]
    st["model"] = m
    if kind == "attention":
        qkv = src.activations(M, (m["Hq"] + 2 * m["Hkv"]) * m["d"])
        st.update(qkv=qkv, causal=case["causal"])
        return st
    for name, N, K in _projections(m):
        st[name] = src.weights(m["qbits"], N, K)
    # what reaches the library from outside it: the layer's input, and the normalised input of the feed-forward block;
    # where attention and gating are the caller's (decode, fp8) also their results
    st.update(x=src.activations(M, m["K"]), x2=src.activations(M, m["K"]))
    if kind != "prefill":
        st.update(attn=src.activations(M, m["Hq"] * m["d"]), act=src.activations(M, m["F"]))
    if kind == "fp8":             # weights are re-encoded once, when the model is loaded
        for name, _, _ in _projections(m):
            st[name] = qg.mx_pack_weights(m["qbits"], *st[name])
    return st


# ------------------------------------------------------------------------------------------------ one pass
def _attend(m, qkv, causal):
    nq, nk = m["Hq"] * m["d"], m["Hkv"] * m["d"]
    return qg.prefill_attention(qkv[:, :nq], qkv[:, nq:nq + nk], qkv[:, nq + nk:], m["Hq"], m["Hkv"], m["d"], causal=causal)


def run(state):
    kind = state["kind"]
    if kind == "decode":
        b = state["model"]["qbits"]
        return (qg.qgemm_small_m(b, state["x"], *state["qkv"]), qg.qgemm_small_m(b, state["attn"], *state["o"]),
                qg.qgemm_small_m(b, state["x2"], *state["gate_up"]), qg.qgemm_small_m(b, state["act"], *state["down"]))
    if kind == "prefill":
        m = state["model"]
        b = m["qbits"]
        qkv = qg.qgemm_dense(b, state["x"], *state["qkv"])
        o = qg.qgemm_dense(b, _attend(m, qkv, True), *state["o"])
        h = qg.qgemm_dense_gate_up_silu(b, state["x2"], *state["gate_up"])
        return qkv, o, qg.qgemm_dense(b, h, *state["down"])
    if kind == "attention":
        return _attend(state["model"], state["qkv"], state["causal"])
    if kind == "fp8":
        x, x2 = qg.mx_quantize(state["x"]), qg.mx_quantize(state["x2"])
        attn, act = qg.mx_quantize(state["attn"]), qg.mx_quantize(state["act"])
        return (qg.qgemm_mx_dense(*x, *state["qkv"]), qg.qgemm_mx_dense(*attn, *state["o"]),
                qg.qgemm_mx_dense(*x2, *state["gate_up"]), qg.qgemm_mx_dense(*act, *state["down"]))
    x, k = state["x"], MOE["k"]
    r = qg.moe_route(qg.moe_router_logits(x, state["router"]), k, X=x)
    h = qg.moe_grouped_qgemm(qg.MODE_GATE_UP_SILU, 4, r["Xperm"], r["offsets"], *state["w1"])
    d = qg.moe_grouped_qgemm(qg.MODE_DOWN_WEIGHTED, 4, h, r["offsets"], *state["w2"], topk_w=r["topk_w"], row_pair=r["row_pair"])
    shared = None
    if "shared1" in state:
        shared = qg.qgemm_dense(4, qg.qgemm_dense_gate_up_silu(4, x, *state["shared1"]), *state["shared2"])
    return dict(y=qg.moe_combine(d, r["pair_row"], k, shared=shared), topk_idx=r["topk_idx"], topk_w=r["topk_w"])


# ------------------------------------------------------------------------------------------------ what a pass needs
def _packed_bytes(qbits, N, K):
    return N * K * (1.0 if qbits == 8 else 0.5) + N * K / 16.0


def work(case):
    kind, M = case["kind"], case["M"]
    if kind == "moe":
        H, E, k, F = MOE["H"], MOE["E"], MOE["k"], MOE["F"]
        used = E * (1.0 - (1.0 - k / E) ** M)           # experts that get a row, for uniform routing
        nbytes = used * (_packed_bytes(4, 2 * F, H) + _packed_bytes(4, H, F)) + 2.0 * E * H + 4.0 * M * H + 8.0 * M * k
        flops = 2.0 * M * k * 3 * F * H + 2.0 * M * E * H
        if case["shared"]:
            nbytes += _packed_bytes(4, 2 * F, H) + _packed_bytes(4, H, F)
            flops += 2.0 * M * 3 * F * H
        return {"bytes": nbytes, "flops": flops}
    m = DENSE[case["model"]]
    pairs = M * (M + 1) / 2.0 if kind == "prefill" or case.get("causal") else float(M) * M
    attend = 4.0 * pairs * m["Hq"] * m["d"]
    if kind == "attention":
        return {"bytes": 2.0 * M * (2 * m["Hq"] + 2 * m["Hkv"]) * m["d"], "flops": attend}
    nbytes = flops = 0.0
    for name, N, K in _projections(m):
        flops += 2.0 * M * N * K
        nbytes += _packed_bytes(m["qbits"], N, K) if kind != "fp8" else N * K * (1.0 + 1.0 / 32)
        if kind != "prefill" or name in ("qkv", "gate_up"):
            nbytes += 2.0 * M * K                        # an input from outside (attention and gating chain inside a prefill)
        if kind != "prefill" or name != "gate_up":
            nbytes += 2.0 * M * N                        # an output that is returned
    if kind == "prefill":
        flops += attend
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Relative 2-norm.  One bf16 rounding is 1.7e-3, and the paths round weights, activations between two calls and
    # outputs once each; block-scaled products are exact, so only the output's rounding is left there.
    if case["kind"] == "fp8":
        return {"rel": 5e-3}
    if case["kind"] == "moe":
        # a token's eighth and ninth expert may be closer than the router sums' rounding
        return {"rel": 1e-2, "differ": 2e-3 if case["M"] >= 64 else 0.1}
    return {"rel": 1e-2}


# ------------------------------------------------------------------------------------------------ the same in 64 bits
def _weights64(qbits, w):
    q, s = w
    if qbits == 4:                # even k in the low nibble, zero point 8
        q = torch.stack((q & 15, q >> 4), -1).flatten(-2).to(torch.int16) - 8
    return (q.double().unflatten(-1, (-1, 32)) * s.double()[..., None]).flatten(-2)


def _silu_mul64(gu):
    g, u = gu.chunk(2, -1)
    return g * torch.sigmoid(g) * u


def _attend64(m, qkv, causal):
    Hq, Hkv, d = m["Hq"], m["Hkv"], m["d"]
    q, k, v = (t.unflatten(-1, (-1, d)) for t in qkv.double().split([Hq * d, Hkv * d, Hkv * d], -1))
    out = torch.empty_like(q)
    mask = torch.ones((len(q), len(q)), dtype=torch.bool, device=q.device).triu(1) if causal else None
    for h in range(Hq):
        p = q[:, h] @ k[:, h * Hkv // Hq].T / math.sqrt(d)
        if causal:
            p.masked_fill_(mask, -math.inf)
        out[:, h] = torch.softmax(p, -1) @ v[:, h * Hkv // Hq]
    return out.flatten(1)


def _block_scaled64(x):
    """Values of a block-scaled FP8 encoding: per 32 values a power of two, floor(log2 of the largest) - 8, and E4M3 codes."""
    b = x.double().unflatten(-1, (-1, 32))
    top = b.abs().amax(-1, keepdim=True)
    scale = torch.ldexp(torch.ones_like(top), torch.frexp(top).exponent - 1 - 8)
    code = torch.where(top > 0, b / scale, b).clamp(-448, 448).float().to(torch.float8_e4m3fn)
    return (code.double() * scale).flatten(-2)


def exact(case, seed):
    kind = case["kind"]
    st = prepare(dict(case, kind="decode") if kind == "fp8" else case, seed)
    if kind != "moe":
        m = DENSE[case["model"]]
    if kind == "attention":
        return _attend64(m, st["qkv"], st["causal"])
    if kind in ("decode", "fp8"):
        enc = _block_scaled64 if kind == "fp8" else torch.Tensor.double
        return tuple(enc(st[x]) @ enc(_weights64(m["qbits"], st[w])).T
                     for x, w in (("x", "qkv"), ("attn", "o"), ("x2", "gate_up"), ("act", "down")))
    if kind == "prefill":
        W = {name: _weights64(m["qbits"], st[name]) for name, _, _ in _projections(m)}
        qkv = st["x"].double() @ W["qkv"].T
        h = _silu_mul64(st["x2"].double() @ W["gate_up"].T)
        return qkv, _attend64(m, qkv, True) @ W["o"].T, h @ W["down"].T
    x = st["x"].double()
    top, idx = (x @ st["router"].double().T).topk(MOE["k"], -1)
    w, y = torch.softmax(top, -1), torch.zeros_like(x)
    for e in range(MOE["E"]):
        t, slot = torch.nonzero(idx == e, as_tuple=True)
        w1, w2 = (_weights64(4, (st[n][0][e], st[n][1][e])) for n in ("w1", "w2"))
        y.index_add_(0, t, w[t, slot, None] * (_silu_mul64(x[t] @ w1.T) @ w2.T))
    if case["shared"]:
        y += _silu_mul64(x @ _weights64(4, st["shared1"]).T) @ _weights64(4, st["shared2"]).T
    return dict(y=y, topk_idx=None, topk_w=w)
