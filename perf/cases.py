"""Workloads of this library that are timed and compared between versions of its code.

Each case is a dict of plain values: its `op`, sizes and options. `listed()` gives the fixed
ones, `draw(rng)` more of the same ranges, `prepare(case, seed)` what a program holds before the
call (inputs, weights, workspaces and output buffers on the GPU), `run(state)` one pass through
the entry points of `paper_2309_00754_gb300.hydra`, `work(case)` the bytes and flops that pass
cannot do without, `tolerance(case)` how far another correct implementation may be off, and
`exact(case, seed)` the same outputs from plain torch in 64 bits.

The operations are those of one experience-scoring and update iteration of Hydra-PPO on a
Llama-7B-shaped model (d 4096, 32 heads of 128, SwiGLU 11008, vocabulary 32000):
  linear    the LoRA linear of 1 to 3 streams over one frozen weight
  lm_head   the dual LM head with log-probabilities and the KL-penalised reward
  attention causal attention over fused q/k/v rows
  update    GAE, then the PPO losses and their gradients
  score     a whole scoring pass (embedding, decoder layers, heads, rewards, advantages)
  generate  prefill and key/value-cached decoding with both streams
Whole passes run three decoder layers, which is every form a layer takes in them (the first,
a middle one, the last)."""
import math

import torch

from paper_2309_00754_gb300 import hydra as H
from paper_2309_00754_gb300 import llama

DEV = "cuda"
D, HEADS, FFN, VOCAB = 4096, 32, 11008, 32000
LAYERS, RANK, SCALE, EPS, THETA = 3, 16, 2.0, 1e-6, 10000.0
BETA, GAMMA, LAM, CLIP = 0.1, 1.0, 0.95, 0.2


def listed():
    return [
        # one token of one sequence through a projection: a decode step's linear
        {"name": "linear_1", "op": "linear", "m": 1, "k": 4096, "n": 4096, "r": 16, "streams": 2,
         "f32": False},
        # a short prompt, or a decode batch, through the gate projection of both streams
        {"name": "linear_40", "op": "linear", "m": 40, "k": 4096, "n": 11008, "r": 8, "streams": 2,
         "f32": False},
        # one medium sequence, first layer: both heads of one input, a larger LoRA rank
        {"name": "linear_300_shared", "op": "linear", "m": 300, "k": 4096, "n": 4096, "r": 64,
         "streams": 1, "f32": False},
        # the down projection of a full scoring batch (4 x 768 tokens)
        {"name": "linear_3072", "op": "linear", "m": 3072, "k": 11008, "n": 4096, "r": 16,
         "streams": 2, "f32": False},
        # log-probabilities and rewards of four 400-token completions of ragged length
        {"name": "lm_head_4x400", "op": "lm_head", "s": 4, "l": 400, "d": D, "v": VOCAB, "r": 0,
         "shared": False},
        # two short sequences (one per stream)
        {"name": "attention_2x97", "op": "attention", "s": 2, "p": 97, "heads": HEADS},
        # both streams of four 400 + 400-token sequences
        {"name": "attention_8x800", "op": "attention", "s": 8, "p": 800, "heads": HEADS},
        # the update side of one small batch: a launch-bound call
        {"name": "update_4x512", "op": "update", "s": 4, "l": 512, "whiten": True},
        # the update side of a large experience buffer at the 400-token completion length
        {"name": "update_16384x400", "op": "update", "s": 16384, "l": 400, "whiten": True},
        # scoring one short sequence: weights bound, every launch counts
        {"name": "score_1x97", "op": "score", "s": 1, "p0": 37, "l": 60, "critic": False},
        # the full scoring batch
        {"name": "score_4x768", "op": "score", "s": 4, "p0": 256, "l": 512, "critic": False},
        # four prompts, 32 tokens each
        {"name": "generate_4x200", "op": "generate", "s": 4, "p0": 200, "steps": 32},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["linear", "linear", "linear", "lm_head", "attention", "attention", "update",
                     "score", "generate"])
    if op == "linear":
        # rows of 16 bytes: widths are multiples of 8
        k = rng.choice([4096, 11008, 8 * _log(rng, 32, 1376)])
        n = rng.choice([4096, 11008, 12288, 8 * _log(rng, 32, 1536)])
        return {"op": op, "m": _log(rng, 1, 3072), "k": k, "n": n,
                "r": rng.choice([0, 8, 16, 32, 64, 128]), "streams": rng.choice([1, 2, 2, 3]),
                "f32": rng.random() < 0.25}
    if op == "lm_head":
        return {"op": op, "s": rng.randint(1, 8), "l": _log(rng, 5, 250), "d": rng.choice([2048, D]),
                "v": 8 * rng.randint(500, 4000), "r": rng.choice([0, 8, 16]),
                "shared": rng.random() < 0.5}
    if op == "attention":
        return {"op": op, "s": rng.randint(1, 8), "p": _log(rng, 20, 1000),
                "heads": rng.choice([12, 16, HEADS])}
    if op == "update":
        return {"op": op, "s": _log(rng, 1, 16384), "l": _log(rng, 16, 400),
                "whiten": rng.random() < 0.5}
    if op == "score":
        return {"op": op, "s": rng.randint(1, 4), "p0": _log(rng, 8, 200), "l": _log(rng, 16, 300),
                "critic": rng.random() < 0.4}
    return {"op": op, "s": _log(rng, 1, 32), "p0": _log(rng, 8, 150), "steps": rng.randint(2, 24)}


# --------------------------------------------------------------------------- inputs


class _Rand:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(seed)

    def f32(self, *shape, std=1.0):
        return std * torch.randn(*shape, device=DEV, generator=self.g)

    def bf16(self, *shape, std=1.0):
        return self.f32(*shape, std=std).to(torch.bfloat16)

    def ints(self, lo, hi, *shape):
        return torch.randint(lo, hi, shape, device=DEV, generator=self.g, dtype=torch.int32)

    def lengths(self, s, l, least=8):
        """Ragged: a `least`-th of the slots to all of them."""
        return self.ints(max(1, l // least), l + 1, s)


def _config(case, response):
    return dict(n_layers=LAYERS, d_model=D, n_heads=HEADS, head_dim=128, ffn=FFN, vocab=VOCAB,
                prompt_len=case["p0"], response_len=response, lora_rank=RANK, lora_scale=SCALE,
                rms_eps=EPS, rope_theta=THETA, beta=BETA, gamma=GAMMA, lam=LAM)


def _empty(*shape, dtype=torch.float32):
    return torch.empty(*shape, dtype=dtype, device=DEV)


# A pass's outputs as views of a few flat buffers, each view on a 256-byte boundary: what
# belongs together is compared together (one score alone says little in 16-bit arithmetic).
_PARTS = {"logp": ("logp_actor", "logp_ref"), "heads": ("values", "score"),
          "credit": ("reward", "advantages", "returns")}


def _parts(op):
    return {k: v for k, v in _PARTS.items() if op == "score" or k != "credit"}


def _flat(parts, s, l, dtype=torch.float32):
    """({flat buffer by name}, {view by output name}), zeroed."""
    flat, view = {}, {}
    for k, names in parts.items():
        size = {n: s if n == "score" else s * l for n in names}
        flat[k] = torch.zeros(sum((v + 63) // 64 * 64 for v in size.values()), dtype=dtype,
                              device=DEV)
        at = 0
        for n in names:
            view[n] = flat[k][at:at + size[n]].view((s,) if n == "score" else (s, l))
            at += (size[n] + 63) // 64 * 64
    return flat, view


def _inputs(case, seed):
    """The seeded tensors of a case (what both `prepare` and `exact` start from)."""
    g = _Rand(seed)
    op = case["op"]
    if op == "linear":
        m, k, n, r, ns = (case[x] for x in ("m", "k", "n", "r", "streams"))
        t = {"x": [g.bf16(m, k) for _ in range(ns)], "W": g.bf16(n, k, std=0.02)}
        lora = 0 if r == 0 else max(1, ns - 1)
        t["A"] = [g.bf16(r, k, std=0.02) for _ in range(lora)]
        t["B"] = [g.bf16(n, r, std=0.02) for _ in range(lora)]
        return t
    if op == "lm_head":
        s, l, d, v, r = (case[x] for x in ("s", "l", "d", "v", "r"))
        t = {"h": [g.bf16(s * l, d) for _ in range(1 if case["shared"] else 2)],
             "W": g.bf16(v, d, std=0.02), "ids": g.ints(0, v, s * l), "lengths": g.lengths(s, l),
             "score": g.f32(s)}
        t["A"] = g.bf16(r, d, std=0.02) if r else None
        t["B"] = g.bf16(v, r, std=0.02) if r else None
        return t
    if op == "attention":
        # q, k and v as the projection of normed rows gives them (std 0.02 sqrt(4096))
        return {"qkv": g.bf16(case["s"] * case["p"], 3 * 128 * case["heads"], std=1.28)}
    if op == "update":
        s, l = case["s"], case["l"]
        lengths = g.lengths(s, l)
        old = -g.f32(s, l).abs() - 0.5
        reward = g.f32(s, l, std=0.02)
        last = torch.arange(l, device=DEV)[None] == (lengths - 1)[:, None]
        reward = torch.where(last, reward + g.f32(s, 1), reward)
        return {"old": old, "new": old + g.f32(s, l, std=0.1), "reward": reward,
                "values": g.f32(s, l, std=0.5), "lengths": lengths}
    t = {"w": llama.random_device_weights(_config(case, 1), seed, DEV)}
    if op == "score":
        t["critic"] = (llama.random_device_lora(_config(case, 1), seed + 1, DEV)
                       if case["critic"] else None)
        t["ids"] = g.ints(0, VOCAB, case["s"], case["p0"] + case["l"])
        t["lengths"] = g.lengths(case["s"], case["l"], 2)
        return t
    # generation: standard Gumbel noise, with one token of each draw raised far above the rest,
    # so that every implementation draws the same sequence and its outputs can be compared
    s, n = case["s"], case["steps"]
    t["ids"] = g.ints(0, VOCAB, s, case["p0"])
    t["tokens"] = g.ints(0, VOCAB, s, n)
    u = torch.rand(n, s, VOCAB, device=DEV, generator=g.g).clamp_(1e-20, 1 - 1e-7)
    noise = -torch.log(-torch.log(u))
    noise.scatter_add_(2, t["tokens"].T.long()[..., None],
                       torch.full((n, s, 1), 1000.0, device=DEV))
    t["noise"] = noise
    return t


def prepare(case, seed):
    t = _inputs(case, seed)
    op = t["op"] = case["op"]
    t["case"] = case
    if op == "linear":
        m, n, r, ns = (case[x] for x in ("m", "n", "r", "streams"))
        dt = torch.float32 if case["f32"] else torch.bfloat16
        t["y"] = [_empty(m, n, dtype=dt) for _ in range(max(2, ns))]
        size = (H.lora_linear_tri_workspace_size if ns == 3 else H.lora_linear_workspace_size)(m, r)
        t["ws"] = _empty(size, dtype=torch.uint8) if size else None
    elif op == "lm_head":
        s, l = case["s"], case["l"]
        t["out"] = [_empty(s * l) for _ in range(5)]
        t["ws"] = _empty(H.lm_head_logprobs_workspace_size(s, l, case["v"], case["r"]),
                         dtype=torch.uint8)
    elif op == "attention":
        t["out"] = _empty(case["s"] * case["p"], 128 * case["heads"], dtype=torch.bfloat16)
    elif op == "update":
        s, l = case["s"], case["l"]
        t["out"] = [_empty(s, l) for _ in range(4)]
        t["stats"] = _empty(7, dtype=torch.float64)
        t["ws"] = _empty(H.ppo_workspace_size(), dtype=torch.uint8)
    elif op == "score":
        t["cfg"] = _config(case, case["l"])
        size = (H.score_llama_hydra_workspace_size if case["critic"]
                else H.score_llama_workspace_size)(t["cfg"], case["s"])
        t["ws"] = _empty(size, dtype=torch.uint8)
        t["flat"], t["out"] = _flat(_parts(op), case["s"], case["l"])
    else:
        s, n = case["s"], case["steps"]
        t["cfg"] = _config(case, n)
        t["ws"] = _empty(H.generate_llama_workspace_size(t["cfg"], s), dtype=torch.uint8)
        t["flat"], t["out"] = _flat(_parts(op), s, n)
        t["out"]["tokens"] = t["flat"]["tokens"] = _empty(s, n, dtype=torch.int32)
    return t


# --------------------------------------------------------------------------- one pass


def run(t):
    case, op = t["case"], t["op"]
    if op == "linear":
        x, A, B, y = t["x"], t["A"] or [None] * 2, t["B"] or [None] * 2, t["y"]
        if case["streams"] == 3:
            H.hydra_lora_linear_tri(x[0], x[1], x[2], t["W"], A[0], B[0], A[1], B[1], SCALE, y[0],
                                    y[1], y[2], t["ws"])
        else:
            H.hydra_lora_linear(x[0], x[1] if len(x) > 1 else None, t["W"], A[0], B[0], SCALE,
                                y[0], y[1], t["ws"])
        return y
    if op == "lm_head":
        h, o = t["h"], t["out"]
        H.hydra_lm_head_logprobs(h[0], h[1] if len(h) > 1 else None, t["W"], t["A"], t["B"], SCALE,
                                 t["ids"], t["lengths"], t["score"], BETA, case["s"], case["l"],
                                 o[0], o[1], o[2], t["ws"], o[3], o[4])
        return o
    if op == "attention":
        H.hydra_causal_attention(t["qkv"], case["s"], case["p"], case["heads"], 128, t["out"])
        return t["out"]
    if op == "update":
        adv, ret, g_logp, g_val = t["out"]
        H.ppo_gae(t["reward"], t["values"], t["lengths"], GAMMA, LAM, adv, ret)
        H.hydra_ppo_loss(t["new"], t["old"], adv, ret, t["values"], t["lengths"], CLIP,
                         case["whiten"], g_logp, g_val, t["stats"], t["ws"])
        return {"adv": adv, "ret": ret, "g_logp": g_logp, "g_val": g_val, "stats": t["stats"]}
    if op == "score":
        if case["critic"]:
            H.hydra_score_llama_hydra(t["cfg"], t["w"], t["critic"], t["ids"], t["lengths"], t["ws"],
                                      t["out"])
        else:
            H.hydra_score_llama(t["cfg"], t["w"], t["ids"], t["lengths"], t["ws"], t["out"])
    else:
        H.hydra_generate_llama(t["cfg"], t["w"], t["ids"], case["steps"], t["noise"], t["ws"],
                               t["out"])
    return t["flat"]


# --------------------------------------------------------------------------- work


def _lora_weights(streams):
    """Elements of one decoder layer's LoRA sets of the streams that carry one."""
    return RANK * ((D + D) + (D + D) + 2 * (D + FFN) + (FFN + D)) * (streams - 1)


def work(case):
    op = case["op"]
    if op == "linear":
        m, k, n, r, ns = (case[x] for x in ("m", "k", "n", "r", "streams"))
        outs, lora = max(2, ns), max(1, ns - 1) if r else 0
        out_bytes = outs * m * n * (4 if case["f32"] else 2)
        return {"bytes": 2 * (ns * m * k + n * k + lora * r * (k + n)) + out_bytes,
                "flops": 2 * m * (ns * k * n + lora * r * (k + n))}
    if op == "lm_head":
        m, d, v, r = case["s"] * case["l"], case["d"], case["v"], case["r"]
        ns = 1 if case["shared"] else 2
        return {"bytes": 2 * (ns * m * d + v * d + r * (d + v)) + 24 * m + 8 * case["s"],
                "flops": 2 * m * (ns * d * v + r * (d + v))}
    if op == "attention":
        s, p, d = case["s"], case["p"], 128 * case["heads"]
        return {"bytes": 2 * s * p * 4 * d, "flops": 4 * s * d * p * (p + 1) // 2}
    if op == "update":
        n = case["s"] * case["l"]  # about 9/16 of the slots hold a token
        valid = n * 9 // 16
        return {"bytes": 16 * valid + 16 * n + 4 * case["s"], "flops": 40 * valid}
    qkv, rest = 3 * D * D, D * D + 3 * D * FFN  # weights of a layer: q/k/v, and o, gate, up, down
    if op == "score":
        ns = 3 if case["critic"] else 2
        s, l = case["s"], case["l"]
        p = case["p0"] + l
        lora = _lora_weights(ns)
        # the first layer's streams share their q/k/v inputs; past its attention, the last layer
        # is needed at the l + 1 positions that the heads read
        dense = s * p * qkv * (ns * (LAYERS - 1) + 1) + ns * s * rest * (p * (LAYERS - 1) + l + 1)
        attn = ns * s * D * p * (p + 1) * LAYERS
        return {"bytes": 2 * ((qkv + rest + lora) * LAYERS + VOCAB * D + s * p * D) + 4 * s * (p + 6 * l),
                "flops": 2 * (dense + s * p * lora * LAYERS + attn + 2 * s * l * D * VOCAB)}
    s, p, n = case["s"], case["p0"], case["steps"]
    once = 2 * (qkv + rest + _lora_weights(2)) * LAYERS
    cache = 2 * 2 * s * D * 2 * LAYERS  # both streams' keys and values of one position
    rows = 2 * s * (p + n) * (qkv + rest) * LAYERS + 2 * s * n * D * VOCAB
    return {"bytes": once * (1 + n) + 2 * VOCAB * D * n + 4 * s * n * VOCAB
            + cache * (p + n + sum(p + i for i in range(n))),
            "flops": 2 * rows}


# --------------------------------------------------------------------------- tolerance


def tolerance(case):
    """About four times what the same operation with its sums in another order shows (the tile
    GEMM with its k-blocks taken last to first: bf16 linear 1.2e-4 to 2.1e-4 and one unit in the
    last place, 7.8e-3, at most; LM head 3.5e-6, 2.2e-5; whole passes 1.1e-2 to 1.3e-2, 0.06)."""
    op = case["op"]
    if op == "linear":
        # bf16 outputs: one unit in the last place (2^-8 relative) at the few sums that round the
        # other way, among them through u, which is stored in bf16; fp32 outputs: u alone
        if case["f32"]:
            return {"rel": 1e-4, "max": 2e-3} if case["r"] else {"rel": 5e-5, "max": 5e-4}
        return {"rel": 1e-3, "max": 3e-2}
    if op == "lm_head":
        return {"rel": 2e-4, "max": 4e-3} if case["r"] else {"rel": 2e-5, "max": 4e-4}
    if op == "attention":
        return {"rel": 4e-3, "max": 3e-2}  # probabilities and outputs rounded to bf16
    if op == "update":
        return {"rel": 1e-5, "max": 1e-3}
    # whole passes: one-unit differences of the bf16 activations travel through the layers
    return {"rel": 3e-2, "max": 3e-1}


# --------------------------------------------------------------------------- 64 bits


def _rms(h, w):
    return h * torch.rsqrt(h.square().mean(-1, keepdim=True) + EPS) * w.double()


def _attend(q, k, v):
    """Causal attention of [P, heads, 128]."""
    q, k, v = (x.transpose(0, 1) for x in (q, k, v))
    z = q @ k.transpose(1, 2) / math.sqrt(128)
    p = z.shape[1]
    z.masked_fill_(torch.ones(p, p, dtype=torch.bool, device=DEV).triu(1), -math.inf)
    return (torch.softmax(z, -1) @ v).transpose(0, 1)


def _lora(x, w, a, b):
    y = x @ w.double().T
    return y if a is None else y + SCALE * (x @ a.double().T) @ b.double().T


def _forward(w, lora, ids):
    """Final normed hidden states [S, P, D] of one stream (lora None: LoRA off)."""
    s, p = ids.shape
    i = torch.arange(64, device=DEV, dtype=torch.float64)
    angle = torch.arange(p, device=DEV).double()[:, None] * THETA ** (-i / 64)
    cos, sin = torch.cos(angle)[None, :, None], torch.sin(angle)[None, :, None]

    def rotate(x):
        x1, x2 = x[..., :64], x[..., 64:]
        return torch.cat([x1 * cos - x2 * sin, x1 * sin + x2 * cos], -1)

    h = w["embed"].double()[ids.long()]
    for j in range(LAYERS):
        ab = [(None, None)] * 3 if lora is None else [(lora["a_" + q][j], lora["b_" + o][j]) for q, o in
                                                      (("qv", "qkv"), ("gu", "gu"), ("down", "down"))]
        qkv = _lora(_rms(h, w["norm_attn"][j]), w["w_qkv"][j], *ab[0]).view(s, p, 3, HEADS, 128)
        q, k = rotate(qkv[:, :, 0]), rotate(qkv[:, :, 1])
        o = torch.stack([_attend(q[n], k[n], qkv[n, :, 2]) for n in range(s)])
        h = h + o.reshape(s, p, D) @ w["w_o"][j].double().T
        gate, up = llama.deinterleave_gate_up(
            _lora(_rms(h, w["norm_ffn"][j]), w["w_gu"][j], *ab[1]).reshape(s * p, -1).T)
        m = (torch.nn.functional.silu(gate) * up).T.reshape(s, p, FFN)
        h = h + _lora(m, w["w_down"][j], *ab[2])
    return _rms(h, w["final_norm"])


def _logp(h, w, ids):
    """Log-probabilities of ids under the head, and the log-sum-exps, a block of rows at a time."""
    wt, lse, z = w.double().T, [], []
    for a, b in zip(h.split(512), ids.split(512)):
        y = a @ wt
        lse.append(torch.logsumexp(y, -1))
        z.append(y.gather(1, b.long()[:, None])[:, 0])
    lse = torch.cat(lse)
    return torch.cat(z) - lse, lse


def _valid(lengths, l):
    return torch.arange(l, device=DEV)[None] < lengths[:, None]


def _gae(reward, values, lengths):
    s, l = reward.shape
    ok = _valid(lengths, l)
    v = torch.where(ok, values, 0.0)
    nxt = torch.cat([v[:, 1:], torch.zeros_like(v[:, :1])], 1)
    delta = torch.where(ok, reward + GAMMA * nxt - v, 0.0)
    adv, a = torch.zeros_like(delta), torch.zeros_like(delta[:, 0])
    for t in range(l - 1, -1, -1):
        a = delta[:, t] + GAMMA * LAM * a
        adv[:, t] = a
    return adv, torch.where(ok, adv + v, 0.0)


def exact(case, seed):
    t = _inputs(case, seed)
    op = case["op"]
    if op == "linear":
        x, w = [v.double() for v in t["x"]], t["W"].double()
        y = [v @ w.T for v in x]
        y = [y[0], y[0].clone()] if len(y) == 1 else y
        x = x * 2 if len(x) == 1 else x
        for i, (a, b) in enumerate(zip(t["A"], t["B"])):
            y[i + 1] += SCALE * (x[i + 1] @ a.double().T) @ b.double().T
        return y
    if op == "lm_head":
        s, l, w = case["s"], case["l"], t["W"].double()
        h = [v.double() for v in t["h"]]
        h = h * 2 if len(h) == 1 else h
        lr, lse_r = _logp(h[0], w, t["ids"])
        if case["r"]:
            w = w + SCALE * t["B"].double() @ t["A"].double()
        la, lse_a = _logp(h[1], w, t["ids"])
        ok = _valid(t["lengths"], l)
        last = torch.arange(l, device=DEV)[None] == (t["lengths"] - 1)[:, None]
        reward = -BETA * (la - lr).view(s, l) + last * t["score"].double()[:, None]
        return [torch.where(ok, v.view(s, l), 0.0).view(-1) for v in (la, lr, reward, lse_a, lse_r)]
    if op == "attention":
        s, p, hd = case["s"], case["p"], case["heads"]
        q, k, v = t["qkv"].double().view(s, p, 3, hd, 128).unbind(2)
        return torch.cat([_attend(q[i], k[i], v[i]).reshape(p, 128 * hd) for i in range(s)])
    if op == "update":
        new, old, r, v = (t[k].double() for k in ("new", "old", "reward", "values"))
        adv, ret = _gae(r, v, t["lengths"])
        ok = _valid(t["lengths"], case["l"])
        n = ok.sum().double()
        mean = adv.sum() / n
        std = (torch.where(ok, adv - mean, 0.0).square().sum() / n).sqrt()
        a = (adv - mean) / (std.square() + 1e-8).sqrt() if case["whiten"] else adv
        ratio = torch.exp(new - old)
        free, held = ratio * a, ratio.clamp(1 - CLIP, 1 + CLIP) * a
        g_logp = torch.where(ok & (free <= held), -free / n, 0.0)
        g_val = torch.where(ok, 2 * (v - ret) / n, 0.0)

        def over(x):
            return torch.where(ok, x, 0.0).sum() / n

        stats = torch.stack([-over(torch.minimum(free, held)), over((v - ret).square()),
                             over(((ratio - 1).abs() > CLIP).double()), over(old - new), mean, std, n])
        return {"adv": adv, "ret": ret, "g_logp": g_logp, "g_val": g_val, "stats": stats}
    # The whole passes. Their distance from 64 bits is that of the activations' bf16 rounding;
    # over a few dozen tokens it is a matter of chance, and no value is given for those.
    w = t["w"]
    if op == "score":
        ids, p0, l, lengths = t["ids"], case["p0"], case["l"], t["lengths"]
    else:
        ids, p0, l = torch.cat([t["ids"], t["tokens"]], 1), case["p0"], case["steps"]
        lengths = torch.full((case["s"],), l, device=DEV)
    s = ids.shape[0]
    if s * l * (1 if op == "generate" else 0.5) < 100:
        return None
    ok = _valid(lengths, l)
    told = ids[:, p0:].reshape(-1)

    def kept(x):
        return torch.where(ok, x.reshape(s, l), 0.0)

    def rows(h):
        return h[:, p0 - 1:-1].reshape(s * l, D)

    rm = w["w_rm"].double()
    h_off, h_on = _forward(w, None, ids), _forward(w, {k: w[k] for k in llama.LORA_KEYS}, ids)
    h_val = _forward(w, t["critic"], ids) if t.get("critic") else h_on
    out = {"logp_actor": kept(_logp(rows(h_on), w["lm_head"], told)[0]),
           "logp_ref": kept(_logp(rows(h_off), w["lm_head"], told)[0]),
           "values": kept(rows(h_val) @ rm)}
    out["score"] = h_off[torch.arange(s, device=DEV), p0 - 1 + lengths.long()] @ rm
    last = torch.arange(l, device=DEV)[None] == (lengths - 1)[:, None]
    out["reward"] = kept(-BETA * (out["logp_actor"] - out["logp_ref"]) + last * out["score"][:, None])
    out["advantages"], out["returns"] = _gae(out["reward"], out["values"], lengths)
    flat, view = _flat(_parts(op), s, l, torch.float64)
    for n, v in view.items():
        v.copy_(out[n])
    return flat if op == "score" else dict(flat, tokens=None)
