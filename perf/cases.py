"""The work that users of this library have it do, as measurable cases.

A case names a call (``call``), a decoder shape and sizes.  Every call goes
through the public entry points: ``Model`` and the functions of ``knapspec``.
The shapes are the configured ones (Llama-3-8B, Qwen3-8B, Qwen3-32B, the tiny
fp32 decoder) and the small ragged ones of the tests, cut to as many layers as
the call needs; the vocabulary of a layer-level case is the tests' 2000.

Weights stand for a trained decoder where it matters: input projections
N(0, 0.02^2), output projections scaled by 1 / sqrt(2 L) and a spread over
the layers (some sublayers contribute more than others, as the layer
selection expects), unit-variance embeddings, norm gains around 1, and an LM head that
prefers one successor per token with a probability around 0.9 rather than
the near-tied logits of plain random weights.

Logits of bf16 models are returned in the model's dtype, the precision its
activations carry; fp32 models return fp32.  The KV cache, which a prefill is
run for, is the head of the caller's workspace: [L][K, V][KV head][max_seq]
[head_dim] in the model's dtype.
"""
from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

from paper_2602_20217_gb300 import configs
from paper_2602_20217_gb300 import knapspec as ks
from paper_2602_20217_gb300.model import Model

SMALL64 = configs.ModelShape("small-hd64", 2, 512, 8, 2, 64, 1368, 2000, dtype="bf16", rope_theta=500000.0)
SMALL128 = configs.ModelShape("small-hd128", 2, 512, 8, 2, 128, 1368, 2000, qk_norm=True, dtype="bf16",
                              rope_theta=500000.0)
WIDE = configs.ModelShape("wide", 2, 1536, 12, 4, 128, 3584, 2000, qk_norm=True, dtype="bf16", rope_theta=500000.0)
SHAPES = {"llama8b": configs.LLAMA3_8B, "qwen8b": configs.QWEN3_8B, "qwen32b": configs.QWEN3_32B,
          "tiny": configs.TINY, "small64": SMALL64, "small128": SMALL128, "wide": WIDE}
MAX_ROWS = 16
LAST_ROWS = 16          # rows of the prefill's last chunk, whose logits are kept


# ------------------------------------------------------------------ cases
def listed():
    return [
        # One knapsack solve with App. C latencies at a 64k context: the call a
        # serving loop makes every resolve interval, all latency.
        {"name": "select_32b", "call": "select", "n_sublayers": 128, "kind": 0, "ratio": 0.58, "budget": 153},
        # Sublayer similarities over a full history (5 steps, 25 rows) of the 8B decoder.
        {"name": "cosine_8b", "call": "cosine", "pairs": 64, "rows": 25, "d": 4096, "plane": 96, "dtype": "f32",
         "indexed": True},
        # The fp32 decoder: one speculation step of the tiny workload, launches and latency.
        {"name": "tiny_step", "call": "verify", "shape": "tiny", "layers": 4, "vocab": 1024, "context": 256,
         "gamma": 4, "right": 3, "draft": "attn_skip"},
        # One Attn sublayer of the 32B shape at a 64k context, four draft tokens.
        {"name": "attn_32b_64k", "call": "draft", "shape": "qwen32b", "layers": 1, "vocab": 2000, "context": 65536,
         "gamma": 4, "mask": "attn_only"},
        # Verify pass of the paper's longest drafts (D = 10: 11 rows) at 32k.
        {"name": "verify11_8b_32k", "call": "verify", "shape": "qwen8b", "layers": 2, "vocab": 2000,
         "context": 32768, "gamma": 10, "right": 7, "draft": ""},
        # Sampling mode (T 0.7, top-k 50, top-p 0.95) with MLP-only drafts, full vocabulary.
        {"name": "sample_8b_4k", "call": "sample", "shape": "llama8b", "layers": 2, "vocab": 128256, "context": 4096,
         "gamma": 4, "mask": "attn_skip"},
        # The TPT stage: eight candidates scored on the history, full vocabulary.
        {"name": "tpt_8b", "call": "tpt", "shape": "llama8b", "layers": 4, "vocab": 128256, "context": 1024,
         "steps": 4, "candidates": 8, "max_gamma": 10},
        # The hidden-state DP of Alg. 1 over 16 sublayers of the 8B decoder.
        {"name": "dp_8b", "call": "dp", "shape": "llama8b", "layers": 8, "vocab": 32000, "context": 1024,
         "attn_units": 1, "mlp_units": 2, "steps": 3, "max_gamma": 10, "max_rows": 32},
        # Prompt processing, two layers: the workload's 4096 tokens, and a long ragged prompt.
        {"name": "prefill_8b_4k", "call": "prefill", "shape": "llama8b", "layers": 2, "vocab": 2000, "context": 4096},
        {"name": "prefill_32b_9k", "call": "prefill", "shape": "qwen32b", "layers": 2, "vocab": 2000,
         "context": 9001},
        # Whole calls: greedy decoding of the full 8B decoder at 4k ...
        {"name": "decode_8b_4k", "call": "decode", "shape": "llama8b", "layers": 32, "vocab": 128256,
         "context": 4096, "tokens": 9},
        # ... and the speculative loop with the knapsack re-solved every step (8 layers of the 32B shape).
        {"name": "spec_32b_8k", "call": "generate", "shape": "qwen32b", "layers": 8, "vocab": 151936,
         "context": 8192, "gamma": 4, "tokens": 16, "ratio": 0.7, "budget_frac": 0.8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _big(rng):
    return rng.choice(["llama8b", "qwen8b", "qwen32b"])


def _any_bf16(rng):
    return rng.choice(["llama8b", "qwen8b", "qwen32b", "small64", "small128", "wide"])


def draw(rng):
    call = rng.choice(["select", "cosine", "tiny", "draft", "verify", "sample", "tpt", "dp", "prefill", "prefill",
                       "decode", "generate"])
    if call == "select":
        n = 2 * _log_int(rng, 1, 128)
        if rng.random() < 0.5:
            return {"call": "select", "n_sublayers": n, "kind": 0, "ratio": round(rng.uniform(0.2, 5.0), 3),
                    "budget": rng.randint(0, 3 * n)}
        return {"call": "select", "n_sublayers": n, "kind": 1, "most_units": _log_int(rng, 4, 1024),
                "budget": _log_int(rng, 8, 16384)}
    if call == "cosine":
        rows = rng.randint(1, 80)
        return {"call": "cosine", "pairs": _log_int(rng, 2, 144), "rows": rows, "d": rng.randint(100, 5120),
                "plane": rows + rng.randint(0, 16), "dtype": rng.choice(["f32", "bf16"]),
                "indexed": rng.random() < 0.5}
    if call == "tiny":
        gamma = rng.randint(1, 15)
        return {"call": "verify", "shape": "tiny", "layers": rng.randint(1, 4), "vocab": 1024,
                "context": _log_int(rng, 2, 1500), "gamma": gamma, "right": rng.randint(0, gamma),
                "draft": rng.choice(["attn_skip", "full"])}
    if call == "prefill":
        shape = _any_bf16(rng)
        return {"call": "prefill", "shape": shape, "layers": rng.randint(1, 2), "vocab": 2000,
                "context": _log_int(rng, 9, 5000 if shape in ("llama8b", "qwen8b", "qwen32b") else 12000)}
    if call == "draft":
        return {"call": "draft", "shape": _any_bf16(rng), "layers": 1, "vocab": 2000,
                "context": _log_int(rng, 5, 24000), "gamma": rng.randint(1, 8),
                "mask": rng.choice(["attn_only", "attn_skip", "full"])}
    if call == "verify":
        gamma = rng.randint(1, 15)
        return {"call": "verify", "shape": _any_bf16(rng), "layers": rng.randint(1, 2), "vocab": 2000,
                "context": _log_int(rng, 5, 12000), "gamma": gamma, "right": rng.randint(0, gamma), "draft": ""}
    if call == "sample":
        return {"call": "sample", "shape": _big(rng), "layers": 1, "vocab": _log_int(rng, 2000, 151936),
                "context": _log_int(rng, 16, 4000), "gamma": rng.randint(1, 8),
                "mask": rng.choice(["attn_skip", "full"])}
    if call == "tpt":
        return {"call": "tpt", "shape": _any_bf16(rng), "layers": rng.randint(2, 4),
                "vocab": _log_int(rng, 2000, 151936), "context": _log_int(rng, 16, 1500),
                "steps": rng.randint(0, 4), "candidates": rng.randint(1, 16), "max_gamma": rng.randint(1, 15)}
    if call == "dp":
        return {"call": "dp", "shape": rng.choice(["llama8b", "small64", "small128", "wide"]),
                "layers": rng.randint(2, 5), "vocab": _log_int(rng, 2000, 32000), "context": _log_int(rng, 64, 1500),
                "attn_units": rng.randint(1, 3), "mlp_units": rng.randint(1, 3), "steps": rng.randint(0, 4),
                "max_gamma": rng.randint(1, 15), "max_rows": rng.randint(4, 40)}
    if call == "decode":
        return {"call": "decode", "shape": _big(rng), "layers": rng.randint(1, 4),
                "vocab": _log_int(rng, 2000, 151936), "context": _log_int(rng, 5, 6000),
                "tokens": rng.randint(2, 24)}
    return {"call": "generate", "shape": _big(rng), "layers": rng.randint(2, 4),
            "vocab": _log_int(rng, 2000, 151936), "context": _log_int(rng, 16, 4000), "gamma": rng.randint(1, 8),
            "tokens": rng.randint(4, 24), "ratio": round(rng.uniform(0.3, 2.0), 2),
            "budget_frac": round(rng.uniform(0.5, 1.0), 2)}


# ----------------------------------------------------------------- inputs
def _shape(case):
    return replace(SHAPES[case["shape"]], n_layers=case["layers"], vocab=case["vocab"])


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _weights(sh, seed):
    """Device tensors in the layout of the library, and the successor table."""
    g = _generator(seed)
    dt = torch.bfloat16 if sh.dtype == "bf16" else torch.float32

    def normal(rows, cols, std):
        return torch.empty(rows, cols, dtype=dt, device="cuda").normal_(0.0, std, generator=g)

    def gain(n):
        return (1.0 + 0.1 * torch.randn(n, generator=g, device="cuda")).to(dt)

    L, d, hd = sh.n_layers, sh.d_model, sh.head_dim
    # contribution of each sublayer: a spread of a factor 8, in a seeded order
    spread = torch.exp(torch.linspace(-1.04, 1.04, 2 * L, dtype=torch.float64))
    spread = spread[torch.randperm(2 * L, generator=torch.Generator().manual_seed(int(seed)))].tolist()
    out = 1.0 / math.sqrt(2 * L)
    layers = []
    for l in range(L):
        w = {"attn_norm": gain(d), "w_qkv": normal(sh.qkv_rows, d, 0.02),
             "w_o": normal(d, sh.n_q_heads * hd, out * spread[2 * l] / math.sqrt(sh.n_q_heads * hd)),
             "mlp_norm": gain(d), "w_gate_up": normal(2 * sh.d_ff, d, 0.02),
             "w_down": normal(d, sh.d_ff, out * spread[2 * l + 1] / math.sqrt(sh.d_ff))}
        if sh.qk_norm:
            w["q_norm"], w["k_norm"] = gain(hd), gain(hd)
        layers.append(w)
    embed = normal(sh.vocab, d, 1.0)
    succ = torch.randperm(sh.vocab, generator=g, device="cuda")      # token t is followed by succ[t]
    head = normal(sh.vocab, d, 0.0195)
    head[succ] += (embed * (24.0 / d)).to(dt)
    return {"layers": layers, "embed": embed, "lm_head": head, "final_norm": gain(d)}, succ


def _prompt(sh, n, seed):
    g = torch.Generator().manual_seed(int(seed) + 7)
    return torch.randint(0, sh.vocab, (n,), generator=g, dtype=torch.int32).numpy()


def _mask(kind, L):
    return np.array({"attn_only": [1, 0], "attn_skip": [0, 1], "full": [1, 1]}[kind] * L, np.uint8)


def _latency(case, L, context):
    """App. C model with t_Attn(context) = ratio * t_MLP, half of it growing with the context."""
    r = case["ratio"]
    return ks.latency(0, 1.0, 0.5 * r / max(1, context), 0.5 * r)


def _chain(succ, start, count):
    """`count` successors of `start`, as the decoder predicts them."""
    out, t = [], int(start)
    for _ in range(count):
        t = int(succ[t])
        out.append(t)
    return out


class _State:
    pass


def _room(case):
    """Positions past the prompt that the call may use."""
    return {"decode": case.get("tokens", 0), "generate": case.get("tokens", 0) + 2 * case.get("gamma", 0) + 4,
            "tpt": 5 * case.get("steps", 0) + 8, "dp": 5 * case.get("steps", 0) + 8}.get(
                case["call"], case.get("gamma", 0)) + 8


def prepare(case, seed):
    s = _State()
    s.case, s.call = case, case["call"]
    if s.call == "select":
        return _prepare_select(s, seed)
    if s.call == "cosine":
        return _prepare_cosine(s, seed)
    s.sh = _shape(case)
    weights, succ = _weights(s.sh, seed)
    s.prompt = _prompt(s.sh, case["context"], seed)
    s.model = Model(s.sh, max_seq=case["context"] + _room(case), weights=weights, max_rows=MAX_ROWS)
    L = s.sh.n_layers
    if s.call == "prefill":
        n = 2 * L * s.sh.n_kv_heads * s.model.cfg.max_seq * s.sh.head_dim
        s.kv = s.model.workspace[: n * s.sh.elem_bytes].view(
            torch.bfloat16 if s.sh.dtype == "bf16" else torch.float32).view(
                L, 2, s.sh.n_kv_heads, s.model.cfg.max_seq, s.sh.head_dim)
        return s
    pending = s.model.prefill(s.prompt)
    if s.call in ("draft", "sample"):
        s.mask = _mask(case["mask"], L)
    if s.call == "sample":
        s.sampling = ks.sampling(0.7, 50, 0.95, seed=int(seed) & 0xFFFF)
    if s.call == "verify":
        s.mask = _mask(case["draft"], L) if case["draft"] else None
        # drafts that agree with the target up to `right`, then leave it
        succ = succ.tolist()
        s.drafts = _chain(succ, pending, case["gamma"])
        for i in range(case["right"], case["gamma"]):
            s.drafts[i] = (s.drafts[i] + 1 + i) % s.sh.vocab
        s.drafts = np.array(s.drafts, np.int32)
    if s.call == "generate":
        s.latency = _latency(case, L, case["context"])
    if s.call == "tpt":
        s.latency = ks.latency(0, 1.0, 0.0, 1.2)
    if s.call == "dp":
        s.latency = ks.latency(1, units=[case["attn_units"], case["mlp_units"]] * L)
        s.states = (case["attn_units"] + case["mlp_units"]) * L // 2 + 1
    for _ in range(case.get("steps", 0)):       # a history of several verify steps
        s.model.draft(_mask("full", L), 4)
        s.model.verify(None, 4)
    return s


def _prepare_select(s, seed):
    c = s.case
    n = c["n_sublayers"]
    g = _generator(seed)
    s.sims = 1.0 - 0.2 * torch.rand(n, generator=g, device="cuda") ** 2
    if c["kind"] == 0:
        s.latency = _latency(c, n // 2, 65536)
    else:
        units = 1 + torch.randint(0, c["most_units"], (n,), generator=torch.Generator().manual_seed(int(seed)))
        s.latency = ks.latency(1, units=units.numpy())
    s.mask = torch.empty(n, dtype=torch.uint8, device="cuda")
    s.objective = torch.empty(1, dtype=torch.float64, device="cuda")
    s.weights = torch.empty(n, dtype=torch.int32, device="cuda")
    s.scratch_bytes = ks.ks_select_scratch_bytes(n, c["budget"])
    s.scratch = torch.empty(s.scratch_bytes, dtype=torch.uint8, device="cuda")
    s.stream = torch.cuda.current_stream()
    return s


def _cosine_inputs(c, seed):
    g = _generator(seed)
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    # a residual stream: every plane adds a sublayer's contribution to the one before
    x = torch.randn(c["pairs"] + 1, c["plane"], c["d"], generator=g, device="cuda")
    x[1:] *= 0.3
    x = x.cumsum(0).to(dt)
    index = torch.randperm(c["plane"], generator=g, device="cuda")[: c["rows"]].to(torch.int32)
    return x, index if c["indexed"] else None


def _prepare_cosine(s, seed):
    s.x, s.index = _cosine_inputs(s.case, seed)
    s.out = torch.empty(s.case["pairs"], dtype=torch.float32, device="cuda")
    s.stream = torch.cuda.current_stream()
    return s


# -------------------------------------------------------------------- run
def _logits(s, rows):
    lg = torch.from_numpy(s.model.logits(rows))
    return lg.to(torch.bfloat16) if s.sh.dtype == "bf16" else lg


def run(s):
    c = s.case
    if s.call == "select":
        lat, _units = s.latency
        ks.ks_select_mask(lat, s.sims, 65536, c["n_sublayers"], c["budget"], s.mask, s.objective, s.weights,
                          s.scratch, s.scratch_bytes, s.stream)
        return {"mask": s.mask, "objective": s.objective, "weights": s.weights}
    if s.call == "cosine":
        ks.ks_cosine(s.x, s.x[1:], ks.KS_DTYPE_F32 if c["dtype"] == "f32" else ks.KS_DTYPE_BF16, c["pairs"],
                     c["rows"], c["d"], c["plane"] * c["d"], s.index, s.out, s.stream)
        return {"cosines": s.out}
    m = s.model
    if s.call == "prefill":
        token = m.prefill(s.prompt)
        return {"next": token, "logits": _logits(s, min(c["context"], LAST_ROWS)), "kv": s.kv}
    if s.call == "draft":
        tokens = m.draft(s.mask, c["gamma"])
        return {"tokens": tokens, "logits": _logits(s, 1)}
    if s.call == "verify":
        m.rewind()
        drafted = m.draft(s.mask, c["gamma"]) if s.mask is not None else None
        accepted, tokens = m.verify(s.drafts, c["gamma"])
        return {"drafted": drafted, "accepted": accepted, "tokens": tokens, "logits": _logits(s, c["gamma"] + 1)}
    if s.call == "sample":
        m.rewind()
        drafts = m.draft_sample(s.mask, c["gamma"], s.sampling, 0)
        accepted, tokens = m.verify_sample(c["gamma"], s.sampling, 0)
        return {"drafts": drafts, "accepted": accepted, "tokens": tokens, "logits": _logits(s, c["gamma"] + 1)}
    if s.call == "decode":
        m.rewind()
        tokens = m.decode_greedy(c["tokens"])
        return {"tokens": tokens, "logits": _logits(s, 1)}
    if s.call == "generate":
        m.rewind()
        tokens, _stats, accepted = m.generate(c["tokens"], c["gamma"], latency=s.latency,
                                              budget_frac=c["budget_frac"], resolve_every=1)
        steps = np.zeros(c["tokens"], np.int32)     # one entry a step, as many as there were
        steps[: len(accepted)] = accepted
        return {"tokens": tokens, "accepted": steps, "logits": _logits(s, c["gamma"] + 1)}
    if s.call == "tpt":
        mask, gamma, tpt, alphas, candidates = m.select_tpt(s.latency, c["candidates"], c["max_gamma"])
        return {"mask": mask, "gamma": gamma, "tpt": tpt, "alphas": alphas, "candidates": candidates}
    mask, gamma, tpt, js, alphas, candidates = m.select_dp(s.latency, c["max_gamma"], 0.5, s.states, c["max_rows"])
    return {"mask": mask, "gamma": gamma, "tpt": tpt, "js": js, "alphas": alphas, "candidates": candidates}


# ------------------------------------------------------------------- work
def _layer_flops(sh, rows, keys):
    """Attn and MLP sublayer of `rows` rows that see `keys` keys each on average."""
    attn = 2.0 * rows * (sh.qkv_rows * sh.d_model + sh.d_model * sh.n_q_heads * sh.head_dim)
    attn += 4.0 * rows * keys * sh.n_q_heads * sh.head_dim
    return attn, 2.0 * rows * 3 * sh.d_ff * sh.d_model


def _pass_work(sh, rows, context, mask, head=True):
    attn, mlp = _layer_flops(sh, rows, context)
    na, nm = int(mask[0::2].sum()), int(mask[1::2].sum())
    b = na * (sh.attn_weight_bytes() + sh.kv_bytes_per_layer(context)) + nm * sh.mlp_weight_bytes()
    f = na * attn + nm * mlp
    if head:
        b += sh.lm_head_bytes() + 4 * rows * sh.vocab
        f += 2.0 * rows * sh.vocab * sh.d_model
    return b, f


def work(case):
    call = case["call"]
    if call == "select":
        n = case["n_sublayers"]
        return {"bytes": 4 * n + n + 4 * n + 8, "flops": 2 * n * (case["budget"] + 1)}
    if call == "cosine":
        e = 4 if case["dtype"] == "f32" else 2
        n = (case["pairs"] + 1) * case["rows"] * case["d"]
        return {"bytes": e * n + 4 * case["pairs"], "flops": 6 * n}
    sh = _shape(case)
    L, ctx = sh.n_layers, case["context"]
    full = _mask("full", L)
    if call == "prefill":
        attn, mlp = _layer_flops(sh, ctx, ctx / 2)
        weights = L * (sh.attn_weight_bytes() + sh.mlp_weight_bytes()) + sh.lm_head_bytes()
        return {"bytes": weights + L * sh.kv_bytes_per_layer(ctx) + sh.elem_bytes * ctx * sh.d_model,
                "flops": L * (attn + mlp) + 2.0 * LAST_ROWS * sh.vocab * sh.d_model}
    passes = []
    if call == "draft":
        passes = [(1, _mask(case["mask"], L))] * case["gamma"]
    elif call == "verify":
        passes = [(case["gamma"] + 1, full)]
        if case["draft"]:
            passes += [(1, _mask(case["draft"], L))] * case["gamma"]
    elif call == "sample":
        passes = [(1, _mask(case["mask"], L))] * case["gamma"] + [(case["gamma"] + 1, full)]
    elif call == "decode":
        passes = [(1, full)] * (case["tokens"] - 1)
    elif call == "generate":
        # the drafts are accepted: gamma + 1 tokens a step after the pending one
        steps = -(-(case["tokens"] - 1) // (case["gamma"] + 1))
        vb, vf = _pass_work(sh, case["gamma"] + 1, ctx, full)
        lb, lf = _pass_work(sh, 1, ctx, full, head=False)       # a draft's layers: the budget's share of them
        hb, hf = _pass_work(sh, 1, ctx, 0 * full)
        share = case["gamma"] * case["budget_frac"]
        return {"bytes": steps * (vb + share * lb + case["gamma"] * hb),
                "flops": steps * (vf + share * lf + case["gamma"] * hf)}
    elif call == "tpt":
        hist = min(8, ctx) + 5 * case["steps"]
        b = sh.lm_head_bytes() + 4 * (2 * L + 1) * hist * sh.d_model
        return {"bytes": b, "flops": 2.0 * (case["candidates"] + 1) * hist * sh.vocab * sh.d_model}
    elif call == "dp":
        states = (case["attn_units"] + case["mlp_units"]) * L // 2
        rows = min(case["max_rows"], min(8, ctx) + 5 * case["steps"])
        b, f = _pass_work(sh, states * rows, ctx, full)
        return {"bytes": b, "flops": f}
    b = f = 0.0
    for rows, mask in passes:
        pb, pf = _pass_work(sh, rows, ctx, mask)
        b, f = b + pb, f + pf
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ exact
class _Reference:
    """The decoder in 64-bit torch with a KV cache, one layer's weights widened at a time."""

    def __init__(self, sh, weights):
        self.sh, self.w = sh, weights
        self.k = [None] * sh.n_layers
        self.v = [None] * sh.n_layers

    @staticmethod
    def norm(x, gain, eps):
        return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * gain.double()

    def rope(self, x, pos):
        half = self.sh.head_dim // 2
        inv = self.sh.rope_theta ** (-2.0 * torch.arange(half, dtype=torch.float64, device="cuda") / self.sh.head_dim)
        ang = pos.double()[:, None, None] * inv
        c, s = torch.cos(ang), torch.sin(ang)
        a, b = x[..., :half], x[..., half:]
        return torch.cat([a * c - b * s, b * c + a * s], -1)

    def attention(self, q, l, p0):
        sh = self.sh
        n = p0 + q.shape[0]
        out = torch.empty_like(q)
        for h in range(sh.n_q_heads):
            k, v = self.k[l][:n, h // sh.group], self.v[l][:n, h // sh.group]
            for r in range(0, q.shape[0], 2048):
                e = min(q.shape[0], r + 2048)
                seen = p0 + e
                sc = q[r:e, h] @ k[:seen].T / math.sqrt(sh.head_dim)
                pos = torch.arange(p0 + r, p0 + e, device="cuda")
                sc.masked_fill_(torch.arange(seen, device="cuda")[None] > pos[:, None], -math.inf)
                out[r:e, h] = torch.softmax(sc, -1) @ v[:seen]
        return out

    def forward(self, tokens, p0, mask=None, cache_only=False):
        """Rows at p0.. : logits; cache_only: only the K/V of every layer (no head, no last layer's rest)."""
        sh, w = self.sh, self.w
        x = w["embed"][torch.as_tensor(np.asarray(tokens), device="cuda").long()].double()
        R = x.shape[0]
        pos = torch.arange(p0, p0 + R, device="cuda")
        for l, lw in enumerate(w["layers"]):
            if mask is None or mask[2 * l]:
                h, nq = self.norm(x, lw["attn_norm"], sh.rms_eps), sh.n_q_heads * sh.head_dim
                k, v = (h @ lw["w_qkv"][nq:].double().T).view(R, -1, sh.head_dim).split(sh.n_kv_heads, 1)
                if sh.qk_norm:
                    k = self.norm(k, lw["k_norm"], sh.rms_eps)
                k = self.rope(k, pos)
                old = p0 if self.k[l] is not None else 0
                self.k[l] = torch.cat([self.k[l][:old], k]) if old else k
                self.v[l] = torch.cat([self.v[l][:old], v]) if old else v
                if cache_only and l == sh.n_layers - 1:
                    return None
                q = (h @ lw["w_qkv"][:nq].double().T).view(R, -1, sh.head_dim)
                if sh.qk_norm:
                    q = self.norm(q, lw["q_norm"], sh.rms_eps)
                o = self.attention(self.rope(q, pos), l, p0).reshape(R, -1)
                x = x + o @ lw["w_o"].double().T
            if mask is None or mask[2 * l + 1]:
                y = self.norm(x, lw["mlp_norm"], sh.rms_eps) @ lw["w_gate_up"].double().T
                g, u = y.split(sh.d_ff, 1)
                x = x + (torch.nn.functional.silu(g) * u) @ lw["w_down"].double().T
        if cache_only:
            return None
        return self.norm(x, w["final_norm"], sh.rms_eps) @ w["lm_head"].double().T


def _exact_select(case, seed):
    s = _prepare_select(_with(case), seed)
    n, B = case["n_sublayers"], case["budget"]
    if n * (B + 1) > 1 << 22:
        return None
    if case["kind"] == 0:
        ta, tm = 0.5 * case["ratio"] / 65536 * 65536 + 0.5 * case["ratio"], 1.0
        dl = min(ta, tm)
        wts = [max(1, int(math.floor(t / dl + 0.5))) for t in (ta, tm)] * (n // 2)
    else:
        wts = s.latency[1].tolist()
    q = np.floor((1.0 - s.sims.double().cpu().numpy()) * 2.0 ** 30 + 0.5).astype(np.int64)
    best = np.zeros(B + 1, np.int64)
    for i in range(n):
        if wts[i] <= B:
            cand = best[: B + 1 - wts[i]] + q[i]
            best[wts[i]:] = np.maximum(best[wts[i]:], cand)
    return {"mask": None, "objective": torch.tensor([best[B] / 2.0 ** 30], dtype=torch.float64), "weights": None}


def _with(case):
    s = _State()
    s.case, s.call = case, case["call"]
    return s


def exact(case, seed):
    call = case["call"]
    if call == "select":
        return _exact_select(case, seed)
    if call == "cosine":
        x, index = _cosine_inputs(case, seed)
        rows = index.long() if index is not None else torch.arange(case["rows"], device="cuda")
        out = torch.empty(case["pairs"], dtype=torch.float64, device="cuda")
        for p in range(case["pairs"]):
            out[p] = torch.nn.functional.cosine_similarity(x[p, rows].double(), x[p + 1, rows].double(), -1,
                                                           1e-300).mean()
        return {"cosines": out}
    if call in ("tpt", "dp", "generate"):
        return None
    sh = _shape(case)
    n, L = case["context"], sh.n_layers
    cache_only = call != "prefill"
    rows_full = L - 1 if cache_only else L
    flops = rows_full * sum(_layer_flops(sh, n, n / 2))
    flops += 4.0 * n * sh.n_kv_heads * sh.head_dim * sh.d_model if cache_only else 0.0
    if flops > 5e12:
        return None
    weights, succ = _weights(sh, seed)
    ref = _Reference(sh, weights)
    prompt = _prompt(sh, n, seed)
    last = min(n, LAST_ROWS)
    if call == "prefill":
        if n > last:
            ref.forward(prompt[: n - last], 0, cache_only=True)
        logits = ref.forward(prompt[n - last:], n - last)
        kv = torch.zeros(L, 2, sh.n_kv_heads, n + _room(case), sh.head_dim, dtype=torch.float64, device="cuda")
        for l in range(L):
            kv[l, 0, :, :n] = ref.k[l].transpose(0, 1)
            kv[l, 1, :, :n] = ref.v[l].transpose(0, 1)
        return {"next": None, "logits": logits, "kv": kv}
    if n > 1:
        ref.forward(prompt[:-1], 0, cache_only=True)
    pending = int(ref.forward(prompt[-1:], n - 1)[0].argmax())
    if call in ("draft", "decode"):
        steps, mask = (case["gamma"], _mask(case["mask"], L)) if call == "draft" else (case["tokens"] - 1, None)
        t, logits = pending, None
        for i in range(steps):
            logits = ref.forward([t], n + i, mask)
            t = int(logits[0].argmax())
        return {"tokens": None, "logits": logits}
    rows = [pending] + _chain(succ.tolist(), pending, case["gamma"])
    if call == "verify":
        for i in range(case["right"], case["gamma"]):
            rows[1 + i] = (rows[1 + i] + 1 + i) % sh.vocab
        return {"drafted": None, "accepted": None, "tokens": None, "logits": ref.forward(rows, n)}
    return None       # sampling: the rows that are scored were drawn
