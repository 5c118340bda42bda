"""Performance cases: the work a program has this library do, through its public entry points.

Three kinds of case:

- "gemm": one projection, `wf_gemm_bf16` (Y = X W^T + b);
- "attn": one attention layer, `wf_attention` (the verify block's causal
  self-attention, the drafter's block attention with RoPE, the cross-attention
  over the encoder frames, a prompt's causal attention);
- "step" / "prefill": a handle's calls (`Session`): a speculative step of the
  decoder at its settled caches, greedy or sampled, one plain greedy step, and
  the admission of requests (acoustic keys and values, prompt, first token).

Sizes are those of the Whisper-large and Whisper-tiny shaped configurations of
`paper_2609_32869_gb300.synthetic` (block of 1 + 8 rows, 1500 encoder frames,
transcripts of up to 448 positions, batches of 1 to 96); `n_layers` reduces the
depth of a handle where a single block, the heads or the sampling are what a
case is about.  Step cases return fp32 logits beside the tokens.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2609_32869_gb300 import binding as B
from paper_2609_32869_gb300 import synthetic as syn
from paper_2609_32869_gb300.session import Session

MODELS = {"large": syn.LARGE, "tiny": syn.TINY}
K1 = syn.LARGE.block_k + 1  # rows of a verify block: the anchor and the proposals


def listed():
    return [
        # the latency of one live transcript: a full speculative step at batch 1
        {"name": "step_b1", "kind": "step", "model": "large", "n_layers": 32, "batch": 1, "lo": 100, "hi": 100,
         "temperature": 0.0, "plain": False},
        # the largest serving batch, ragged transcripts
        {"name": "step_b96", "kind": "step", "model": "large", "n_layers": 32, "batch": 96, "lo": 10, "hi": 220,
         "temperature": 0.0, "plain": False},
        # a middle-sized batch, one block in eight of the decoder
        {"name": "step_b16_4l", "kind": "step", "model": "large", "n_layers": 4, "batch": 16, "lo": 20, "hi": 220,
         "temperature": 0.0, "plain": False},
        # temperature sampling: the heads, the draws and the rejection rule weigh most
        {"name": "sample_b32_4l", "kind": "step", "model": "large", "n_layers": 4, "batch": 32, "lo": 20, "hi": 220,
         "temperature": 0.7, "plain": False},
        # admission of new requests with a four-token prompt (language, task)
        {"name": "prefill_b8_4l", "kind": "prefill", "model": "large", "n_layers": 4, "batch": 8, "prompt": 4},
        # one projection of a single sequence's verify block (QKV)
        {"name": "gemm_qkv_b1", "kind": "gemm", "M": 9, "N": 3840, "K": 1280},
        # feed-forward in at batch 16
        {"name": "gemm_fc1_b16", "kind": "gemm", "M": 144, "N": 5120, "K": 1280},
        # feed-forward out at batch 96 with three sequences already finished
        {"name": "gemm_fc2_b93", "kind": "gemm", "M": 837, "N": 1280, "K": 5120},
        # the drafter's block attention of one sequence, RoPE on queries and keys
        {"name": "attn_draft_b1", "kind": "attn", "mode": 1, "rope": True, "n_seq": 1, "rps": 9, "heads": 20,
         "ctx": 448, "lo": 150, "hi": 150},
        # cross-attention over the audio at batch 16
        {"name": "attn_cross_b16", "kind": "attn", "mode": 2, "rope": False, "n_seq": 16, "rps": 9, "heads": 20,
         "ctx": 1500, "lo": 0, "hi": 0},
        # the verify block's causal self-attention at batch 96, ragged caches
        {"name": "attn_verify_b96", "kind": "attn", "mode": 0, "rope": False, "n_seq": 96, "rps": 9, "heads": 20,
         "ctx": 448, "lo": 10, "hi": 220},
        # a long prompt (the previous window's text) at admission
        {"name": "attn_prompt_b8", "kind": "attn", "mode": 0, "rope": False, "n_seq": 8, "rps": 223, "heads": 20,
         "ctx": 448, "lo": 0, "hi": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    model = "large" if rng.random() < 0.75 else "tiny"
    cfg = MODELS[model]
    d, f = cfg.d_model, cfg.d_ff
    kind = rng.choice(("gemm", "attn", "step"))
    if kind == "gemm":
        # every projection of a block, the history projection and the head (at most 96 blocks of rows)
        n, k = rng.choice(((3 * d, d), (d, d), (f, d), (d, f), (2 * d, d), (d, 5 * d), (cfg.vocab, d)))
        return {"kind": kind, "M": _log_int(rng, 1, 96 * K1 if n == cfg.vocab else 12000), "N": n, "K": k}
    if kind == "attn":
        form = rng.choice(("verify", "draft", "cross", "prompt"))
        c = {"kind": kind, "mode": {"verify": 0, "draft": 1, "cross": 2, "prompt": 0}[form], "rope": form == "draft",
             "n_seq": _log_int(rng, 1, 16 if form == "prompt" else 96), "rps": rng.choice((1, K1, K1, K1)),
             "heads": cfg.n_heads, "ctx": 448, "lo": rng.randint(4, 120), "hi": rng.randint(121, 430)}
        if form == "draft":
            c["rps"] = K1
        elif form == "cross":
            c.update(ctx=rng.choice((1500, 1500, _log_int(rng, 100, 1500))), lo=0, hi=0)
        elif form == "prompt":
            c.update(rps=_log_int(rng, 4, 224), lo=0, hi=0)
        return c
    n_layers = rng.choice((4, 8, 16)) if model == "large" else cfg.n_layers
    if rng.random() < 0.2:
        n = _log_int(rng, 1, 16)  # prompts that one pass of the handle takes together (its rows: 448)
        return {"kind": "prefill", "model": model, "n_layers": n_layers, "batch": n,
                "prompt": _log_int(rng, 3, min(224, 448 // n))}
    return {"kind": "step", "model": model, "n_layers": n_layers, "batch": _log_int(rng, 1, 96),
            "lo": rng.randint(4, 60), "hi": rng.randint(61, 400), "temperature": rng.choice((0.0, 0.0, 0.7, 1.0)),
            "plain": rng.random() < 0.2}


# ------------------------------------------------------------------ inputs --
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, shape, std):
    return (torch.randn(shape, generator=g, device="cuda") * std).to(torch.bfloat16)


def _config(case):
    cfg = MODELS[case["model"]]
    if case["n_layers"] == cfg.n_layers:
        return cfg
    n = case["n_layers"]
    return dataclasses.replace(cfg, n_layers=n, taps=tuple(min(n - 1, i * n // 5) for i in range(4)) + (n - 1,))


def _weights(g, cfg):
    """Seeded parameters: matrices N(0, 0.02), LayerNorm gains N(1, 0.1) and biases N(0, 0.05)."""
    d, f = cfg.d_model, cfg.d_ff

    def ln(t, name):
        t[name + "_g"] = (1.0 + 0.1 * torch.randn(d, generator=g, device="cuda")).to(torch.bfloat16)
        t[name + "_b"] = _normal(g, (d,), 0.05)

    def layer():
        t = {}
        for name in ("ln1", "ln2", "ln3"):
            ln(t, name)
        for name, rows, cols in (("qkv", 3 * d, d), ("out", d, d), ("xq", d, d), ("xkv", 2 * d, d), ("xout", d, d),
                                 ("fc1", f, d), ("fc2", d, f)):
            t[name + "_w"], t[name + "_b"] = _normal(g, (rows, cols), 0.02), _normal(g, (rows,), 0.02)
        t["qkv_b"][d:2 * d] = 0  # Whisper's key projections carry no bias
        t["xkv_b"][:d] = 0
        return t

    target = {"tok_emb": _normal(g, (cfg.vocab, d), 0.02), "pos_emb": _normal(g, (cfg.max_pos, d), 0.02)}
    ln(target, "lnf")
    drafter = {"proj_w": _normal(g, (d, cfg.n_taps * d), 0.02), "proj_b": _normal(g, (d,), 0.02),
               "mask_emb": _normal(g, (d,), 0.02)}
    ln(drafter, "hln")
    return {"target": target, "target_layers": [layer() for _ in range(cfg.n_layers)], "drafter": drafter,
            "drafter_layers": [layer() for _ in range(cfg.n_draft_layers)]}


def _prompt(rs, cfg, n, length):
    ids = rs.randint(0, cfg.vocab - 1, (n, length))
    return np.where(ids >= cfg.eos_id, ids + 1, ids).astype(np.int32)


def _bases(case):
    """Cache lengths of an attention case's sequences: spread evenly over [lo, hi], within the cache."""
    n, top = case["n_seq"], case["ctx"] - case["rps"]
    return [min(top, case["lo"] + (case["hi"] - case["lo"]) * i // max(1, n - 1)) for i in range(n)]


def _groups(case):
    """(sequences, transcript length) of a step case: up to four groups spread over [lo, hi]."""
    n = min(4, case["batch"])
    size = [case["batch"] // n + (1 if i < case["batch"] % n else 0) for i in range(n)]
    return [(s, case["lo"] + (case["hi"] - case["lo"]) * i // max(1, n - 1)) for i, s in enumerate(size)]


def prepare(case, seed):
    g, rs = _gen(seed), np.random.RandomState(seed)
    if case["kind"] == "gemm":
        m, n, k = case["M"], case["N"], case["K"]
        return {"case": case, "x": _normal(g, (m, k), 1.0), "w": _normal(g, (n, k), 0.02), "b": _normal(g, (n,), 0.02),
                "y": torch.empty(m, n, dtype=torch.float32, device="cuda"),
                "scratch": torch.empty(max(256, B.wf_gemm_scratch_bytes(m, n, k)), dtype=torch.uint8, device="cuda")}
    if case["kind"] == "attn":
        n, rps, heads, ctx = case["n_seq"], case["rps"], case["heads"], case["ctx"]
        order = rs.permutation(n)
        base = np.zeros(n, np.int32)
        base[order] = _bases(case)
        return {"case": case, "q": _normal(g, (n * rps, heads * 64), 1.0), "k": _normal(g, (n, heads, ctx, 64), 1.0),
                "v": _normal(g, (n, heads, ctx, 64), 1.0),
                "slot": torch.from_numpy(order.astype(np.int32)).cuda(), "base": torch.from_numpy(base).cuda(),
                "out": torch.zeros(n * rps, heads * 64, dtype=torch.bfloat16, device="cuda"),
                "scratch": torch.empty(B.wf_attention_scratch_bytes(n, rps, heads, ctx), dtype=torch.uint8,
                                       device="cuda")}
    cfg, n = _config(case), case["batch"]
    s = Session(cfg, _weights(g, cfg), max_batch=n, keep_logits=True)
    enc = _normal(g, (n, cfg.enc_frames, cfg.d_model), 1.0)
    state = {"case": case, "cfg": cfg, "s": s, "all": torch.arange(n, dtype=torch.int32, device="cuda")}
    if case["kind"] == "prefill":
        # one output token allowed: the slots are free again after the first token
        state.update(enc=enc, slots=np.arange(n, dtype=np.int32), prompt=_prompt(rs, cfg, n, case["prompt"]),
                     budget=np.ones(n, np.int32))
        return state
    at = 0
    for size, length in _groups(case):
        s.prefill(np.arange(at, at + size, dtype=np.int32), enc[at:at + size], _prompt(rs, cfg, size, length),
                  np.full(size, 448, np.int32))
        at += size
    state["sp"] = B.sample_params(case["temperature"], seed=seed) if case["temperature"] > 0 else None
    return state


# -------------------------------------------------------------------- runs --
def run(state):
    case = state["case"]
    if case["kind"] == "gemm":
        B.wf_gemm_bf16(state["x"], state["w"], state["b"], state["y"], case["M"], case["N"], case["K"],
                       state["scratch"], state["scratch"].numel())
        return state["y"]
    if case["kind"] == "attn":
        B.wf_attention(state["q"], state["k"], state["v"], state["slot"], state["base"], case["n_seq"], case["rps"],
                       case["heads"], case["ctx"], case["mode"], case["rope"], syn.LARGE.rope_base, state["out"],
                       state["scratch"], state["scratch"].numel())
        return state["out"]
    s, cfg, n = state["s"], state["cfg"], case["batch"]
    if case["kind"] == "prefill":
        first = s.prefill(state["slots"], state["enc"], state["prompt"], state["budget"])
        s.compact()
        return {"logits": s.view(B.WF_VIEW_TARGET_LOGITS, torch.float32, (n, cfg.vocab)), "first": first}
    # back to where the prompt ended, then one step from there
    B.wf_reset_slots(s.h, n, state["all"])
    if case["plain"]:
        tokens, count = s.greedy_step(state["sp"])
        return {"logits": s.view(B.WF_VIEW_TARGET_LOGITS, torch.float32, (n, cfg.vocab)), "tokens": tokens,
                "count": count}
    tokens, count = s.step(sp=state["sp"])
    return {"logits": s.view(B.WF_VIEW_TARGET_LOGITS, torch.float32, (n * K1, cfg.vocab)),
            "draft_logits": s.view(B.WF_VIEW_DRAFT_LOGITS, torch.float32, (n * K1, cfg.vocab)),
            "taps": s.view(B.WF_VIEW_TAPS, torch.bfloat16, (n * K1, cfg.n_taps * cfg.d_model)),
            "tokens": tokens, "count": count}


# -------------------------------------------------------------------- work --
def work(case):
    if case["kind"] == "gemm":
        m, n, k = case["M"], case["N"], case["K"]
        return {"bytes": 2 * (m * k + n * k + n) + 4 * m * n, "flops": 2 * m * n * k}
    if case["kind"] == "attn":
        rps, d = case["rps"], case["heads"] * 64
        keys = pairs = 0
        for base in _bases(case):
            seen = case["ctx"] if case["mode"] == 2 else base + rps
            keys += seen
            pairs += sum(base + j + 1 for j in range(rps)) if case["mode"] == 0 else seen * rps
        return {"bytes": 4 * keys * d + 4 * case["n_seq"] * rps * d, "flops": 4 * pairs * d}
    cfg, n = _config(case), case["batch"]
    d, f, v, nl, nd, frames = cfg.d_model, cfg.d_ff, cfg.vocab, cfg.n_layers, cfg.n_draft_layers, cfg.enc_frames
    block = 6 * d * d + 2 * d * f  # QKV, out, cross query, cross out, feed-forward
    if case["kind"] == "prefill":
        rows = n * case["prompt"]
        history = (cfg.n_taps + 2 * nd) * d * d
        weights = nl * block + (nl + nd) * 2 * d * d + history + v * d
        kv = (nl + nd) * n * frames * 2 * d
        pairs = nl * n * (case["prompt"] * frames + case["prompt"] * (case["prompt"] + 1) // 2)
        return {"bytes": 2 * weights + 2 * n * frames * d + 4 * kv + 4 * n * v,
                "flops": 2 * kv * d + 2 * rows * (nl * block + history) + 2 * n * v * d + 4 * pairs * d}
    lengths = [length for size, length in _groups(case) for _ in range(size)]
    rows = n * (1 if case["plain"] else K1)
    passes = nl if case["plain"] else nl + nd
    heads = 1 if case["plain"] else 2
    history = 0 if case["plain"] else (cfg.n_taps + 2 * nd) * d * d
    keys = passes * (n * frames + sum(length + rows // n for length in lengths))
    return {"bytes": 2 * (passes * block + history + heads * v * d) + 4 * keys * d + heads * 4 * rows * v,
            "flops": 2 * rows * (passes * block + history + heads * v * d) + 4 * keys * (rows // n) * d}


# ------------------------------------------------------------------- exact --
def _exact_attention(q, k, v, see=None):
    """softmax(q k^T / 8) v per head; q [.., rows, 64], k and v [.., keys, 64], see [rows, keys]."""
    s = q @ k.transpose(-1, -2) / 8.0
    if see is not None:
        s = s.masked_fill(~see, -math.inf)
    return torch.softmax(s, -1) @ v


def _exact_rope(x, at, base):
    inv = (base ** (-torch.arange(0, 64, 2, dtype=torch.float64, device="cuda") / 64)).float()
    a = (at.float()[:, None] * inv).double()  # the phase is formed in fp32
    lo, hi = x[..., :32], x[..., 32:]
    return torch.cat((lo * a.cos() - hi * a.sin(), hi * a.cos() + lo * a.sin()), -1)


def _exact_prefill(case, state):
    """The first tokens' logits: the target's causal pass over the prompts, in 64 bits."""
    cfg, n, w = state["cfg"], case["batch"], state["s"].dev_weights
    d, heads, rows = cfg.d_model, cfg.n_heads, case["prompt"]
    split = lambda x: x.view(n, -1, heads, 64).transpose(1, 2)  # noqa: E731
    join = lambda x: x.transpose(1, 2).reshape(n, rows, d)  # noqa: E731
    ln = lambda x, t, name: torch.nn.functional.layer_norm(  # noqa: E731
        x, (d,), t[name + "_g"].double(), t[name + "_b"].double(), cfg.ln_eps)
    lin = lambda x, t, name: x @ t[name + "_w"].double().T + t[name + "_b"].double()  # noqa: E731
    t = w["target"]
    enc = state["enc"].double()
    ids = torch.from_numpy(state["prompt"]).cuda().long()
    x = t["tok_emb"].double()[ids] + t["pos_emb"].double()[:rows]
    see = torch.ones(rows, rows, dtype=torch.bool, device="cuda").tril()
    for lw in w["target_layers"]:
        q, k, v = lin(ln(x, lw, "ln1"), lw, "qkv").split(d, -1)
        x = x + lin(join(_exact_attention(split(q), split(k), split(v), see)), lw, "out")
        k, v = lin(enc, lw, "xkv").split(d, -1)
        x = x + lin(join(_exact_attention(split(lin(ln(x, lw, "ln2"), lw, "xq")), split(k), split(v))), lw, "xout")
        x = x + lin(torch.nn.functional.gelu(lin(ln(x, lw, "ln3"), lw, "fc1")), lw, "fc2")
    return {"logits": ln(x[:, -1], t, "lnf") @ t["tok_emb"].double().T, "first": None}


def exact(case, seed):
    if case["kind"] == "step":
        # every row hangs on tokens that the rounding of earlier logits picked
        # (the anchor, the proposals), so no value is independent of it
        return None
    state = prepare(case, seed)
    if case["kind"] == "prefill":
        return _exact_prefill(case, state)
    if case["kind"] == "gemm":
        return state["x"].double() @ state["w"].double().T + state["b"].double()
    n, rps, heads, ctx, mode = (case[k] for k in ("n_seq", "rps", "heads", "ctx", "mode"))
    out = torch.empty(n * rps, heads * 64, dtype=torch.float64, device="cuda")
    slots, bases = state["slot"].tolist(), state["base"].tolist()
    for i, slot in enumerate(slots):
        base = 0 if mode == 2 else bases[slot]
        keys = ctx if mode == 2 else base + rps
        q = state["q"][i * rps:(i + 1) * rps].double().view(rps, heads, 64).transpose(0, 1)
        k, v = state["k"][slot][:, :keys].double(), state["v"][slot][:, :keys].double()
        at = base + torch.arange(rps, device="cuda")
        if case["rope"]:
            q = _exact_rope(q, at, syn.LARGE.rope_base)
            k = _exact_rope(k, torch.arange(keys, device="cuda"), syn.LARGE.rope_base)
        see = torch.arange(keys, device="cuda") <= at[:, None] if mode == 0 else None
        out[i * rps:(i + 1) * rps] = _exact_attention(q, k, v, see).transpose(0, 1).reshape(rps, heads * 64)
    return out
