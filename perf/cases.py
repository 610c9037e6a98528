"""The work that users of this library have it do, as cases that can be timed and compared.

Four kinds of call, each through the Python binding as a decoding program makes it:
  step      one denoising step of a stepping program: `Model.denoise_step` on a partly decoded canvas, then
            `accept_freeze` on the block that is being decoded
  cached    the same under the block-wise KV cache: `Model.denoise_step_cached` over the block's rows only, against the
            keys and values an earlier full pass left in the cache
  head      the LM head with its statistics on hidden states the caller has (`Model.lm_head_stats`), with or without
            a draw at a temperature, then `accept_freeze`
  generate  Algorithm 1 from prompt to tokens: `Model.generate`, with or without the KV cache

Weights are random (no trained ones exist here): N(0, 0.02), gains N(1, 0.1).  A trained head is mostly sure of its
token, a random one never, so every canvas position gets a planted logit (the library's bump arguments), in units of
the random head's own logit spread `sigma`:
  step, cached, head   6.25 sigma + U(0, 12): from "just ahead of 100k other tokens" to "certain", so that both the early
                       exit and the transfer schedule have work
  generate             `hard` positions of a block get 8.6 sigma (always the argmax, never above the threshold: they wait for the
                       schedule, one per step), the others 30 (they exit at once), so that how many steps a generation
                       takes is known from the case and does not hang on the last bit of a logit
"""
import math
import random

import torch

from paper_2602_11133_b200 import inputs, jot

GEOMETRIES = {"tiny": inputs.TINY, "llada8b": inputs.LLADA_8B, "dream7b": inputs.DREAM_7B}
THRESHOLDS = {"tiny": (90.0, 1.0, 0.5, 8), "llada8b": (30.0, 1.0, 0.5, 8), "dream7b": (90.0, 1.0, 0.5, 8)}
GENERATE_TAU = 1e6          # between the hard positions' top-2 ratio (below e^10) and the easy ones' (above e^20)


def _case(name, kind, model, batch, prompt, gen, block, *, temperature=0.0, hard=0):
    c = {"kind": kind, "model": model, "batch": batch, "prompt": prompt, "gen": gen, "block": block,
         "temperature": temperature, "hard": hard}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest step there is: a toy model whose kernels take microseconds, so launches and latency are the cost
        _case("tiny_step", "step", "tiny", 1, 32, 64, 64),
        # the same model decoding its 64 tokens through the library's own loop, 16 steps
        _case("tiny_generate", "generate", "tiny", 1, 32, 64, 64, hard=15),
        # interactive decoding of one sequence, semi-autoregressive blocks of 32: the usual call
        _case("llada8b_step", "step", "llada8b", 1, 128, 256, 32),
        # the same canvas decoded as one block: up to 256 rows go through the LM head
        _case("llada8b_step_one_block", "step", "llada8b", 1, 128, 256, 256),
        # a small batch of a length that fits no tile
        _case("llada8b_step_ragged", "step", "llada8b", 3, 101, 230, 23),
        # offline decoding of a full batch of long answers: the largest call
        _case("llada8b_step_b16", "step", "llada8b", 16, 192, 512, 32),
        # a batch under grouped-query attention, each answer one block
        _case("dream7b_step_b8", "step", "dream7b", 8, 256, 256, 256),
        # a multiple-choice question: a short prompt and five tokens of answer
        _case("dream7b_step_short", "step", "dream7b", 1, 128, 5, 5),
        # decoding with the KV cache: one pass over a block of 32 against the cached canvas
        _case("llada8b_cached_block", "cached", "llada8b", 1, 128, 256, 32),
        # two blocks from prompt to tokens with the KV cache: 2 full passes and 14 block passes
        _case("llada8b_generate_cached", "generate_cached", "llada8b", 1, 128, 64, 32, hard=7),
        # the head alone on a batch of half-decoded answers (a caller with a network of its own)
        _case("head_b8", "head", "llada8b", 8, 128, 256, 256),
        # the head on one block with sampled tokens
        _case("head_block_sampled", "head", "llada8b", 1, 128, 256, 32, temperature=0.7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """A call of the same ranges: any model, one to sixteen sequences, canvases from 40 positions to 704, blocks of any
    length; never more rows than the largest listed batch."""
    kind = rng.choice(["step", "step", "step", "cached", "cached", "head", "generate", "generate_cached"])
    model = "llada8b" if kind == "head" else rng.choice(["tiny", "llada8b", "llada8b", "dream7b"])
    batch = _log_int(rng, 1, 4 if kind.startswith("generate") else 16)
    prompt = _log_int(rng, 32, 256)
    block = _log_int(rng, 5, 256)
    if kind.startswith("generate"):
        block = _log_int(rng, 5, 64)
        return _case(None, kind, model, batch, prompt, block * rng.randint(1, 2), block, hard=rng.randint(1, min(block - 1, 7)))
    gen = block * rng.randint(1, max(1, min(16, 448 // block)))
    return _case(None, kind, model, batch, prompt, gen, block,
                 temperature=rng.choice([0.0, 0.7]) if kind == "head" else 0.0)


# ------------------------------------------------------------------------------------------------ inputs
def _weights(g, n_layers, gen):
    def normal(*shape, std=0.02):
        return torch.empty(*shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=gen)

    def gain():
        return (1.0 + 0.1 * torch.randn(g.d_model, device="cuda", generator=gen)).to(torch.bfloat16)

    layers = [{"attn_norm": gain(), "wqkv": normal(g.qkv_rows, g.d_model), "wo": normal(g.d_model, g.n_q_heads * g.head_dim),
               "mlp_norm": gain(), "w_gate_up": normal(2 * g.d_ff, g.d_model), "w_down": normal(g.d_model, g.d_ff)}
              for _ in range(n_layers)]
    # (a caller that only uses the head has no embedding table: the head stands in for the pointer)
    head = normal(g.vocab, g.d_model)
    return {"embed": normal(g.vocab, g.d_model) if n_layers else head, "lm_head": head, "final_norm": gain(), "layers": layers}


def _token_ids(g, shape, gen):
    t = torch.randint(0, g.vocab - 1, shape, dtype=torch.int32, device="cuda", generator=gen)
    return t + (t >= g.mask_id).to(torch.int32)


def _first_undecided_block(case):
    """Decoding is half-way through the answer: the middle block is the current one."""
    lo = case["prompt"] + case["gen"] // case["block"] // 2 * case["block"]
    return lo, lo + case["block"]


def _hard_counts(case):
    """Hard positions per block of each sequence: from 1 up to the case's `hard`, so that a batch ends staggered."""
    B = case["batch"]
    return [1 + (case["hard"] - 1) * (b + 1) // B for b in range(B)]


def _inputs(case, seed):
    """Weights and inputs of a case; everything is drawn here, in this order."""
    g = GEOMETRIES[case["model"]]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    B, P, G, Lb = case["batch"], case["prompt"], case["gen"], case["block"]
    L, kind = P + G, case["kind"]
    sigma = 0.02 * math.sqrt(g.d_model)
    s = {"weights": _weights(g, 0 if kind == "head" else g.n_layers, gen), "bump_id": _token_ids(g, (B, L), gen)}
    uniform = torch.rand(B, L, device="cuda", generator=gen)
    if kind.startswith("generate"):
        order = torch.argsort(uniform[:, P:].reshape(B, G // Lb, Lb), dim=2)
        n_hard = torch.tensor(_hard_counts(case), device="cuda").view(B, 1, 1)
        val = torch.full((B, L), 30.0, device="cuda")
        val[:, P:] = torch.where(order < n_hard, 8.6 * sigma, 30.0).reshape(B, G)
        s.update(bump_val=val, prompt=_token_ids(g, (B, P), gen))
        return s
    s["bump_val"] = 6.25 * sigma + 12.0 * uniform
    lo, hi = _first_undecided_block(case)
    canvas = _token_ids(g, (B, L), gen)
    canvas[:, lo:] = g.mask_id                           # blocks before the current one are decided, later ones are not
    if kind == "head" and Lb > 32:                       # ... and so are some positions inside a long block
        decided = torch.rand(B, Lb, device="cuda", generator=gen) < 0.5
        canvas[:, lo:hi] = torch.where(decided, _token_ids(g, (B, Lb), gen), canvas[:, lo:hi])
    s["canvas"] = canvas
    if kind == "head":
        s["hidden"] = torch.empty(B * L, g.d_model, dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=gen)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    B, L, kind = case["batch"], case["prompt"] + case["gen"], case["kind"]
    model = jot.Model(GEOMETRIES[case["model"]], s.pop("weights"), B, L)
    s.update(case=case, model=model)
    if kind.startswith("generate"):
        s["params"] = jot.Params(GENERATE_TAU, GENERATE_TAU, 0.5, 8)
        if kind == "generate_cached":
            model.attach_kv_cache()
        return s
    lo, hi = _first_undecided_block(case)
    s.update(params=jot.Params(*THRESHOLDS[case["model"]]), tokens=s["canvas"].clone(), stats=jot.Stats.empty(B, L, "cuda"),
             lo=lo, hi=hi, n_masked=torch.zeros(B, dtype=torch.int32, device="cuda"))
    if kind == "head":
        s["sampling"] = jot.Sampling(case["temperature"], int(seed), 3) if case["temperature"] > 0 else None
    if kind == "cached":
        model.attach_kv_cache()
        model.denoise_step_cached(s["canvas"], lo, hi, True)
    return s


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    case, model = s["case"], s["model"]
    bump = {"bump_id": s["bump_id"], "bump_val": s["bump_val"]}
    if case["kind"].startswith("generate"):
        tokens, used, passes = model.generate(s["prompt"], case["gen"], case["gen"], s["params"], case["block"],
                                              kv_cache=case["kind"] == "generate_cached", **bump)
        return {"tokens": tokens, "steps_used": used, "passes": passes}
    tokens, stats, lo, hi = s["tokens"], s["stats"], s["lo"], s["hi"]
    tokens.copy_(s["canvas"])                            # accept_freeze decides on the canvas in place
    if case["kind"] == "step":
        model.denoise_step(tokens, lo, hi, out=stats, **bump)
    elif case["kind"] == "cached":
        model.denoise_step_cached(tokens, lo, hi, False, out=stats, **bump)
    else:
        model.lm_head_stats(s["hidden"], tokens, lo, hi, out=stats, sampling=s["sampling"], **bump)
    jot.accept_freeze(s["params"], model.cfg.mask_id, tokens, lo, hi, 1, stats, s["n_masked"], step_index=1)
    # the largest probability rather than its reciprocal `sumexp`: that is what a program shows and ranks by
    out = {"tokens": tokens, "top1": stats.top1, "top2": stats.top2, "argmax": stats.argmax, "p1": 1.0 / stats.sumexp}
    if stats.sampled is not None:
        out["sampled"] = stats.sampled
    return out


# ------------------------------------------------------------------------------------------------ the same in 64 bits
def _norm64(h, gain, eps):
    return h * torch.rsqrt((h * h).mean(-1, keepdim=True) + eps) * gain.double()


def _hidden64(g, w, canvas):
    """The network on the whole canvas, with no activation rounded; final-normalised, [B * L, d]."""
    B, L = canvas.shape
    nq, nkv, hd = g.n_q_heads, g.n_kv_heads, g.head_dim
    h = w["embed"][canvas.long()].double().reshape(B * L, -1)
    inv = g.rope_theta ** (-torch.arange(hd // 2, dtype=torch.float64, device="cuda") * 2.0 / hd)
    angle = torch.arange(L, dtype=torch.float64, device="cuda")[:, None, None] * inv
    cos, sin = torch.cos(angle), torch.sin(angle)

    def turn(t):
        a, b = t[..., :hd // 2], t[..., hd // 2:]
        return torch.cat([a * cos - b * sin, b * cos + a * sin], dim=-1)

    for lw in w["layers"]:
        qkv = (_norm64(h, lw["attn_norm"], g.rms_eps) @ lw["wqkv"].double().T).reshape(B, L, nq + 2 * nkv, hd)
        o = torch.empty(B, L, nq * hd, dtype=torch.float64, device="cuda")
        for b in range(B):
            q, k, v = turn(qkv[b, :, :nq]), turn(qkv[b, :, nq:nq + nkv]), qkv[b, :, nq + nkv:]
            q = q.reshape(L, nkv, nq // nkv, hd).permute(1, 2, 0, 3)                       # [kv head, its queries, L, hd]
            scores = q @ k.permute(1, 2, 0)[:, None] / math.sqrt(hd)
            o[b] = (torch.softmax(scores, -1) @ v.permute(1, 0, 2)[:, None]).permute(2, 0, 1, 3).reshape(L, nq * hd)
        h = h + o.reshape(B * L, -1) @ lw["wo"].double().T
        gate_up = _norm64(h, lw["mlp_norm"], g.rms_eps) @ lw["w_gate_up"].double().T
        act = torch.nn.functional.silu(gate_up[:, :g.d_ff]).mul_(gate_up[:, g.d_ff:])
        h = h + act @ lw["w_down"].double().T
        del gate_up, act
    return _norm64(h, w["final_norm"], g.rms_eps)


def exact(case, seed):
    """Statistics of the masked positions of the block as 64 bits give them.  Tokens and argmax have no such value
    (a tie or a threshold decides them); a block pass right after the full pass sees what the full pass saw."""
    if case["kind"].startswith("generate"):
        return None
    g, s = GEOMETRIES[case["model"]], _inputs(case, seed)
    lo, hi = _first_undecided_block(case)
    canvas, w = s["canvas"], s["weights"]
    masked = torch.zeros_like(canvas, dtype=torch.bool)
    masked[:, lo:hi] = canvas[:, lo:hi] == g.mask_id
    rows = masked.flatten().nonzero().flatten()
    hidden = s["hidden"].double() if case["kind"] == "head" else _hidden64(g, w, canvas)
    hidden, head = hidden[rows], w["lm_head"].double()
    out = {"top1": torch.zeros(canvas.shape, dtype=torch.float64, device="cuda"), "p1": torch.ones(canvas.shape, dtype=torch.float64, device="cuda")}
    out["top2"] = out["top1"].clone()
    for at in range(0, len(rows), 256):
        r = rows[at:at + 256]
        logits = hidden[at:at + 256] @ head.T
        logits[torch.arange(len(r), device="cuda"), s["bump_id"].flatten()[r].long()] += s["bump_val"].flatten()[r].double()
        logits[:, g.mask_id] = -math.inf
        best = logits.topk(2, dim=1).values
        out["top1"].view(-1)[r], out["top2"].view(-1)[r] = best[:, 0], best[:, 1]
        out["p1"].view(-1)[r] = torch.exp(best[:, 0] - torch.logsumexp(logits, 1))
    out.update(tokens=None, argmax=None)
    if case["temperature"] > 0:
        out["sampled"] = None
    return out


# ------------------------------------------------------------------------------------------------ what it cannot do without
def _pass_work(g, batch, queries, keys, head_rows):
    """(bytes, flops) of one pass: `queries` positions of each sequence through the network, attending to `keys`."""
    rows, d = batch * queries, g.d_model
    params = g.qkv_rows * d + d * g.n_q_heads * g.head_dim + 3 * g.d_ff * d
    attention = 4 * batch * g.n_q_heads * queries * keys * g.head_dim
    kv = 2 * batch * (keys - queries) * g.n_kv_heads * g.head_dim * 2             # what is read from a cache
    nbytes = g.n_layers * (2 * params + 4 * d + kv) + 2 * g.vocab * d + 2 * d + rows * (2 * d + 4)
    flops = g.n_layers * (2 * rows * params + attention) + 2 * head_rows * d * g.vocab
    return nbytes, flops


def work(case):
    g = GEOMETRIES[case["model"]]
    B, P, G, Lb, kind = case["batch"], case["prompt"], case["gen"], case["block"], case["kind"]
    L = P + G
    io = B * L * 24                                      # canvas, planted logits, statistics
    if kind == "head":
        rows = B * Lb // (2 if Lb > 32 else 1)
        return {"bytes": 2 * g.vocab * g.d_model + rows * g.d_model * 2 + io, "flops": 2 * rows * g.d_model * g.vocab}
    if kind == "step":
        nbytes, flops = _pass_work(g, B, L, L, B * Lb)
        return {"bytes": nbytes + io, "flops": flops}
    if kind == "cached":
        nbytes, flops = _pass_work(g, B, Lb, L, B * Lb)
        return {"bytes": nbytes + io, "flops": flops}
    nbytes, flops = io, 0
    hard, blocks = _hard_counts(case), G // Lb
    for step in range(1 + max(hard)):                    # a sequence needs 1 + its hard positions steps per block
        if kind == "generate_cached":
            b, f = _pass_work(g, B, L if step == 0 else Lb, L, B * Lb if step == 0 else sum(max(0, h + 1 - step) for h in hard))
            nbytes, flops = nbytes + blocks * b, flops + blocks * f
    if kind == "generate":
        for step in range(blocks * (1 + max(hard))):     # every sequence on its own block, finished ones drop out
            live = [h for h in hard if step < blocks * (1 + h)]
            rows = sum(Lb if step % (1 + h) == 0 else h + 1 - step % (1 + h) for h in live)
            b, f = _pass_work(g, len(live), L, L, rows)
            nbytes, flops = nbytes + b, flops + f
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"].startswith("generate"):
        return "exact"                                   # by construction of the planted logits (above)
    if case["kind"] == "head":
        # against the same logits in 64 bits: rel 4.7e-5 (p1), max 1.3e-4, no other argmax; one position of a canvas may tie
        return {"rel": 2e-4, "max": 5e-4, "differ": 3e-3}
    if case["model"] == "tiny":
        # two layers: the activations' bf16 rounding moves a logit by 2.2e-3 to 4.3e-3 of its scale
        return {"rel": 1e-2, "max": 3e-2, "differ": 1e-2}
    # 28 to 32 layers, the same sequences in a batch of three (other tiles, other summation order): rel up to 7.7e-3,
    # max up to 2.1e-2, one decision in 384 on the other side of its threshold
    return {"rel": 3e-2, "max": 8e-2, "differ": 1e-2}
