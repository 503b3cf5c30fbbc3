"""The work that users of this library have it do, as cases that can be timed and compared.

Four kinds of pass, each through the public entry points of ``binding`` and ``loop``:

* ``verify``   one verification step of a batch (``binding.verify``), committed, and the cut back to the
               cache it started from (``KVCache.rollback``), as a serving loop with a fixed cache does it;
* ``prefill``  a prompt appended to an empty sequence (``KVCache.prefill``), then the first drafted block on it;
* ``score``    semantic-preservation scores of token replacements (``KVCache.semantic_score``), the labelling
               of a verifier's training data;
* ``cycle``    one cycle of the host loop (``loop.SpeculativeDecoder.cycle``): the draft model's passes, the
               target's verification, both caches cut back.

Model shapes are the repository's own (``synth``), large ones with fewer layers where several copies of the
state have to fit one GPU.  Weights, caches and drafts are random with the distributions of ``synth``.
``prepare`` draws inputs again whose outcome would hang on the last bits of a float (two best logits, or a
judge score and its threshold, closer than rounding errors move them), so that two correct implementations
decide alike; ``settle_*`` below does that with the library's own debug outputs.
"""
import math

import numpy as np
import torch

from paper_2510_02329_b200 import binding, loop, synth

MODELS = {"tiny": synth.TINY, "1b": synth.LLAMA_1B, "8b": synth.LLAMA_8B, "32b": synth.QWEN_32B}
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}

# What a case does not say.  layers 0: all of them; kv_min < kv: lengths drawn from [kv_min, kv].
DEFAULTS = {"kind": "verify", "model": "8b", "layers": 0, "dtype": "bf16", "batch": 1, "gamma": 8, "kv": 1024,
            "kv_min": 0, "sampling": False, "top_k": 0, "full_outputs": False, "draft": "", "replacements": 0,
            "future": 20}


def listed():
    return [
        # The smallest call there is: the repository's first configuration, a step of a toy model.  Launches,
        # copies and barriers are all of its time.
        {"name": "tiny_b1", "model": "tiny", "kv": 128, "gamma": 4},
        # One chat user on a small model (second configuration).
        {"name": "1b_b1", "model": "1b", "kv": 2048, "gamma": 8},
        # One chat user on the model the benchmark is quoted on (third configuration).
        {"name": "8b_b1", "model": "8b", "kv": 4096, "gamma": 8},
        # The same user at temperature 1 with long drafts and a cache of odd length.
        {"name": "8b_b1_sampling", "model": "8b", "kv": 3001, "gamma": 16, "sampling": True},
        # A few users on a small model, ragged caches; hidden states and logits kept as well: what gathering a
        # verifier's training data, or distilling a draft model, asks for.
        {"name": "1b_b8_outputs", "model": "1b", "batch": 8, "kv": 1500, "kv_min": 100, "gamma": 5,
         "full_outputs": True},
        # A busy server (fourth configuration): 32 ragged caches, 288 rows.
        {"name": "8b_b32", "model": "8b", "batch": 32, "kv": 8192, "kv_min": 512, "gamma": 8},
        # Long documents on a large model (fifth configuration), a quarter of its layers.
        {"name": "32b_b8", "model": "32b", "layers": 16, "batch": 8, "kv": 8192, "gamma": 8},
        # The widest steps: many short conversations at once, top-2 alignment, 342 rows.
        {"name": "8b_b38", "model": "8b", "layers": 8, "batch": 38, "kv": 1000, "kv_min": 64, "gamma": 8, "top_k": 2},
        # A prompt of a thousand tokens and the first block on it (time to the first tokens).
        {"name": "8b_prefill", "kind": "prefill", "model": "8b", "kv": 1000, "gamma": 8},
        # Labelling: three replacements in a response, 20 future tokens each as in the paper.
        {"name": "8b_score", "kind": "score", "model": "8b", "kv": 777, "replacements": 3, "future": 20},
        # A whole cycle of the paper's smaller pair: draft passes of the 1B shape, verification by the 8B shape.
        {"name": "8b_1b_cycle", "kind": "cycle", "model": "8b", "draft": "1b", "kv": 1024, "gamma": 8},
        # The 32-bit storage type: checking a deployment against exact arithmetic.
        {"name": "1b_f32", "model": "1b", "layers": 4, "dtype": "f32", "batch": 2, "kv": 512, "gamma": 4},
    ]


def log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """Another case of the ranges the listed ones stand for."""
    kind = rng.choices(["verify", "prefill", "score", "cycle", "f32"], [12, 2, 2, 2, 2])[0]
    if kind == "f32":
        model = rng.choice(["tiny", "1b"])
        return {"model": model, "layers": rng.randint(1, 2 if model == "tiny" else 6), "dtype": "f32",
                "batch": rng.randint(1, 4), "kv": log_uniform(rng, 16, 1024), "gamma": rng.randint(1, 8)}
    if kind == "cycle":
        target = rng.choice(["1b", "8b"])
        return {"kind": "cycle", "model": target, "layers": rng.randint(6, MODELS[target].n_layers), "draft": "1b",
                "batch": rng.choice([1, 1, 2, 3]), "kv": log_uniform(rng, 32, 2048), "gamma": rng.randint(3, 12)}
    model = rng.choice(["tiny", "1b", "1b", "8b", "8b", "32b"])
    shape = MODELS[model]
    layers = rng.randint(max(1, min(4, shape.n_layers)), min(shape.n_layers, 16 if model == "32b" else 32))
    if kind == "prefill":
        return {"kind": "prefill", "model": model, "layers": layers, "kv": log_uniform(rng, 24, 900),
                "gamma": rng.randint(1, 12)}
    if kind == "score":
        return {"kind": "score", "model": model, "layers": layers, "kv": log_uniform(rng, 16, 2000),
                "replacements": rng.randint(1, 3), "future": rng.randint(4, 17)}
    most_rows = 96 // (shape.n_q_heads // shape.n_kv_heads)      # query rows of a KV head that one step may have
    gamma = log_uniform(rng, 1, min(31, most_rows - 1))
    batch = log_uniform(rng, 1, min(48, 340 // (gamma + 1)))
    kv = log_uniform(rng, 16, 8192)
    while batch > 1 and batch * kv * shape.cut(layers).kv_bytes_per_token() > 16e9:
        batch //= 2
    sampling = rng.random() < 0.25 and batch * (gamma + 1) <= 160
    return {"model": model, "layers": layers, "batch": batch, "kv": kv,
            "kv_min": 0 if rng.random() < 0.4 else max(1, int(kv * rng.uniform(0.05, 0.9))), "gamma": gamma,
            "sampling": sampling, "top_k": 2 if not sampling and rng.random() < 0.2 else 0,
            "full_outputs": rng.random() < 0.15 and batch * (gamma + 1) <= 160}


# --------------------------------------------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------------------------------------------


def full(case):
    return {**DEFAULTS, **case}


def shape_of(case, model=None):
    s = MODELS[model or case["model"]]
    return s.cut(case["layers"]) if case["layers"] and not model else s


def lengths(case, seed):
    """Tokens in each sequence's cache when the pass starts."""
    r = np.random.default_rng([seed, 1])
    if case["kv_min"]:
        return [int(x) for x in r.integers(case["kv_min"], case["kv"] + 1, size=case["batch"])]
    return [case["kv"]] * case["batch"]


class Draws:
    """Seeded random numbers on the GPU."""

    def __init__(self, seed, stream):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed * 1000003 + stream)

    def normal(self, shape, std, dtype):
        return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=self.g)

    def tokens(self, shape, vocab):
        return torch.randint(0, vocab, shape, dtype=torch.int32, device="cuda", generator=self.g)


def make_model(shape, dtype, seed, max_rows):
    """Random-init weights of a shape (N(0, 0.02^2), norm gains 1, judge weights N(0, 1/d)) and a target on them."""
    d = Draws(seed, 2)
    std = synth.WEIGHT_STD
    embed = d.normal((shape.vocab, shape.d_model), std, dtype)
    top = {"embed": embed, "final_norm": torch.ones(shape.d_model, dtype=dtype, device="cuda"),
           "lm_head": embed if shape.tied_embeddings else d.normal((shape.vocab, shape.d_model), std, dtype)}
    layers = []
    for _ in range(shape.n_layers):
        layer = {name: d.normal(s, std, dtype) for name, s in synth.layer_tensor_shapes(shape).items()}
        layer["norm_attn"] = torch.ones(shape.d_model, dtype=dtype, device="cuda")
        layer["norm_ffn"] = torch.ones(shape.d_model, dtype=dtype, device="cuda")
        layers.append(layer)
    target = binding.Target(shape, top, layers, max_rows=max_rows)
    target.load_judge_head(d.normal((shape.d_model,), 1.0 / math.sqrt(shape.d_model), torch.float32), 0.0, 0.5)
    return target


def make_cache(target, lens, extra, seed, filled=True):
    """A paged cache with `lens` tokens per sequence (pages of different sequences interleaved) and room for
    `extra` more."""
    shape, n = target.shape, len(lens)
    kv = binding.KVCache(target, n, sum((length + extra + 15) // 16 + 1 for length in lens) + 8)
    if filled:
        d = Draws(seed, 3)
        std = synth.WEIGHT_STD * math.sqrt(shape.d_model)
        starts = np.concatenate([[0], np.cumsum(lens)])
        for layer in range(shape.n_layers):
            k, v = (d.normal((int(starts[-1]), shape.n_kv_heads, shape.head_dim), std, target.dtype) for _ in range(2))
            piece = 256 if layer == 0 else max(lens)    # layer 0 reserves the pages
            for s0 in range(0, max(lens), piece):
                for b, length in enumerate(lens):
                    m, at = min(piece, length - s0), int(starts[b]) + s0
                    if m > 0:
                        kv.fill(b, layer, s0, k[at:at + m], v[at:at + m])
        kv.set_len(list(range(n)), lens)
    return kv


LOGIT_GAP, SCORE_GAP = 0.03, 2e-3     # several times what the two-plane bf16 path is off by at its largest sizes


def look(target, kv, ids, pending, drafts):
    """Two best logits of every row, their tokens, the logits, and the judge scores of a block."""
    out = binding.VerifyBuffers(*drafts.shape, target.shape.d_model, target.shape.vocab, debug=True)
    kv.set_pending(ids, pending.tolist())
    binding.verify(target, kv, ids, drafts, out, commit=False, accept_all=True)
    target.sync()
    best = out.dbg_logits.topk(2, dim=2)
    return best.values, best.indices, out.dbg_logits, out.judge_scores


def pick_threshold(scores, near):
    """The middle of the widest gap between judge scores within 0.1 of `near` (a calibrated threshold)."""
    s = scores.flatten().sort().values
    s = torch.cat([s.new_tensor([near - 0.1]), s[(s > near - 0.1) & (s < near + 0.1)], s.new_tensor([near + 0.1])])
    i = int((s[1:] - s[:-1]).argmax())
    return float((s[i] + s[i + 1]) / 2)


def first_rejection(ok):
    return (ok.int().cumprod(dim=1)).sum(dim=1)


def settle_greedy(d, target, kv, ids, pending, drafts, top_k, near=0.4):
    """Pending tokens, drafts and a threshold with no decision on a near-tie; some first drafts follow the target."""
    vocab, gamma, rows = target.shape.vocab, drafts.shape[1], torch.arange(len(ids), device="cuda")
    follow = torch.rand(len(ids), device="cuda", generator=d.g) < 0.6
    _, best, _, _ = look(target, kv, ids, pending, drafts)
    drafts[:, 0] = torch.where(follow, best[:, 0, 0].int(), drafts[:, 0])
    theta = near
    for _ in range(8):
        two, best, logits, scores = look(target, kv, ids, pending, drafts)
        theta = pick_threshold(scores, near)
        mine = logits[:, :gamma].gather(2, drafts[:, :, None].long())[:, :, 0]
        edges = logits[:, :gamma].topk(3, dim=2).values
        aligned = (drafts[:, :, None] == best[:, :gamma, :max(1, top_k)]).any(dim=2)
        n = first_rejection(aligned | (scores > theta))
        reached = torch.arange(gamma, device="cuda")[None] <= n[:, None]
        # the token a draft would have to overtake, or not to be overtaken by
        k = max(1, top_k)
        edge = torch.where(aligned, edges[:, :, k], edges[:, :, k - 1])
        close = ((mine - edge).abs() < LOGIT_GAP) | ((scores - theta).abs() < SCORE_GAP)
        gap = (two[:, :, 0] - two[:, :, 1])[rows, n]
        bad = (close & reached).any(dim=1) | (gap < LOGIT_GAP)
        del logits
        if not bool(bad.any()):
            break
        pending = torch.where(bad, d.tokens(pending.shape, vocab), pending)
        drafts = torch.where(bad[:, None], d.tokens(drafts.shape, vocab), drafts)
    return pending, drafts, theta


def settle_sampling(d, target, kv, ids, pending, drafts, q, theta_near=0.4):
    """A threshold and uniforms with no acceptance on a near-tie, the emitted token in the middle of its interval."""
    B, gamma = drafts.shape
    rows = torch.arange(B, device="cuda")
    _, _, logits, scores = look(target, kv, ids, pending, drafts)
    theta = pick_threshold(scores, theta_near)
    p = logits.double().softmax(dim=2)
    at = drafts[:, :, None].long()
    p_tok, q_tok = p[:, :gamma].gather(2, at)[:, :, 0], q.gather(2, at)[:, :, 0]
    u = torch.rand((B, gamma + 1), device="cuda", generator=d.g)
    ratio = u[:, :gamma] * q_tok / p_tok
    u[:, :gamma] = torch.where((ratio - 1).abs() < 0.05, u[:, :gamma] * 0.8, u[:, :gamma])
    n = first_rejection((u[:, :gamma] * q_tok < p_tok) | (scores > theta))
    rest = torch.where((n < gamma)[:, None], (p[rows, n] - q[rows, n.clamp(max=gamma - 1)].double()).clamp(min=0), p[rows, gamma])
    cdf = rest.cumsum(dim=1)
    cdf = cdf / cdf[:, -1:]
    tok = torch.searchsorted(cdf, u[:, gamma:].double().contiguous()).clamp(max=cdf.shape[1] - 1)
    below = torch.where(tok > 0, cdf.gather(1, (tok - 1).clamp(min=0)), torch.zeros_like(cdf[:, :1]))
    u[:, gamma:] = ((below + cdf.gather(1, tok)) / 2).float()
    return theta, q_tok.contiguous(), u.contiguous()


def prepare(case, seed):
    c = full(case)
    seed = int(seed)
    shape, dtype, gamma = shape_of(c), DTYPES[c["dtype"]], c["gamma"]
    d = Draws(seed, 5)
    lens = lengths(c, seed)
    B, ids = len(lens), list(range(len(lens)))
    s = {"case": c, "ids": ids, "lens": lens}
    if c["kind"] == "score":
        s["target"] = make_model(shape, dtype, seed, 64)
        s["kv"] = make_cache(s["target"], lens, c["future"] + 2, seed)
        t = d.tokens((c["replacements"], c["future"] + 3), shape.vocab).tolist()
        s["replacements"] = [(x[0], x[1], x[2], x[3:]) for x in t]      # y_{i-1}, y_i, z_i, the future tokens
    elif c["kind"] == "prefill":
        s["target"] = make_model(shape, dtype, seed, 64)
        s["kv"] = make_cache(s["target"], lens, gamma + 2, seed, filled=False)
        s["prompt"] = d.tokens((c["kv"],), shape.vocab).tolist()
        s["out"] = binding.VerifyBuffers(1, gamma)
        s["pending"], s["drafts"] = d.tokens((1,), shape.vocab), d.tokens((1, gamma), shape.vocab)
        s["kv"].prefill(0, s["prompt"], want_next=False)
        s["pending"], s["drafts"], s["theta"] = settle_greedy(d, s["target"], s["kv"], ids, s["pending"], s["drafts"], 0)
        s["pending"] = s["pending"].tolist()
    elif c["kind"] == "cycle":
        target = make_model(shape, dtype, seed, 64)
        draft = make_model(shape_of(c, c["draft"]), dtype, seed + 7, 64)
        # the host knows only an upper bound of a draft pass's length (two rows each) until the roll-back
        target_kv, draft_kv = make_cache(target, lens, gamma + 2, seed), make_cache(draft, lens, 2 * gamma + 4, seed + 7)
        s["loop"] = loop.SpeculativeDecoder(draft, draft_kv, target, target_kv, ids, gamma)
        settle_cycle(d, s, B, gamma)
    else:
        s["target"] = make_model(shape, dtype, seed, max(16, B * (gamma + 1)))
        s["kv"] = make_cache(s["target"], lens, 2 * (gamma + 1), seed)
        s["out"] = binding.VerifyBuffers(B, gamma, shape.d_model, shape.vocab, debug=c["full_outputs"])
        pending = d.tokens((B,), shape.vocab)
        if c["sampling"]:
            q = torch._standard_gamma(torch.full((B * gamma, shape.vocab), 0.1, device="cuda"), generator=d.g)
            q /= q.sum(dim=1, keepdim=True)
            s["drafts"] = torch.multinomial(q, 1, generator=d.g).int().view(B, gamma)
            s["q"] = q.view(B, gamma, shape.vocab)
            s["theta"], s["q_tok"], s["u"] = settle_sampling(d, s["target"], s["kv"], ids, pending, s["drafts"], s["q"])
        else:
            pending, s["drafts"], s["theta"] = settle_greedy(d, s["target"], s["kv"], ids, pending,
                                                             d.tokens((B, gamma), shape.vocab), c["top_k"])
        s["pending"] = pending.tolist()
    torch.cuda.synchronize()
    return s


def settle_cycle(d, s, B, gamma):
    """Pending tokens whose draft chain and verification decide nothing on a near-tie."""
    dec, vocab = s["loop"], s["loop"].target.shape.vocab
    pending, s["theta"] = d.tokens((B,), vocab), 0.4
    for _ in range(8):
        s["pending"] = pending.tolist()
        chain, at = torch.zeros((B, gamma), dtype=torch.int32, device="cuda"), pending
        # the draft model's greedy chain from its logits, position by position as one growing block
        for j in range(gamma):
            block = chain[:, :j].contiguous() if j else torch.zeros((B, 1), dtype=torch.int32, device="cuda")
            two, best, _, _ = look(dec.draft, dec.draft_kv, s["ids"], at, block)
            chain[:, j] = best[:, j, 0].int()
            gap = two[:, j, 0] - two[:, j, 1] if j == 0 else torch.minimum(gap, two[:, j, 0] - two[:, j, 1])
        two, best, _, scores = look(dec.target, dec.target_kv, s["ids"], at, chain)
        s["theta"] = pick_threshold(scores, 0.4)
        n = first_rejection((chain == best[:, :gamma, 0]) | (scores > s["theta"]))
        rows = torch.arange(B, device="cuda")
        bad = (gap < LOGIT_GAP) | ((two[:, :, 0] - two[:, :, 1])[rows, n] < LOGIT_GAP)
        if not bool(bad.any()):
            break
        pending = torch.where(bad, d.tokens((B,), vocab), pending)


# --------------------------------------------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------------------------------------------


def outputs(out):
    got = {k: getattr(out, k) for k in ("accepted_len", "next_token", "judge_scores", "p_draft", "new_kv_len", "logp_draft")}
    if out.dbg_hidden is not None:
        got["hidden"], got["logits"] = out.dbg_hidden, out.dbg_logits
    return got


def run(s):
    c = s["case"]
    if c["kind"] == "score":
        got = []
        for y_prev, y, z, future in s["replacements"]:
            s["kv"].set_pending([0], [y_prev])
            got.append(s["kv"].semantic_score(0, y, z, future))
        return np.array(got)
    if c["kind"] == "cycle":
        dec = s["loop"]
        dec.draft_kv.rollback(s["ids"], s["lens"])
        dec.target_kv.rollback(s["ids"], s["lens"])
        dec.lens, dec.pending = list(s["lens"]), list(s["pending"])
        tokens = np.full((len(s["ids"]), c["gamma"] + 1), -1, dtype=np.int64)
        for row, made in zip(tokens, dec.cycle(theta=s["theta"])):
            row[:len(made)] = made
        return tokens
    kv, ids = s["kv"], s["ids"]
    if c["kind"] == "prefill":
        kv.rollback(ids, [0])
        kv.prefill(0, s["prompt"], want_next=False)
        kv.set_pending(ids, s["pending"])
        binding.verify(s["target"], kv, ids, s["drafts"], s["out"], theta=s["theta"])
        return outputs(s["out"])
    kv.set_pending(ids, s["pending"])
    if c["sampling"]:
        binding.verify(s["target"], kv, ids, s["drafts"], s["out"], mode=binding.MODE_SAMPLING, draft_q_tok=s["q_tok"],
                       draft_q_full=s["q"], uniforms=s["u"], theta=s["theta"])
    else:
        binding.verify(s["target"], kv, ids, s["drafts"], s["out"], theta=s["theta"], top_k=c["top_k"])
    kv.rollback(ids, s["lens"])
    return outputs(s["out"])


# --------------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far two correct ones are apart
# --------------------------------------------------------------------------------------------------------------


def step_work(shape, esz, rows, keys, lm_rows):
    """Bytes and operations of `rows` rows that attend to `keys` (row, key) pairs in all; one read of the weights."""
    params = shape.n_layers * shape.layer_params()
    return {"bytes": shape.streamed_params() * esz + rows * shape.kv_bytes_per_token(esz),
            "flops": 2.0 * params * rows + 2.0 * shape.vocab * shape.d_model * lm_rows + 4.0 * shape.n_layers * shape.q_dim * keys}


def verify_work(shape, esz, lens, gamma):
    rows = gamma + 1
    w = step_work(shape, esz, rows * len(lens), sum(rows * n + rows * (rows + 1) // 2 for n in lens), rows * len(lens))
    w["bytes"] += sum(lens) * shape.kv_bytes_per_token(esz)
    return w


def work(case):
    c = full(case)
    shape, esz, gamma = shape_of(c), 4 if c["dtype"] == "f32" else 2, c["gamma"]
    mean = (c["kv"] + (c["kv_min"] or c["kv"])) // 2        # ragged lengths: the middle of their range
    lens = [mean] * c["batch"]
    if c["kind"] == "score":      # two blocks of future + 2 rows over one cache, per call
        w = verify_work(shape, esz, lens * 2, c["future"] + 1)
        w["bytes"] -= mean * shape.kv_bytes_per_token(esz)
        parts = [w] * c["replacements"]
    elif c["kind"] == "cycle":
        d = shape_of(c, c["draft"])
        parts = [verify_work(d, esz, [n + j for n in lens], 0) for j in range(gamma)] + [verify_work(shape, esz, lens, gamma)]
    elif c["kind"] == "prefill":
        n = c["kv"]
        parts = [step_work(shape, esz, n, n * (n + 1) // 2, 1), verify_work(shape, esz, [n], gamma)]
    else:
        parts = [verify_work(shape, esz, lens, gamma)]
        if c["sampling"]:         # the draft distribution of the rejected row, the logits of the row drawn from
            parts.append({"bytes": 4.0 * shape.vocab * c["batch"], "flops": 0.0})
        if c["full_outputs"]:
            parts.append({"bytes": 4.0 * (shape.vocab + shape.d_model) * c["batch"] * (gamma + 1), "flops": 0.0})
    return {"bytes": float(sum(p["bytes"] for p in parts)), "flops": float(sum(p["flops"] for p in parts))}


def tolerance(case):
    """Four times what was seen between the library's own alternatives on the same inputs (one kernel per stage
    against the persistent kernel, mma.sync against tcgen05 attention, one- against two-term attention operands):
    bf16 steps at most 1.3e-4 (largest value 4e-4), scores 2e-4, a step on a prefilled cache 1.1e-3 (its rows were
    rounded to bf16 block by block).  32-bit: the rounding of sums over a few thousand terms."""
    c = full(case)
    if c["dtype"] == "f32":
        return {"rel": 2e-5, "max": 2e-4, "differ": 0.0}
    if c["kind"] == "prefill":
        return {"rel": 5e-3, "max": 1e-2, "differ": 0.0}
    return {"rel": 1e-3, "max": 4e-3, "differ": 0.0}
