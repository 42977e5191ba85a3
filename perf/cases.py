"""The work that users of this package have it do, as measurable cases.

Everything goes through the public entry points of the binding (`Context` and its methods).  A case names

  entry     "request"   new input ids in hand: encode them, then generate (what a summarization or translation service
                        does for every request)
            "generate"  the input is encoded already: generate only (another threshold, another mode, another draw)
            "prefill"   encode, then the first pass of both models: time to first token, scoring of an input
            "step"      one single-token step of the small model from a host program (smallest call)
            "round"     a host program's own draft / verify policy: `draft` single steps, one block pass of the large
                        model over them, both caches cut back
  pair      which two models (the shapes of workloads.MODEL_SHAPES)
  enc, gen  encoder ids and generated tokens; max_enc, max_dec: the capacities the context was created with
  mode      "bild" (Algorithm 1), "small" or "large" (one model alone); top_p > 0: the sampling variant
  draft     the most small-model tokens in a row; eos: generation ends on the end-of-sequence token
  rate      share of the positions at which the small model is unsure (fallbacks); wrong: share at which it is sure of
            a token that the large model rejects (rollbacks)

The models are random models of those shapes whose heads carry a planted next-token relation, as trained pairs have one:
both are sure of the next token at most positions, the small one hesitates between two at some and is mistaken at a few.
So the confidences, fallback and rollback rates are those of an aligned pair, and every decision has a margin far above
what rounding moves: the tokens are a property of the case and not of the order of the additions.
"""
import math
import random

import numpy as np
import torch

from paper_2302_07863_b200 import binding as B
from workloads import MODEL_SHAPES
from workloads.gen import tensor_names

# name: (small, large, type of the weights, decoder layers of an early-exit small model or 0)
PAIRS = {
    "t5": ("t5_s", "t5_l", "bf16", 0),
    "mt5": ("mt5_s", "mt5_l", "bf16", 0),
    "mt5_exit": ("mt5_s", "mt5_s", "bf16", 1),
    "wide": ("wide_s", "wide_l", "bf16", 0),
    "odd": ("odd_s", "odd_l", "bf16", 0),
    "odd_fp32": ("odd_s", "odd_l", "fp32", 0),
    "tiny_fp32": ("tiny_s", "tiny_l", "fp32", 0),
}
MODES = {"bild": B.MODE_BILD, "small": B.MODE_SMALL_ONLY, "large": B.MODE_LARGE_ONLY}
START, EOS = 0, 1
ALPHA_FB, ALPHA_RB = 0.8, 3.0
EMB_STD = 4.0    # trained tables have wide rows; a token's own row then stays visible in the last hidden state
PLANT = 0.1      # weight of the planted direction in a head row (the other entries have a deviation of 0.02)
SECOND = 0.98    # weight of the second choice where the small model hesitates


def _case(name, entry, pair, enc, gen, max_enc, max_dec, mode="bild", draft=10, top_p=0.0, eos=False, rate=0.2, wrong=0.03):
    return {"name": name, "entry": entry, "pair": pair, "enc": enc, "gen": gen, "max_enc": max_enc, "max_dec": max_dec,
            "mode": mode, "draft": draft, "top_p": top_p, "eos": eos, "rate": rate, "wrong": wrong}


def listed():
    return [
        # one token of the small model on the host's own loop, in the middle of a summary
        _case("step", "step", "t5", 512, 31, 512, 65),
        # a host-driven speculative round: four drafts, one verification of five rows
        _case("round", "round", "t5", 512, 31, 512, 65, draft=4),
        # a document comes in: both encoders and the first token (long input, nothing generated yet)
        _case("prefill_long", "prefill", "t5", 1024, 1, 1024, 257),
        # summarization, the package's benchmark shape, per request
        _case("summarize", "request", "t5", 512, 64, 512, 65),
        # the same, generation alone (a second pass over an encoded input)
        _case("summarize_again", "generate", "t5", 512, 64, 512, 65),
        # what the method is compared with: the large model alone
        _case("large_only", "generate", "t5", 512, 64, 512, 65, mode="large"),
        # the sampling variant, on a context that also takes longer inputs
        _case("summarize_sampled", "request", "t5", 389, 75, 1024, 257, top_p=0.8),
        # translation: a short sentence, a large vocabulary, ends on the end-of-sequence token
        _case("translate", "request", "mt5", 64, 64, 64, 97, eos=True),
        # a very short sentence (ragged sizes, everything is latency)
        _case("translate_short", "request", "mt5", 17, 13, 256, 129, eos=True),
        # long summaries of long documents
        _case("summarize_long", "request", "t5", 1024, 256, 1024, 257),
        # early exit: the small model is the first layer of the large one
        _case("early_exit", "request", "mt5_exit", 64, 64, 64, 97, eos=True, wrong=0.0),
        # the fp32 configuration
        _case("fp32", "request", "tiny_fp32", 32, 32, 32, 33),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    entry = rng.choices(["request", "generate", "prefill", "step", "round"], [10, 4, 2, 1, 2])[0]
    pair = rng.choices(list(PAIRS), [10, 6, 2, 1, 1, 1, 1])[0]
    mode = rng.choices(["bild", "large", "small"], [8, 1, 1])[0] if entry == "generate" else "bild"
    small_vocab = pair not in ("t5", "mt5", "mt5_exit")
    enc = _log_int(rng, 8, 200 if small_vocab else 1024)
    longest = 48 if small_vocab else 80 if mode == "large" or pair == "mt5" else 180
    gen = _log_int(rng, 4, longest)
    # a service creates its context for the longest input it takes, or for the one at hand
    max_enc = rng.choice([enc, 1 << (enc - 1).bit_length(), 256 if small_vocab else 1024])
    max_dec = rng.choice([gen + 1, gen + 1 + rng.randrange(1, 32), 257])
    draft = rng.choice([10, 10, 10, 15, 7, 4]) if entry != "round" else rng.choice([2, 3, 4, 6, 8, 11])
    return {"entry": entry, "pair": pair, "enc": enc, "gen": gen, "max_enc": max(enc, max_enc),
            "max_dec": max(gen + 1 + (draft + 1 if entry == "round" else 1), max_dec), "mode": mode, "draft": draft,
            "top_p": 0.8 if entry in ("request", "generate") and mode == "bild" and rng.random() < 0.15 else 0.0,
            "eos": entry == "request" and rng.random() < 0.3,
            "rate": round(rng.uniform(0.08, 0.3), 3), "wrong": 0.0 if pair == "mt5_exit" else round(rng.uniform(0.0, 0.06), 3)}


# ---- what happens at each position: the same for every seed, so that a case is the same amount of work ------------------
def _script(case):
    """Per position of the output: "sure", "torn" (the small model hesitates) or the length of the wrong continuation that
    the small model is sure of there."""
    rng = random.Random("%(pair)s %(gen)d %(rate)g %(wrong)g %(mode)s" % case)
    more = case["draft"] + 2 if case["entry"] in ("step", "round") else 0
    lost = 0.0 if case["entry"] in ("step", "round") or case["mode"] == "small" else case["wrong"]
    kinds = []
    for _ in range(case["gen"] + more):
        u, run = rng.random(), rng.randrange(1, 7)
        kinds.append("torn" if u < case["rate"] else run if u < case["rate"] + lost else "sure")
    kinds[-1] = "sure"
    return kinds


def _passes(case):
    """The passes of one run(): rows already cached by small steps, and (rows cached, rows of the block) of large passes."""
    if case["entry"] == "prefill":
        return [0], [(0, 1)]
    p = case["gen"]
    if case["entry"] == "step":
        return [p], []
    if case["entry"] == "round":
        return [p + i for i in range(case["draft"])], [(p, case["draft"] + 1)]
    if case["mode"] == "large":
        return [], [(i, 1) for i in range(p)]
    if case["mode"] == "small":
        return list(range(p)), []
    kinds, small, large = _script(case), [], []
    n = done = drafts = 0          # last token, rows of the large model's cache, drafts since its last pass
    astray = None                  # (position of the mistake, drafts until the small model doubts)
    while n < p:
        small.append(n)
        kind = kinds[n] if astray is None else "sure" if n - astray[0] < astray[1] else "torn"
        if kind == "torn" or drafts == case["draft"]:
            large.append((done, n - done + 1))
            n = (n if astray is None else astray[0]) + 1
            done, drafts, astray = n, 0, None
        else:
            if kind != "sure":
                astray = (n, kind)
            n, drafts = n + 1, drafts + 1
    return small, large


def _shapes(case):
    small, large, dtype, exit_layers = PAIRS[case["pair"]]
    return MODEL_SHAPES[small], MODEL_SHAPES[large], dtype, exit_layers


def work(case):
    """Weights once per pass, keys and values at the weights' width; the encoders' weights once per input."""
    small, large, dtype, exit_layers = _shapes(case)
    wb = 2 if dtype == "bf16" else 4
    nbytes = flops = 0
    E = case["enc"]

    def passes(s, layers, rows):
        nonlocal nbytes, flops
        I, d, F = s.inner, s.d_model, s.d_ff
        weights = layers * (6 * I * d + (3 if s.ffn == "gated_gelu" else 2) * d * F) + s.vocab * d
        for cached, k in rows:
            nbytes += wb * (weights + layers * 2 * I * (cached + k + E) + k * d)
            flops += 2 * k * (weights + layers * 2 * I * (cached + k + E))

    steps, blocks = _passes(case)
    passes(small if not exit_layers else large, exit_layers or small.n_layers, [(c, 1) for c in steps])
    passes(large, large.n_layers, blocks)
    if case["entry"] in ("request", "prefill"):
        for s in ([large] if exit_layers else [small, large]):
            I, d, F = s.inner, s.d_model, s.d_ff
            layer = 4 * I * d + (3 if s.ffn == "gated_gelu" else 2) * d * F
            nbytes += wb * s.n_layers * (layer + 2 * I * d + 2 * I * E) + wb * E * d
            flops += 2 * E * s.n_layers * (layer + 2 * I * d + 2 * I * E)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Tokens, positions and counts are whole numbers with wide margins (a tie between two of the small model's hesitant
    candidates may fall either way).  Confidences and distances: fp32 sums in fp32 configurations; with bf16 weights the
    activations go through the products with 16 mantissa bits, over up to 48 layers."""
    return {"rel": 1e-4 if PAIRS[case["pair"]][2] == "fp32" else 2e-3, "max": 1e-3 if PAIRS[case["pair"]][2] == "fp32" else 2e-2,
            "differ": 0.01}


# ---- models and inputs ---------------------------------------------------------------------------------------------------
# what the head is scaled by so that a planted token's logit is about ln V + 6: the correlation of the last hidden state with
# the embedding of the token fed in
CORR = {"tiny_s": 0.9, "tiny_l": 0.9, "odd_s": 0.9, "odd_l": 0.9, "wide_s": 0.9, "wide_l": 0.9, "t5_s": 0.9, "t5_l": 0.8,
        "mt5_s": 0.9, "mt5_l": 0.8}


def _scale(shape):
    return (math.log(shape.vocab) + 6.0) / (PLANT * shape.d_model * CORR[shape.name])


def _model(shape, dtype, g):
    """Random weights of one model on the GPU: matrices N(0, 0.02), gains 1 + N(0, 0.02), bias tables N(0, 1)."""
    w = {}
    for name, (size, kind) in tensor_names(shape).items():
        x = torch.empty(size, device="cuda", dtype=torch.bfloat16 if dtype == "bf16" and kind in ("matrix", "embedding") else torch.float32)
        x.normal_(1.0 if kind == "gain" else 0.0, {"matrix": 0.02, "gain": 0.02, "bias": 1.0, "embedding": EMB_STD}[kind], generator=g)
        w[name] = x
    return w


def _plant(w, pairs):
    """Head row b gets the direction of token a's embedding, for every (a, b, weight)."""
    src, dst, weight = (torch.tensor(v, device="cuda") for v in zip(*pairs))
    rows = w["emb"][src].float() * (PLANT / EMB_STD) * weight.float()[:, None]
    head = w["lm_head"]
    block = torch.zeros(len(pairs), head.shape[1], device="cuda")
    to, at = torch.unique(dst, return_inverse=True)
    block.index_add_(0, at, rows)
    head[to] = (head[to].float() + block[:len(to)]).to(head.dtype)


def _language(case, vocab, seed):
    """The token sequence, and what to plant in the small and in the large model's head."""
    kinds = _script(case)
    rng = random.Random(seed)
    fresh = iter(rng.sample(range(2, vocab), min(vocab - 2, 12 * len(kinds) + 16)))
    y, small, large, here = [START], [], [], [START]
    for i, kind in enumerate(kinds):
        last = i == len(kinds) - 1
        nxt = EOS if case["eos"] and last else next(fresh)
        for a in here:
            large.append((a, nxt, 1.0))
        if kind == "torn":
            other = next(fresh)
            for a in here:
                small += [(a, nxt, 1.0), (a, other, SECOND)]
            here = [nxt, other]
        elif kind == "sure":
            small += [(a, nxt, 1.0) for a in here]
            here = [nxt]
        else:
            branch = [next(fresh) for _ in range(kind + 2)]
            small += [(a, branch[0], 1.0) for a in here] + [(branch[j], branch[j + 1], 1.0) for j in range(kind)]
            small.append((branch[kind - 1], branch[kind + 1], SECOND))
            here = [nxt]
        y.append(nxt)
    return y, small, large


def prepare(case, seed):
    small, large, dtype, exit_layers = _shapes(case)
    g = torch.Generator("cuda").manual_seed(seed)
    y, plant_s, plant_l = _language(case, large.vocab, seed)
    wl = _model(large, dtype, g)
    if exit_layers:   # one model: what the small one is unsure of, the large one is too
        import dataclasses
        small, ws = dataclasses.replace(large, n_layers=exit_layers), wl
        _plant(wl, plant_s)
    else:
        ws = _model(small, dtype, g)
        _plant(ws, plant_s)
        _plant(wl, plant_l)
    eos = EOS if case["eos"] else -1
    cfg = B.Config(B.model_cfg(small, _scale(small)), B.model_cfg(large, _scale(large)), B.BF16 if dtype == "bf16" else B.FP32,
                   case["max_enc"], case["max_dec"], min(15, case["draft"]), START, eos, exit_layers)
    ctx = B.Context(cfg, small, ws, large, wl)
    rng = np.random.default_rng(seed)
    st = {"case": case, "ctx": ctx, "ids": rng.integers(2, large.vocab, size=case["enc"], dtype=np.int32),
          "mode": MODES[case["mode"]], "max_len": case["max_dec"] - 1 if case["eos"] else case["gen"], "y": y,
          "u": (rng.random(case["max_dec"] + 1, dtype=np.float32), rng.random(case["max_dec"] + 1, dtype=np.float32))}
    ctx.encode(st["ids"])
    if case["entry"] in ("step", "round"):      # the sequence so far is in both caches
        for t in y[:case["gen"]]:
            ctx.small_step(t, ALPHA_FB)
        for i in range(0, case["gen"], B.MAX_BLOCK):
            ctx.large_verify(y[i:min(i + B.MAX_BLOCK, case["gen"])], ALPHA_RB)
    else:                                       # a service is warmed up before it takes requests
        _generate(st, 1)
    return st


def _generate(st, max_len):
    case, ctx = st["case"], st["ctx"]
    if case["top_p"] > 0:
        return ctx.generate_sampled(st["mode"], ALPHA_FB, ALPHA_RB, max_len, case["top_p"], *st["u"])
    return ctx.generate(st["mode"], ALPHA_FB, ALPHA_RB, max_len)


def _step_out(o):
    return {"argmax": o.argmax, "max_logit": o.max_logit, "lse": o.lse, "pmax": o.pmax, "fallback": o.fallback}


def _verify_out(o, k):
    return {"argmax": np.array(o.argmax[:k]), "lse": np.array(o.lse[:k]), "d": np.array(o.d[:k - 1]),
            "first_violation": o.first_violation, "next_token": o.next_token}


def run(st):
    case, ctx = st["case"], st["ctx"]
    entry = case["entry"]
    if entry == "step":
        ctx.rewind(0, case["gen"])
        return _step_out(ctx.small_step(st["y"][case["gen"]], ALPHA_FB))
    if entry == "round":
        token, block, steps = st["y"][case["gen"]], [], []
        for _ in range(case["draft"]):
            block.append(token)
            steps.append(ctx.small_step(token, ALPHA_FB))
            token = steps[-1].argmax
        block.append(token)
        v = ctx.large_verify(block, ALPHA_RB)
        ctx.rewind(0, case["gen"])
        ctx.rewind(1, case["gen"])
        return {"drafts": np.array(block), "pmax": np.array([s.pmax for s in steps]), "lse": np.array([s.lse for s in steps]),
                "verify": _verify_out(v, len(block))}
    if entry in ("request", "prefill"):
        ctx.encode(st["ids"])
    if entry == "prefill":
        return {"small": _step_out(ctx.small_step(START, ALPHA_FB)), "large": _verify_out(ctx.large_verify([START], ALPHA_RB), 1)}
    r = _generate(st, st["max_len"])
    return {"tokens": np.array(r["tokens"]), "trace": np.array([t[:5] for t in r["trace"]]), "values": np.array([t[5] for t in r["trace"]]),
            "stats": np.array([r["stats"][k] for k in sorted(r["stats"])])}
