"""What a user of this library has it do, as cases that can be timed and compared.

Three kinds of pass, all through the binding of the C ABI:

  layer   one whole-path call for one prompt (lookm_compress_layer / _opt): what a prefill does once
          per model layer
  batch   one whole-path call for a packed ragged batch (lookm_compress_varlen)
  score   the cumulative attention scores alone (lookm_score), for a caller that selects by itself
  decode  one generation step of one layer over one or several caches (lookm_decode_step /
          _varlen): what a server does once per model layer and generated token

Head counts, prompt lengths, budgets, windows and prompt layouts are those of the package's own
workloads (`synth.py`) and of the ranges between and around them: 576-token images between short
text segments, about a seventh of the tokens text, budgets from 5 % to 40 % of the prompt.

Values.  Queries and values are N(0, 1); text keys are N(0, 1), image keys lie around 24 centres per
(image, head) with noise 0.3, and some layers have a few channels eight times as large, as in
`synth.py`.  On top of that keys have importance, as prompts do: the first four tokens (attention
sinks) and a set of salient tokens, drawn per head, receive some 150 times the attention of the
others.  There are as many salient tokens as the budget has room for in the class that the method
ranks, so the threshold lies where attention drops.  That keeps outputs comparable: without a drop
the weakest kept and the strongest evicted token differ by about 1e-4 in score at 8192 tokens, in
one head or another rounding decides between them, and every row between the two moves by one.
"""
import math
import random

import torch

from paper_2406_18139_b200 import binding as B

D = 128                    # head_dim, the only one the library has
IMAGE = 576                # tokens per image
CENTRES = 24               # key centres per (image, KV head)
SINKS = 4                  # first tokens that draw attention whatever they are
SALIENT_LOGIT = 5.0        # extra logit of sinks and salient tokens ...
OUTLIER_LOGIT = 9.0        # ... in layers whose outlier channels spread the others' logits
MODES = {"averaged": B.MERGE_AVERAGE, "pivotal": B.MERGE_PIVOTAL, "weighted": B.MERGE_WEIGHTED,
         "eviction": B.MERGE_NONE}
MERGES = ("averaged", "pivotal", "weighted")
HEADS = ((8, 8), (32, 32), (40, 40), (32, 8))      # (query heads, KV heads)


def listed():
    return [
        # One image and a question: the shortest prompt that is worth compressing.  Launches and
        # latency, hardly any arithmetic.
        layer("layer_700_32h", 700, 32, 32, mode="weighted"),
        # The 2048-token, 8-head workload: few heads, so few independent units.
        layer("layer_2048_8h", 2048, 8, 8),
        # The 8192-token layer of 32 heads with outlier channels, the headline shape.
        layer("layer_8192_32h", 8192, 32, 32, mode="pivotal", outliers=True),
        # The 16384-token layer of 40 heads.
        layer("layer_16384_40h", 16384, 40, 40, window=64, mode="weighted"),
        # The 32768-token prompt with grouped queries (4 query heads per KV head).
        layer("layer_32768_32h_8kv", 32768, 32, 8, window=64, mode="pivotal"),
        # An odd length at 5 % of the prompt, with the log-sum-exp that the caller's own prefill
        # attention left, and without the text prior.
        layer("layer_7777_lse_5pct", 7777, 32, 8, ratio=0.05, lse=True, prior=False),
        # A serving batch: 16 ragged prompts of 2048 to 16384 tokens, merge modes mixed.  The largest.
        batch("batch_16_ragged_32h", 16, 2048, 16384, 32, 32),
        # Scores of a few ragged prompts for a caller with a selection of its own.
        score("score_3_ragged_32h_8kv", 3, 1500, 6000, 32, 8),
        # Token generation over a cache at 5 % of an 8192-token prompt: the smallest call there is.
        decode("decode_409_32h", 1, 409, 409, 32, 32),
        # ... over the same prompt's whole cache.
        decode("decode_8192_32h", 1, 8192, 8192, 32, 32),
        # ... over a long cache with grouped queries.
        decode("decode_32768_32h_8kv", 1, 32768, 32768, 32, 8),
        # ... for a batch of 16 requests whose prompts were compressed to 20 %.
        decode("decode_16_ragged_32h", 16, 400, 3300, 32, 32),
    ]


def layer(name, length, hq, hkv, ratio=0.2, window=32, mode="averaged", prior=True, lse=False, outliers=False):
    return {"name": name, "kind": "layer", "length": length, "hq": hq, "hkv": hkv, "ratio": ratio, "window": window,
            "mode": mode, "prior": prior, "lse": lse, "outliers": outliers}


def batch(name, n, shortest, longest, hq, hkv, ratio=0.2, window=32, mode="mixed", lengths=0):
    return {"name": name, "kind": "batch", "n": n, "shortest": shortest, "longest": longest, "hq": hq, "hkv": hkv,
            "ratio": ratio, "window": window, "mode": mode, "prior": True, "lse": False, "outliers": False,
            "lengths": lengths}


def score(name, n, shortest, longest, hq, hkv, lengths=0):
    return {"name": name, "kind": "score", "n": n, "shortest": shortest, "longest": longest, "hq": hq, "hkv": hkv,
            "lengths": lengths}


def decode(name, n, shortest, longest, hq, hkv, lengths=0):
    return {"name": name, "kind": "decode", "n": n, "shortest": shortest, "longest": longest, "hq": hq, "hkv": hkv,
            "lengths": lengths}


def draw(rng):
    """Sizes over the whole range of their kind, by logarithm; odd ones are the rule."""
    def between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["layer", "layer", "layer", "batch", "score", "decode", "decode", "decode"])
    hq, hkv = rng.choice(HEADS)
    ratio = rng.choice([0.05, 0.1, 0.2, 0.2, 0.4])
    window = rng.choice([16, 32, 64])
    if kind == "layer":
        prior = rng.random() < 0.75
        mode = rng.choice(MERGES + ("eviction",))
        length = between(640, 32768)
        window = min(window, length // 20)
        case = layer("", length, hq, hkv, ratio, window, mode, prior, rng.random() < 0.33, rng.random() < 0.33)
    elif kind == "batch":
        lo = between(640, 4000)
        case = batch("", rng.randint(2, 16), lo, between(lo, 12000), hq, hkv, ratio, min(window, lo // 20),
                     rng.choice(MERGES + ("mixed", "eviction")), rng.randrange(1 << 20))
    elif kind == "score":
        lo = between(100, 4000)
        case = score("", rng.randint(1, 4), lo, between(lo, 12000), hq, hkv, rng.randrange(1 << 20))
    else:
        n = rng.choice([1, 1, rng.randint(2, 16)])
        lo = between(100, 32768 if n == 1 else 4000)
        case = decode("", n, lo, lo if n == 1 else between(lo, 8192), hq, hkv, 0 if n == 1 else rng.randrange(1 << 20))
    del case["name"]
    return case


def lengths_of(case):
    """The prompt (or cache) lengths of a case, fixed by the case alone."""
    if case["kind"] == "layer":
        return [case["length"]]
    if case["shortest"] == case["longest"]:
        return [case["longest"]] * case["n"]
    rng = random.Random(case["lengths"])
    return [rng.randint(case["shortest"], case["longest"]) for _ in range(case["n"])]


def budget_of(case, length):
    return max(1, int(case["ratio"] * length))


def modes_of(case):
    if case["mode"] == "mixed":
        return [MODES[MERGES[r % 3]] for r in range(case["n"])]
    return [MODES[case["mode"]]] * case.get("n", 1)


# ---- inputs -------------------------------------------------------------------------------------

def layout_of(length):
    """(mask, centre index): 1 = image token; an image token's key centre, -1 for text.  15 % of the
    prompt is text, spread around the images; the last image is cropped to what is left."""
    images = (length - (3 * length + 19) // 20 + IMAGE - 1) // IMAGE
    left = length - (3 * length + 19) // 20
    text = length - left
    mask, centre = torch.zeros(length, dtype=torch.uint8), torch.full((length,), -1, dtype=torch.long)
    for i in range(images):
        at = text * (2 * i + 3) // (2 * images + 3) + i * IMAGE
        n = min(IMAGE, left - i * IMAGE)
        mask[at:at + n] = 1
        centre[at:at + n] = i * CENTRES + torch.arange(n) // (IMAGE // CENTRES)
    return mask.cuda(), centre.cuda()


def prompt(gen, length, hq, hkv, outliers, budget, window, prior):
    """q [L, hq, D], k, v [L, hkv, D] in bf16 and the modality mask of one prompt."""
    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    mask, centre = layout_of(length)
    k = normal(length, hkv, D)
    at = (centre >= 0).nonzero()[:, 0]
    k[at] = normal(int(centre.max()) + 1, hkv, D)[centre[at]] + 0.3 * k[at]
    if outliers:
        chan = torch.rand(hkv, D, generator=gen, device="cuda").topk(4, dim=1).indices
        k *= torch.ones(hkv, D, device="cuda").scatter_(1, chan, 8.0)
    # salient tokens: the sinks, and as many of the ranked class as the budget has room for, in the
    # first 75 % of the prompt (later tokens are seen by too few queries to rank high)
    window = min(window, budget)
    room, candidates = budget - window, length - window
    text = int((mask[:candidates] == 0).sum())
    early = torch.arange(length, device="cuda") < 0.75 * length
    if prior and text <= room:
        allowed, n = early & (mask == 1), room - text
    else:
        allowed, n = early & ((mask == 0) if prior else torch.ones_like(early)), room - SINKS
    allowed[:SINKS] = False
    n = max(0, min(n, int(allowed.sum())))
    chance = torch.rand(hkv, length, generator=gen, device="cuda") * allowed
    salient = torch.zeros(hkv, length, dtype=torch.bool, device="cuda")
    if n:
        salient.scatter_(1, chance.topk(n, dim=1).indices, True)
    salient[:, :SINKS] = True
    # one direction per KV head: every query has a component of 5 along it, keys have none unless
    # they are salient
    u = torch.nn.functional.normalize(normal(hkv, D), dim=-1)
    k -= (k * u).sum(-1, keepdim=True) * u
    k += ((OUTLIER_LOGIT if outliers else SALIENT_LOGIT) * math.sqrt(D) / 5.0) * salient.t()[:, :, None] * u
    q = normal(length, hq, D)
    q += 5.0 * u.repeat_interleave(hq // hkv, dim=0)
    return q.bfloat16(), k.bfloat16(), normal(length, hkv, D).bfloat16(), mask


def row_lse(q, k, hkv):
    """Natural-log row log-sum-exp of the prompt's causal attention, [hq, L] fp32: what a caller's
    prefill attention leaves."""
    length, hq = q.shape[0], q.shape[1]
    out = torch.empty(hq, length, device="cuda")
    for i in range(0, length, 1024):
        n = min(1024, length - i)
        later = torch.arange(i + n, device="cuda")[None, :] > torch.arange(i, i + n, device="cuda")[:, None]
        for h in range(hkv):
            g = hq // hkv
            rows = q[i:i + n, h * g:(h + 1) * g].float().transpose(0, 1)
            s = torch.matmul(rows, k[:i + n, h].float().t()) / math.sqrt(D)
            out[h * g:(h + 1) * g, i:i + n] = s.masked_fill_(later, -math.inf).logsumexp(-1)
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    hq, hkv, lens = case["hq"], case["hkv"], lengths_of(case)
    s = {"case": case, "lens": lens}
    if case["kind"] == "decode":
        return prepare_decode(s, gen)
    total = sum(lens)
    s["q"], s["k"], s["v"] = (torch.empty(total, h, D, dtype=torch.bfloat16, device="cuda") for h in (hq, hkv, hkv))
    s["mask"] = torch.empty(total, dtype=torch.uint8, device="cuda")
    s["cu"] = [sum(lens[:i]) for i in range(len(lens) + 1)]
    for length, at in zip(lens, s["cu"]):
        part = slice(at, at + length)
        room = length // 5 if case["kind"] == "score" else budget_of(case, length)
        s["q"][part], s["k"][part], s["v"][part], s["mask"][part] = prompt(
            gen, length, hq, hkv, case.get("outliers", False), room, case.get("window", 32), case.get("prior", True))
    s["layout"] = B.make_layout(s["q"], s["k"])
    s["workspace"] = B.alloc_workspace(s["layout"], lens)
    if case["kind"] == "score":
        s["scores"], s["lse"] = torch.empty(hkv, total, device="cuda"), torch.empty(hq, total, device="cuda")
        return s
    s["budgets"] = [budget_of(case, n) for n in lens]
    s["windows"], s["modes"] = [case["window"]] * len(lens), modes_of(case)
    kept = sum(s["budgets"])
    shape = (hkv, kept, D) if case["kind"] == "layer" else (kept, hkv, D)
    s["out_k"], s["out_v"] = (torch.empty(*shape, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    if not case["prior"] or case["lse"]:
        s["options"] = B.make_options(no_text_prior=not case["prior"],
                                      lse=s.setdefault("lse", row_lse(s["q"], s["k"], hkv)) if case["lse"] else None)
    return s


def prepare_decode(s, gen):
    """Caches [hkv, rows, D], each request's rows with room for the appended one behind them."""
    case, lens = s["case"], s["lens"]
    hq, hkv, n = case["hq"], case["hkv"], len(lens)
    rows = sum(lens) + n
    s["begin"] = [sum(lens[:i]) + i for i in range(n)]
    s["cache_k"], s["cache_v"] = (torch.randn(hkv, rows, D, generator=gen, device="cuda").bfloat16() for _ in range(2))
    s["q"] = torch.randn(n, hq, D, generator=gen, device="cuda").bfloat16()
    s["k_new"], s["v_new"] = (torch.randn(n, hkv, D, generator=gen, device="cuda").bfloat16() for _ in range(2))
    s["out"] = torch.empty(n, hq, D, device="cuda")
    s["layout"] = B.CacheLayout(hq, hkv, D, D, rows * D, 0.0)
    s["workspace"] = B.alloc_decode_workspace(s["layout"], n)
    return s


# ---- the pass -----------------------------------------------------------------------------------

def run(s):
    kind = s["case"]["kind"]
    if kind == "decode":
        if len(s["lens"]) == 1:
            status = B.lookm_decode_step(s["q"], s["k_new"], s["v_new"], s["cache_k"], s["cache_v"], s["lens"][0],
                                         s["layout"], s["out"], s["workspace"])
        else:
            status = B.lookm_decode_step_varlen(s["q"], s["k_new"], s["v_new"], s["cache_k"], s["cache_v"], s["begin"],
                                                s["lens"], s["layout"], s["out"], s["workspace"])
        B.check(status)
        return {"out": s["out"], "cache_k": s["cache_k"], "cache_v": s["cache_v"]}
    if kind == "score":
        B.check(B.lookm_score(s["q"], s["k"], s["cu"], s["layout"], s["scores"], s["lse"], False, s["workspace"]))
        return {"scores": s["scores"], "lse": s["lse"]}
    if kind == "batch":
        status, _ = B.lookm_compress_varlen(s["q"], s["k"], s["v"], s["mask"], s["cu"], s["budgets"], s["windows"],
                                            s["modes"], s["layout"], s["out_k"], s["out_v"], s["workspace"])
    elif "options" in s:
        status, _ = B.lookm_compress_layer_opt(s["q"], s["k"], s["v"], s["mask"], s["lens"][0], s["budgets"][0],
                                               s["windows"][0], s["modes"][0], s["layout"], s["options"], s["out_k"],
                                               s["out_v"], s["workspace"])
    else:
        status, _ = B.lookm_compress_layer(s["q"], s["k"], s["v"], s["mask"], s["lens"][0], s["budgets"][0],
                                           s["windows"][0], s["modes"][0], s["layout"], s["out_k"], s["out_v"],
                                           s["workspace"])
    B.check(status)
    return {"out_k": s["out_k"], "out_v": s["out_v"]}


# ---- what a pass cannot do without ----------------------------------------------------------------

def work(case):
    """Bytes: every input read once, every output written once.  Operations: one causal Q K^T for the
    scores (the softmax normaliser and the column sums could share it), evicted x kept cosines for
    the matching; Q K^T and P V for a generation step."""
    hq, hkv, lens = case["hq"], case["hkv"], lengths_of(case)
    total = sum(lens)
    row = 2 * D                                          # bytes of one bf16 row
    if case["kind"] == "decode":
        n = len(lens)
        moved = 2 * hkv * (total + n) * row + 2 * hkv * n * row + n * hq * (row + 4 * D)
        return {"bytes": moved, "flops": 4 * D * hq * (total + n)}
    causal = sum(D * n * (n + 1) for n in lens) * hq
    if case["kind"] == "score":
        return {"bytes": total * (hq + hkv) * row + 4 * total * (hq + hkv), "flops": causal}
    moved = total * (hq + hkv) * row + (total if case["prior"] else 0) + (4 * hq * total if case["lse"] else 0)
    flops = causal
    for n, mode in zip(lens, modes_of(case)):
        kept = budget_of(case, n)
        merged = mode != B.MERGE_NONE
        moved += hkv * ((n if merged else kept) + 2 * kept) * row      # values read, rows written
        flops += 2 * D * hkv * (n - kept) * kept if merged else 0
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    """Scores and generation: 32-bit sums of up to 32768 terms.  With other shares of the exponentials
    on the two units, other splits and other orders of the sums, the library differed from itself by
    4e-8 (scores) and 3e-7 (generation) of the norm, 3e-7 and 1e-6 of single values.
    Compressed caches: bf16 rows.  Another order of the sums turns a few roundings (1e-6 of the norm);
    with the key norms rounded otherwise some evicted tokens whose two best cosines tie to the last
    bit move from one kept row to another, which changes two rows each: 7e-4 of the norm, 0.6 of
    single values, in the largest batch."""
    if case["kind"] == "score":
        return {"rel": 1e-6, "max": 1e-5}
    if case["kind"] == "decode":
        return {"rel": 2e-6, "max": 1e-5}
    return {"rel": 3e-3, "max": 0.99}
