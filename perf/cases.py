"""Performance cases of the SpecDec library: what a user's program calls, over the sizes it calls it at.

A case is one call (or one short fixed sequence of calls) of the public Python binding:

  generate      SpecDec.generate / generate_host: encode, then draft -> verify -> commit until every sequence has ended
                (k = 0: greedy decoding with the verifier alone)
  first_tokens  encode, then one draft -> verify -> commit and the session's output: the time to the first tokens
  verify, draft one step of a program that runs the loop itself, on a session with a committed prefix
  accept        the acceptance rule alone, on logits that the caller has

The model pairs have the shapes of workloads.py (Transformer-base verifier with the 12+2 drafter, the BART-base-shaped
pair, the tiny fp32 pair).  Their weights are random except for the last decoder layer's cross-attention, which is set so that the
target at position p is the source token at position p: the output then depends on the source, decoding ends at the source's [EOS] the
way a trained model ends, every decision has a wide margin, and the drafter, whose embedding confuses every seventh
id with its neighbour, is wrong about once in seven tokens -- the accepted lengths of the paper's regime (5 to 8
tokens an iteration) without any test hook.
"""
import math
import random

import numpy as np
import torch

from paper_2203_16487_b200 import binding, workloads as W

PAIRS = {"base": (W.BASE_V, W.BASE_D), "bart": (W.BART_V, W.BART_D), "tiny": (W.TINY_V, W.TINY_D)}
BETA, TAU = 3, 1.0
P_WRONG = 1.0 / 7.0                 # share of target tokens that the drafter gets wrong


def listed():
    gen = dict(kind="generate", pair="base", host=False, cached=False)
    return [
        # one sentence at a time, the paper's online translation setting
        dict(gen, name="sentence", batch=1, k=25, lo=29, hi=29),
        # a few sentences from host memory with short drafts and the drafter that caches its prefix
        dict(gen, name="sentences_host", batch=4, k=10, lo=15, hi=37, host=True, cached=True),
        # ragged batches of sentences, up to the largest batch of the benchmark
        dict(gen, name="batch_32", batch=32, k=25, lo=10, hi=80),
        dict(gen, name="batch_128", batch=128, k=25, lo=10, hi=80),
        # greedy decoding without a drafter: one row per sequence and step
        dict(gen, name="greedy_16", batch=16, k=0, lo=20, hi=40),
        # summarisation: long sources, outputs cut at 128 tokens
        dict(gen, name="summaries", batch=8, k=25, lo=300, hi=512),
        # time to the first tokens of long documents with the BART-base-shaped pair (GELU, 768 wide)
        dict(name="bart_first_tokens", kind="first_tokens", pair="bart", batch=4, k=25, lo=300, hi=478),
        # the fp32 handle, on the pair small enough to be checked against anything
        dict(gen, name="tiny_fp32", pair="tiny", batch=2, k=8, lo=13, hi=16),
        # steps of a program that runs the loop itself: the least and the most rows
        dict(name="verify_1", kind="verify", pair="base", batch=1, k=25, prefix=64),
        dict(name="verify_128", kind="verify", pair="base", batch=128, k=50, prefix=256),
        dict(name="draft_24", kind="draft", pair="base", batch=24, k=25, prefix=40, cached=False),
        # the acceptance rule on a caller's logits
        dict(name="accept_32", kind="accept", batch=32, k=25, vocab=32768, static=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["generate"] * 5 + ["verify", "verify", "draft", "first_tokens", "accept"])
    if kind == "accept":
        static = rng.random() < 0.3                      # (its scratch array holds at most 4096 rows)
        batch, k = _log_int(rng, 1, 78 if static else 128), _log_int(rng, 5, 50)
        return dict(kind=kind, batch=batch, k=k, vocab=rng.choice([1000, 32768, 50265]), static=static)
    if kind in ("verify", "draft"):
        c = dict(kind=kind, pair=rng.choice(["base", "base", "base", "bart"]), k=_log_int(rng, 4, 50), prefix=rng.randint(0, 256))
        c["batch"] = _log_int(rng, 1, 128 if c["pair"] == "base" else 32)
        if kind == "draft":
            c["cached"] = rng.random() < 0.3
        return c
    if kind == "first_tokens":
        if rng.random() < 0.5:
            lo = rng.randint(10, 40)
            return dict(kind=kind, pair="base", batch=_log_int(rng, 1, 64), k=_log_int(rng, 5, 50), lo=lo, hi=rng.randint(lo, 80))
        lo = rng.randint(200, 400)
        return dict(kind=kind, pair=rng.choice(["base", "bart"]), batch=rng.randint(1, 4), k=_log_int(rng, 5, 50), lo=lo, hi=rng.randint(lo, 512))
    c = dict(kind="generate", pair="base", host=rng.random() < 0.3, cached=rng.random() < 0.25, k=_log_int(rng, 5, 50))
    shape = rng.random()
    if shape < 0.12:                                     # fp32
        c.update(pair="tiny", batch=_log_int(rng, 1, 16), k=rng.randint(4, 12), lo=rng.randint(6, 10), hi=rng.randint(11, 20))
    elif shape < 0.27:                                   # greedy decoding
        c.update(batch=_log_int(rng, 1, 64), k=0, cached=False, lo=rng.randint(10, 20), hi=rng.randint(20, 40))
    elif shape < 0.42:                                   # long sources
        c.update(pair=rng.choice(["base", "base", "bart"]), lo=rng.randint(150, 300), hi=rng.randint(300, 450))
        c["batch"] = _log_int(rng, 1, 4 if c["pair"] == "base" else 2)
        c["k"] = max(c["k"], 15)
    else:                                                # sentences
        c.update(batch=_log_int(rng, 1, 128), lo=rng.randint(10, 30), hi=rng.randint(30, 80))
        c["k"] = max(c["k"], 10) if c["batch"] <= 48 else min(max(c["k"], 10), 25)
    return c


# ------------------------------------------------------------------------------------------------ models
_weights = {}                       # one entry per pair, as a program loads its checkpoint once


def _model(dims, seed, drafter, bf16):
    """Weights of one model on the GPU (names as in specdec.h), then as host arrays for the binding."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    d, f, half = dims.d_model, dims.d_ffn, dims.d_model // 2
    std = 0.02 if d > 64 else 0.06
    w = {}

    def rand(*shape, s=0.02):
        return torch.randn(shape, generator=g, device="cuda") * s

    def norm(name):
        w[name + ".g"], w[name + ".b"] = 1.0 + rand(d), rand(d)

    def attn(name):
        for p in "qkv":
            w[f"{name}.{p}.w"], w[f"{name}.{p}.b"] = rand(d, d), rand(d)
        w[name + ".o.w"], w[name + ".o.b"] = rand(d, d, s=0.002), rand(d)

    def ffn(name):
        w[name + ".w1"], w[name + ".b1"] = rand(f, d), rand(f)
        w[name + ".w2"], w[name + ".b2"] = rand(d, f, s=0.002), rand(d)

    w["embed"] = rand(dims.vocab, d, s=std)
    # learned positions in the first half of the width; the drafter's [MASK] at position t looks for source token t - 1
    pos = torch.randn((dims.max_pos, d), generator=torch.Generator(device="cuda").manual_seed(77), device="cuda")
    pos[:, half:] = 0
    w["pos_enc"], w["pos_dec"] = pos, pos.clone()
    if drafter:
        w["pos_dec"][1:] = pos[:-1]
    for l in range(dims.enc_layers):
        norm(f"enc.{l}.ln1"); attn(f"enc.{l}.self"); norm(f"enc.{l}.ln2"); ffn(f"enc.{l}.ffn")
    norm("enc.ln_f")
    for l in range(dims.dec_layers):
        norm(f"dec.{l}.ln1"); attn(f"dec.{l}.self"); norm(f"dec.{l}.ln_cross"); attn(f"dec.{l}.cross")
        norm(f"dec.{l}.ln2"); ffn(f"dec.{l}.ffn")
    norm("dec.ln_f")
    # the last cross-attention: match positions, copy the token half of the encoder memory
    cg = torch.Generator().manual_seed(seed + 9)
    q1, q2 = (torch.linalg.qr(torch.randn((d, d), generator=cg))[0].cuda() for _ in range(2))
    match, copy = q1 * 8.0, q2.clone()
    match[:, half:] = 0
    copy[:, :half] = 0
    last = f"dec.{dims.dec_layers - 1}.cross"
    w[last + ".q.w"], w[last + ".k.w"] = match, match.clone()
    w[last + ".v.w"], w[last + ".o.w"] = copy, 8.0 * copy.t()
    if drafter:
        u = torch.arange(7, dims.vocab - 1, 7, device="cuda")
        w["embed"][u] = w["embed"][u + 1] / 1.3
    if bf16:                                             # matrices hold bf16 values, as a bf16 checkpoint does
        w = {n: a.bfloat16().float() if a.ndim == 2 and not n.startswith("pos_") else a for n, a in w.items()}
    return {n: a.cpu().numpy() for n, a in w.items()}


def _handle(pair, **caps):
    v, d = PAIRS[pair]
    bf16 = pair != "tiny"
    if pair not in _weights:
        _weights[pair] = _model(v, 1001, False, bf16), _model(d, 1002, True, bf16)
    wv, wd = _weights[pair]
    return binding.SpecDec(v, wv, d, wd, bf16=bf16, activation="gelu" if pair == "bart" else "relu", **caps)


_kept = {}                          # the handle that the program decodes with, one at a time


def _shared_handle(pair, cached, **caps):
    key = (pair, cached) + tuple(sorted(caps.items()))
    if key not in _kept:
        _kept.clear()               # (closed by its destructor once its last state is gone)
        sd = _handle(pair, **caps)
        if cached:
            sd.set_option("drafter_prefix_causal", 1)
        _kept[key] = sd
    return _kept[key]


# ------------------------------------------------------------------------------------------------ inputs
def _lengths(c):
    """Source lengths: evenly spread over lo..hi, in a fixed shuffled order, so that they are the case's and not the seed's."""
    b, lo, hi = c["batch"], c["lo"], c["hi"]
    n = [hi] if b == 1 else [lo + (hi - lo) * i // (b - 1) for i in range(b)]
    random.Random(5).shuffle(n)
    return n


def _sources(seed, lens, vocab):
    """Zipf ids ending in [EOS], right-padded: (ids [B, max], lengths [B])."""
    rng = np.random.default_rng(seed)
    flat = W.zipf_ids(rng, sum(lens), vocab)
    out = np.full((len(lens), max(lens)), W.PAD_ID, np.int32)
    at = 0
    for b, n in enumerate(lens):
        out[b, :n] = flat[at:at + n]
        out[b, n - 1] = W.EOS_ID
        at += n
    return out, np.asarray(lens, np.int32)


def _max_tgt(c):
    return [min(int(1.2 * n) + 10, 128) if c["pair"] != "tiny" else 32 for n in _lengths(c)]


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "accept":
        g = torch.Generator(device="cuda").manual_seed(seed)
        logits = torch.randn((c["batch"], c["k"] + 1, c["vocab"]), generator=g, device="cuda") * 3.0
        best = logits[:, :-1].argmax(-1).to(torch.int32)
        wrong = torch.rand(best.shape, generator=g, device="cuda") < P_WRONG
        other = torch.randint(0, c["vocab"], best.shape, generator=g, device="cuda", dtype=torch.int32)
        i32 = dict(dtype=torch.int32, device="cuda")
        return dict(c=c, logits=logits, drafts=torch.where(wrong, other, best).contiguous(),
                    acc=torch.zeros(c["batch"], **i32), bif=torch.zeros(c["batch"], **i32))
    vocab = PAIRS[c["pair"]][0].vocab
    if kind in ("generate", "first_tokens"):
        src, lens = _sources(seed, _lengths(c), vocab)
        mt = np.asarray(_max_tgt(c), np.int32)
        sd = _shared_handle(c["pair"], c.get("cached", False), k_max=max(c["k"], 1), max_batch=c["batch"], max_src=src.shape[1], max_tgt=int(mt.max()))
        if c.get("host"):
            pin = lambda a: torch.from_numpy(a).pin_memory()  # noqa: E731
            return dict(c=c, sd=sd, src=pin(src), lens=pin(lens), mt=pin(mt),
                        out=torch.zeros((c["batch"], int(mt.max())), dtype=torch.int32).pin_memory(),
                        n=torch.zeros(c["batch"], dtype=torch.int32).pin_memory())
        return dict(c=c, sd=sd, src=_dev(src), lens=_dev(lens), mt=_dev(mt))
    # verify / draft: a session with `prefix` committed tokens (the source's own), so the handle is this state's
    b, k, j = c["batch"], c["k"], c["prefix"]
    src, lens = _sources(seed, [j + k + 8] * b, vocab)
    sd = _handle(c["pair"], k_max=k, max_batch=b, max_src=src.shape[1], max_tgt=j + k + 2)
    if c.get("cached"):
        sd.set_option("drafter_prefix_causal", 1)
    sd.encode(_dev(src), _dev(lens))
    if kind == "draft" and c.get("cached"):
        sd.draft(k)
    done = 0
    while done < j:
        n = min(k, j - done - 1)
        block = np.zeros((b, k), np.int32)
        block[:, :n] = src[:, done:done + n]
        sd.verify(_dev(block), 1, 0.0)
        sd.commit(_dev(np.full(b, n)), _dev(src[:, done + n]))
        done += n + 1
        if kind == "draft" and c.get("cached"):
            sd.draft(k)             # the drafter's cache follows the prefix, as in a decoding loop
    drafts = src[:, j:j + k].copy()
    rej = np.random.default_rng(seed + 1).geometric(P_WRONG, size=b)
    for i in range(b):              # one wrong draft per sequence, at the mean distance of the paper's regime
        if rej[i] <= k:
            drafts[i, rej[i] - 1] = 4 + (drafts[i, rej[i] - 1] + 13) % (vocab - 4)
    return dict(c=c, sd=sd, drafts=_dev(drafts), acc=_dev(np.zeros(b)), bif=_dev(np.zeros(b)))


def run(s):
    c, kind = s["c"], s["c"]["kind"]
    if kind == "accept":
        if c["static"]:
            return binding.accept_scan_static(s["logits"], s["drafts"], BETA, TAU, s["acc"], s["bif"])
        return binding.accept_scan(s["logits"], s["drafts"], BETA, TAU)
    sd = s["sd"]
    if kind == "verify":
        return sd.verify_raw(s["drafts"], BETA, TAU, s["acc"], s["bif"])
    if kind == "draft":
        return sd.draft(c["k"])
    if kind == "first_tokens":
        sd.encode(s["src"], s["lens"], s["mt"])
        sd.verify(sd.draft(c["k"]), BETA, TAU)
        sd.commit()
        return sd.output()
    if c["host"]:
        sd.generate_host(s["src"], s["lens"], s["mt"], s["out"], s["n"], c["k"], BETA, TAU)
        return s["out"], s["n"]
    out, n, stats = sd.generate(s["src"], s["lens"], s["mt"], c["k"], BETA, TAU)
    return out, n, stats["emitted"]


# ------------------------------------------------------------------------------------------------ work and tolerance
def _tokens_per_iteration(k):
    """Accepted drafts and the verifier's own token, when each draft is wrong with probability P_WRONG."""
    q = 1.0 - P_WRONG
    return 1.0 + sum(q ** i for i in range(1, k + 1))


def _encode(dims, lens):
    d, f = dims.d_model, dims.d_ffn
    layer = 4 * d * d + 2 * d * f
    params = dims.enc_layers * layer + dims.dec_layers * 2 * d * d
    flops = sum(2.0 * n * params + 4.0 * n * n * d * dims.enc_layers for n in lens)
    return params, sum(lens) * (4 * d + dims.dec_layers * 2 * d), flops        # parameters, values read and written, flops


def _decode(dims, rows, keys, mask_rows=None):
    """One decoder pass: `rows`, and for each of them `keys` self- and cross-attended positions in all."""
    d, f, layers = dims.d_model, dims.d_ffn, dims.dec_layers
    layer = 6 * d * d + 2 * d * f
    top = rows if mask_rows is None else mask_rows       # (the drafter's last layer and the vocabulary: [MASK] rows only)
    params = layers * layer + dims.vocab * d
    flops = 2.0 * (rows * (layers - 1) + top) * layer + 2.0 * top * dims.vocab * d + 4.0 * keys * d * (rows * (layers - 1) + top)
    return params, flops


def _step(c, kind, b, prefix, src_len):
    """Bytes and flops of one verify or draft step of `b` sequences with `prefix` committed tokens each."""
    v, d = PAIRS[c["pair"]]
    size, k = 4 if c["pair"] == "tiny" else 2, c["k"]
    if kind == "verify":
        params, flops = _decode(v, b * (k + 1), prefix + (k + 1) / 2 + src_len)
        kv = b * v.dec_layers * (prefix + k + 1 + src_len) * 2 * v.d_model
    else:
        rows = k + 1 if c.get("cached") else prefix + 1 + k
        params, flops = _decode(d, b * rows, prefix + 1 + k + src_len, b * k)
        kv = b * d.dec_layers * (src_len + (prefix if c.get("cached") else 0)) * 2 * d.d_model
    return (params + kv) * size, flops


def work(case):
    c = case
    if c["kind"] == "accept":       # rows up to the first rejected draft, fp32
        rows = c["batch"] * _tokens_per_iteration(c["k"])
        return {"bytes": rows * c["vocab"] * 4 + c["batch"] * (c["k"] + 2) * 4, "flops": rows * c["vocab"] * 3}
    if c["kind"] in ("verify", "draft"):
        bytes_, flops = _step(c, c["kind"], c["batch"], c["prefix"], c["prefix"] + c["k"] + 8)
        return {"bytes": bytes_, "flops": flops}
    lens, size, total_b, total_f = _lengths(c), 4 if c["pair"] == "tiny" else 2, 0.0, 0.0
    for m in PAIRS[c["pair"]][:1 if c["k"] == 0 else 2]:
        params, values, flops = _encode(m, lens)
        total_b += (params + values) * size
        total_f += flops
    # every step reads the weights of both decoders once: together with the caches they exceed what stays on the chip
    per = _tokens_per_iteration(c["k"])
    want = [min(n, t) for n, t in zip(lens, _max_tgt(c))]
    steps = 1 if c["kind"] == "first_tokens" else math.ceil(max(want) / per)
    for i in range(steps):
        live = [n for n, t in zip(lens, want) if t > i * per]
        for kind in ("verify",) if c["k"] == 0 else ("draft", "verify"):
            bytes_, flops = _step(c, kind, len(live), i * per, sum(live) / len(live))
            total_b += bytes_
            total_f += flops
    return {"bytes": total_b, "flops": total_f}


def tolerance(case):
    # token ids, lengths and accepted counts only; every decision that they rest on has a margin far above the rounding of the
    # logits, except that a tie between two near-equal logits of the tiny pair may fall either way
    return {"rel": 0.0, "differ": 0.005}
