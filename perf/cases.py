"""What is measured: the calls a decoding loop makes into the library, over the sizes it meets.

Every case holds a compiled grammar x vocabulary (the handle a program keeps), a batch of parser
states advanced through prefixes of sampled sentences, and fresh logits.  Prefixes, cut points and
logits come from the seed; grammars and prefix lengths are those of `workloads/`, batches 1-1024 and
vocabularies 512-262,145 those of the benchmark and of the paper's tokenizers (151,665 and 262,145
are odd: rows of contiguous logits are then not 16-byte aligned).

A pass that advances the states starts by restoring them with `psc_state_copy`, so it can be called
again; masking the same logits with the same masks again writes the same values.
"""
from __future__ import annotations

import collections
import functools
import math

import numpy as np
import torch

from paper_2608_03065_gb300 import psc
from workloads import grammars, sample

# grammar -> (rules, longest prefix in bytes, derivation depth, nesting bias, largest vocabulary)
GRAMMARS = {
    "arith": (grammars.arithmetic, 64, 40, 1.0, 1024),
    "json": (grammars.json_grammar, 512, 40, 1.0, 262145),
    "schema": (grammars.schema_json, 1024, 40, 1.0, 262145),
    "c": (grammars.c_like, 2048, 500, 4.0, 262145),
    "java": (grammars.java_like, 2048, 60, 1.0, 262145),
}
CAP = 256            # parser stack capacity, as in the benchmark
TEXTS = 32           # sentences the prefixes of a grammar are cut from
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


# ------------------------------------------------------------------ grammar, vocabulary, prefixes
@functools.lru_cache(maxsize=None)
def _grammar(name):
    return GRAMMARS[name][0]()


@functools.lru_cache(maxsize=None)
def _pieces(name):
    """Token strings of a grammar's vocabularies, the most frequent first: single bytes, the
    pre-tokens of sampled sentences and their prefixes, numbers and indentation runs."""
    rng = np.random.default_rng([101, len(name)])
    sampler = sample.SentenceSampler(_grammar(name), max_depth=30)
    count = collections.Counter()
    size = 0
    while size < 1 << 17:
        text, _ = sampler.text(rng, 4096)
        size += len(text)
        for m in sample.PRETOKEN.finditer(text):
            p = m.group(0)
            count[p] += 5
            for k in range(2, len(p)):
                count[p[:k]] += 1
    ranked = [p for p, _ in sorted(count.items(), key=lambda kv: (-kv[1], kv[0])) if len(p) <= 24]
    more = [str(i).encode() for i in range(1000)]
    more += [lead + b" " * w for w in range(2, 17) for lead in (b"", b"\n")]
    return list(dict.fromkeys(sample.PRINTABLE + ranked + more))


@functools.lru_cache(maxsize=None)
def _vocabulary(name, V):
    """V unique byte strings in a shuffled order; words with at most one leading non-letter after
    the grammar's own pieces, the end-of-sequence token (no bytes) last."""
    rng = np.random.default_rng([102, V])
    toks = dict.fromkeys(_pieces(name)[:V - 1])
    lead = [b"", b" ", b" ", b" ", b".", b"(", b"_", b'"']
    while len(toks) < V - 1:
        n = V - 1 - len(toks)
        letters = rng.integers(ord("a"), ord("z") + 1, 10 * n, dtype=np.uint8).tobytes()
        for i, (w, k) in enumerate(zip(rng.integers(2, 11, n).tolist(), rng.integers(0, len(lead), n).tolist())):
            toks[lead[k] + letters[10 * i:10 * i + w]] = None
    toks = list(toks)
    return [toks[i] for i in rng.permutation(V - 1).tolist()] + [b""]


@functools.lru_cache(maxsize=None)
def _handle(name, V):
    return psc.psc_compile(_grammar(name).text(), _vocabulary(name, V), V - 1)


@functools.lru_cache(maxsize=None)
def _tokenized(name, V):
    """Sampled sentences of the grammar (cut at up to the longest prefix) as token ids."""
    spec, (_, longest, depth, bias, _) = _grammar(name), GRAMMARS[name]
    texts = sample.build_prefixes(spec, TEXTS, longest // 2, longest, [103, len(name)], max_depth=depth, nest_bias=bias)
    ids = {t: i for i, t in enumerate(_vocabulary(name, V)) if t}
    out = []
    for text in texts:
        row, i = [], 0
        while i < len(text):
            n = next(n for n in range(min(24, len(text) - i), 0, -1) if text[i:i + n] in ids)
            row.append(ids[text[i:i + n]])
            i += n
        out.append(row)
    return out


# ------------------------------------------------------------------ cases
def listed():
    return [
        # one pass of the fused masking and greedy choice on the tiny arithmetic grammar: the smallest call
        dict(name="arith_b8_choose", op="choose", grammar="arith", V=512, B=8, dtype="f32", pad=0, steps=1),
        # one interactive sequence decoded from Python, call by call
        dict(name="json_b1_decode", op="decode", grammar="json", V=32000, B=1, dtype="bf16", pad=0, steps=8),
        # one interactive sequence in a program grammar, the decode loop captured in a CUDA graph
        dict(name="c_b1_graph", op="graph", grammar="c", V=262144, B=1, dtype="bf16", pad=0, steps=16),
        # a server's batch with continuous batching: before each step one finished row starts anew
        dict(name="schema_b32_serve", op="serve", grammar="schema", V=128256, B=32, dtype="bf16", pad=0, steps=4),
        # the benchmark's large batch
        dict(name="c_b1024_decode", op="decode", grammar="c", V=262144, B=1024, dtype="bf16", pad=0, steps=2),
        # engines that hold logits in 32 bits
        dict(name="json_b128_f32_decode", op="decode", grammar="json", V=151936, B=128, dtype="f32", pad=0, steps=2),
        # an odd vocabulary, logits as the model's head leaves them: contiguous rows, most not 16-byte aligned
        dict(name="json_b64_odd_decode", op="decode", grammar="json", V=262145, B=64, dtype="bf16", pad=0, steps=2),
        # an engine that samples itself: bitmask out, bitmask applied, its tokens fed back
        dict(name="schema_b256_engine", op="engine", grammar="schema", V=128256, B=256, dtype="bf16", pad=0, steps=2),
        # a bitmask that the caller has, applied to odd rows of 32-bit logits
        dict(name="b16_odd_apply", op="apply", grammar="json", V=151665, B=16, dtype="f32", pad=0, steps=1),
        # the three calls of a step apart: masking, greedy choice, advance
        dict(name="c_b64_apart", op="apart", grammar="c", V=262144, B=64, dtype="bf16", pad=0, steps=2),
        # prompts and forced tokens taken in, in a Java-sized grammar: one advance per token, then the masks
        dict(name="java_b64_prefill", op="prefill", grammar="java", V=128256, B=64, dtype="bf16", pad=0, steps=64),
        # parser states that the caller holds, masked without allocating
        dict(name="c_b256_noalloc", op="noalloc", grammar="c", V=262144, B=256, dtype="bf16", pad=0, steps=1),
    ]


def draw(rng):
    op = rng.choice(["choose", "decode", "decode", "decode", "graph", "serve", "engine", "apply", "apart", "prefill", "noalloc"])
    grammar = rng.choice(["json", "json", "schema", "c", "java", "arith"])
    most = GRAMMARS[grammar][4]
    V = rng.choice([32000, 50257, 128256, 151665, 151936, 262144, 262145, 0, 0, 0, 0])
    if not 0 < V <= most:
        V = int(math.exp(rng.uniform(math.log(512), math.log(most))))
    dtype = rng.choice(["bf16", "bf16", "f32"])
    pad = rng.choice([0, 0, 64])       # rows contiguous, or padded to a multiple of 64 columns
    steps = {"choose": 1, "apply": 1, "noalloc": 1, "prefill": rng.randint(8, 64), "graph": rng.randint(2, 16)}.get(op) or rng.randint(1, 4)
    row = V * (2 if dtype == "bf16" else 4) * (1 if op == "prefill" else steps)
    B = int(math.exp(rng.uniform(0, math.log(min(1024, max(1, (1 << 29) // row)) + 0.99))))
    return dict(op=op, grammar=grammar, V=V, B=B, dtype=dtype, pad=pad, steps=steps)


def prepare(case, seed):
    name, V, B, op = case["grammar"], case["V"], case["B"], case["op"]
    steps, dtype = case["steps"], DTYPES[case["dtype"]]
    rng = np.random.default_rng([104, seed])
    gen = torch.Generator(device="cuda").manual_seed(seed)
    W = (V + 31) // 32
    ld = V if not case["pad"] else -(-V // case["pad"]) * case["pad"]
    s = {"op": op, "steps": steps, "V": V, "B": B}

    def logits():
        return (torch.randn(B, ld, generator=gen, device="cuda", dtype=dtype) * math.sqrt(2))[:, :V]

    if op == "apply":
        # masks as grammars make them: rows from nearly empty to nearly full
        keep = torch.from_numpy(rng.random(B).astype(np.float32)).cuda()
        bits = torch.rand(B, 32 * W, generator=gen, device="cuda") < keep[:, None]
        bits[:, V:] = False
        word = (bits.view(B, W, 32).long() << torch.arange(32, device="cuda")).sum(-1)
        s["logits"], s["bitmask"] = [logits()], word.to(torch.int32)
        s["first"] = s["logits"][0].clone()
        return s

    # rows at random places of the sampled sentences; the tokens that follow are the forced ones
    h, texts = _handle(name, V), _tokenized(name, V)
    forced = steps if op in ("engine", "prefill") else 0
    at = rng.integers(0, TEXTS, B)
    cut = [int(rng.integers(1, max(2, len(texts[t]) - forced))) for t in at]
    tokens = np.full((max(cut) + forced, B), -1, dtype=np.int32)
    for b, (t, n) in enumerate(zip(at, cut)):
        tokens[:n, b] = texts[t][:n]
        tail = texts[t][n:n + forced]
        tokens[max(cut):max(cut) + len(tail), b] = tail
    tokens = torch.from_numpy(tokens).cuda()
    st = psc.psc_state_init(h, B, CAP)
    for row in tokens[:max(cut)]:
        psc.psc_advance(h, st, row)
    s.update(h=h, kept=st, forced=[t.clone() for t in tokens[max(cut):]])
    if op == "noalloc":
        got = psc.psc_states_download(st)
        s["arrays"] = [torch.from_numpy(got[k]).cuda() for k in ("q", "depth", "status")]
        s["arrays"].append(torch.from_numpy(got["stack"].view(np.int16)).cuda())
    if op not in ("choose", "noalloc"):
        s["states"] = psc.psc_state_init(h, B, CAP)
    if op != "prefill":
        s["logits"] = [logits() for _ in range(steps)]
    s["bitmask"] = [torch.zeros(B, W, dtype=torch.int32, device="cuda") for _ in range(1 if op == "prefill" else steps)]
    s["tokens"] = [torch.zeros(B, dtype=torch.int32, device="cuda") for _ in range(steps)]
    s["status"] = torch.zeros(B, dtype=torch.int32, device="cuda")
    s["rows"] = [torch.from_numpy(rng.integers(0, B, 1).astype(np.int32)).cuda() for _ in range(steps)]
    if op == "graph":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _decode(s)
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _decode(s)
    return s


def _decode(s):
    h, st = s["h"], s["states"]
    psc.psc_state_copy(st, s["kept"])
    for x, bits, tok in zip(s["logits"], s["bitmask"], s["tokens"]):
        psc.psc_decode_step(h, st, x, tok, bits, s["status"])


def run(s):
    op = s["op"]
    if op == "graph":
        s["graph"].replay()
        return s["logits"], s["bitmask"], s["tokens"], s["status"]
    if op == "decode":
        _decode(s)
        return s["logits"], s["bitmask"], s["tokens"], s["status"]
    if op == "apply":
        psc.psc_apply_mask(s["logits"][0], s["bitmask"], s["B"], s["V"])
        return s["logits"]
    h = s["h"]
    if op == "choose":
        psc.psc_fill_apply_argmax(h, s["kept"], s["logits"][0], s["tokens"][0], s["bitmask"][0])
        return s["logits"], s["bitmask"], s["tokens"]
    if op == "noalloc":
        psc.psc_fill_apply_noalloc(h, *s["arrays"], s["logits"][0], s["bitmask"][0])
        return s["logits"], s["bitmask"]
    st = s["states"]
    psc.psc_state_copy(st, s["kept"])
    if op == "prefill":
        for tok in s["forced"]:
            psc.psc_advance(h, st, tok, s["status"])
        psc.psc_fill_mask(h, st, s["bitmask"][0])
        return s["bitmask"], s["status"]
    if op == "serve":
        for x, bits, tok, rows in zip(s["logits"], s["bitmask"], s["tokens"], s["rows"]):
            psc.psc_state_reset(st, rows)
            psc.psc_decode_step(h, st, x, tok, bits, s["status"])
    elif op == "engine":
        for x, bits, tok in zip(s["logits"], s["bitmask"], s["forced"]):
            psc.psc_fill_mask(h, st, bits)
            psc.psc_apply_mask(x, bits, s["B"], s["V"])
            psc.psc_advance(h, st, tok, s["status"])
    else:
        for x, bits, tok in zip(s["logits"], s["bitmask"], s["tokens"]):
            psc.psc_fill_apply(h, st, x, bits)
            psc.psc_argmax_masked(h, st, x, tok)
            psc.psc_advance(h, st, tok, s["status"])
    return s["logits"], s["bitmask"], s["tokens"], s["status"]


def work(case):
    """Logits read and written once and the bitmask written once per step; token ids and statuses."""
    B, V, steps = case["B"], case["V"], case["steps"]
    mask = B * ((V + 31) // 32) * 4
    if case["op"] == "prefill":
        return {"bytes": steps * B * 4 + mask + B * 4, "flops": 0}
    return {"bytes": steps * (2 * B * V * (2 if case["dtype"] == "bf16" else 4) + mask + 8 * B), "flops": 0}


def tolerance(case):
    """Masks, tokens and statuses are whole numbers, and an allowed logit keeps its bits."""
    return "exact"


def exact(case, seed):
    """The masked logits where the bitmask is an input.  In every other case the outputs are the
    grammar's decisions, which a brute force over the vocabulary takes far over 20 seconds for."""
    if case["op"] != "apply":
        return None
    s = prepare(case, seed)
    bits = (s["bitmask"].long()[:, :, None] >> torch.arange(32, device="cuda")) & 1
    keep = bits.reshape(s["B"], -1)[:, :s["V"]].bool()
    return [torch.where(keep, s["first"].double(), -math.inf)]
