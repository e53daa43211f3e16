"""The cases that this library's speed is measured on.

Each case is a piece of work that a serving program has the library do, through
its Python entry points, on sets, vocabularies and batches of the sizes that
the repository's workloads name, from the smallest (one request, 100 strings,
32,000 tokens) to the largest (74,719 strings, 262,144 tokens). The kinds:

decode   the decode loop of a batch on a compiled schema: step 0 masks its
         logits, every later step advances the states by the tokens sampled
         from the step before and masks its own logits.
compile  the masks of a schema whose handle is kept, into memory set aside for
         the masks of whichever schema is active (they are compiled again each
         time the schema comes back).
schema   a schema that the server has not seen: its trie built from the
         strings, uploaded, its masks compiled into that memory, and the
         handle released.
forest   a batch of requests that each bring their own set: one forest built
         on the GPU, its valid lists, the decode loop, the release.
lazy     the decode loop without a mask of all nodes: rows computed when a
         state first reaches them, with or without a row cache.
format   a fixed format (a date, a UUID): its masks compiled, then decoded.

Sampled tokens are random tokenizations of random members of the sets, so
every sampled token is one that the mask allows, as a sampler's are; a request
that has spelled its string samples end-of-sequence from then on. Logits are
returned as the integers of their bits: allowed ones have to keep every bit.
"graph" loops are captured once and replayed, as servers do where a step's
launches would cost more than its kernels; the others are called step by step.
"""
from __future__ import annotations

import bisect
import functools

import numpy as np
import torch

from paper_2608_12574_gb300 import triemask as T
from paper_2608_12574_gb300 import workloads as W

_TYPES = {"f32": (torch.float32, torch.int32), "bf16": (torch.bfloat16, torch.int16)}
_SIZE = {"f32": 4, "bf16": 2}
_FINISHED = -2


def listed():
    return [
        # one interactive request that picks one of 100 tools: latency of the smallest call
        dict(name="decode-K100-V32000-B1-f32", kind="decode", sets="tools", K=100, V=32000, B=1, steps=32,
             dtype="f32", graph=True),
        # a mid-sized batch with a vocabulary of an odd size (added tokens, no padding): rows of
        # logits that start at any two-byte boundary
        dict(name="decode-K1000-V128011-B64-bf16", kind="decode", sets="tools", K=1000, V=128011, B=64, steps=16,
             dtype="bf16", graph=False),
        # a full batch on a code list, as a classification service decodes it
        dict(name="decode-K10000-V152064-B256-bf16", kind="decode", sets="codes", K=10000, V=152064, B=256,
             steps=8, dtype="bf16", graph=True),
        # masks of a tool list small enough that launches and dependent loads are what counts
        dict(name="compile-K100-V32000", kind="compile", sets="tools", K=100, V=32000),
        # masks of a code list, 0.44 GB
        dict(name="compile-K10000-V152064", kind="compile", sets="codes", K=10000, V=152064),
        # the largest: every code of a coding system, 3.6 GB of masks
        dict(name="compile-K74719-V262144", kind="compile", sets="codes", K=74719, V=262144),
        # a new tool list arrives with a request
        dict(name="schema-K1000-V128000", kind="schema", sets="tools", K=1000, V=128000),
        # every request of a full batch has its own 300-2,000 strings
        dict(name="forest-M256-V128000-bf16", kind="forest", M=256, k_lo=300, k_hi=2000, V=128000, steps=32,
             dtype="bf16"),
        # a small batch of such requests, an odd vocabulary, logits kept in 32 bits
        dict(name="forest-M16-V50021-f32", kind="forest", M=16, k_lo=50, k_hi=700, V=50021, steps=16, dtype="f32"),
        # no memory for the masks at all: every row computed in the step that needs it
        dict(name="lazy-K10000-V152064-B256-bf16", kind="lazy", sets="codes", K=10000, V=152064, B=256, steps=8,
             dtype="bf16", cache=0, graph=True),
        # the largest set without its 3.6 GB of masks: the rows in use are cached
        dict(name="lazy-K74719-V262144-B64-f32", kind="lazy", sets="codes", K=74719, V=262144, B=64, steps=8,
             dtype="f32", cache=4096, graph=False),
        # an identifier field
        dict(name="format-uuid-V152064-B64-bf16", kind="format", format="UUID v4", V=152064, B=64, steps=16,
             dtype="bf16"),
    ]


def _spread(rng, lo, hi):
    """A whole number, spread over the logarithm of lo..hi."""
    return min(hi, int(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["decode", "decode", "compile", "schema", "forest", "lazy", "format"])
    V = _spread(rng, 32000, 262144)
    if rng.random() < 0.6:  # most vocabularies are padded to a multiple of 64, the others are of any size
        V = max(32000, V // 64 * 64)
    sets = rng.choice(["tools", "codes"])
    K = _spread(rng, 100, 4000 if sets == "tools" else 74719)
    B = _spread(rng, 1, 256)
    dtype = rng.choice(["f32", "bf16"])
    case = dict(kind=kind, V=V)
    if kind in ("decode", "lazy"):
        case.update(sets=sets, K=K, B=B, steps=rng.randrange(4, 17), dtype=dtype, graph=rng.random() < 0.5)
    if kind == "lazy":
        case.update(cache=rng.choice([0, _spread(rng, 64, 4096)]))
    if kind in ("compile", "schema"):
        case.update(sets=sets, K=K)
    if kind == "forest":
        k_lo = _spread(rng, 20, 500)
        case.update(M=B, k_lo=k_lo, k_hi=_spread(rng, k_lo, 2000), steps=rng.randrange(4, 33), dtype=dtype)
    if kind == "format":
        case.update(format=rng.choice(sorted(W.FORMATS)), B=B, steps=rng.randrange(4, 17), dtype=dtype)
    if "steps" in case:  # at most 2 GB of logits
        case["steps"] = min(case["steps"], max(2, int(2e9 / (B * V * _SIZE[dtype]))))
    return case


# ------------------------------------------------------------------- inputs

@functools.lru_cache(maxsize=6)
def _vocab(sets, V):
    """A tokenizer: (bytes, offsets, {token bytes: id}, longest token). One per kind of set and size."""
    if sets == "tools":
        spec = W.VocabSpec(V=V, max_len=16, substr_frac=0.30, run_frac=0.0, run_len=(2, 4), upper=False, mixed=False)
        vb, vo = W.byte_vocab(1, spec, substr_src=W.tool_stems(1, 200))
    else:
        spec = W.VocabSpec(V=V, max_len=16, substr_frac=0.0, run_frac=0.20, run_len=(2, 4), upper=True, mixed=False)
        vb, vo = W.byte_vocab(3, spec)
    ids = {t: i for i, t in enumerate(W.unpack(vb, vo)[:-1])}
    return vb, vo, ids, max(len(t) for t in ids)


@functools.lru_cache(maxsize=1)
def _pool():
    return W.tool_names(5, 20000, 800)


def _strings(case, seed):
    if case["sets"] == "tools":
        return W.tool_names(seed + 100, case["K"], max(40, case["K"] // 5))
    return W.icd_codes(seed + 100, case["K"], 4 if case["K"] <= 20000 else 3)


def _request_sets(case, seed):
    rng = np.random.default_rng([seed, 7])
    pool, sets = _pool(), []
    for _ in range(case["M"]):
        pick = np.sort(rng.choice(len(pool), int(rng.integers(case["k_lo"], case["k_hi"] + 1)), replace=False))
        sets.append([pool[i] for i in pick])
    return sets


def _spell(s, ids, longest, eos, steps, rng):
    """`steps` tokens that spell s by a random tokenization, then end-of-sequence."""
    out, at = [], 0
    while at < len(s) and len(out) < steps:
        fits = [k for k in range(1, min(longest, len(s) - at) + 1) if s[at:at + k] in ids]
        k = fits[int(rng.integers(len(fits)))]
        out.append(ids[s[at:at + k]])
        at += k
    return out + [eos] * (steps - len(out))


def _member(pattern, rng):
    pick = {"#": "0123456789", "x": "0123456789abcdef", "y": "89ab"}
    return "".join(c if c not in pick else pick[c][int(rng.integers(len(pick[c])))] for c in pattern).encode()


def _decode_inputs(case, seed, members):
    """Logits of every step ([steps, B * V and a little room], each step's start aligned as an
    allocator's blocks are), and the tokens int32[steps, B] that spell the members."""
    B, V, steps = len(members), case["V"], case["steps"]
    _, _, ids, longest = _vocab(case.get("sets", "tools"), V)
    rng = np.random.default_rng([seed, 9])
    tokens = np.array([_spell(m, ids, longest, V - 1, steps, rng) for m in members], np.int32).T.copy()
    g = torch.Generator(device="cuda")
    g.manual_seed(1000 + seed)
    buf = torch.randn(steps, (B * V + 127) // 128 * 128, generator=g, device="cuda", dtype=_TYPES[case["dtype"]][0])
    return buf.mul_(2.0), torch.from_numpy(tokens).cuda()


def _members(case, seed, strings):
    rng = np.random.default_rng([seed, 8])
    if case["kind"] == "format":
        return [_member(W.FORMATS[case["format"]], rng) for _ in range(case["B"])]
    if case["kind"] == "forest":
        return [s[int(rng.integers(len(s)))] for s in strings]
    return [strings[int(rng.integers(len(strings)))] for _ in range(case["B"])]


def prepare(case, seed):
    kind, V = case["kind"], case["V"]
    vb, vo, _, _ = _vocab(case.get("sets", "tools"), V)
    st = {"kind": kind, "V": V, "vocab": (vb, vo), "voc": T.trie_vocab_create(vb, vo, V)}
    strings = None
    if kind == "forest":
        strings = _request_sets(case, seed)
        st["set"] = W.pack([x for s in strings for x in s])
        st["index"] = np.cumsum([0] + [len(s) for s in strings]).astype(np.int32)
        st["roots"] = torch.empty(case["M"], dtype=torch.int32, pin_memory=True)
    elif kind == "format":
        st["fmt"] = T.fmt_build(W.format_classes(W.FORMATS[case["format"]]))
        st["mask"] = T.fmt_alloc_mask(st["fmt"], V)
    else:
        strings = _strings(case, seed)
        st["set"] = W.pack(strings)
        if kind != "schema":
            st["h"] = T.trie_build(*st["set"])
    if kind == "decode":
        st["mask"] = T.alloc_mask(st["h"], V)
    if kind in ("compile", "schema"):
        st["masks"] = torch.zeros(_mask_rows(case), T.mask_words(V), dtype=torch.int32, device="cuda")
    if kind == "compile":
        st["mask"] = st["masks"][:st["h"].num_nodes]
    if kind in ("compile", "decode"):
        T.trie_compile_masks_vocab(st["h"], st["voc"], st["mask"])
    if kind == "lazy":
        T.trie_lazy_init(st["h"], vb, vo, V, case["cache"], case["B"])
    if "steps" in case:
        buf, st["tokens"] = _decode_inputs(case, seed, _members(case, seed, strings))
        B = st["tokens"].shape[1]
        st["logits"] = [row[:B * V].view(B, V) for row in buf]
        st["bits"] = buf.view(_TYPES[case["dtype"]][1])
        st["states"] = torch.zeros(case["steps"], B, dtype=torch.int32, device="cuda")
        st["err"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    if case.get("graph"):
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _loop(st)  # what the library does on a first call is done outside of the capture
        torch.cuda.current_stream().wait_stream(side)
        st["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st["graph"]):
            _loop(st)
    return st


# ---------------------------------------------------------------------- run

def _loop(st):
    apply, step = {"decode": (T.trie_apply_mask, T.trie_advance_apply),
                   "lazy": (T.trie_lazy_apply, T.trie_lazy_advance_apply),
                   "forest": (T.trie_apply_lists, T.trie_advance_apply_lists)}[st["kind"]]
    h, logits, states, tokens, err = st["h"], st["logits"], st["states"], st["tokens"], st["err"]
    apply(h, logits[0], states[0])
    for t in range(1, len(logits)):
        step(h, states[t - 1], tokens[t - 1], states[t], logits[t], err)


def run(st):
    kind = st["kind"]
    if kind == "compile":
        T.trie_compile_masks_vocab(st["h"], st["voc"], st["mask"])
        return st["masks"]
    if kind == "schema":
        h = T.trie_build(*st["set"])
        T.trie_compile_masks_vocab(h, st["voc"], st["masks"][:h.num_nodes])
        h.destroy_async()
        return st["masks"]
    if kind == "format":
        states = torch.zeros_like(st["states"][0])
        T.fmt_compile_masks(st["fmt"], *st["vocab"], st["V"], st["mask"])
        for t, logits in enumerate(st["logits"]):
            T.fmt_apply_mask(st["fmt"], logits, states)
            T.fmt_advance(st["fmt"], states, st["tokens"][t], st["err"])
        return [st["mask"], st["bits"], states, st["err"]]
    if kind == "forest":
        h = st["h"] = T.trie_build_many_device(*st["set"], st["index"])
        st["roots"].copy_(torch.from_numpy(h.roots()))
        st["states"][0].copy_(st["roots"], non_blocking=True)
        T.trie_compile_lists_vocab(h, st["voc"], count=False)
        _loop(st)
        h.destroy_async()
    elif "graph" in st:
        st["graph"].replay()
    else:
        _loop(st)
    return [st["bits"], st["states"], st["err"]]


# --------------------------------------------------------- work and tolerance

def _mask_rows(case):
    """Rows of the memory set aside for masks: more than the nodes of any set of the case."""
    return 16 * case["K"] + 64 if case["sets"] == "tools" else 3 * case["K"] + 4000


def _nodes_about(case):
    """Trie nodes, about: from the workloads' own counts (11.5 a name, 2.3 to 1.5 a code)."""
    if case["sets"] == "tools":
        return 12 * case["K"]
    return int(case["K"] * (2.3 if case["K"] <= 20000 else 1.5))


def work(case):
    kind, V = case["kind"], case["V"]
    n_bytes = 0
    if "steps" in case:  # every logit of the loop written once; allowed ones are a few
        n_bytes = case["steps"] * case.get("B", case.get("M", 0)) * V * _SIZE[case["dtype"]]
    if kind in ("compile", "schema"):  # the masks written once
        n_bytes = 4 * _nodes_about(case) * T.mask_words(V)
    if kind == "forest":  # the strings read, an entry of parent, label and end flag a node, 3 listed tokens a node
        names = case["M"] * (case["k_lo"] + case["k_hi"]) // 2
        n_bytes += names * 25 + names * 16 * (6 + 3 * 4)
    if kind == "format":
        n_bytes += 4 * (len(W.FORMATS[case["format"]]) + 1) * T.mask_words(V) + 16 * V
    return {"bytes": n_bytes, "flops": 0}


def tolerance(case):
    return "exact"  # bits, node ids and whole masks: there is nothing to round


# -------------------------------------------------------------------- exact

class _Set:
    """valid[p] and breadth-first node ids of a set of strings, by definition."""

    def __init__(self, strings, base=0):
        self.s = sorted(set(strings))
        self.len = np.array([len(x) for x in self.s])
        common = [0]
        for a, b in zip(self.s, self.s[1:]):
            n = 0
            while n < len(a) and n < len(b) and a[n] == b[n]:
                n += 1
            common.append(n)
        self.common = np.array(common)
        self.base = base
        self.nodes = 1 + int((self.len - self.common).sum())
        self.rows = {}

    def node(self, p):
        """The id of prefix p: the prefixes that are shorter, or as long and smaller, come first."""
        if not p:
            return self.base
        d, i = len(p), bisect.bisect_left(self.s, p)
        shorter = 1 + int((np.minimum(self.len, d - 1) - np.minimum(self.common, d - 1)).sum())
        return self.base + shorter + int(((self.len[:i] >= d) & (self.common[:i] < d)).sum())

    def valid(self, p, ids, longest, eos):
        got = self.rows.get(p)
        if got is None:
            lo = bisect.bisect_left(self.s, p)
            found = set()
            for x in self.s[lo:]:
                if not x.startswith(p):
                    break
                if x == p:
                    found.add(eos)
                for k in range(len(p) + 1, min(len(x), len(p) + longest) + 1):
                    t = ids.get(x[len(p):k])
                    if t is not None:
                        found.add(t)
            got = self.rows[p] = np.fromiter(found, np.int64, len(found))
        return got


def _masks(strings, case):
    """Every row of the masks, from every (node, token that ends there)."""
    _, _, ids, longest = _vocab(case["sets"], case["V"])
    nodes = sorted({x[:k] for x in strings for k in range(len(x) + 1)}, key=lambda p: (len(p), p))
    at, ends = {p: i for i, p in enumerate(nodes)}, set(strings)
    row, tok = [], []
    for i, p in enumerate(nodes):
        if p in ends:
            row.append(i)
            tok.append(case["V"] - 1)
        for k in range(1, min(len(p), longest) + 1):
            t = ids.get(p[len(p) - k:])
            if t is not None:
                row.append(at[p[:len(p) - k]])
                tok.append(t)
    row, tok, words = np.array(row), np.array(tok), T.mask_words(case["V"])
    key, where = np.unique(row * words + tok // 32, return_inverse=True)
    value = np.zeros(len(key), np.uint32)
    np.bitwise_or.at(value, where, np.uint32(1) << (tok % 32).astype(np.uint32))
    masks = torch.zeros(_mask_rows(case) * words, dtype=torch.int32, device="cuda")
    masks[torch.from_numpy(key).cuda()] = torch.from_numpy(value.view(np.int32)).cuda()
    return masks.view(-1, words)


def exact(case, seed):
    kind, V = case["kind"], case["V"]
    if kind in ("compile", "schema"):
        return _masks(_strings(case, seed), case)
    vb, vo, ids, longest = _vocab(case.get("sets", "tools"), V)
    eos, words, out_mask = V - 1, W.unpack(vb, vo), None
    if kind == "format":
        classes = np.unpackbits(W.format_classes(W.FORMATS[case["format"]]), axis=1, bitorder="little")
        L = len(classes)
        fits = [[] for _ in range(L + 1)]
        for t, i in ids.items():
            for p in range(L - len(t) + 1):
                if all(classes[p + j, c] for j, c in enumerate(t)):
                    fits[p].append(i)
        fits[L].append(eos)
        bits = np.zeros((L + 1, T.mask_words(V) * 32), np.uint8)
        for p in range(L + 1):
            bits[p, fits[p]] = 1
        out_mask = torch.from_numpy(np.packbits(bits, axis=1, bitorder="little").view(np.int32)).cuda()
        members = _members(case, seed, None)
    elif kind == "forest":
        strings = _request_sets(case, seed)
        sets, base = [], 0
        for s in strings:
            sets.append(_Set(s, base))
            base += sets[-1].nodes
        members = _members(case, seed, strings)
    else:
        strings = _strings(case, seed)
        sets = [_Set(strings)] * case["B"]
        members = _members(case, seed, strings)
    buf, tokens = _decode_inputs(case, seed, members)
    bits = buf.view(_TYPES[case["dtype"]][1])
    tok, B = tokens.cpu().numpy(), tokens.shape[1]
    masked = {"f32": -8388608, "bf16": -128}[case["dtype"]]  # the bits of -inf
    at, states = [b""] * B, np.zeros((case["steps"], B), np.int32)
    for t in range(case["steps"]):
        keep_r, keep_v = [], []
        for b in range(B):
            if at[b] is None:
                states[t, b], ok = _FINISHED, np.array([eos])
            elif kind == "format":
                states[t, b], ok = len(at[b]), np.array(fits[len(at[b])])
            else:
                states[t, b], ok = sets[b].node(at[b]), sets[b].valid(at[b], ids, longest, eos)
            keep_r.append(np.full(len(ok), b * V))
            keep_v.append(ok)
            at[b] = None if at[b] is None or tok[t, b] == eos else at[b] + words[tok[t, b]]
        keep = torch.from_numpy(np.concatenate(keep_r) + np.concatenate(keep_v)).cuda()
        kept = bits[t, keep]
        bits[t, :B * V] = masked
        bits[t, keep] = kept
    err = torch.zeros(1, dtype=torch.int32)
    if kind == "format":
        last = np.array([_FINISHED if a is None else len(a) for a in at], np.int32)
        return [out_mask, bits, torch.from_numpy(last), err]
    return [bits, torch.from_numpy(states), err]
