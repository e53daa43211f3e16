"""The one-launch set-up of a single trie (child links, compile tables, cleared
transition table and summary) at sizes around its warps' and CTAs' shares."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2608_12574_gb300 import triemask as T
from paper_2608_12574_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 255, 256, 257, 2049, 40000])
def test_setup_sizes(n):
    """A trie of exactly n nodes: masks and moves equal the oracle's, from
    memory that an earlier trie of the same size has used."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    oracle.build()
    rng = np.random.default_rng(n)
    toks = [bytes([b]) for b in range(256)] + [bytes(rng.integers(97, 100, k)) for k in (2, 3, 5, 9, 17)] + [b""]
    vb, vo = W.pack(toks)
    V = len(toks)
    for turn in range(2):
        strings, nodes = [], {b""}
        while len(nodes) < n:  # random strings, the last one cut to fit
            s = bytes(rng.integers(97, 100, rng.integers(1, 40)))
            new = [s[:k] for k in range(1, len(s) + 1) if s[:k] not in nodes][:n - len(nodes)]
            nodes.update(new)
            strings.append(new[-1] if new else s)
        sb, so = W.pack(strings)
        h, ot, ov = T.trie_build(sb, so), oracle.Trie(sb, so), oracle.Vocab(vb, vo)
        assert h.num_nodes == n
        m = T.alloc_mask(h, V, "cuda")
        T.trie_compile_masks(h, vb, vo, V, m)
        assert np.array_equal(m.cpu().numpy().view(np.uint32), oracle.mask_all(ot, ov))
        s0 = rng.integers(0, n, 500).astype(np.int32)
        t0 = rng.integers(97, 262, 500).astype(np.int32)
        want, _ = oracle.advance(ot, ov, s0, t0)
        ds = torch.as_tensor(s0, device="cuda")
        T.trie_advance(h, ds, torch.as_tensor(t0, device="cuda"))
        assert np.array_equal(ds.cpu().numpy(), want)
        h.destroy()


@pytest.mark.parametrize("n", [16384, 16385])
def test_one_block_limit(n):
    """The largest trie that gets the arrays of its first dense compile in one
    block and the smallest that gets them apart: a compile, one with a larger
    vocabulary (whose segment summary is larger), and the first one again. Masks
    equal the pairwise derivation's, applies (which read the summary) the mask's."""
    import itertools

    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(n)
    strings, nodes = [], {b""}
    while len(nodes) < n:
        s = bytes(rng.integers(97, 100, rng.integers(1, 60)))
        new = [s[:k] for k in range(1, len(s) + 1) if s[:k] not in nodes][:n - len(nodes)]
        nodes.update(new)
        strings.append(new[-1] if new else s)
    h = T.trie_build(*W.pack(strings))
    assert h.num_nodes == n
    words = [bytes(t) for k in range(1, 11) for t in itertools.product(b"abc", repeat=k)]
    states = np.concatenate([[-1, -2, n], rng.integers(0, n, 40)]).astype(np.int32)
    ds = torch.as_tensor(states, device="cuda")
    for V in (33_000, 70_001, 33_000):
        vb, vo = W.pack(words[:V - 1] + [b""])
        m, want = T.alloc_mask(h, V, "cuda"), T.alloc_mask(h, V, "cuda")
        T.trie_compile_masks(h, vb, vo, V, m)
        T.trie_compile_masks_pairwise(h, vb, vo, V, want)
        assert torch.equal(m, want)
        rows = m[ds.clamp(0, n - 1).long()].cpu().numpy().view(np.uint8)
        bits = np.unpackbits(rows, axis=1, bitorder="little")[:, :V].astype(bool)
        bits[(states < 0) | (states >= n)] = False
        bits[(states < 0) | (states >= n), V - 1] = True
        x = torch.randn((len(states), V), device="cuda")
        ref = np.where(bits, x.cpu().numpy(), -np.inf)
        T.trie_apply_mask(h, x, ds)
        assert np.array_equal(x.cpu().numpy(), ref)
    h.destroy()
