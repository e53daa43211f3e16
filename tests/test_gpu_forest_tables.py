"""A forest has no compile tables until a call reads them: lists first, then
the dense compile or the lazy rows of the same handle, and a synchronous and
a stream-ordered release of each."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2608_12574_gb300 import triemask as T
from paper_2608_12574_gb300 import workloads as W
from pins import random_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("then", ["masks", "lazy"])
@pytest.mark.parametrize("device_build", [False, True])
@pytest.mark.parametrize("lists_first", [False, True])
def test_tables_on_first_use(then, device_build, lists_first):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    oracle.build()
    strings, toks = random_case(91)
    sets = [strings, strings[:3] + [b""], [x + b"a" * 20 for x in strings]]
    sb, so = W.pack([x for s in sets for x in s])
    si = np.cumsum([0] + [len(s) for s in sets]).astype(np.int32)
    vb, vo = W.pack(toks)
    V = len(toks)
    h = (T.trie_build_many_device if device_build else T.trie_build_many)(sb, so, si)
    ov = oracle.Vocab(vb, vo)
    want = np.concatenate([oracle.mask_all(oracle.Trie(*W.pack(s)), ov) for s in sets])
    if lists_first:
        n = T.trie_compile_lists(h, vb, vo, V)
        assert n == int(np.unpackbits(want.view(np.uint8)).sum())
    if then == "masks":
        m = T.alloc_mask(h, V, "cuda")
        T.trie_compile_masks(h, vb, vo, V, m)
    else:
        T.trie_lazy_init(h, vb, vo, V, cache_rows=0, max_batch=h.num_nodes)
        m = T.trie_lazy_rows(h, torch.arange(h.num_nodes, dtype=torch.int32, device="cuda"), V)
    assert np.array_equal(m.cpu().numpy().view(np.uint32), want)
    (h.destroy_async if lists_first else h.destroy)()


def test_lazy_setup_behind_an_upload_on_another_stream():
    """The lists' upload waits on a busy stream while the lazy set-up asks for
    the tables, which come from the arrays that it uploads."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    oracle.build()
    strings, toks = random_case(91)
    sb, so = W.pack(strings + strings[:3])
    vb, vo = W.pack(toks)
    V = len(toks)
    h = T.trie_build_many(sb, so, np.array([0, len(strings), len(strings) + 3], np.int32))
    ov = oracle.Vocab(vb, vo)
    want = np.concatenate([oracle.mask_all(oracle.Trie(*W.pack(s)), ov) for s in (strings, strings[:3])])
    voc = T.trie_vocab_create(vb, vo, V)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)  # about 10 ms
        T.trie_compile_lists_vocab(h, voc, side, count=False)
    T.trie_lazy_init(h, vb, vo, V, cache_rows=0, max_batch=h.num_nodes)
    m = T.trie_lazy_rows(h, torch.arange(h.num_nodes, dtype=torch.int32, device="cuda"), V)
    assert np.array_equal(m.cpu().numpy().view(np.uint32), want)
    h.destroy()


@pytest.mark.parametrize("build", ["single", "host", "device"])
@pytest.mark.parametrize("uploaded", [False, True])
def test_first_compile_captured(build, uploaded):
    """A handle's first dense compile (and, if nothing did it before, its upload)
    is captured, and the graph has not run yet when calls outside it need the
    same arrays, tables and buffers."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    oracle.build()
    strings, toks = random_case(91)
    sets = [strings] if build == "single" else [strings, strings[:3]]
    sb, so = W.pack([x for s in sets for x in s])
    si = np.cumsum([0] + [len(s) for s in sets]).astype(np.int32)
    vb, vo = W.pack(toks)
    V = len(toks)
    voc = T.trie_vocab_create(vb, vo, V)
    h = T.trie_build(sb, so) if build == "single" else \
        (T.trie_build_many_device if build == "device" else T.trie_build_many)(sb, so, si)
    ov = oracle.Vocab(vb, vo)
    want = np.concatenate([oracle.mask_all(oracle.Trie(*W.pack(s)), ov) for s in sets])
    if uploaded:
        T.trie_compile_lists_vocab(h, voc)
    first, second = torch.empty((2, h.num_nodes, T.mask_words(V)), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        T.trie_compile_masks_vocab(h, voc, first)
    T.trie_compile_masks_vocab(h, voc, second)
    assert np.array_equal(second.cpu().numpy().view(np.uint32), want)
    T.trie_lazy_init(h, vb, vo, V, cache_rows=0, max_batch=h.num_nodes)
    m = T.trie_lazy_rows(h, torch.arange(h.num_nodes, dtype=torch.int32, device="cuda"), V)
    assert np.array_equal(m.cpu().numpy().view(np.uint32), want)
    for _ in range(2):
        first.fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(first.cpu().numpy().view(np.uint32), want)
    del g
    h.destroy()


@pytest.mark.parametrize("then", ["masks", "lazy"])
def test_moves_after_a_captured_compile(then):
    """A single trie's transition table, whose clear and fill were captured but
    have not run, in memory where an earlier handle's table lies: the same rows
    and tokens with the moves of another vocabulary."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    oracle.build()
    strings, toks = random_case(91)
    sb, so = W.pack(strings)
    V = len(toks)
    other = T.trie_vocab_create(*W.pack(toks[-2::-1] + toks[-1:]), V)  # every token but EOS under another id
    vb, vo = W.pack(toks)
    voc = T.trie_vocab_create(vb, vo, V)
    ot, ov = oracle.Trie(sb, so), oracle.Vocab(vb, vo)
    n = ot.num_nodes
    masks = torch.empty((2, n, T.mask_words(V)), dtype=torch.int32, device="cuda")
    for _ in range(3):  # the pool's next block of this size is one of these
        old = T.trie_build(sb, so)
        T.trie_compile_lists_vocab(old, other)
        T.trie_compile_masks_vocab(old, other, masks[0])
        old.destroy()
    h = T.trie_build(sb, so)
    T.trie_compile_lists_vocab(h, voc)  # the upload, as the old handle's
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        T.trie_compile_masks_vocab(h, voc, masks[1])
    s0 = np.repeat(np.arange(n, dtype=np.int32), V)
    t0 = np.tile(np.arange(V, dtype=np.int32), n)
    want, _ = oracle.advance(ot, ov, s0, t0)
    states, tokens = torch.as_tensor(s0, device="cuda"), torch.as_tensor(t0, device="cuda")
    for k in range(2):
        if k == 1:
            g.replay()
        elif then == "masks":
            T.trie_compile_masks_vocab(h, voc, masks[0])
        else:
            T.trie_lazy_init(h, vb, vo, V, cache_rows=0, max_batch=8)
        got = states.clone()
        T.trie_advance(h, got, tokens)
        assert np.array_equal(got.cpu().numpy(), want)
    del g
    h.destroy()
