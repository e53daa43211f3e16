"""trie_destroy_async: a handle released right after its last queued kernel.

The work queued before the release must still run on the handle's device
memory and host arrays (the upload of a host-built trie reads the host arrays
from a kernel where the GPU reads host memory coherently), so every result is
checked after the stream is synchronised, over several handles built and
released in turn on one stream."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2608_12574_gb300 import triemask as T
from paper_2608_12574_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_12574_gb300 import _build
    _build.build()
    oracle.build()
    return torch.device("cuda:0")


def test_release_after_queued_work(cuda):
    import torch
    w = W.config(1)
    ot = oracle.Trie(w.set_bytes, w.set_offsets)
    ov = oracle.Vocab(w.vocab_bytes, w.vocab_offsets)
    want = oracle.mask_all(ot, ov)
    stream = torch.cuda.Stream(cuda)
    B = 4
    logits = [W.logits(w, i, device="cuda", batch=B) for i in range(6)]
    states = [torch.tensor([0, 1, 2, 3 + i], dtype=torch.int32, device=cuda) for i in range(6)]
    wants = []
    for i, x in enumerate(logits):
        bits = x.cpu().view(torch.int32).numpy().view(np.uint32).copy()
        masked, _, _, _ = oracle.decode(ot, ov, [bits], np.array([0, 1, 2, 3 + i], np.int32))
        wants.append(masked[0])
    masks = [torch.empty((ot.num_nodes, T.mask_words(w.V)), dtype=torch.int32, device=cuda) for _ in range(6)]
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for i in range(6):  # no synchronisation inside: each release follows its queued work
            h = T.trie_build(w.set_bytes, w.set_offsets)
            T.trie_compile_masks(h, w.vocab_bytes, w.vocab_offsets, w.V, masks[i], stream)
            T.trie_apply_mask(h, logits[i], states[i], stream)
            h.destroy_async(stream)
    stream.synchronize()
    for m, x, wx in zip(masks, logits, wants):
        assert np.array_equal(m.cpu().view(torch.int32).numpy().view(np.uint32), want)
        assert np.array_equal(x.cpu().view(torch.int32).numpy().view(np.uint32), wx)


def test_release_beside_a_capture(cuda):
    """One thread captures a graph in the default mode (in which an event query
    by any thread is refused and makes the capture fail) while this one builds
    handles and releases others whose queued work has not run yet."""
    import threading

    import torch
    w = W.config(1)
    names = W.unpack(w.set_bytes, w.set_offsets)
    fb, fo = W.pack(names + names[:50])
    index = np.array([0, len(names), len(names) + 50], np.int32)
    voc = T.trie_vocab_create(w.vocab_bytes, w.vocab_offsets, w.V)
    side = torch.cuda.Stream(cuda)

    def forest():
        f = T.trie_build_many_device(fb, fo, index, side)
        T.trie_compile_lists_vocab(f, voc, side, count=False)
        return f
    forests = [forest() for _ in range(4)]
    h = T.trie_build(w.set_bytes, w.set_offsets)
    m = T.alloc_mask(h, w.V, cuda)
    T.trie_compile_masks(h, w.vocab_bytes, w.vocab_offsets, w.V, m)
    x = torch.randn((4, w.V), device=cuda)
    states = torch.arange(4, dtype=torch.int32, device=cuda)
    want = x.clone()
    T.trie_apply_mask(h, want, states)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)  # about 10 ms
    forests.pop().destroy_async(side)
    g, cap = torch.cuda.CUDAGraph(), torch.cuda.Stream(cuda)
    begun, go_on, failed = threading.Event(), threading.Event(), []

    def capture():
        try:
            with torch.cuda.stream(cap):
                g.capture_begin(capture_error_mode="global")
                begun.set()
                T.trie_apply_mask(h, x, states, cap)
                go_on.wait(30)
                g.capture_end()
        except Exception as e:  # noqa: BLE001 -- reported by the test's thread
            failed.append(repr(e))
        begun.set()
    t = threading.Thread(target=capture)
    t.start()
    assert begun.wait(30)
    t2 = T.trie_build(w.set_bytes, w.set_offsets)  # looks through the released handles
    for f in forests:                              # and through the kept blocks of their lists
        f.destroy_async(side)
    go_on.set()
    t.join()
    assert not failed, failed
    assert t2.num_nodes == h.num_nodes
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(x, want)
