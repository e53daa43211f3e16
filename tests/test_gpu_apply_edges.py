"""The apply kernels at the edges of how they cut a row of logits: rows that
start at every offset from a 16-byte boundary, sizes around a 16-byte chunk, a
1,024-token segment and an 8,192-token part, against the CPU oracle's masks."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2608_12574_gb300 import triemask as T
from paper_2608_12574_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NINF = {"f32": 0xFF800000, "bf16": 0xFF80}


@pytest.fixture(scope="module")
def cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_12574_gb300 import _build
    _build.build()
    oracle.build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V", [2, 5, 9, 31, 33, 1023, 1024, 1025, 1031, 8191, 8193, 8199, 16385, 32768, 32775, 33799])
def test_apply_row_cuts(cuda, V, dtype):
    """Every entry point that masks logits, B rows of V logits that begin 0..7
    elements into a buffer: allowed logits keep their bits, the others are
    -inf, and the elements around the rows are untouched."""
    import torch
    toks = [bytes([97 + i % 26, 97 + i // 26 % 26, 97 + i // 676 % 26, 97 + i // 17576]) for i in range(V - 1)] + [b""]
    rng = np.random.default_rng(V)
    edge = [x for c in (0, 8, 1024, 2048, 8192, 16384, 32768, V - 1) for x in range(c - 9, c + 9)]
    pick = sorted({x for x in edge + list(rng.integers(0, V, 20)) if 0 <= x < V - 1 and rng.random() < 0.6} | {V - 2})
    strings = [toks[i] for i in pick] + [toks[pick[0]] + toks[i] for i in pick[::3]] + [toks[pick[-1]] + toks[0]]
    sb, so = W.pack(strings)
    vb, vo = W.pack(toks)
    ot, ov = oracle.Trie(sb, so), oracle.Vocab(vb, vo)
    h = T.trie_build(sb, so)
    mask = T.alloc_mask(h, V, cuda)
    T.trie_compile_masks(h, vb, vo, V, mask)
    T.trie_compile_lists(h, vb, vo, V)
    s0 = np.array([0, 0, -2, -1, 0, 1, h.num_nodes - 1], np.int32)
    t0 = np.array([pick[0], pick[-1], V - 1, 0, V - 2, 0, V - 1], np.int32)
    B = len(s0)
    s1, _ = oracle.advance(ot, ov, s0, t0)
    ds0, dt0 = torch.as_tensor(s0, device=cuda), torch.as_tensor(t0, device=cuda)
    ds1 = torch.empty_like(ds0)
    calls = {"apply": (s0, lambda x: T.trie_apply_mask(h, x, ds0)),
             "advance_apply": (s1, lambda x: T.trie_advance_apply(h, ds0, dt0, ds1, x)),
             "lists": (s0, lambda x: T.trie_apply_lists(h, x, ds0)),
             "advance_lists": (s1, lambda x: T.trie_advance_apply_lists(h, ds0, dt0, ds1, x))}
    it, ut = (torch.int32, np.uint32) if dtype == "f32" else (torch.int16, np.uint16)
    for off in range(8 if dtype == "bf16" else 4):
        raw = rng.integers(0, 2 ** (32 if dtype == "f32" else 16), B * V + 64, dtype=np.uint64).astype(ut)
        for name, (states, call) in calls.items():
            words = oracle.mask_rows(ot, ov, np.where(states < 0, 0, states).astype(np.int32))
            bits = np.unpackbits(words.view(np.uint8), axis=1, bitorder="little")[:, :V].astype(bool)
            bits[states < 0] = False
            bits[states < 0, V - 1] = True
            want = raw.copy()
            want[off:off + B * V][~bits.reshape(-1)] = NINF[dtype]
            buf = torch.from_numpy(raw.view(np.int32 if dtype == "f32" else np.int16).copy()).to(cuda)
            call(buf.view(torch.float32 if dtype == "f32" else torch.bfloat16)[off:off + B * V].view(B, V))
            got = buf.view(it).cpu().numpy().view(ut)
            assert np.array_equal(got, want), (name, off, np.flatnonzero(got != want)[:5])
            if "advance" in name:
                assert np.array_equal(ds1.cpu().numpy(), s1)


@pytest.mark.parametrize("V,B", [(32767, 32), (65533, 32), (65533, 120)])
def test_apply_summary_unaligned(cuda, V, B):
    """Unaligned rows of a mask with a segment summary whose words are full (32
    or 64 segments): the last segment has no next one to take bits from. 120
    rows take CTAs of 256 threads, 32 rows CTAs of 128."""
    import torch
    names = W.tool_names(1, 1000, 200)
    sb, so = W.pack(names)
    spec = W.VocabSpec(V=V, max_len=16, substr_frac=0.3, run_frac=0.0, run_len=(2, 4), upper=False, mixed=False)
    vb, vo = W.byte_vocab(1, spec, substr_src=W.tool_stems(1, 200))
    h = T.trie_build(sb, so)
    mask = T.alloc_mask(h, V, cuda)
    T.trie_compile_masks(h, vb, vo, V, mask)
    ot, ov = oracle.Trie(sb, so), oracle.Vocab(vb, vo)
    rng = np.random.default_rng(V)
    n = h.num_nodes
    s0 = np.concatenate([[0, n - 1, n - 2, -1, -2], rng.integers(0, n, B)]).astype(np.int32)
    raw = rng.integers(0, 2 ** 16, (len(s0), V), dtype=np.uint32).astype(np.uint16)
    want = oracle.apply(ot, ov, raw, s0)
    x = torch.from_numpy(raw.view(np.int16)).view(torch.bfloat16).to(cuda)
    T.trie_apply_mask(h, x, torch.as_tensor(s0, device=cuda))
    assert np.array_equal(x.view(torch.int16).cpu().numpy().view(np.uint16), want)
