"""Forests of very different set sizes built on the device from several threads
at once: every build succeeds and equals the host builder's forest."""
from __future__ import annotations

import random
import threading

import numpy as np
import pytest

from paper_2608_12574_gb300 import triemask as T
from paper_2608_12574_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_builds_of_different_sizes_from_threads():
    """One thread builds sets of 4,000 strings, the others sets of a few, each on
    its own stream (the kernels of a large set need more dynamic shared memory
    than the default limit, those of a small set hardly any)."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = random.Random(4)
    word = lambda: bytes(rng.randrange(97, 123) for _ in range(rng.randrange(1, 12)))
    want, packed = [], []
    for k in (4000, 3, 40, 2000):
        sets = [[word() for _ in range(k)], [word(), b""]]
        sb, so = W.pack([x for s in sets for x in s])
        si = np.cumsum([0] + [len(s) for s in sets]).astype(np.int32)
        packed.append((sb, so, si))
        want.append(T.trie_build_many(sb, so, si).csr())
    T.trie_build_many_device(*packed[0]).destroy()  # library and pool set up
    failed = []

    def work(k):
        s = torch.cuda.Stream()
        try:
            with torch.cuda.stream(s):
                for _ in range(150):
                    h = T.trie_build_many_device(*packed[k], stream=s)
                    s.synchronize()
                    h.destroy_async(s)
                h = T.trie_build_many_device(*packed[k], stream=s)
                got = h.csr()
                assert all(np.array_equal(got[x], v) for x, v in want[k].items())
                h.destroy()
        except Exception as e:  # noqa: BLE001 -- reported by the test's thread
            failed.append((k, repr(e)))

    th = [threading.Thread(target=work, args=(k,)) for k in (0, 1, 2, 3, 0, 1)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not failed, failed
