"""Which freed list blocks the library keeps (csrc/spare_blocks.h), run on the
host: sequences of batches, each taking the smallest kept block that fits or a
new one, and giving it back."""
from __future__ import annotations

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "spare_blocks.h"
#include <stdio.h>
#include <string.h>

static tmk::SpareBlocks cache;
static size_t made = 0, live = 0;   // blocks allocated; bytes allocated and not freed
static int busy;                    // an event that has not completed

static bool done(void *e) { return e != &busy; }

static tmk::SpareBlock take(size_t bytes) {
    tmk::SpareBlock b = cache.take(0, bytes, done);
    if (b.p) return b;
    made++;
    live += bytes;
    b.dev = 0;
    b.p = reinterpret_cast<void *>(made);
    b.bytes = bytes;
    b.ready = nullptr;
    return b;
}

static void give(tmk::SpareBlock b) {
    const tmk::SpareBlock out = cache.give(b, done);
    if (out.p) live -= out.bytes;
}

static void batch(size_t bytes) { give(take(bytes)); }

static void two(size_t bytes) {
    tmk::SpareBlock a = take(bytes), b = take(bytes);
    give(a);
    give(b);
}

int main(int argc, char **argv) {
    const char *t = argv[1];
    if (!strcmp(t, "alternating")) {  // sizes in turn: the largest two serve them all
        for (int i = 0; i < 3; i++) batch(350), batch(500), batch(650);
        made = 0;
        for (int i = 0; i < 30; i++) batch(350), batch(500), batch(650);
    } else if (!strcmp(t, "size")) {  // a large block that served a small batch is still a large one
        batch(600);
        made = 0;
        for (int i = 0; i < 30; i++) batch(350), batch(600);
    } else if (!strcmp(t, "shrunk")) {  // after a peak, small batches find their block again
        for (int i = 0; i < 4; i++) two(2000);
        for (int i = 0; i < 20; i++) batch(100);
        made = 0;
        for (int i = 0; i < 30; i++) batch(100);
    } else if (!strcmp(t, "shrunk two")) {  // the same with two batches in flight; the peak's memory is given back
        for (int i = 0; i < 4; i++) two(2000);
        for (int i = 0; i < 20; i++) two(100);
        made = 0;
        for (int i = 0; i < 30; i++) two(100);
    } else if (!strcmp(t, "now and then")) {  // a large batch between a few small ones keeps its block
        for (int i = 0; i < 3; i++) batch(2000), batch(100), batch(100), batch(100);
        made = 0;
        for (int i = 0; i < 30; i++) batch(2000), batch(100), batch(100), batch(100);
    } else if (!strcmp(t, "pending")) {  // a block in use is neither handed out nor freed
        tmk::SpareBlock a = take(100);
        a.ready = &busy;
        give(a);
        tmk::SpareBlock b = take(100);
        printf("%d ", b.p != a.p);
        a = take(100);
        a.ready = &busy;
        give(a);
        for (int i = 0; i < 20; i++) batch(1000);
        give(b);
        made = 0;
    }
    printf("%zu %zu\n", made, live);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("spare")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_2608_12574_gb300", "csrc"),
                    str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    return lambda name: subprocess.run([str(d / "t"), name], check=True, capture_output=True, text=True).stdout.split()


@pytest.mark.parametrize("name,most_live", [("alternating", 1300), ("size", 1200), ("shrunk", 2100),
                                            ("shrunk two", 200), ("now and then", 2100)])
def test_no_new_blocks_once_settled(run, name, most_live):
    made, live = map(int, run(name))
    assert made == 0
    assert live <= most_live


def test_blocks_in_use_stay(run):
    other, _, live = map(int, run("pending"))
    assert other == 1 and live == 200
