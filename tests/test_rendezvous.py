"""The outcome of a rendezvous whose waits are bounded (csrc/lbm_rendezvous.h,
compiled for the host): every order of arrivals, expired waits and decisions of
three warps, over two rendezvous.  The block's warps must all take the same
branch, whatever each saw of its own wait, and may cut only when all arrived."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "lbm_rendezvous.h"
extern "C" int met(unsigned* word, int own, unsigned c) {
    return lbm::rendezvous_met(own != 0, c, [&](unsigned e, unsigned d) {
        const unsigned before = *word;
        if (before == e) *word = d;
        return before;
    });
}
"""


@pytest.fixture(scope="module")
def met(tmp_path_factory):
    d = tmp_path_factory.mktemp("rendezvous")
    (d / "r.cpp").write_text(SRC)
    so = str(d / "r.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared",
                    "-I", os.path.join(ROOT, "paper_0705_4371_gb300", "csrc"), "-o", so, str(d / "r.cpp")], check=True)
    f = C.CDLL(so).met
    f.argtypes = [C.POINTER(C.c_uint), C.c_int, C.c_uint]
    return f


def _orders(n, met, word, c):
    """Every interleaving of n warps, each arriving, ending its wait (met once
    all have arrived; given up at any time) and deciding.  Yields (own, outcome)
    of each warp and the word afterwards."""
    def go(stage, own, out, w):
        if all(s == 3 for s in stage):
            yield tuple(own), tuple(out), w
            return
        for i in range(n):
            if stage[i] == 0:
                yield from go(stage[:i] + [1] + stage[i + 1:], own, out, w)
            elif stage[i] == 1:
                full = all(s >= 1 for s in stage)
                for seen in ([1, 0] if full else [0]):
                    yield from go(stage[:i] + [2] + stage[i + 1:], own[:i] + [seen] + own[i + 1:], out, w)
            elif stage[i] == 2:
                word = C.c_uint(w)
                r = met(C.byref(word), own[i], c)
                yield from go(stage[:i] + [3] + stage[i + 1:], own, out[:i] + [r] + out[i + 1:], word.value)
    yield from go([0] * n, [None] * n, [None] * n, word)


def test_every_warp_takes_the_same_branch(met):
    mixed = 0
    for own, out, w in set(_orders(3, met, 0, 0)):
        assert len(set(out)) == 1, (own, out)
        mixed += len(set(own)) == 2
        if all(own):
            assert all(out)            # met everywhere: the block cuts
        if not any(own):
            assert not any(out)        # nobody met: it leaves
        assert w == (2 if out[0] else 1)
    # the waits alone do disagree in some orders (what the one word is for)
    assert mixed > 0


def test_the_next_rendezvous_starts_open(met):
    for own, out, w in set(_orders(2, met, 2, 1)):
        assert len(set(out)) == 1, (own, out)
        assert w == (4 if out[0] else 3)
