"""Rings in shared memory whose slots are used again: that a slot is not written while another warp still reads it, and not
read before it has been written.  The kernels' constants and conditions are taken from their sources and walked on the host."""
from __future__ import annotations

import os
import re

import paper_1911_00472_b200

CSRC = os.path.join(os.path.dirname(paper_1911_00472_b200.__file__), "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _constants(text):
    return {m[0]: int(m[1]) for m in re.findall(r"constexpr (?:int|uint32_t) (k\w+) = (\d+);", text)}


def _value(expression, names):
    """An expression of the sources: unsigned literals, whole divisions, `&&`."""
    py = re.sub(r"\b(\d+)u\b", r"\1", expression).replace("/", "//").replace("&&", " and ")
    return eval(py, {"__builtins__": {}, "min": min, "max": max}, names)


def _one(pattern, text):
    found = re.findall(pattern, text)
    assert len(found) == 1, (pattern, found)
    return found[0]


def test_sequential_block_beginnings():
    """Blocks of two symbols, the fewest there can be: in a round warp 0 stores where the blocks behind its own begin, while the
    other warps read where the blocks of the round before began."""
    text = _source("pcr_sequential.cuh")
    const = _constants(text)
    slots, steps = const["kSeqSlots"], const["kSeqSteps"]
    m_end = _one(r"m_end = ([^;]+);", text)
    n, m, handed, rounds = 1000, 0, 0, 0
    while m < n:
        stop = _value(m_end, {**const, "n": n, "m": m}) // 32
        read = {j % slots for j in range(handed, m)}             # the helpers' blocks
        handed, k = m, 0
        for _ in range(steps):
            if m >= stop:
                break
            k += 1
            if k == 2:
                m, k = m + 1, 0
                assert m % slots not in read, (rounds, m)
        assert m > handed
        rounds += 1
    assert rounds <= n // (steps // 2 - 1) + 1


def test_refinement_mask_queue():
    """Intervals of 1 to 40 blocks, any number of blocks finished between two top-ups: a lane loads its next block's entry only
    if the queue holds that block's."""
    text = _source("pcr_entropy.cuh")
    size = _constants(text)["kMaskQueue"]
    load = _one(r"lds128_if\(([^,]+), queue \+ \(\(m & \(kMaskQueue - 1\)\) << 9\), Z\)", text)
    for blocks in range(1, 41):
        for most in range(1, size + 1):
            held, m, hm = [None] * size, 0, 0
            while m < blocks:
                while hm < blocks and hm - m < size:             # top-up
                    held[hm % size] = hm
                    hm += 1
                for _ in range(most):
                    if m >= hm:
                        break
                    m += 1
                    if _value(load, {"end": True, "m": m, "hm": hm}):
                        assert held[m % size] == m, (blocks, most, m, hm)
