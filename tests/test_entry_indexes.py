"""Entry indexes of the kernels that read a list a chunk at a time (CPU).

A table may hold up to 2^31 - 2 entries, so a list may begin in the last few
of them, and the index of a chunk's last lane, and the next chunk's first,
pass 2^31: they are 32-bit unsigned, where a signed one would turn negative,
compare below the list's end and be read. Shown on the arithmetic of the last
lists of the largest table, and on the declarations in the source."""
from __future__ import annotations

import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2605_02224_gb300", "csrc")
LAST = 2**31 - 2  # the end of the largest table's last list


def _read(first, end, lanes, dtype):
    """The indexes that lanes of chunk after chunk read, in `dtype` arithmetic."""
    got, base = [], np.array(first).astype(dtype)
    end = np.array(end).astype(dtype)
    for _ in range(4):
        if not base < end:
            break
        e = (base + np.arange(lanes).astype(dtype)).astype(dtype)
        got += [int(x) for x in e[e < end]]
        if base + dtype(lanes) >= end:
            break
        base = base + dtype(lanes)
    return got


@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
@pytest.mark.parametrize("length", [1, 2, 31, 32, 33, 40])
def test_chunks_of_the_last_lists(lanes, length):
    with np.errstate(over="ignore"):
        got = _read(LAST - length, LAST, lanes, np.uint32)
        assert got == list(range(LAST - length, LAST))[: 4 * lanes]
        if length < lanes - 1:  # what signed indexes would read
            assert min(_read(LAST - length, LAST, lanes, np.int32)) < 0


def test_kernels_keep_entry_indexes_unsigned():
    with open(os.path.join(CSRC, "knn_device.cuh")) as f:
        src = f.read()
    body = src[src.index("void knn_query("):]
    loops = re.findall(r"for \((\w+) (?:e = [^;]*, )?base = ", body) + \
        re.findall(r"^\s+(\w+) base = rr\.x;", body, re.M)
    entries = re.findall(r"const (\w+) e = base \+", body)
    assert len(loops) == 4 and set(loops) == {"uint32_t"}, loops
    assert len(entries) == 3 and set(entries) == {"uint32_t"}, entries
