"""The lookup tables of the centres' order (csrc/order.cuh) against the curve
they were generated from: Skilling's Hilbert index, computed here level by
level from its published definition."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_11775_gb300", "csrc")


def hilbert(c, bits):
    c, n = list(c), len(c)
    q = 1 << (bits - 1)
    while q > 1:
        for i in range(n):
            if c[i] & q:
                c[0] ^= q - 1
            else:
                t = (c[0] ^ c[i]) & (q - 1)
                c[0] ^= t
                c[i] ^= t
        q >>= 1
    for i in range(1, n):
        c[i] ^= c[i - 1]
    t, q = 0, 1 << (bits - 1)
    while q > 1:
        if c[n - 1] & q:
            t ^= q - 1
        q >>= 1
    key = 0
    for b in range(bits - 1, -1, -1):
        for v in c:
            key = key << 1 | ((v ^ t) >> b & 1)
    return key


def tables():
    with open(os.path.join(CSRC, "order.cuh")) as f:
        text = f.read()
    two = int(re.search(r"kCurve2 = (0x[0-9a-f]+)ull", text).group(1), 16)
    words = re.search(r"kCurve3\[48\] = \{(.*?)\}", text, re.S).group(1)
    three = np.array([int(w, 16) for w in re.findall(r"0x[0-9a-f]+", words)], dtype="<u4").tobytes()
    assert len(three) == 192
    return two, three


@pytest.mark.parametrize("d,bits", [(2, 1), (2, 3), (2, 6), (3, 1), (3, 4)])
def test_the_tables_walk_the_curve(d, bits):
    two, three = tables()
    n = 1 << bits
    for cell in np.ndindex(*(n,) * d):
        key = s = 0
        for b in range(bits - 1, -1, -1):
            q = 0
            for v in cell:
                q = q << 1 | (v >> b & 1)
            if d == 2:
                e = two >> 4 * (4 * s + q)
                key, s = key << 2 | e & 3, e >> 2 & 3
            else:
                e = three[8 * s + q]
                key, s = key << 3 | e & 7, e >> 3
        assert key == hilbert(cell, bits)
