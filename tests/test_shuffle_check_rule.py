"""The check of a finished shuffling sample, replayed on the CPU with its words and
masks: it passes tilings and finds every single wrong edge beside a cell."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O


def is_tiling(st, n):
    W = 2 * n + 1
    K = (n + 1 + 127) // 128 * 128
    planes = np.zeros((4, W, K), dtype=bool)   # He, Ho, Ve, Vo
    for t in range(2):
        for r in range(2):
            part = st[t][:, r::2]
            planes[2 * t + r, :, :part.shape[1]] = part
    for y in range(2 * n):
        w = y + 1 if y < n else 2 * n - y
        for r in range(2):
            a, b, c = planes[r, y], planes[r, y + 1], planes[2 + r, y]
            d = np.append(planes[2, y, 1:], False) if r else planes[3, y]
            inside = np.zeros(K, dtype=bool)
            inside[(n - w + 1 - r) >> 1:((n + w - 1 - r) >> 1) + 1] = True
            one = (a ^ b ^ c ^ d) & ~((a & b) | (c & d))
            if (one != inside).any() or ((a | b | c | d) & ~inside).any():
                return False
    return True


@pytest.mark.parametrize("n", [1, 2, 3, 16, 33, 70, 130])
def test_check(n):
    st = O.aztec_shuffle(n, n, 1) if n < 60 else O.aztec(n)
    assert is_tiling(st, n)
    rng = np.random.default_rng(n)
    for _ in range(20):
        t, y, x = rng.integers(2), rng.integers(2 * n), rng.integers(2 * n)
        bad = st.copy()
        bad[t, y, x] ^= 1
        assert not is_tiling(bad, n)
