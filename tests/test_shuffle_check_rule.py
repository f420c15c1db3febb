"""The check of a finished shuffling sample, replayed on the CPU over its units of 16
columns at every alignment: it passes tilings and finds every single wrong edge
beside a cell."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O


def is_tiling(st, n, lead):
    W, bit = 2 * n + 1, np.arange(16)

    def bits(row, x0):
        x = x0 + np.arange(17)
        return np.where((x >= 0) & (x < W), row[np.clip(x, 0, W - 1)], 0).astype(bool)
    for y in range(2 * n):
        w = y + 1 if y < n else 2 * n - y
        for x0 in range(-lead, W, 16):
            a, b, v = bits(st[0, y], x0)[:16], bits(st[0, y + 1], x0)[:16], bits(st[1, y], x0)
            c, d = v[:16], v[1:]
            inside = (bit >= n - w - x0) & (bit <= n + w - 1 - x0)
            one = (a ^ b ^ c ^ d) & ~((a & b) | (c & d))
            if ((one ^ inside) | ((a | b | c | d) & ~inside)).any():
                return False
    return True


@pytest.mark.parametrize("n", [1, 2, 3, 16, 33])
def test_check(n):
    st = O.aztec_shuffle(n, n, 1)
    assert all(is_tiling(st, n, lead) for lead in range(16))
    rng = np.random.default_rng(n)
    for i in range(20):
        t, y, x = rng.integers(2), rng.integers(2 * n), rng.integers(2 * n)
        bad = st.copy()
        bad[t, y, x] ^= 1
        assert not is_tiling(bad, n, i % 16)
