"""Domino shuffling in several launches against a sampler that shares no code with
it: the destroy, slide and fill steps on whole arrays of cells, itself pinned to
the oracle at small orders."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O


def philox_word0(c0, c1, c2, c3, seed):
    """First output word of Philox4x32-10 (Salmon et al., SC'11)."""
    m = np.uint64(0xFFFFFFFF)
    x = [np.asarray(v, dtype=np.uint64) for v in (c0, c1, c2, c3)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = x[0] * np.uint64(0xD2511F53), x[2] * np.uint64(0xCD9E8D57)
        x = [(b >> np.uint64(32)) ^ x[1] ^ np.uint64(k0), b & m, (a >> np.uint64(32)) ^ x[3] ^ np.uint64(k1), a & m]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x[0]


def shuffle_cells(n, seed, stream):
    H = np.zeros((2, 2), dtype=bool)   # left cells of horizontal dominoes, cells (x, y) at [y + K, x + K]
    V = np.zeros((2, 2), dtype=bool)   # bottom cells of vertical ones
    for K in range(1, n + 1):
        k, s = K - 1, 2 * K
        if k:
            H, V = np.pad(H, 1), np.pad(V, 1)
        y, x = np.ogrid[-K:K, -K:K]
        north = (x + y + k) % 2 == 0   # north of an even cell, else south; east, else west
        bad = H & north
        bad[:-1] &= H[1:]
        bad[-1] = False
        H &= ~bad
        H[1:] &= ~bad[:-1]
        bad = V & north
        bad[:, :-1] &= V[:, 1:]
        bad[:, -1] = False
        V &= ~bad
        V[:, 1:] &= ~bad[:, :-1]
        h, v = np.zeros((s, s), dtype=bool), np.zeros((s, s), dtype=bool)
        h[1:] |= (H & north)[:-1]
        h[:-1] |= (H & ~north)[1:]
        v[:, 1:] |= (V & north)[:, :-1]
        v[:, :-1] |= (V & ~north)[:, 1:]
        empty = (abs(2 * x + 1) + abs(2 * y + 1) <= 2 * K) & ~h & ~v
        empty[:, 1:] &= ~h[:, :-1]
        empty[1:] &= ~v[:-1]
        # blocks are stacked from the bottom of every run of empty cells in a column
        row = np.arange(s, dtype=np.int32)[:, None]
        last = np.maximum.accumulate(np.where(empty, -1, row), axis=0)
        corner = empty & ((row - last) % 2 == 1) & ((x + y + K) % 2 == 1)
        cy, cx = np.nonzero(corner)
        assert 4 * len(cy) == empty.sum() and empty[cy + 1, cx].all() and empty[cy, cx + 1].all() and empty[cy + 1, cx + 1].all()
        hor = philox_word0(((cy - K + n) << 16) | (cx - K + n), K, 0xFFFE0000, stream, seed) < 1 << 31
        h[cy[hor], cx[hor]] = h[cy[hor] + 1, cx[hor]] = True
        v[cy[~hor], cx[~hor]] = v[cy[~hor], cx[~hor] + 1] = True
        H, V = h, v
    st = np.zeros((2, 2 * n + 1, 2 * n + 1), dtype=np.uint8)
    st[1, :-1, 1:] = H                # a horizontal domino crosses the edge between its cells
    st[0, 1:, :-1] = V
    return st


@pytest.mark.parametrize("n", [1, 2, 3, 8, 25, 60])
def test_cells_match_the_oracle(n):
    assert np.array_equal(shuffle_cells(n, 5 + n, 2), O.aztec_shuffle(n, 5 + n, 2))


@pytest.mark.gpu
@pytest.mark.parametrize("n", [561, 640])
def test_several_launches(n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_07250_gb300 as T
    assert np.array_equal(T.aztec_shuffle(T.Context(0), n, seed=17, stream_id=2), shuffle_cells(n, 17, 2))
