"""Hashes and heights of small states on both sides of the line between one block
and several launches, against the oracle; heights say which by their launches."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_07250_gb300 as T
    return T


@pytest.mark.parametrize("kind,size,launches", [
    ("aztec", (32,), 1), ("aztec", (64,), 1), ("aztec", (70,), 1), ("aztec", (71,), 4), ("aztec", (127,), 4),
    ("dwbc", (40,), 1), ("dwbc", (42,), 1), ("dwbc", (44,), 1), ("dwbc", (140,), 1), ("dwbc", (141,), 4),
    ("rect", (10, 319), 1), ("rect", (10, 320), 4), ("rect", (1022, 5), 1), ("rect", (1024, 5), 4), ("rect", (15000, 1), 4),
    ("hexagon", (10, 11, 12), 1), ("hexagon", (70, 70, 70), 1), ("hexagon", (71, 71, 71), 4)])
def test_hash_and_heights(T, kind, size, launches):
    ctx, dom = T.Context(0), getattr(T.Domain, kind)(*size)
    lat = {"aztec": O.DOMINO, "rect": O.DOMINO, "hexagon": O.LOZENGE, "dwbc": O.SIXV}[kind]
    th = T.thresholds(table16=T.sixv_thresholds(np.ones(6))) if kind == "dwbc" else T.thresholds(scalar=3 << 29)
    kw = {"t16": O.sixv_thresholds(np.ones(6))} if kind == "dwbc" else {"t_scalar": 3 << 29}
    ch = T.Chain(ctx, dom, seed=5, th=th)
    st = getattr(O, kind)(*size)
    O.sweeps(lat, st, seed=5, k=40, **kw)
    ch.run(40)
    assert ch.state_hash() == O.state_hash(st)
    before = ch.launches
    h, off = O.height(lat, st)
    assert off == 0 and np.array_equal(ch.read_height(), h)
    assert ch.launches - before == launches
