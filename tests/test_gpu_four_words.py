"""Four words a thread of the word kernel: taken where they beat launches per pass,
or when a plan asks for them, and then equal to the oracle after every sweep."""
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


@pytest.fixture(scope="module")
def ctx(T):
    return T.Context(0)


def _chain(T, ctx, kind, size, t):
    dom = getattr(T.Domain, kind)(*size)
    if t == "table":
        t16 = T.sixv_thresholds([1.3, 0.7, 0.9, 1.6, 1.1, 2.0])
        th, kw = T.thresholds(table16=t16), {"t16": t16}
    elif t == "site":
        site = np.random.default_rng(9).integers(0, 1 << 32, size=dom.canon_shape[1:], dtype=np.uint32)
        th, kw = T.thresholds(site=site), {"t_site": site}
    else:
        th, kw = T.thresholds(scalar=t), {"t_scalar": t}
    return T.Chain(ctx, dom, seed=19, stream_id=3, th=th), kw


@pytest.mark.parametrize("kind,size,t,kernel", [
    ("hexagon", (2800, 2800, 2800), "site", 1), ("rect", (4600, 4600), 19 << 27, 1), ("rect", (16000, 26), "site", 1),
    ("hexagon", (3200, 3200, 3200), 5 << 29, 1), ("rect", (4600, 4600), 0x9E3779B9, 2), ("dwbc", (4000,), "table", 2)])
def test_rule(T, ctx, kind, size, t, kernel):
    assert _chain(T, ctx, kind, size, t)[0].plan()["kernel"] == kernel


@pytest.mark.parametrize("kind,size,t", [("rect", (16000, 26), "site"), ("rect", (16000, 26), 19 << 27),
                                         ("rect", (16000, 26), 0x9E3779B9), ("dwbc", (2100,), "table")])
def test_parity_under_plan_2(T, ctx, kind, size, t):
    ch, kw = _chain(T, ctx, kind, size, t)
    ch.set_plan(2)
    assert ch.plan()["kernel"] == 2
    st = getattr(O, kind)(*size)
    ring = ch.run_hashed(6)
    want = O.sweeps(O.SIXV if kind == "dwbc" else O.DOMINO, st, seed=19, stream=3, k=6, want_hashes=True, **kw)
    assert np.array_equal(ring, want)
    assert np.array_equal(ch.read_state(), st)
