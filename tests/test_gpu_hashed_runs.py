"""Hashed runs of the word kernel: more threads than the passes need, warps that
do not fall on the same planes of every row, and large stripes hashed by a
launch of their own, against the oracle after every sweep."""
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


@pytest.mark.parametrize("kind,size,k,apart", [
    ("aztec", (3,), 20, False), ("aztec", (128,), 20, False), ("aztec", (900,), 6, False), ("hexagon", (60, 50, 70), 20, False),
    ("rect", (16380, 30), 6, False), ("aztec", (1200,), 6, True)])
def test_against_oracle(T, kind, size, k, apart):
    ctx, dom = T.Context(0), getattr(T.Domain, kind)(*size)
    site = np.random.default_rng(4).integers(0, 1 << 32, size=dom.canon_shape[1:], dtype=np.uint32)
    ch = T.Chain(ctx, dom, seed=11, stream_id=1, th=T.thresholds(site=site))
    ref = T.Chain(ctx, dom, seed=11, stream_id=1, th=T.thresholds(site=site))
    for c in (ch, ref):
        c.count_flips(True)
        c.density_begin(2, 0)
        c.plan()
    before = ch.launches
    ring = ch.run_hashed(k)
    if ch.plan()["kernel"] == 2:
        assert ch.launches - before == (2 * k if apart else 1)
    ref.run(k)
    st = getattr(O, kind)(*size)
    want = O.sweeps(O.LOZENGE if kind == "hexagon" else O.DOMINO, st, seed=11, stream=1, k=k, t_site=site, want_hashes=True)
    assert np.array_equal(ring, want)
    assert np.array_equal(ch.read_state(), st)
    assert ch.flips == ref.flips
    a, b = ch.read_density(), ref.read_density()
    assert a[1] == b[1] and np.array_equal(a[0], b[0])
