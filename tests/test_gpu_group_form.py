"""Large stripes with one threshold of few set bits (and lozenges with one a site)
take the kernel of a thread per 128 sites: the rule's choice, and parity with the oracle after every sweep
at the edges of its planes (one, four and more than were drawn ahead), of its
lattices and thread counts, in both pass orders."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

HALF = 1 << 31


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


def _thresholds(T, dom, t):
    if t == "site":
        site = np.random.default_rng(8).integers(0, 1 << 32, size=dom.canon_shape[1:], dtype=np.uint32)
        return T.thresholds(site=site), {"t_site": site}
    return T.thresholds(scalar=t), {"t_scalar": t}


def _plan(T, ctx, kind, size, t):
    dom = getattr(T.Domain, kind)(*size)
    p = T.Chain(ctx, dom, seed=3, th=_thresholds(T, dom, t)[0]).plan()
    return p["kernel"], p["halo"], p["threads"]


@pytest.mark.parametrize("kind,size,t,groups", [
    ("rect", (6000, 6000), HALF, (2, 6, 1024)), ("rect", (2000, 2000), 1 << 30, (2, 8, 512)),
    ("rect", (2000, 2000), 19 << 27, (2, 8, 512)), ("aztec", (2000,), 3 << 30, (2, 8, 512)),
    ("hexagon", (1400, 1400, 1400), HALF, (2, 6, 512)), ("hexagon", (1400, 1400, 1400), "site", (2, 6, 512)), ("hexagon", (2800, 2800, 2800), HALF, (2, 6, 512))])
def test_rule(T, ctx, kind, size, t, groups):
    assert _plan(T, ctx, kind, size, t) == groups


@pytest.mark.parametrize("kind,size,t", [("rect", (900, 900), 1 << 30), ("rect", (2000, 2000), 0x9E3779B9),
                                         ("hexagon", (900, 900, 900), HALF), ("hexagon", (900, 900, 900), "site")])
def test_rule_keeps_words(T, ctx, kind, size, t):
    assert _plan(T, ctx, kind, size, t) not in ((2, 8, 512), (2, 6, 512), (2, 6, 1024))


@pytest.mark.parametrize("kind,size,t,npre,threads", [
    ("rect", (16000, 26), HALF, 0, 0), ("rect", (8000, 60), 1 << 30, 0, 0), ("rect", (8000, 60), 3 << 30, 1, 1024),
    ("rect", (8000, 60), 5 << 29, 0, 0), ("rect", (8000, 60), 11 << 28, 2, 0), ("rect", (8000, 60), 19 << 27, 0, 512),
    ("rect", (12000, 26), 37 << 26, 0, 0), ("aztec", (520,), 0, 0, 0), ("hexagon", (9000, 20, 15), HALF, 0, 0),
    ("hexagon", (9000, 20, 15), 5 << 29, 0, 0), ("hexagon", (9000, 20, 15), "site", 0, 0), ("hexagon", (9000, 20, 15), 19 << 27, 3, 1024)])
@pytest.mark.parametrize("random_order", [False, True])
def test_parity(T, ctx, kind, size, t, npre, threads, random_order):
    lat = O.LOZENGE if kind == "hexagon" else O.DOMINO
    dom, st = getattr(T.Domain, kind)(*size), getattr(O, kind)(*size)
    th, kw = _thresholds(T, dom, t)
    ch = T.Chain(ctx, dom, seed=41, stream_id=6, th=th)
    if random_order:
        ch.set_order(True)
    ch.set_plan(0, 0, 0, threads, npre)
    ch.count_flips(True)
    ring = ch.run_hashed(9)
    want = O.sweeps(lat, st, seed=41, stream=6, k=9, want_hashes=True, random_order=random_order, **kw)
    assert np.array_equal(ring, want)
    assert np.array_equal(ch.read_state(), st)
    ch.run(3)
    O.sweeps(lat, st, seed=41, stream=6, sweep0=9, k=3, random_order=random_order, **kw)
    assert np.array_equal(ch.read_state(), st)
    per_pass = T.Chain(ctx, dom, seed=41, stream_id=6, th=th)
    if random_order:
        per_pass.set_order(True)
    per_pass.set_plan(1)
    per_pass.count_flips(True)
    per_pass.run(12)
    assert ch.flips == per_pass.flips > 0 or t == 0
