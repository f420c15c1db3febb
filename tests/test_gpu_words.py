"""The word kernel where its shape changes, against the oracle after every
sweep: domains that one block holds, stripes of one, two and four words per
thread, whole and broken sweeps per exchange, and both pass orders."""
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


W6 = [1.3, 0.7, 0.9, 1.6, 1.1, 2.0]


def _check(T, ctx, kind, size, thr, *, k, halo=0, random_order=False, threads=0):
    lat = {"aztec": O.DOMINO, "rect": O.DOMINO, "hexagon": O.LOZENGE, "dwbc": O.SIXV}[kind]
    dom, st = getattr(T.Domain, kind)(*size), getattr(O, kind)(*size)
    if thr == "site":
        site = np.random.default_rng([len(kind), *size]).integers(0, 1 << 32, size=st.shape[1:], dtype=np.uint32)
        th, kw = T.thresholds(site=site), {"t_site": site}
    elif thr == "table":
        t16 = T.sixv_thresholds(W6)
        th, kw = T.thresholds(table16=t16), {"t16": t16}
    elif thr == "count":
        t16 = T.sixv_thresholds([1, 1, 1, 1, 2 ** 0.5, 2 ** 0.5])
        th, kw = T.thresholds(table16=t16), {"t16": t16}
    else:
        th, kw = T.thresholds(scalar=thr), {"t_scalar": thr}
    ch = T.Chain(ctx, dom, seed=77, stream_id=5, th=th)
    if random_order:
        ch.set_order(True)
        kw["random_order"] = True
    if halo or threads:
        ch.set_plan(0, 0, halo, threads)
    ch.count_flips(True)
    ring = ch.run_hashed(k)
    want = O.sweeps(lat, st, seed=77, stream=5, k=k, want_hashes=True, **kw)
    assert np.array_equal(ring, want)
    assert np.array_equal(ch.read_state(), st)
    return ch.plan()


@pytest.mark.parametrize("kind,size,thr", [
    ("aztec", (1,), "site"), ("aztec", (5,), "site"), ("aztec", (9,), 0x9E3779B9), ("rect", (2, 3), 1 << 30),
    ("rect", (256, 2), "site"), ("rect", (258, 3), 3), ("hexagon", (1, 1, 1), 0x9E3779B9), ("hexagon", (3, 1, 7), "site"),
    ("hexagon", (20, 17, 23), 1 << 31), ("dwbc", (2,), "table"), ("dwbc", (31,), "count"),
    ("dwbc", (64,), "table")])
@pytest.mark.parametrize("random_order", [False, True])
def test_one_block(T, ctx, kind, size, thr, random_order):
    _check(T, ctx, kind, size, thr, k=40, random_order=random_order)


@pytest.mark.parametrize("kind,size,thr", [("rect", (8000, 31), 0x9E3779B9), ("rect", (16000, 26), "site"),
                                           ("hexagon", (3000, 8, 9), "site"), ("dwbc", (700,), "table")])
@pytest.mark.parametrize("halo,threads", [(0, 0), (12, 0), (5, 512)])
def test_words_per_thread(T, ctx, kind, size, thr, halo, threads):
    _check(T, ctx, kind, size, thr, k=10, halo=halo, threads=threads)


def test_random_order_in_stripes(T, ctx):
    _check(T, ctx, "hexagon", (90, 120, 70), "site", k=30, random_order=True)
    _check(T, ctx, "dwbc", (200,), "count", k=30, random_order=True)
    _check(T, ctx, "aztec", (140,), "site", k=30, random_order=True)
