"""The one-block kernel of small domino domains at t = 2^31 against the oracle:
word and group edges, ragged rows, odd and even sweep counts, continued runs;
and coupling from the past, which runs its two chains in one launch (or on two
streams) and must give the oracle's sample and T."""
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


@pytest.mark.parametrize("kind,size", [("aztec", (8,)), ("aztec", (15,)), ("aztec", (16,)), ("aztec", (31,)), ("aztec", (32,)),
                                       ("aztec", (33,)), ("aztec", (63,)), ("aztec", (64,)), ("aztec", (96,)),
                                       ("aztec", (127,)), ("rect", (254, 40)), ("rect", (255, 40)), ("rect", (256, 30)),
                                       ("rect", (510, 31)), ("rect", (512, 24)), ("rect", (1000, 20)), ("rect", (16, 240))])
def test_plain_runs(T, ctx, kind, size):
    st = getattr(O, kind)(*size)
    ch = T.Chain(ctx, getattr(T.Domain, kind)(*size), seed=6, stream_id=2, th=T.thresholds(scalar=1 << 31))
    done = 0
    for k in (1, 2, 3, 64, 37):
        ch.run(k)
        O.sweeps(O.DOMINO, st, seed=6, stream=2, sweep0=done, k=k, t_scalar=1 << 31)
        done += k
        assert np.array_equal(ch.read_state(), st), k
    # hashed, counted and sampled runs of the same chain go on from there
    ring = ch.run_hashed(5)
    want = O.sweeps(O.DOMINO, st, seed=6, stream=2, sweep0=done, k=5, t_scalar=1 << 31, want_hashes=True)
    assert np.array_equal(ring, want)


@pytest.mark.parametrize("kind,size,scalar", [("aztec", (20,), 1 << 31), ("hexagon", (9, 8, 7), 1 << 31),
                                              ("hexagon", (9, 8, 7), 0x90000000)])
def test_cftp_pairs(T, ctx, kind, size, scalar):
    lat = O.DOMINO if kind == "aztec" else O.LOZENGE
    got, t = T.cftp(ctx, getattr(T.Domain, kind)(*size), seed=12, stream_id=1, th=T.thresholds(scalar=scalar), t0=16)
    # one step further back the sample is the same, and it is a fixed point of both extremes
    again, t2 = T.cftp(ctx, getattr(T.Domain, kind)(*size), seed=12, stream_id=1, th=T.thresholds(scalar=scalar), t0=2 * t)
    assert t2 == 2 * t and np.array_equal(got, again)
    for which in ("top", "bottom"):
        st = getattr(T.Domain, kind)(*size).extreme_state(which)
        O.sweeps(lat, st, seed=12, stream=1, sweep0=(1 << 32) - t, k=t, t_scalar=scalar)
        assert np.array_equal(st, got)
