"""Launches so short that the stripes never exchange rows: a stripe must not
write its rows back before its neighbours have loaded them.  Runs of one to
twelve sweeps on domains of many stripes, on every resident kernel, with
another stream keeping SMs busy so that the blocks of a launch start apart."""
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


def _chain(T, ctx, kind, size, thr, kernel):
    dom, st = getattr(T.Domain, kind)(*size), getattr(O, kind)(*size)
    if thr == "table":
        t16 = T.sixv_thresholds([1, 1, 1, 1, 2 ** 0.5, 2 ** 0.5])
        th, kw = T.thresholds(table16=t16), {"t16": t16}
    else:
        th, kw = T.thresholds(scalar=thr), {"t_scalar": thr}
    ch = T.Chain(ctx, dom, seed=31, stream_id=2, th=th)
    if kernel:
        ch.set_plan(kernel)
    assert ch.plan()["ctas"] > 1
    return ch, st, kw


@pytest.mark.parametrize("kind,size,thr,kernel,lattice", [
    ("aztec", (300,), 1 << 31, 3, O.DOMINO),        # halo 24: up to 12 sweeps without an exchange
    ("aztec", (500,), 1 << 31, 2, O.DOMINO), ("aztec", (400,), 0x6A09E667, 0, O.DOMINO),
    ("hexagon", (200, 150, 170), 0x6A09E667, 0, O.LOZENGE), ("dwbc", (400,), "table", 0, O.SIXV)])
def test_short_runs_match(T, kind, size, thr, kernel, lattice):
    import torch
    ctx = T.Context(0)
    ch, st, kw = _chain(T, ctx, kind, size, thr, kernel)
    lens = [1, 1, 2, 1, 3, 1, 2, 4, 1, 5, 12, 1, 2, 3, 1, 1]
    stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    busy = torch.rand(1 << 22, device="cuda")
    for k in lens:
        with torch.cuda.stream(other):
            for _ in range(3):
                busy = busy * 1.0001 + 0.5
        ch.run(k, stream=stream)
    ch.sync(stream)
    O.sweeps(lattice, st, seed=31, stream=2, k=sum(lens), **kw)
    assert np.array_equal(ch.read_state(stream=stream), st)
    torch.cuda.synchronize()


@pytest.mark.parametrize("kind,size,thr,kernel", [("aztec", (1000,), 1 << 31, 3), ("aztec", (1333,), 0x6A09E667, 0),
                                                  ("hexagon", (600, 500, 550), 1 << 30, 0), ("dwbc", (1500,), "table", 0)])
def test_many_short_runs_match_one_long(T, kind, size, thr, kernel):
    # the long run exchanges; 400 sweeps one and two at a time never do
    import torch
    ctx = T.Context(0)
    short, _, _ = _chain(T, ctx, kind, size, thr, kernel)
    long_, _, _ = _chain(T, ctx, kind, size, thr, kernel)
    stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    busy = torch.rand(1 << 24, device="cuda")
    for i in range(266):
        if i % 4 == 0:
            with torch.cuda.stream(other):
                busy = busy * 1.0001 + 0.5
        short.run(1 + i % 2, stream=stream)
    short.sync(stream)
    long_.run(399)
    assert short.state_hash() == long_.state_hash()
    torch.cuda.synchronize()
