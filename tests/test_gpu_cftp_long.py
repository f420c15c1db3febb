"""Coupling from the past where its launches differ from a chain's: one launch of
both chains is bounded in sweeps, and two chains of many stripes run at the same
time on two streams."""
from __future__ import annotations

import re

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


def test_pair_launches_are_bounded(T, ctx):
    # a launch takes 60,000 cycles of at most 64 passes
    from torch.profiler import ProfilerActivity, profile
    dom, th, k = T.Domain.aztec(20), T.thresholds(scalar=1 << 31), 1 << 21
    assert T.Chain(ctx, dom, seed=5, th=th).kernel == "small_kernel"
    with profile(activities=[ProfilerActivity.CUDA]):   # the first one of a process records nothing
        T.cftp(ctx, dom, seed=5, th=th, t0=1)
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        got, used = T.cftp(ctx, dom, seed=5, th=th, t0=k)
    launches = sum(e.count for e in p.key_averages() if re.search(r"(?<!\w)small_kernel", e.key))
    if not launches:
        pytest.skip("the profiler records no kernels here")
    assert used == k and launches >= k * 2 // (60000 * 64) + 1
    ch = T.Chain(ctx, dom, seed=5, th=th)
    ch.seek((1 << 32) - k)
    ch.run(k)
    assert np.array_equal(ch.read_state(), got)


@pytest.mark.parametrize("kind,size,t,kernel", [("aztec", (140,), 1 << 31, 3), ("hexagon", (90, 80, 70), 0x00100000, 2)])
def test_two_chains_of_many_stripes(T, ctx, kind, size, t, kernel):
    dom, th = getattr(T.Domain, kind)(*size), T.thresholds(scalar=t)
    probe = T.Chain(ctx, dom, seed=1, th=th).plan()
    assert probe["kernel"] == kernel and 1 < probe["ctas"] <= 76   # two fit the SMs
    got, used = T.cftp(ctx, dom, seed=29, stream_id=4, th=th, t0=32)
    ends = []
    for which in ("top", "bottom"):
        ch = T.Chain(ctx, dom, seed=29, stream_id=4, th=th, init=dom.extreme_state(which))
        ch.seek((1 << 32) - used)
        ch.run(used)
        ends.append(ch.read_state())
        if used > 32:   # half the range had not coalesced
            ch.reset()
            ch.seek((1 << 32) - used // 2)
            ch.run(used // 2)
            ends.append(ch.read_state())
    assert np.array_equal(ends[0], got) and np.array_equal(ends[len(ends) // 2], got)
    if used > 32:
        assert not np.array_equal(ends[1], ends[3])
    if t != 1 << 31:
        lat = O.DOMINO if kind == "aztec" else O.LOZENGE
        st = O.extreme(lat, getattr(O, kind)(*size), True)
        O.sweeps(lat, st, seed=29, stream=4, sweep0=(1 << 32) - used, k=used, t_scalar=t)
        assert np.array_equal(st, got)
