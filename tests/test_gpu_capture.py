"""Sweeps captured into a CUDA graph: a chain that has not run before is captured
too (planning its resident kernel would allocate), and a planned one."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_07250_gb300 as T
    return T


@pytest.mark.parametrize("kind,size,t", [("aztec", (3,), 3 << 29), ("aztec", (1200,), 0x9E3779B9), ("rect", (40, 30), 1 << 31),
                                         ("hexagon", (4, 3, 2), 1 << 31)])
@pytest.mark.parametrize("planned", [False, True])
def test_captured_sweeps(T, kind, size, t, planned):
    import torch
    ctx = T.Context(0)
    th = T.thresholds(scalar=t)
    ch = T.Chain(ctx, getattr(T.Domain, kind)(*size), seed=6, th=th)
    ref = T.Chain(ctx, getattr(T.Domain, kind)(*size), seed=6, th=th)
    if planned:
        ch.plan()
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        ch.run(30, stream=stream)
    graph.replay()
    torch.cuda.synchronize()
    ref.run(30)
    assert np.array_equal(ch.read_state(), ref.read_state())
    ch.run(10)
    ref.run(10)
    assert ch.state_hash() == ref.state_hash()
