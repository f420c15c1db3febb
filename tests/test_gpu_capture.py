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


@pytest.mark.parametrize("planned", [False, True])
def test_captured_hashed_run(T, planned):
    import torch
    ctx, dom, th = T.Context(0), T.Domain.aztec(3), T.thresholds(scalar=3 << 29)
    ch, ref = (T.Chain(ctx, dom, seed=6, th=th) for _ in range(2))
    if planned:
        ch.plan()
    ring = torch.zeros(12, dtype=torch.int64, device="cuda")
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        ch.run_hashed(12, ring, stream=stream)
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(ring.cpu().numpy().view(np.uint64), ref.run_hashed(12))
