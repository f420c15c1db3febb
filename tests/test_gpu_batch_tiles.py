"""Batches of few and of many tiles (lower tiles and more threads per tile when
they are few), odd tile heights and every threshold kind: every chain must end
as the same chain run alone."""
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


def _chain(T, ctx, i):
    rng = np.random.default_rng([19, i])
    kind = ("aztec", "hexagon", "dwbc", "rect")[i % 4]
    size = {"aztec": (int(rng.integers(1, 300)),), "hexagon": tuple(int(v) for v in rng.integers(1, 200, 3)),
            "dwbc": (int(rng.integers(2, 280)),), "rect": (2 * int(rng.integers(1, 150)), int(rng.integers(1, 250)))}[kind]
    dom = getattr(T.Domain, kind)(*size)
    if kind == "dwbc":
        w6 = [1, 1, 1, 1, 1.5, 1.5] if i % 8 < 4 else np.exp(0.4 * rng.standard_normal(6))
        th = T.thresholds(table16=T.sixv_thresholds(w6))
    elif (i // 4) % 3 == 0:
        th = T.thresholds(site=rng.integers(0, 1 << 32, size=dom.canon_shape[1:], dtype=np.uint32))
    else:
        th = T.thresholds(scalar=1 << 31 if (i // 4) % 3 == 1 else 0x51EB851F)
    return T.Chain(ctx, dom, seed=23, stream_id=i, th=th)


@pytest.mark.parametrize("chains,tile_rows,R,threads", [(1, 128, 4, 256), (2, 33, 3, 128), (12, 128, 4, 256),
                                                        (24, 7, 1, 128), (48, 64, 8, 128), (48, 31, 2, 256)])
def test_tiles_match_alone(T, chains, tile_rows, R, threads):
    ctx = T.Context(0)
    cs = [_chain(T, ctx, i) for i in range(chains)]
    alone = [_chain(T, ctx, i) for i in range(chains)]
    b = T.Batch(ctx, cs)
    b.set_plan(tile_rows, R, -1, threads)
    assert b.plan()["tile_rows"] == tile_rows and b.plan()["threads"] == threads
    b.run(25)
    got = b.hashes()
    for i, c in enumerate(alone):
        c.run(25)
        assert int(got[i]) == c.state_hash(), i
        assert np.array_equal(cs[i].read_state(), c.read_state()), i


def test_plans_of_other_batches_leave_a_batch_runnable(T):
    # a batch of lower tiles made later must not shrink the first one's limit
    ctx = T.Context(0)
    big = T.Batch(ctx, [T.Chain(ctx, T.Domain.rect(4000, 700), seed=1, th=T.thresholds(scalar=3 << 29))])
    big.set_plan(128, 8, -1)
    small = T.Batch(ctx, [T.Chain(ctx, T.Domain.aztec(20), seed=1)])
    small.set_plan(8, 1, -1)
    big.run(8)
    assert len(big.hashes()) == 1


@pytest.mark.parametrize("graph_block", [-1, 1026])
def test_more_launches_than_tile_cursors(T, graph_block):
    # 1,024 cursors are cleared together: launches beyond them, with more tiles
    # than blocks so that the blocks read them
    ctx = T.Context(0)
    cs = [T.Chain(ctx, T.Domain.aztec(8 + i % 5), seed=3, stream_id=i, th=T.thresholds(scalar=3 << 29))
          for i in range(320)]
    b = T.Batch(ctx, cs)
    b.set_plan(8, 1, graph_block, 256)
    p = b.plan()
    assert p["ntiles"] > p["grid"]
    import torch
    stream = torch.cuda.Stream()
    b.run(1030, stream=stream)
    got = b.hashes(stream=stream)
    for i in (0, 1, 158, 317, 318, 319):
        alone = T.Chain(ctx, T.Domain.aztec(8 + i % 5), seed=3, stream_id=i, th=T.thresholds(scalar=3 << 29))
        alone.run(1030)
        assert int(got[i]) == alone.state_hash(), i
