"""Batches of chains so wide that the rows of a tile fit the shared memory and the
table of its groups beside them does not: they run, in lower tiles or fewer
sweeps a launch, and end as the chains run alone."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_07250_gb300 as T
    return T


# 232,448 bytes a block: 72 rows of 3,136 bytes leave no room for their table; nor
# do one row and its 68 halo rows
@pytest.mark.parametrize("width,height,rows,R", [(12500, 300, 64, 2), (12500, 300, 0, 0), (12500, 200, 1, 17)])
def test_wide_chain(T, width, height, rows, R):
    ctx = T.Context(0)
    th = T.thresholds(scalar=3 << 29)
    chain = T.Chain(ctx, T.Domain.rect(width, height), seed=7, th=th)
    alone = T.Chain(ctx, T.Domain.rect(width, height), seed=7, th=th)
    b = T.Batch(ctx, [chain])
    b.set_plan(rows, R, -1)
    b.run(20)
    alone.run(20)
    assert int(b.hashes()[0]) == alone.state_hash()


def test_rows_that_do_not_fit_stay_refused(T):
    ctx = T.Context(0)
    b = T.Batch(ctx, [T.Chain(ctx, T.Domain.rect(12500, 300), seed=7, th=T.thresholds(scalar=3 << 29))])
    with pytest.raises(T.TilingError) as e:
        b.set_plan(64, 8, -1)
    assert e.value.code == T.TL_EUNSUPPORTED
