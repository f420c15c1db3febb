"""Plans of one chain leave the others runnable: a kernel's shared-memory limit
is not lowered by a smaller chain planned later."""
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


@pytest.mark.parametrize("kernel,big,small,threads", [
    (2, 700, 60, 0), (2, 700, 60, 512), (3, 1500, 200, 0)])
def test_smaller_plan_later(T, kernel, big, small, threads):
    ctx = T.Context(0)
    th = T.thresholds(scalar=1 << 31)

    def chain(n):
        c = T.Chain(ctx, T.Domain.aztec(n), seed=3, th=th)
        c.set_plan(kernel, 0, 0, threads)
        return c
    first, alone = chain(big), chain(big)
    alone.run(40)
    want = alone.state_hash()
    second = chain(small)
    if kernel == 2:
        assert second.plan()["smem_bytes"] < first.plan()["smem_bytes"]
    second.run(40)
    first.run(40)
    first.sync()
    assert first.state_hash() == want
