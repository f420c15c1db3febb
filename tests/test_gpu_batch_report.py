"""What a batch launches: reported beside the plan that was asked for, and told
apart by the autotuner (one trial per different launch, picks kept apart for
batches for which the settings come to something else)."""
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


def _batch(T, ctx, count, n):
    th = T.thresholds(scalar=3 << 29)
    return T.Batch(ctx, [T.Chain(ctx, T.Domain.aztec(n), seed=2, stream_id=i, th=th) for i in range(count)])


@pytest.mark.parametrize("count,n,plan,launch", [
    (3, 60, (128, 4, 256), (64, 4, 512)),      # 6 tiles of 64 rows
    (100, 60, (128, 4, 128), (64, 4, 256)),    # 100 tiles of 128 rows: lowered, 200
    (100, 60, (64, 2, 128), (64, 2, 256)), (160, 60, (128, 2, 128), (128, 2, 256)),
    (320, 60, (128, 2, 128), (128, 2, 128)), (320, 60, (32, 1, 256), (32, 1, 256))])
def test_launch_shape(T, count, n, plan, launch):
    ctx = T.Context(0)
    b = _batch(T, ctx, count, n)
    b.set_plan(plan[0], plan[1], -1, plan[2])
    p, s = b.plan(), b.launch_shape()
    assert (p["tile_rows"], p["sweeps_per_launch"], p["threads"]) == plan
    assert (s["tile_rows"], s["sweeps_per_launch"], s["threads"]) == launch


def _trial_launches(shapes, trial):
    # two runs a trial: launches of R sweeps, an even number of them (the last
    # one split or a copy back), and the counters' advance
    total = 0
    for _, R, _ in shapes:
        n = -(-trial // R)
        total += 2 * (n + n % 2 + 1)
    return total


@pytest.mark.parametrize("count,n", [(3, 60), (100, 60), (200, 20), (320, 60)])
def test_one_trial_per_launch_shape(T, count, n):
    import torch
    ctx = T.Context(0)
    b = _batch(T, ctx, count, n)
    shapes = set()
    for threads in (256, 128):
        for rows in (32, 64, 128):
            for R in (1, 2, 4, 8):
                b.set_plan(rows, R, 0, threads)
                s = b.launch_shape()
                shapes.add((s["tile_rows"], s["sweeps_per_launch"], s["threads"]))
    T.Batch.autotune_cache_clear()
    before = b.launches
    b.autotune(8, stream=torch.cuda.Stream())
    assert b.launches - before == _trial_launches(shapes, 8)
    T.Batch.autotune_cache_clear()


def test_pick_is_not_taken_by_a_batch_of_another_form(T):
    # rows in all between 2^14 and 2^15 for both: 137 and 248 tiles of 128 rows,
    # fewer and more than the SMs
    import torch
    ctx, stream = T.Context(0), torch.cuda.Stream()
    few, many, again = _batch(T, ctx, 137, 60), _batch(T, ctx, 248, 60), _batch(T, ctx, 247, 60)
    T.Batch.autotune_cache_clear()
    few.autotune(8, stream=stream)
    many.autotune(8, stream=stream)
    assert many.launches > 0
    again.autotune(8, stream=stream)
    assert again.launches == 0
    T.Batch.autotune_cache_clear()
