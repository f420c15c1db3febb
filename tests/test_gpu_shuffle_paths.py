"""Domino shuffling where its kernels change shape: orders at the edges of the
packed words and of the 128-site groups against the oracle, and orders that
take several launches against the per-step kernel (a context of one SM, whose
shared memory the rows do not fit)."""
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


@pytest.mark.parametrize("n", [15, 16, 31, 32, 33, 63, 64, 65, 126, 127, 128])
def test_word_and_group_edges(T, n):
    ctx = T.Context(0)
    assert np.array_equal(T.aztec_shuffle(ctx, n, seed=n, stream_id=3), O.aztec_shuffle(n, n, 3))


def test_one_stripe_and_per_step_kernel(T):
    # one SM: order 100 in a single stripe, order 300 one launch per step
    ctx = T.Context(0, max_sms=1)
    assert np.array_equal(T.aztec_shuffle(ctx, 100, seed=4), O.aztec_shuffle(100, 4, 0))
    assert np.array_equal(T.aztec_shuffle(ctx, 300, seed=5), T.aztec_shuffle(T.Context(0), 300, seed=5))


@pytest.mark.parametrize("n", [561, 1023])
def test_several_launches(T, n):
    assert np.array_equal(T.aztec_shuffle(T.Context(0), n, seed=n), T.aztec_shuffle(T.Context(0, max_sms=1), n, seed=n))
