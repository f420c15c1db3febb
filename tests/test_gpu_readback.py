"""Packing, unpacking, validation, heights and density read-back at widths
around the 16-byte stores, the words and the groups, into buffers of every
alignment."""
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


SIZES = [("aztec", (1,)), ("aztec", (7,)), ("aztec", (8,)), ("aztec", (130,)), ("rect", (15, 2)), ("rect", (16, 31)),
         ("rect", (254, 9)), ("rect", (255, 8)), ("rect", (257, 12)), ("hexagon", (1, 1, 1)), ("hexagon", (5, 9, 11)),
         ("hexagon", (40, 300, 57)), ("dwbc", (2,)), ("dwbc", (14,)), ("dwbc", (255,)), ("dwbc", (300,))]


@pytest.mark.parametrize("kind,size", SIZES)
def test_state_and_heights(T, kind, size):
    import torch
    ctx, dom = T.Context(0), getattr(T.Domain, kind)(*size)
    lat = {"aztec": O.DOMINO, "rect": O.DOMINO, "hexagon": O.LOZENGE, "dwbc": O.SIXV}[kind]
    th = T.thresholds(table16=T.sixv_thresholds(np.ones(6))) if kind == "dwbc" else T.thresholds(scalar=1 << 31)
    ch = T.Chain(ctx, dom, seed=3, th=th)
    st = getattr(O, kind)(*size)
    kw = {"t16": O.sixv_thresholds(np.ones(6))} if kind == "dwbc" else {"t_scalar": 1 << 31}
    O.sweeps(lat, st, seed=3, k=30, **kw)
    n = st.size
    for shift in (0, 1, 7, 13):
        src = torch.zeros(n + 64, dtype=torch.uint8, device="cuda")[shift:shift + n]
        src.copy_(torch.from_numpy(st.reshape(-1)))
        ch.write_state(src)
        dst = torch.full((n + 64,), 9, dtype=torch.uint8, device="cuda")
        ch.read_state(dst[shift:shift + n])
        got = dst.cpu().numpy()
        assert np.array_equal(got[shift:shift + n], st.reshape(-1))
        assert (got[:shift] == 9).all() and (got[shift + n:] == 9).all()
        bad = src.clone()
        bad[n - 1] = 2
        with pytest.raises(T.TilingError) as e:
            ch.write_state(bad)
        assert "byte %d" % (n - 1) in str(e.value)
    h, off = O.height(lat, st)
    assert off == 0 and np.array_equal(ch.read_height(), h)


@pytest.mark.parametrize("n,stride,k", [(1, 1, 3), (9, 1, 300), (130, 1, 20), (40, 1, 2100), (33, 2, 5)])
def test_nsew_counts(T, n, stride, k):
    # the densities of the four types are those of the edges around each face
    ctx, dom = T.Context(0), T.Domain.aztec(n)
    ch = T.Chain(ctx, dom, seed=8)
    ch.density_begin(stride, 0)
    ch.run(k)
    dens, samples = ch.read_density()
    nsew = ch.read_nsew()
    hz, vt = dens
    F = 2 * n
    left, right, bottom, top = vt[:F, :F], vt[:F, 1:], hz[:F, :F], hz[1:, :F]
    y, x = np.mgrid[0:F, 0:F]
    ck = (x + y) % 2 == n % 2
    assert samples == k // stride
    assert np.array_equal(nsew, np.stack([np.where(ck, right, left), np.where(ck, left, right),
                                          np.where(ck, top, bottom), np.where(ck, bottom, top)]))
