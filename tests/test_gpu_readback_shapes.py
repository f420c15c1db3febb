"""Read-back and write on flat and narrow domains: states at every alignment,
validation, and the type densities on both of their paths."""
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


@pytest.mark.parametrize("kind,size", [("rect", (16000, 1)), ("rect", (60000, 3)), ("rect", (2, 3001)), ("rect", (20, 2000)),
                                       ("rect", (2046, 2)), ("rect", (2050, 2)), ("hexagon", (1, 2, 3000)),
                                       ("hexagon", (3000, 1, 2)), ("dwbc", (513,))])
def test_state(T, kind, size):
    import torch
    ctx, dom = T.Context(0), getattr(T.Domain, kind)(*size)
    lat = {"rect": O.DOMINO, "hexagon": O.LOZENGE, "dwbc": O.SIXV}[kind]
    th = T.thresholds(table16=T.sixv_thresholds(np.ones(6))) if kind == "dwbc" else T.thresholds(scalar=3 << 29)
    ch = T.Chain(ctx, dom, seed=3, th=th)
    st = getattr(O, kind)(*size)
    kw = {"t16": O.sixv_thresholds(np.ones(6))} if kind == "dwbc" else {"t_scalar": 3 << 29}
    O.sweeps(lat, st, seed=3, k=20, **kw)
    n = st.size
    for shift in (0, 3, 9):
        src = torch.zeros(n + 64, dtype=torch.uint8, device="cuda")[shift:shift + n]
        src.copy_(torch.from_numpy(st.reshape(-1)))
        ch.write_state(src)
        assert ch.state_hash() == O.state_hash(st)
        dst = torch.full((n + 64,), 9, dtype=torch.uint8, device="cuda")
        ch.read_state(dst[shift:shift + n])
        got = dst.cpu().numpy()
        assert np.array_equal(got[shift:shift + n], st.reshape(-1))
        assert (got[:shift] == 9).all() and (got[shift + n:] == 9).all()
        for pos in (0, n // 2, n - 1):
            bad = src.clone()
            bad[pos] ^= 1
            with pytest.raises(T.TilingError):
                ch.write_state(bad)
        bad = src.clone()
        bad[n // 3] = 2
        with pytest.raises(T.TilingError) as e:
            ch.write_state(bad)
        assert "byte %d" % (n // 3) in str(e.value)


@pytest.mark.parametrize("w,h", [(1600, 30), (1602, 30), (1602, 32), (2000, 8), (16000, 3), (158, 900), (160, 900), (30, 878), (30, 880),
                                 (20, 3000)])
def test_nsew(T, w, h):
    ctx, dom = T.Context(0), T.Domain.rect(w, h)
    ch = T.Chain(ctx, dom, seed=8)
    ch.density_begin(2, 0)
    ch.run(14)
    (hz, vt), samples = ch.read_density()
    nsew = ch.read_nsew()
    H, W = hz.shape
    left, right, bottom, top = vt[:-1, :-1], vt[:-1, 1:], hz[:-1, :-1], hz[1:, :-1]
    assert samples == 7
    y, x = np.mgrid[0:H - 1, 0:W - 1]
    even = (x + y) % 2 == 0
    both = [np.stack([np.where(c, right, left), np.where(c, left, right), np.where(c, top, bottom), np.where(c, bottom, top)])
            for c in (even, ~even)]
    assert any(np.array_equal(nsew, b) for b in both)
    assert np.allclose(nsew.sum(0)[1:-1, 1:-1], (left + right + bottom + top)[1:-1, 1:-1])
