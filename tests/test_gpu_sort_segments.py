"""The general sort's per-cell fix-up at the edges of its register and shared
memory networks: cells of every segment length around 32, 64, 128, 256, the
shared-memory limits and the block network, filled in random slot order; the
result is the stable sort by cell, exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("nr,nth,lengths", [
    (16, 8, [0, 1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257]),
    (37, 10, [3, 100, 200, 2047, 2048, 2049, 5]),
    (200, 160, [7, 40, 0, 90]),
    (8, 4, [16384, 16385, 1]),
])
def test_sort_is_stable_for_every_segment_length(prec, nr, nth, lengths):
    import torch
    from paper_2503_04558_gb300 import grpic as G
    cfg = G.Config(nr, nth, 0.9, 1.2, 20.0, precision=prec)
    ctx = G.Context(cfg)
    rng = np.random.default_rng(5)
    ncell = nr * nth
    per = np.resize(np.array(lengths), ncell) if max(lengths) < 2000 else np.zeros(ncell, np.int64)
    if max(lengths) >= 2000:
        per[rng.choice(ncell, len(lengths), replace=False)] = lengths
    cells = rng.permutation(np.repeat(np.arange(ncell, dtype=np.int32), per))
    n = len(cells)
    o = (0.25 + 0.5 * rng.random((2, n))).astype(np.float32)
    u = rng.standard_normal((3, n))
    tag = (rng.integers(0, 2, n).astype(np.uint32) | np.where(rng.random(n) < 0.05, np.uint32(G.DEAD), np.uint32(0)))
    P = G.ParticleSet(cfg, n)
    if prec == 32:
        P.load(o[0], o[1], *u.astype(np.float32), tag, cells)
    else:
        P.load(cfg.r_in * np.exp((cells % nr + o[0]) * cfg.dx1), (cells // nr + o[1]) * cfg.dth, *u, tag)
    ctx.sort(P)
    assert ctx.sync() == 0
    live = np.nonzero(tag < G.DEAD)[0]
    want = live[np.argsort(cells[live], kind="stable")]
    h = P.host()
    assert len(h["u1"]) == len(want)
    assert np.array_equal(h["u1"], u[0][want].astype(h["u1"].dtype))
    assert np.array_equal(h["u3"], u[2][want].astype(h["u3"].dtype))
    assert np.array_equal(h["tag"], tag[want])
