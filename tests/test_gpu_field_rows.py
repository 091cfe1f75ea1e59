"""grpic_field_update_rows: the rows outside the range are left as they are, bit for
bit, and feed the range's edge rows with the values they have at the call, whatever
the context updated before."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _fields(gc, seed):
    import torch
    from paper_2503_04558_gb300 import grpic as G
    rng = np.random.default_rng(seed)
    F = G.Fields(gc)
    for t in F.D + F.B + F.J:
        t.copy_(torch.from_numpy(rng.standard_normal(tuple(t.shape))).to(t.dtype))
    return F


def _rows(ctx, F, j0, j1):
    fc = F.c()
    assert ctx.lib.grpic_field_update_rows(ctx.h, C.byref(fc), j0, j1, None) == 0
    assert ctx.sync() == 0
    return [t.cpu().numpy() for t in F.D + F.B]


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("nr,nth,N", [(66, 40, 7), (130, 90, 2), (57, 30, 0)])
@pytest.mark.parametrize("where", ["low", "middle", "one row", "high"])
def test_rows_outside_stay_and_history_does_not_matter(prec, nr, nth, N, where):
    from paper_2503_04558_gb300 import grpic as G
    j0, j1 = {"low": (0, 9), "middle": (8, 23), "one row": (11, 12), "high": (nth - 9, nth + 1)}[where]
    gc = G.Config(nr, nth, 0.9, 1.3, 20.0, precision=prec, n_field_iter=N, damp_cells=8)
    new, used = G.Context(gc), G.Context(gc)
    before = [t.cpu().numpy() for t in (lambda F: F.D + F.B)(_fields(gc, 1))]
    a = _rows(new, _fields(gc, 1), j0, j1)
    for seed in (2, 3):
        used.field_update(_fields(gc, seed))
        _rows(used, _fields(gc, seed + 2), max(j0 - 3, 0), min(j1 + 4, nth + 1))
    b = _rows(used, _fields(gc, 1), j0, j1)
    for k, (x, y, z) in enumerate(zip(a, b, before)):
        top = nth + (k not in (1, 3, 5))   # half-theta components end one row earlier
        assert np.array_equal(x[:top], y[:top]), k
        assert np.array_equal(x[:j0], z[:j0]) and np.array_equal(x[j1:], z[j1:]), k
        assert not np.array_equal(x[j0:j1], z[j0:j1]), k


@pytest.mark.parametrize("prec", [64, 32])
def test_edge_rows_read_the_rows_outside(prec):
    """One row at a time from copies of the same state: its update with its two
    neighbours held equals the whole grid's predictor (N = 0), and with a corrector
    it differs from a call whose neighbour rows differ."""
    from paper_2503_04558_gb300 import grpic as G
    nr, nth = 40, 24
    for N in (0, 1):
        gc = G.Config(nr, nth, 0.9, 1.3, 20.0, precision=prec, n_field_iter=N, damp_cells=8)
        ctx = G.Context(gc)
        F = _fields(gc, 5)
        full = _fields(gc, 5)
        ctx.field_update(full)
        full = [t.cpu().numpy() for t in full.D + full.B]
        one = _rows(ctx, F, 10, 11)
        if N == 0:
            assert all(np.array_equal(x[10], y[10]) for x, y in zip(one, full))
        else:
            F2 = _fields(gc, 5)
            for t in F2.D + F2.B:
                t[9].mul_(1.5)
                t[11].mul_(1.5)
            two = _rows(ctx, F2, 10, 11)
            # D^r, D^phi read H of the row below; B^r, B^theta, B^phi E of the row above
            assert not np.array_equal(one[0][10], two[0][10]) and not np.array_equal(one[5][10], two[5][10])
