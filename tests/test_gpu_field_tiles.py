"""The field update at the edges of its tiles and strips: grids one point
around their widths, the smallest grid, row strides that are no multiple of 16
bytes and beyond n_r + 4, few and many correctors, row ranges; against the
oracle's update on random fields and currents."""
import numpy as np
import pytest

import oracle as O
from gpu_common import configs, flux_form

pytestmark = pytest.mark.gpu

# FP64: a few hundred roundings of values of the fields' size.  FP32: the
# tables' and values' 6e-8 over 8 stages of differences, dt / cell ~ 0.5.
TOL = {64: 1e-12, 32: 2e-5}


def _run(prec, nr, nth, N, pad=0, rows=None, fused=True):
    import torch
    from paper_2503_04558_gb300 import grpic as G
    oc, gc = configs(nr, nth, 0.9, 1.3, 20.0, precision=prec, n_fld_iter=N, damp_cells=min(8, nr))
    rng = np.random.default_rng(nr * 1000 + nth)
    dt = np.float64 if prec == 64 else np.float32
    D, B = O.init_fields(oc, O.WALD, 1.0)
    D = [(x + 0.05 * rng.standard_normal(x.shape) * (np.abs(x).max() + 0.1)).astype(dt).astype(np.float64) for x in D]
    B = [x.astype(dt).astype(np.float64) for x in B]
    J = [1e-3 * rng.standard_normal(x.shape) for x in D]
    ctx = G.Context(gc)
    ctx.set_field_path(fused)
    F = G.Fields(gc, ld=gc.ld + pad)
    Jf = flux_form(oc, J)
    for dst, src in zip(F.D + F.B + F.J, D + B + Jf):
        dst.fill_(7.0)
        dst[:, :gc.ld] = torch.from_numpy(src.astype(dt))
    if rows is None:
        ctx.field_update(F)
    else:
        import ctypes as C
        fc = F.c()
        assert ctx.lib.grpic_field_update_rows(ctx.h, C.byref(fc), rows[0], rows[1], None) == 0
        torch.cuda.synchronize()
    assert ctx.sync() == 0
    got = [t.cpu().numpy() for t in F.D + F.B]
    O.field_update(oc, D, B, J)
    return oc, gc, got, D + B


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("nr,nth,N,pad", [(4, 4, 7, 0), (57, 14, 7, 1), (58, 16, 3, 0), (59, 30, 2, 2), (118, 62, 1, 0),
                                          (121, 40, 7, 3), (249, 254, 7, 0), (600, 402, 7, 1), (70, 20, 12, 0)])
def test_update_matches_oracle(prec, nr, nth, N, pad):
    oc, gc, got, want = _run(prec, nr, nth, N, pad)
    for k, (x, y) in enumerate(zip(got, want)):
        top = nth if k in (1, 3, 5) else nth + 1   # half-theta components end one row earlier
        assert np.max(np.abs(x[:top, :gc.ld] - y[:top])) <= TOL[prec] * max(1.0, np.max(np.abs(y))), k
        assert np.all(x[:, gc.ld:] == 7.0), k      # columns past the guards are the caller's


@pytest.mark.parametrize("nr,nth,N", [(57, 14, 7), (301, 182, 7), (64, 48, 2)])
def test_fp32_launch_shapes_agree_bit_for_bit(nr, nth, N):
    a = _run(32, nr, nth, N)[2]
    b = _run(32, nr, nth, N, fused=False)[2]
    assert all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("j0,j1", [(0, 9), (12, 25), (30, 41)])
def test_row_range_leaves_the_rest_and_updates_its_inside(prec, j0, j1):
    N, nr, nth = 2, 66, 40
    oc, gc, got, want = _run(prec, nr, nth, N, rows=(j0, j1))
    full = _run(prec, nr, nth, N)[2]
    lo = j0 + 2 if j0 > 0 else 0          # a wrong row moves half a row inwards per stage
    hi = j1 - 2 if j1 < nth + 1 else nth
    for k, (x, y) in enumerate(zip(got, full)):
        assert np.array_equal(x[lo:hi], y[lo:hi]), k
