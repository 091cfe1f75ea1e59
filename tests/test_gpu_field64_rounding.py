"""One FP64 field update rounds a value of the fields' size once: with a step so short
that the update moves a field by about a thousandth of its size, the correctly
rounded sum is the oracle's in all but a few entries per cent (where the two
increments, which agree to a few 1e-16 of themselves, fall on either side of a
tie: about 1e-3 of the entries, more where a field's value is small).  A second
rounding of that size would change about a quarter of them."""
import numpy as np
import pytest

import oracle as O
from gpu_common import configs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nr,nth,N", [(57, 14, 7), (128, 128, 7), (130, 62, 2), (40, 30, 1)])
def test_update_rounds_a_field_once(nr, nth, N):
    import torch
    from paper_2503_04558_gb300 import grpic as G
    oc, gc = configs(nr, nth, 0.9, 1.3, 20.0, dt=1e-5, n_fld_iter=N, damp_cells=0)
    rng = np.random.default_rng(nr)
    X = [rng.uniform(0.5, 2.0, (nth + 1, oc.ld)) for _ in range(6)]
    for x in X:
        x[:, :2], x[:, nr:] = x[:, 2:3], x[:, nr - 1:nr]  # guard copies
    J = [np.zeros((nth + 1, oc.ld)) for _ in range(3)]
    ctx = G.Context(gc)
    F = G.Fields(gc)
    for t, x in zip(F.D + F.B, X):
        t.copy_(torch.from_numpy(x))
    ctx.field_update(F)
    assert ctx.sync() == 0
    got = [t.cpu().numpy() for t in F.D + F.B]
    D, B = [x.copy() for x in X[:3]], [x.copy() for x in X[3:]]
    O.field_update(oc, D, B, J)
    for k, (x, y, x0) in enumerate(zip(got, D + B, X)):
        x, y, x0 = (v[2:nth - 2, 6:nr - 4] for v in (x, y, x0))
        assert np.median(np.abs(y - x0)) > 1e-8, k   # the fields do move
        assert np.mean(x == y) > 0.95, (k, np.mean(x == y))
