"""The FP64 push's cell search, row sines and deposit across the grids that pick
their form: columns by the series (1 to 16 terms) or the logarithm, row sines
from the table or the library (n_theta below 63), both shapes and pushers, cell
edges and the rows at the axis.  One push against the oracle; then steps whose
neighbour sorts rely on the push and the sort agreeing on every cell."""
import numpy as np
import pytest

import oracle as O
from gpu_common import configs, flux_form, relerr

pytestmark = pytest.mark.gpu

GRIDS = [(4, 4, 1.3, 30.0),       # dx1 = 0.78: logarithm, library sines
         (16, 62, 1.3, 20.0),     # dx1 = 0.171: 16 terms, library sines
         (16, 64, 1.3, 20.0),     # the same columns, row table
         (12, 100, 1.3, 20.0),    # dx1 = 0.228: logarithm, row table
         (90, 64, 1.3, 50.0),
         (700, 130, 1.3, 1.5),    # dx1 = 2e-4: 2 to 3 terms
         (2000, 64, 1.3, 1.4)]    # dx1 = 3.7e-5: logarithm (too narrow for the FP32 guess)


def _particles(oc, n, seed):
    rng = np.random.default_rng(seed)
    x1 = rng.random(n) * oc.nr
    x2 = rng.random(n) * oc.nth
    k = n // 8
    x1[:k] = np.minimum(np.round(x1[:k]) + 1e-9, oc.nr - 1e-3)       # just above a column's edge
    x1[k:2 * k] = np.maximum(np.round(x1[k:2 * k]) - 1e-9, 1e-3)     # just below one
    x2[2 * k:3 * k] = np.clip(np.round(x2[2 * k:3 * k]) + 1e-9, 0.3, oc.nth - 0.3)
    x2[3 * k:4 * k] = rng.choice([0.2, oc.nth - 0.2], k) + 0.1 * rng.random(k) - 0.05   # the axis rows
    r = oc.r_in * np.exp(x1 * oc.dx1)
    th = np.clip(x2, 0.1, oc.nth - 0.1) * oc.dth
    u = 0.1 * rng.standard_normal((3, n))
    tag = (np.arange(n) % 2).astype(np.uint32)
    tag[::17] = 3
    return O.Particles(r, th, u[0], u[1] * r, u[2] * r * np.sin(th), tag)


@pytest.mark.parametrize("shape,pusher", [(1, 0), (1, 1), (3, 0)])
@pytest.mark.parametrize("nr,nth,r_in,r_out", GRIDS)
def test_one_push_matches_oracle(nr, nth, r_in, r_out, shape, pusher):
    import torch
    from paper_2503_04558_gb300 import grpic as G
    oc, gc = configs(nr, nth, 0.9, r_in, r_out, shape=shape, pusher=pusher, damp_cells=min(8, nr))
    ctx = G.Context(gc)
    F = G.Fields(gc)
    ctx.init_fields(F, G.WALD, 1.0)
    D, B = O.init_fields(oc, O.WALD, 1.0)
    P = _particles(oc, 20000, nr)
    S = G.ParticleSet(gc, P.n)
    S.load(P.r, P.th, P.u1, P.u2, P.u3, P.tag)
    ctx.push(S, F)
    st = ctx.sync()
    so, J, _ = O.push_deposit(oc, P, D, B)
    assert st == so
    t = S.a.tag.cpu().numpy().view(np.uint32)
    assert np.array_equal(t, P.tag)
    for k, ref in (("x1", P.r), ("x2", P.th), ("u1", P.u1), ("u2", P.u2), ("u3", P.u3)):
        assert relerr(getattr(S.a, k).cpu().numpy(), ref) < 1e-12, k
    for k, ref in enumerate(flux_form(oc, J)):
        assert relerr(F.J[k].cpu().numpy(), ref) < 1e-11, ("J", k)


@pytest.mark.parametrize("nr,nth,r_in,r_out", [GRIDS[1], GRIDS[2], GRIDS[3], GRIDS[4]])
def test_steps_keep_every_particle_and_its_order(nr, nth, r_in, r_out):
    """Four steps in one call (deferred sorts): the neighbour sorts place every
    live particle once, in the order of the oracle's stable sort."""
    from paper_2503_04558_gb300 import grpic as G
    oc, gc = configs(nr, nth, 0.9, r_in, r_out)
    ctx = G.Context(gc)
    F = G.Fields(gc)
    ctx.init_fields(F, G.WALD, 1.0)
    D, B = O.init_fields(oc, O.WALD, 1.0)
    P = _particles(oc, 20000, 7)
    S = G.ParticleSet(gc, P.n)
    S.load(P.r, P.th, P.u1, P.u2, P.u3, P.tag)
    ctx.step(S, F, 4)
    st = ctx.sync()
    for _ in range(4):
        so, P, _ = O.step(oc, P, D, B)
    assert st in (0, 4, 5)
    h = S.host()
    assert len(h["tag"]) == P.n
    assert np.array_equal(h["tag"], P.tag)
    assert np.median(np.abs(h["x1"] - P.r) / P.r) < 1e-13
    assert np.mean(np.abs(h["x2"] - P.th) < 1e-8) > 0.999


@pytest.mark.parametrize("sigma", [0.05, 0.6])
@pytest.mark.parametrize("n_iter", [1, 2, 3, 5])
def test_correctors_in_pairs_keep_fp64(n_iter, sigma):
    """The early correctors run in double-FP32 pairs where their error leaves the
    last one under an eighth of a rounding (dt <= 0.02, off the axis).  Positions
    then agree with the oracle's to a few roundings of FP64 (2^-53 = 1.1e-16; the
    two push formulas round differently in about ten places of a step whose move
    is at most 1e-2), near the axis, where FP64 takes over, included."""
    from paper_2503_04558_gb300 import grpic as G
    oc, gc = configs(128, 128, 0.9, 1.3, 50.0, n_push_iter=n_iter)
    assert gc.dt <= 0.02
    ctx = G.Context(gc)
    F = G.Fields(gc)
    ctx.init_fields(F, G.WALD, 1.0)
    D, B = O.init_fields(oc, O.WALD, 1.0)
    P = _particles(oc, 40000, 11)
    f = sigma / 0.1
    P.u1, P.u2, P.u3 = P.u1 * f, P.u2 * f, P.u3 * f
    S = G.ParticleSet(gc, P.n)
    S.load(P.r, P.th, P.u1, P.u2, P.u3, P.tag)
    ctx.push(S, F)
    st = ctx.sync()
    so, J, _ = O.push_deposit(oc, P, D, B)
    assert st == so
    mid = np.abs(P.th - np.pi / 2) < 1.2
    for k, ref, tol in (("x1", P.r, 2e-15), ("x2", P.th, 2e-15), ("u1", P.u1, 1e-13), ("u2", P.u2, 1e-13)):
        got = getattr(S.a, k).cpu().numpy()
        assert relerr(got[mid], ref[mid]) < tol, k
        assert relerr(got, ref) < 1e-12, k
