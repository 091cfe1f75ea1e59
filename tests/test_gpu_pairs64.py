"""The FP64 push's early correctors at the edges of the range in which they run in
double-FP32 pairs: small radii at high spin with the largest step, either side of the
angular limit, photons of very small and very large momentum.  No fields, so that the momentum
before the geodesic step is the loaded one."""
import numpy as np
import pytest

import oracle as O
from gpu_common import configs

pytestmark = pytest.mark.gpu


def _push(gc, r, th, u, tag):
    from paper_2503_04558_gb300 import grpic as G
    ctx = G.Context(gc)
    F = G.Fields(gc)
    S = G.ParticleSet(gc, len(r))
    S.load(r, th, *u, tag)
    ctx.push(S, F)
    assert ctx.sync() == 0
    return [getattr(S.a, k).cpu().numpy() for k in ("x1", "x2", "u1", "u2", "u3")]


def _oracle(oc, r, th, u, tag):
    P = O.Particles(r.copy(), th.copy(), *(x.copy() for x in u), tag.copy())
    Z = [np.zeros((oc.nth + 1, oc.ld)) for _ in range(6)]
    st, _, _ = O.push_deposit(oc, P, Z[:3], Z[3:])
    assert st == 0
    return P.r, P.th, P.u1, P.u2, P.u3


@pytest.mark.parametrize("dt", [0.002, 0.0125, 0.02])
@pytest.mark.parametrize("sigma", [0.1, 3.0])
def test_every_particle_to_a_few_roundings(dt, sigma):
    """r_in = 0.95 at a = 0.995: dt/2 / r on both sides of 2^-7.  Per particle:
    positions within 1e-15 of themselves (4 roundings: one of the value on each
    side, the changes' errors are hundreds of times below), momenta within 4e-15 of
    the momentum's size (changes of up to a tenth of it, each formed in ten to
    twenty roundings on each side)."""
    oc, gc = configs(20, 64, 0.995, 0.95, 2.0, dt=dt)
    rng = np.random.default_rng(int(dt * 1e5))
    n = 20000
    r = 0.96 + 0.9 * rng.random(n)
    # theta where dt/2 dphi/dt spreads over 1/10 .. 10 times its limit, away from
    # the pole by ten times a step's move
    th = np.clip(np.arccos(rng.uniform(-1, 1, n)), 0.25, np.pi - 0.25)
    u = [sigma * rng.standard_normal(n), sigma * rng.standard_normal(n) * r,
         sigma * rng.standard_normal(n) * r * np.sin(th)]
    tag = np.array([0, 1, 2, 3], np.uint32)[np.arange(n) % 4]
    got, ref = _push(gc, r, th, u, tag), _oracle(oc, r, th, u, tag)
    size = np.sqrt(ref[2] ** 2 + (ref[3] / r) ** 2 + (ref[4] / (r * np.sin(th))) ** 2)
    size = np.maximum(size, np.where(tag == 3, 0.0, 0.1))
    assert np.max(np.abs(got[0] - ref[0]) / ref[0]) < 1e-15
    assert np.max(np.abs(got[1] - ref[1]) / ref[1]) < 1e-15
    for k, s in ((2, 1.0), (3, r), (4, r * np.sin(th))):
        assert np.max(np.abs(got[k] - ref[k]) / (s * size)) < 4e-15, k


@pytest.mark.parametrize("power", [-10, -29, -31, -41, -55, -62, 29, 31, 45, 55, 62, 100, 130, 140])
def test_a_photon_path_does_not_depend_on_its_energy(power):
    """The massless right-hand side is homogeneous in u, so momenta scaled by a power
    of two give the same path and scaled momenta, to the roundings above."""
    oc, gc = configs(24, 64, 0.995, 1.2, 3.0, dt=0.015)
    rng = np.random.default_rng(8)
    n = 20000
    r, th = 1.25 + rng.random(n), np.clip(np.arccos(rng.uniform(-1, 1, n)), 0.4, np.pi - 0.4)
    u = [rng.standard_normal(n), rng.standard_normal(n) * r, rng.standard_normal(n) * r * np.sin(th)]
    tag = np.full(n, 3, np.uint32)
    f = 2.0 ** power
    a, b = _push(gc, r, th, u, tag), _push(gc, r, th, [x * f for x in u], tag)
    size = np.sqrt(u[0] ** 2 + (u[1] / r) ** 2 + (u[2] / (r * np.sin(th))) ** 2)
    assert np.max(np.abs(b[0] - a[0]) / a[0]) < 1e-15
    assert np.max(np.abs(b[1] - a[1]) / a[1]) < 1e-15
    for k, s in ((2, 1.0), (3, r), (4, r * np.sin(th))):
        assert np.max(np.abs(b[k] / f - a[k]) / (s * size)) < 4e-15, k
