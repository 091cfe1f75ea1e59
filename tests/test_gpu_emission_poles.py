"""Emission next to the poles (FP64 push with radiation): momenta carried by u_phi,
so that Gamma depends on sin(theta) at 1e-7 .. 1e-5 rad from either pole.  A step
too short to move anything takes the oracle's decision for every particle."""
import numpy as np
import pytest

import oracle as O
from gpu_common import configs, relerr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pole", ["north", "south"])
def test_emission_at_a_pole_is_the_oracles(pole):
    from paper_2503_04558_gb300 import grpic as G
    oc, gc = configs(32, 32, 0.9, 1.3, 20.0, dt=1e-13, qw=(0.0, 0.0, 0.0, 0.0), radiation=1, gamma_thr=100.0,
                     eps_ph=4.0, tau=0.0)
    for k in ("radiation", "gamma_thr", "eps_ph", "tau"):
        setattr(gc, k, getattr(oc, k))
    rng = np.random.default_rng(3)
    n = 4000
    r = 1.4 + 10.0 * rng.random(n)
    d = 10.0 ** rng.uniform(-7.0, -5.0, n)
    th = d if pole == "north" else np.pi - d
    gam = np.where(np.arange(n) % 4 == 0, 90.0 + 9.9 * rng.random(n), 100.1 + 19.9 * rng.random(n))
    gpp = 1.0 / ((r * r + 0.81 * np.cos(th) ** 2) * np.sin(th) ** 2)  # gamma^phph
    u3 = np.sqrt((gam * gam - 1.0) / gpp) * np.where(rng.random(n) < 0.5, -1.0, 1.0)
    P = O.Particles(r, th, np.zeros(n), np.zeros(n), u3, (np.arange(n) % 2).astype(np.uint32))
    ctx = G.Context(gc)
    F = G.Fields(gc)
    D, B = ([np.zeros((oc.nth + 1, oc.ld)) for _ in range(3)] for _ in range(2))
    S = G.ParticleSet(gc, 2 * n)
    S.load(P.r, P.th, P.u1, P.u2, P.u3, P.tag)
    ev = []
    st, P, _ = O.step(oc, P, D, B, events=ev)
    assert st == 0 and ev[0][0] == int(np.sum(gam > 100.0))
    ctx.step(S, F, 1)
    assert ctx.sync() == 0
    h = S.host()
    assert np.array_equal(h["tag"], P.tag)  # a photon behind every emitter, the slots in the oracle's order
    assert relerr(h["u3"], P.u3) < 1e-10
