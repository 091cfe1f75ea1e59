"""Steps of one call against a host stable sort, particle by particle.  Photons keep
their u_phi to the bit, so distinct values name them; a push alone (the same kernel,
slots in place) gives every step's cells, and the stable sorts of those cells in
turn give the order that the call has to end with.  Grids below and above the size
where the scan takes a third launch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("nr,nth,n,steps", [(4, 4, 500, 3), (37, 62, 30000, 5), (128, 128, 200000, 4),
                                            (1100, 1000, 1500000, 3)])
def test_every_particle_in_its_place(prec, nr, nth, n, steps):
    import torch
    from paper_2503_04558_gb300 import grpic as G
    gc = G.Config(nr, nth, 0.9, 1.3, 1.3 * 1.02 ** min(nr, 150) + 0.5, precision=prec,
                  damp_cells=min(8, nr))
    rng = np.random.default_rng(nr)
    i = np.minimum((nr * rng.random(n) ** 2).astype(np.int32), nr - 1)   # many next to r_in, where the steps cross cells
    j = rng.integers(0, nth, n).astype(np.int32)
    o = rng.uniform(0.05, 0.95, (2, n))
    r, th = gc.r_in * np.exp((i + o[0]) * gc.dx1), (j + o[1]) * gc.dth
    dt = np.float32 if prec == 32 else np.float64
    u3 = ((np.arange(n) + 1.0) / n).astype(dt)          # distinct in FP32 too (n < 2^24)
    u3 *= np.where(rng.random(n) < 0.5, -1, 1).astype(dt)
    u = [(4 * rng.standard_normal(n)).astype(dt), (4 * r * rng.standard_normal(n)).astype(dt), u3]
    tag = np.full(n, 3, np.uint32)

    def state():
        ctx, F, S = G.Context(gc), G.Fields(gc), G.ParticleSet(gc, n)
        if prec == 32:
            o2 = np.where(j == nth - 1, 1.0 - o[1], o[1])
            S.load(o[0].astype(dt), o2.astype(dt), *u, tag, j * nr + i)
        else:
            S.load(r, th, *u, tag)
        return ctx, F, S

    ctx, F, S = state()
    order, moved = np.arange(n), 0
    last = j * nr + i
    for _ in range(steps):
        ctx.push(S, F)
        assert ctx.sync() == 0
        live = S.a.tag.cpu().numpy().view(np.uint32) < G.DEAD
        if prec == 32:
            cell = S.a.cell.cpu().numpy()
        else:
            x1, x2 = S.a.x1.cpu().numpy(), S.a.x2.cpu().numpy()
            ci = np.clip(np.floor((np.log(x1) - np.log(gc.r_in)) / gc.dx1), 0, nr - 1).astype(np.int64)
            cell = np.minimum(np.floor(x2 / gc.dth), nth - 1).astype(np.int64) * nr + ci
        order = order[live[order]]
        order = order[np.argsort(cell[order], kind="stable")]
        moved += int(np.sum(cell[order] != last[order]))
        last = cell
    assert moved > n // 50
    ctx, F, S = state()
    ctx.step(S, F, steps)
    assert ctx.sync() == 0
    h = S.host()
    assert len(h["u3"]) == len(order)
    assert np.array_equal(h["u3"], u3[order])
