"""grpic_horizon_flux: calls on one context from several threads and streams at a
time."""
import threading

import pytest

pytestmark = pytest.mark.gpu


def _setup(nf):
    from paper_2503_04558_gb300 import grpic as G
    gc = G.Config(48, 64, 0.9, 1.3, 20.0)
    ctx = G.Context(gc)
    out = []
    for k in range(nf):
        F = G.Fields(gc)
        ctx.init_fields(F, G.SPLIT_MONOPOLE, 1.0 + k)
        for i, t in enumerate(F.D + F.B):
            t.mul_(1.0 + 0.01 * i)
        out.append(F)
    return G, ctx, out


def test_threads_on_one_context():
    import torch
    nt, calls, iH = 4, 200, 8
    G, ctx, Fs = _setup(nt)
    want = [G.horizon_flux(ctx, F, iH) for F in Fs]
    assert len(set(want)) == nt
    torch.cuda.synchronize()
    bad = []

    def work(k):
        torch.cuda.set_device(0)
        s = torch.cuda.Stream()
        for _ in range(calls):
            v = G.horizon_flux(ctx, Fs[k], iH, stream=s)
            if v != want[k]:
                bad.append((k, v))
                return

    ts = [threading.Thread(target=work, args=(k,)) for k in range(nt)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad, bad
