"""The FP32 form's roundings.  Next to the axis J^phi is decided by a few particles
whose angular velocity goes like 1 / sin(theta): one FP32 rounding of the fields or
currents of a step moves it by up to 1e-3 of its size in the next one, so a change
in the order of operations shows in a run's outputs however small it is.  The
checksums are those of the first kernels of the FP32 form (sm_103a), on inputs from
integer hashes: a field update alone, and one push of particles so far apart that
every entry of J is a single particle's."""
import zlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _hash(shape, seed, scale=1.0):
    """Values in [-scale, scale), the same on every machine."""
    x = (np.arange(int(np.prod(shape)), dtype=np.uint64) + np.uint64(seed * 1000003 + 12345)) & np.uint64(0xFFFFFFFF)
    for m in (0x7FEB352D, 0x846CA68B):
        x ^= x >> np.uint64(16)
        x = (x * np.uint64(m)) & np.uint64(0xFFFFFFFF)
    x ^= x >> np.uint64(15)
    return (scale * (x.astype(np.float64) * 2.0 ** -31 - 1.0)).astype(np.float32).reshape(shape)


def _crc(arrays):
    c = 0
    for a in arrays:
        c = zlib.crc32(np.ascontiguousarray(a).tobytes(), c)
    return c


def field_bits(nr, nth, N):
    import torch
    from paper_2503_04558_gb300 import grpic as G
    cfg = G.Config(nr, nth, 0.9, 1.3, 20.0, precision=32, n_field_iter=N, damp_cells=8)
    ctx = G.Context(cfg)
    F = G.Fields(cfg)
    for k, t in enumerate(F.D + F.B + F.J):
        t.copy_(torch.from_numpy(_hash((nth + 1, cfg.ld), k, 1.0 if k < 6 else 1e-2)))
    ctx.field_update(F)
    assert ctx.sync() == 0
    # half-theta components end one row earlier; + 0 makes -0 and 0 alike
    return _crc([t.cpu().numpy()[:nth + (k not in (1, 3, 5))] + np.float32(0) for k, t in enumerate(F.D + F.B)])


def push_bits(pusher, tol):
    import torch
    from paper_2503_04558_gb300 import grpic as G
    nr, nth = 192, 96
    cfg = G.Config(nr, nth, 0.9, 1.3, 20.0, precision=32, pusher=pusher, fp64_radius=3.0, push_tol=tol)
    ctx = G.Context(cfg)
    F = G.Fields(cfg)
    for k, t in enumerate(F.D + F.B):
        t.copy_(torch.from_numpy(_hash((nth + 1, cfg.ld), 20 + k, 0.3)))
    out = []
    for s in range(6):
        ii, jj = (x.ravel() for x in np.meshgrid(np.arange(3, nr - 3, 6), np.arange(3 * (s % 2), nth, 6)))
        n = len(ii)
        o1, o2 = 0.5 + _hash(n, 40 + s, 0.5), 0.5 + _hash(n, 50 + s, 0.5)
        for o, m in ((o1, 60), (o2, 70)):  # two thirds next to an edge, so that many leave their cell
            near = np.arange(n) % 3
            o[near == 0] = 0.03 + 0.03 * _hash(n, m + s)[near == 0]
            o[near == 1] = 0.97 - 0.029 * np.abs(_hash(n, m + s)[near == 1])
        r = (1.3 * np.exp((ii + 0.5) * cfg.dx1)).astype(np.float32).round(3)
        u = [_hash(n, 80 + s), _hash(n, 90 + s) * r, _hash(n, 100 + s) * r]
        S = G.ParticleSet(cfg, n)
        S.load(o1, o2, *u, (np.arange(n) % 2).astype(np.uint32), (jj * nr + ii).astype(np.int32))
        for t in F.J:
            t.zero_()
        ctx.push(S, F)
        assert ctx.sync() == 0
        a = S.a
        out += [t.cpu().numpy() for t in (a.x1, a.x2, a.u1, a.u2, a.u3, a.tag, a.cell)]
        out += [t.cpu().numpy() + np.float32(0) for t in F.J]
    return _crc(out)


# one launch, two (16-byte rows and odd ones; small and wide tiles), three, four
FIELD = {(60, 20, 1): 0x94804699, (60, 20, 7): 0x0d65abe0, (57, 14, 7): 0xdf8b6efc, (700, 200, 7): 0x025bccdf,
         (301, 182, 7): 0x533892e0, (60, 20, 9): 0xf113978c, (702, 202, 9): 0x35490453, (130, 44, 12): 0x103327f8}
PUSH = {(0, 0.0): 0xdcc8fa17, (0, 1e-06): 0xb62e13bf, (1, 0.0): 0xf506967d, (1, 1e-06): 0x80033e84}


@pytest.mark.parametrize("nr,nth,N", list(FIELD))
def test_field_update_keeps_its_bits(nr, nth, N):
    assert field_bits(nr, nth, N) == FIELD[nr, nth, N]


@pytest.mark.parametrize("pusher,tol", list(PUSH))
def test_push_and_deposit_keep_their_bits(pusher, tol):
    assert push_bits(pusher, tol) == PUSH[pusher, tol]
