"""The FP32 form's roundings.  Next to the axis J^phi is decided by a few particles
whose angular velocity goes like 1 / sin(theta): one FP32 rounding of the fields or
currents of a step moves it by up to 1e-3 of its size in the next one, so a change
in the order of operations shows in a run's outputs however small it is.  The
checksums are those of the first kernels of the FP32 form (sm_103a), on inputs from
integer hashes."""
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


# one launch, two (16-byte rows and odd ones; small and wide tiles), three, four
FIELD = {(60, 20, 1): 0x94804699, (60, 20, 7): 0x0d65abe0, (57, 14, 7): 0xdf8b6efc, (700, 200, 7): 0x025bccdf,
         (301, 182, 7): 0x533892e0, (60, 20, 9): 0xf113978c, (702, 202, 9): 0x35490453, (130, 44, 12): 0x103327f8}


@pytest.mark.parametrize("nr,nth,N", list(FIELD))
def test_field_update_keeps_its_bits(nr, nth, N):
    assert field_bits(nr, nth, N) == FIELD[nr, nth, N]
