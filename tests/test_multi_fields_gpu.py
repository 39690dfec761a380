"""flbm_mmoments into the caller's arrays: by either route (copied from device
scratch, stored by the kernel) and after an error."""
import ctypes

import numpy as np
import pytest

from paper_1410_5584_gb300 import D2Q9, MultiLattice
from paper_1410_5584_gb300 import flbm as F
from paper_1410_5584_gb300 import inputs
import oracle

pytestmark = pytest.mark.gpu


def _state(shape, ns=3, seed=4):
    c, w, T, N = oracle.tables(D2Q9)
    return inputs.random_populations(np.stack([w * r for r in (1.0, 0.8, 0.6)[:ns]]), shape, 0.02, seed=seed)


def _moments_into(g, *arrays):
    ptrs = [None if a is None else a.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for a in arrays]
    return F.lib().flbm_mmoments(g._h, *ptrs)


@pytest.mark.parametrize("shape", [(1, 40, 30), (1, 1100, 1030)])
def test_arrays_are_left_alone_when_the_state_is_not_finite(shape):
    """A small box and one of 27 MB of densities."""
    nz, ny, nx = shape
    f0 = _state(shape)
    f0[1, :, 0, 3, 3] = -0.01
    g = MultiLattice(D2Q9, 3, nx, ny, 1, [1.0, 0.8, 1.1], 1e-4, 0.3 * (1 - np.eye(3)), 1)
    g.set_populations(f0)
    g.step(1)
    rng = np.random.default_rng(2)
    out = [rng.random(3 * nx * ny), rng.random(2 * nx * ny), rng.random(6)]
    before = [o.copy() for o in out]
    assert _moments_into(g, *out) == F.ENONFINITE
    assert all(np.array_equal(o, b) for o, b in zip(out, before))
    g.close()


@pytest.mark.parametrize("shape", [(1, 40, 30), (1, 1100, 1030)])
def test_fields_into_arrays_at_odd_bytes_and_without_some(shape):
    """The fields are copied: an array may start at any byte, and each may be left out (a small box and one of 27 MB of
    densities)."""
    nz, ny, nx = shape
    N = nx * ny
    g = MultiLattice(D2Q9, 3, nx, ny, 1, [1.0, 0.8, 1.1], 1e-4, 0.3 * (1 - np.eye(3)), 1)
    g.set_populations(_state(shape))
    g.step(2)
    rho, u, cons = (a.ravel() for a in g.moments())
    raw = np.zeros(5 * N * 8 + 64, dtype=np.uint8)
    odd = [np.frombuffer(raw.data, np.float64, n, offset) for n, offset in ((3 * N, 4), (2 * N, 3 * N * 8 + 13))]
    got = np.empty(6)
    assert _moments_into(g, odd[0], odd[1], got) == F.OK
    assert np.array_equal(odd[0], rho) and np.array_equal(odd[1], u) and np.array_equal(got, cons)
    assert not raw[:4].any() and not raw[-64 + 13:].any()
    for keep in ((0,), (1,), (2,), (0, 2), ()):
        out = [np.full(a.size, 7.0) for a in (rho, u, cons)]
        assert _moments_into(g, *(o if k in keep else None for k, o in enumerate(out))) == F.OK
        for k, (o, want) in enumerate(zip(out, (rho, u, cons))):
            assert np.array_equal(o, want) if k in keep else np.all(o == 7.0)
    g.close()
