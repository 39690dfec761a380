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
