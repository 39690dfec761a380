"""The ends of the densities' range in two-species boxes: steps on a uniform flow,
one species subnormal or the sum so large that its reciprocal is."""
import numpy as np
import pytest

import oracle
from paper_1410_5584_gb300 import D2Q9, D3Q19, Lattice

pytestmark = pytest.mark.gpu


def _flow(lat, shape, rho, v=(0.05, 0.02, -0.03)):
    """f = w rho (1 + 3 c.v + 9/2 (c.v)^2 - 3/2 v^2): a uniform flow, which a step leaves as it is."""
    c, w, T, N = oracle.tables(lat)
    v = np.array(v[:2] + ((v[2],) if lat == D3Q19 else (0.0,)))
    cv = c.astype(float) @ v
    f = w * (1 + 3 * cv + 4.5 * cv ** 2 - 1.5 * (v @ v))
    return np.stack([np.broadcast_to((r * f)[:, None, None, None], (len(w),) + shape) for r in rho]), v


@pytest.mark.parametrize("rho", [(1.0, 5e-39), (1e-38, 0.5), (1.0, 1.5e-38), (2e-38, 0.7), (3e-30, 2e-5), (0.4, 8e37),
                                 (0.7, 1e38), (1.2e38, 0.8)])
@pytest.mark.parametrize("lat,shape", [(D2Q9, (1, 6, 33)), (D3Q19, (3, 4, 33))])
@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("options", [{}, {"noise_rho": 1}, {"streaming": 0}])
def test_uniform_flow_at_extreme_densities(lat, shape, rho, tau, options):
    """Momentum and masses after three steps.  Float steps round by 1e-7 of a population, subnormal ones of 1e-40 by
    1e-5 of themselves, 19 of them a site."""
    nz, ny, nx = shape
    f0, v = _flow(lat, shape, rho)
    g = Lattice(lat, nx, ny, nz, tau, 1.0, 0.0, 0.0, 3, rho0_a=rho[0], rho0_b=rho[1], **options)
    g.set_populations(f0)
    g.step(3)
    g.sync()
    f = g.get_populations()
    g.close()
    c, w, T, N = oracle.tables(lat)
    for s in range(2):
        mass = f[s].sum(axis=0) / rho[s]
        assert np.max(np.abs(mass - 1)) <= (5e-4 if rho[s] < 1e-36 else 5e-6)
    j = sum(np.tensordot(c.T.astype(float), f[s] / sum(rho), axes=(1, 0)) for s in range(2))
    assert np.max(np.abs(j - v.reshape(3, 1, 1, 1))) <= 5e-6
