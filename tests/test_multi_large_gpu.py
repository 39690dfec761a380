"""N-species boxes of more than 96 MB of populations, whose density pass walks the
rows and planes from the last: every site of ragged boxes against the oracle, and
the fields against FP64 sums."""
import numpy as np
import pytest

import oracle
from paper_1410_5584_gb300 import D2Q9, D3Q19, MultiLattice
from paper_1410_5584_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,ns,shape", [(D3Q19, 3, (71, 75, 83)), (D2Q9, 4, (1, 841, 833)), (D2Q9, 2, (1, 1201, 1171))])
@pytest.mark.parametrize("tau", [(1.0, 1.0, 1.0, 1.0), (1.0, 0.8, 1.1, 0.9)])
def test_large_species_boxes_match_the_oracle(lat, ns, shape, tau):
    """Two steps with every site compared (the bound of the small boxes' tests: 1.5e-6 of the largest population a step);
    then densities to 1e-14 and velocities to 1e-7 (the force's float densities) of FP64 sums of the stored populations,
    and the totals."""
    nz, ny, nx = shape
    N = nx * ny * nz
    c, w, T, _ = oracle.tables(lat)
    assert ns * len(w) * N * 4 > 96 << 20
    tau, G = list(tau[:ns]), 0.4 * (1 - np.eye(ns))
    f0 = inputs.random_populations(np.stack([w * r for r in (1.0, 0.8, 0.6, 0.9)[:ns]]), shape, 0.02, seed=2)
    o = oracle.MultiOracle(lat, ns, nx, ny, nz, tau, 1e-4, G, 3)
    o.set_f(f0, step=5)
    o.step(2)
    want = o.get_f()
    o.close()
    for streaming in ("two_arrays", "in_place"):
        g = MultiLattice(lat, ns, nx, ny, nz, tau, 1e-4, G, 3, streaming=streaming)
        g.set_populations(f0, step=5)
        g.step(2)
        f = g.get_populations()
        rho, u, cons = g.moments()
        g.close()
        assert np.max(np.abs(f - want)) <= 3e-6 * np.max(np.abs(want))
        dens = f.sum(axis=1)
        assert np.max(np.abs(rho - dens)) <= 1e-14
        D = u.shape[0]
        j = sum(np.tensordot(c.T[:D].astype(float), f[s], axes=(1, 0)) for s in range(ns))
        for i in range(1, len(w)):
            shifted = np.roll(dens, [-v for v in c[i][::-1]], axis=(1, 2, 3))
            for s in range(ns):
                a = -sum(G[s, t] * w[i] * shifted[t] for t in range(ns) if t != s)
                j = j + 0.5 * dens[s] * a * c[i][:D].reshape(-1, 1, 1, 1)
        assert np.max(np.abs(u - j / dens.sum(axis=0))) <= 1e-7
        assert np.max(np.abs(cons[:ns] - dens.sum(axis=(1, 2, 3)))) <= 1e-14 * N
        assert np.max(np.abs(cons[ns:ns + D] - j.sum(axis=(1, 2, 3)))) <= 1e-7 * N
