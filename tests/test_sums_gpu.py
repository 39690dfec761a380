"""Sums over many sites and over the populations of a site, against exact sums
of the same stored floats: no fewer bits than sums in FP64."""
import math

import numpy as np
import pytest

import oracle
from paper_1410_5584_gb300 import D2Q9, D3Q19, Lattice, MultiLattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,axis,terms", [((510, 1023, 10), 0, 4076), ((2, 1022, 2050), 2, 9198),
                                              ((1024, 4, 2050), 1, 9216)])
def test_snapshots_of_thousands_of_terms_a_thread(shape, axis, terms):
    """Profiles of `terms` values a thread of sizes from 0.6 down to 6e-7, positive in the first half of the terms and
    negative in the second, so that the sums pass far from where they end.  Each run of 128 values is summed to
    (256 2^-24)^3 = 2^-48 of their magnitudes; the runs and the 256 or 1024 threads are added in FP64, fewer than 90
    roundings by 2^-53 of partial sums of which most are below half of a thread's magnitudes: less than 2^-47 in all
    (pairs of floats come to about 2^-43 here).  The transform multiplies by numbers of at most 1 and rounds n times."""
    nz, ny, nx = shape
    n = (nx, ny, nz)[axis]
    rng = np.random.default_rng(terms)
    g = Lattice(D3Q19, nx, ny, nz, 1.0, 1.0, 0.0, 0.0, 6, sf_axis=axis)
    rho = []
    for s in range(2):
        r = 1.0 + 0.6 * np.exp2(-20 * rng.random(shape))
        half = (slice(nz // 2, None),) if axis != 2 else (slice(None), slice(ny // 2, None))
        r[half] = 2.0 - r[half]
        rho.append(r)
    g.init(*(r.ravel() for r in rho))
    g.sf_sample()
    got = g.structure_factor(axis=axis)[:3]
    # rho0 = 1 plus a float of at most 1/2 in magnitude that is a sum of floats: the difference is exact
    dev = [np.asarray(f).reshape(shape) - 1.0 for f in g.moments()[:2]]
    g.close()
    prof, size = [], []
    for d in dev:
        rows = np.moveaxis(d, 2 - axis, 0).reshape(n, -1)
        prof.append(np.array([math.fsum(r) for r in rows]))
        size.append(np.abs(rows).sum())
    k = 2 * np.pi * np.outer(np.arange(1, n // 2 + 1), np.arange(n)) / n
    hat = [(p * np.exp(-1j * k)).sum(axis=1) for p in prof]
    err = [(2.0 ** -47 + 3 * n * 2.0 ** -53) * z for z in size]
    N = nx * ny * nz
    for q, (a, b) in enumerate(((0, 0), (0, 1), (1, 1))):
        want = (hat[a] * hat[b].conj()).real / N
        bound = (np.abs(hat[a]) * err[b] + np.abs(hat[b]) * err[a] + 2 * err[a] * err[b]) / N + 1e-15 * np.abs(want)
        assert np.all(np.abs(got[q] - want) <= bound), np.max(np.abs(got[q] - want) / bound)


@pytest.mark.parametrize("lat,shape", [(D2Q9, (1, 33, 51)), (D3Q19, (4, 9, 33))])
@pytest.mark.parametrize("ns", [2, 3, 4])
def test_species_velocities_are_the_rounded_quotients(lat, shape, ns):
    """Without forces, from deviations that are multiples of 2^-44 of very different sizes: every sum is a multiple of
    2^-44 below 8, so momenta and densities are exact and the velocity is one rounded division."""
    nz, ny, nx = shape
    c, w, T, N = oracle.tables(lat)
    g = MultiLattice(lat, ns, nx, ny, nz, [1.0] * ns, 0.0, np.zeros((ns, ns)), 3)
    rng = np.random.default_rng(ns)
    base = (w.astype(np.float32) * np.float32(1.0)).astype(np.float64)
    size = np.exp2(-rng.integers(6, 20, (ns, len(w)) + shape).astype(float))
    dev = np.round(rng.uniform(-1, 1, size.shape) * size * 2.0 ** 24) * 2.0 ** -24
    tiny = np.round(rng.uniform(-1, 1, size.shape) * 2.0 ** 20) * 2.0 ** -44
    dev = np.where(rng.random(size.shape) < 0.5, dev, tiny)
    f = base[None, :, None, None, None] + dev
    assert np.array_equal(f - base[None, :, None, None, None], dev) and np.array_equal(dev, dev.astype(np.float32))
    g.set_populations(f)
    rho, u, cons = g.moments()
    assert np.array_equal(g.get_populations(), f)
    g.close()
    total = base.sum() * ns + dev.sum(axis=(0, 1))
    D = 2 if lat == D2Q9 else 3
    assert np.array_equal(rho.reshape((ns,) + shape), base.sum() + dev.sum(axis=1))
    for d in range(D):
        j = np.tensordot(c[:, d].astype(float), dev.sum(axis=0), axes=(0, 0))
        assert np.array_equal(u.reshape((D,) + shape)[d], j / total)
