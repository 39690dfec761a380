"""The first snapshot of a box, which also makes and uploads the tables of the
transforms, against later ones of the same state: the mean of two equal
snapshots is the first one, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1410_5584_gb300 import D2Q9, Lattice
from paper_1410_5584_gb300 import inputs

pytestmark = pytest.mark.gpu


def _box(nx, ny, **options):
    c, w, T, N = oracle.tables(D2Q9)
    g = Lattice(D2Q9, nx, ny, 1, 1.0, 1.0, 1e-4, 0.9, 6, **options)
    g.set_populations(inputs.random_populations(np.stack([w, 0.8 * w]), (1, ny, nx), 0.02, seed=nx))
    g.step(1)
    return g


def _first_and_second(sample, read):
    out = []
    for n in (1, 2):
        sample()
        got = read()
        assert got[-1] == n
        out.append(got[:-1])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [64, 1000, 32749])
@pytest.mark.parametrize("axis", [0, 1])
def test_axis_structure_factors(n, axis):
    g = _box(*((n, 5) if axis == 0 else (5, n)), sf_axis=axis)
    _first_and_second(g.sf_sample, lambda: g.structure_factor(axis=axis))


@pytest.mark.parametrize("nx,ny", [(64, 32), (33, 600), (15, 1999)])
def test_full_structure_factors(nx, ny):
    g = _box(nx, ny)
    _first_and_second(g.sfk_sample, g.sfk)


@pytest.mark.parametrize("nx,ny", [(64, 33), (40, 8191)])
@pytest.mark.parametrize("columns", [(-1, -1), (20, 0)])
def test_capillary_spectra(nx, ny, columns):
    g = Lattice(D2Q9, nx, ny, 1, 1.0, 1.0, 1e-5, 1.5, 3, rho0_a=1.18, rho0_b=1.18)
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    shift = 0.3 * np.sin(2 * np.pi * y / ny)
    phi = 0.25 * (1 + np.tanh((x - shift - nx / 4) / 2)) * (1 - np.tanh((x - shift - 3 * nx / 4) / 2))
    g.init((0.2 + 2.0 * phi).ravel(), (2.2 - 2.0 * phi).ravel())
    _first_and_second(lambda: g.cap_sample(*columns), g.cap_spectrum)


@pytest.mark.parametrize("columns", [(-1, -1), (20, 0)])
def test_a_first_capillary_snapshot_that_is_captured_and_never_run(columns):
    """The buffers of the first snapshot are ready for the next even if the snapshot itself, recorded into a graph that
    is dropped, never ran: its share of the mean is zero."""
    import torch

    got = []
    for captured in (False, True):
        g = Lattice(D2Q9, 40, 96, 1, 1.0, 1.0, 1e-5, 1.5, 3, rho0_a=1.18, rho0_b=1.18)
        x, y = np.arange(40)[None, :], np.arange(96)[:, None]
        shift = 0.3 * np.sin(2 * np.pi * y / 96)
        phi = 0.25 * (1 + np.tanh((x - shift - 10) / 2)) * (1 - np.tanh((x - shift - 30) / 2))
        g.init((0.2 + 2.0 * phi).ravel(), (2.2 - 2.0 * phi).ravel())
        g.sync()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=g.stream, capture_error_mode="relaxed"):
                g.cap_sample(*columns)
            del graph
        g.cap_sample(*columns)
        s, hm, n = g.cap_spectrum()
        got.append((s * n, hm * n, n))
        g.close()
    assert [k[2] for k in got] == [1, 2]
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
