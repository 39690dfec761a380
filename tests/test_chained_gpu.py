"""Step launches that may begin before the stream's previous launch ends
(programmatic stream serialization) against launches that run one at a time
(kernel timing on): the same bits, directly, from graphs and in a caller's
capture."""
import numpy as np
import pytest

import oracle
from paper_1410_5584_gb300 import D2Q9, D3Q19, Lattice, MultiLattice, inputs

pytestmark = pytest.mark.gpu


def _state(lat, shape, ns=2, seed=4):
    c, w, T, N = oracle.tables(lat)
    return inputs.random_populations(np.stack([w * r for r in (1.0, 0.8, 0.6)[:ns]]), shape, 0.02, seed=seed)


@pytest.mark.parametrize("lat,shape", [(D2Q9, (1, 2, 64)), (D2Q9, (1, 200, 130)), (D3Q19, (9, 20, 33)),
                                       (D3Q19, (40, 48, 64))])
@pytest.mark.parametrize("tau,options", [(1.0, {}), (0.8, {}), (1.0, {"streaming": 0}), (0.8, {"streaming": 0}),
                                         (1.0, {"schedule": 3}), (0.8, {"storage": "bf16"})])
@pytest.mark.parametrize("graph_steps", [0, 7])
def test_chained_steps_are_bitwise_those_of_plain_launches(lat, shape, tau, options, graph_steps):
    nz, ny, nx = shape
    got = []
    for extra in ({"kernel_timing": 1}, {"graph_steps": graph_steps}):
        g = Lattice(lat, nx, ny, nz, tau, 1.0, 1e-4, 0.9, 6, **options, **extra)
        g.set_populations(_state(lat, shape), step=3)
        for n in (1, 40, 22):
            g.step(n)
        got.append(g.get_populations())
        g.close()
    assert np.array_equal(*got)


@pytest.mark.parametrize("lat,shape,storage", [(D3Q19, (83, 85, 97), "f32"), (D3Q19, (71, 75, 130), "f32"),
                                               (D3Q19, (131, 83, 130), "bf16"), (D2Q9, (1, 1171, 1201), "f32"),
                                               (D2Q9, (1, 44001, 33), "f32")])
@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_density_passes_from_the_end_are_bitwise_the_fused_step(lat, shape, storage, tau):
    """Boxes of more than 96 MB of populations, whose density pass walks the rows
    and planes from the last (ragged in x and in y), against the schedules of one
    launch a step: the fused one and, in 2D, the tiled one, whose steps walk the
    rows from either end in turn."""
    nz, ny, nx = shape
    width = 4 if storage == "f32" else 2
    assert 2 * (9 if lat == D2Q9 else 19) * nx * ny * nz * width > 96 << 20
    got = []
    for schedule in (1, 0) + ((3,) if lat == D2Q9 else ()):
        g = Lattice(lat, nx, ny, nz, tau, 1.0, 1e-4, 0.9, 6, schedule=schedule, storage=storage)
        g.init()
        g.step(5)
        sites = np.concatenate([np.arange(300), nx * ny * nz - 1 - np.arange(300),
                                np.random.default_rng(1).integers(0, nx * ny * nz, 5000)])
        got.append((g.site_populations(sites), g.moments(fields=False)))
        g.close()
    for populations, totals in got[1:]:
        assert np.array_equal(populations, got[0][0])
        assert np.array_equal(totals, got[0][1])


@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("streaming", ["two_arrays", "in_place"])
def test_chained_species_steps_are_bitwise_those_of_plain_launches(tau, streaming):
    from paper_1410_5584_gb300 import flbm as F

    got = []
    for timing in (1, 0):
        g = MultiLattice(D3Q19, 3, 33, 20, 9, [tau, 1.0, 1.0], 1e-4, 0.9 * (1 - np.eye(3)), 6, streaming=streaming)
        g.set_option(F.OPT_KERNEL_TIMING, timing)
        g.set_populations(_state(D3Q19, (9, 20, 33), 3), step=3)
        g.step(41)
        got.append(g.get_populations())
        g.close()
    assert np.array_equal(*got)


def test_two_boxes_in_turn_on_one_stream():
    """Each box's launches follow the other's; a step reads what the same
    stream's last step but one wrote."""
    import torch

    shape, s = (9, 20, 33), torch.cuda.Stream()
    make = lambda seed, **k: Lattice(D3Q19, 33, 20, 9, 1.0, 1.0, 1e-4, 0.9, seed, **k)
    want = []
    for seed in (6, 7):
        g = make(seed, kernel_timing=1)
        g.set_populations(_state(D3Q19, shape, seed=seed))
        g.step(30)
        want.append(g.get_populations())
    boxes = [make(6, stream=s), make(7, stream=s)]
    for seed, g in zip((6, 7), boxes):
        g.set_populations(_state(D3Q19, shape, seed=seed))
    for _ in range(30):
        for g in boxes:
            g.step(1)
    for g, w in zip(boxes, want):
        assert np.array_equal(g.get_populations(), w)


@pytest.mark.parametrize("lat,shape", [(D2Q9, (1, 96, 100)), (D3Q19, (9, 20, 33))])
def test_steps_in_a_callers_capture_after_a_join(lat, shape):
    """The first captured launch depends on two streams at once."""
    import torch

    nz, ny, nx = shape
    ref, g = (Lattice(lat, nx, ny, nz, 1.0, 1.0, 1e-4, 0.9, 6) for _ in range(2))
    for box in (ref, g):
        box.set_populations(_state(lat, shape))
        box.step(1)
        box.sync()
    ref.step(3)
    other, x = torch.cuda.Stream(), torch.zeros(1 << 20, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=g.stream):
        x.add_(1.0)
        other.wait_stream(g.stream)
        with torch.cuda.stream(other):
            x.mul_(2.0)
        x2 = x + 1.0
        g.stream.wait_stream(other)
        g.step(3)
        x2.add_(x)
    with torch.cuda.stream(g.stream):
        graph.replay()
    g.sync()
    assert np.array_equal(g.get_populations(), ref.get_populations())


@pytest.mark.parametrize("lat,shape", [(D2Q9, (1, 2, 64)), (D2Q9, (1, 37, 130)), (D2Q9, (1, 300, 3)), (D3Q19, (5, 6, 7)),
                                       (D3Q19, (12, 33, 70)), (D3Q19, (40, 3, 260))])
def test_structure_factor_snapshots_are_those_of_the_fields(lat, shape):
    """Two snapshots along every axis, on boxes that leave remainders of the
    profile kernels' blocks, against the FP64 transform of the fields that
    flbm_moments returns.  The fields are the same floats; sums of M < 2e4 values
    of order 1 and their transform over n <= 300 rows round by less than
    n M 2^-50 <= 1e-8 of a value, and with fluctuations of 0.02 an amplitude is of
    order sqrt(N) 0.02: 1e-8 of the largest mode covers it."""
    nz, ny, nx = shape
    for axis in range(2 if lat == D2Q9 else 3):
        n = (nx, ny, nz)[axis]
        g = Lattice(lat, nx, ny, nz, 0.8, 1.0, 1e-4, 0.9, 6, sf_axis=axis)
        g.set_populations(_state(lat, shape), step=3)
        want = np.zeros((4, n // 2))
        for _ in range(2):
            g.step(3)
            g.sf_sample()
            fields = [np.asarray(f).reshape(-1, nz, ny, nx) for f in g.moments()[:3]]
            prof = [f.sum(axis=tuple(k for k in (1, 2, 3) if k != 3 - axis)) for f in fields]
            a, b, u = (np.fft.fft(p, axis=1)[:, 1:n // 2 + 1] for p in prof)
            N = nx * ny * nz
            want += 0.5 / N * np.stack([np.abs(a[0]) ** 2, (a[0] * b[0].conj()).real, np.abs(b[0]) ** 2,
                                        (np.abs(u) ** 2).mean(axis=0)])
        got = np.stack(g.structure_factor(axis=axis)[:4])
        assert np.max(np.abs(got[:3] - want[:3])) <= 1e-8 * np.max(want[:3])
        assert np.max(np.abs(got[3] - want[3])) <= 1e-8 * np.max(want[3])
        g.close()
