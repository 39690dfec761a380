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
