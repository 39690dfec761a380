"""The schedules of one launch a step on boxes of 2^29 sites and more: the tiled
step runs there at full relaxation, otherwise both run the two-kernel step; in
either case the bits of the two-kernel step."""
import numpy as np
import pytest

from paper_1410_5584_gb300 import D2Q9, D3Q19, Lattice
from paper_1410_5584_gb300 import flbm as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,shape,schedules", [(D2Q9, (1, 65535, 8193), ("tiled", "fused")),
                                                 (D3Q19, (513, 1025, 1023), ("fused",))])
@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_one_launch_schedules_beyond_32_bit_offsets(lat, shape, schedules, tau):
    nz, ny, nx = shape
    N = nx * ny * nz
    assert N >= 2 ** 29
    sites = np.concatenate([np.arange(64), N - 1 - np.arange(64), 2 ** 29 + np.arange(-64, 64),
                            np.random.default_rng(1).integers(0, N, 2000)])
    got = {}
    for schedule in ("two_kernels",) + schedules:
        g = Lattice(lat, nx, ny, nz, tau, 1.0, 1e-4, 0.9, 6, storage="f16", schedule=F.SCHEDULE[schedule], kernel_timing=1)
        g.init()
        g.step(1)
        g.step(2)
        launches = g.kernel_times()[1]
        assert launches == {"density": 0 if schedule == "tiled" and tau == 1.0 else 3, "collide": 3}
        got[schedule] = g.site_populations(sites)
        g.close()
        del g
    for schedule in schedules:
        assert np.array_equal(got[schedule], got["two_kernels"])
