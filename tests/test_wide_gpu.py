"""Boxes of 2^29 sites and more, whose arrays pass the reach of the step kernels' 32-bit byte offsets."""
import numpy as np
import pytest

from paper_1410_5584_gb300 import D2Q9, Batch, Lattice
from paper_1410_5584_gb300 import inputs
from test_parity_gpu import _block_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [(1.0, 1.0), (0.8, 1.0)])
def test_sampled_parity_beyond_32_bit_offsets(tau, monkeypatch):
    """Sampled sites (the last ones among them) of a box just above 2^29 sites against the oracle, moment-fed and
    general collide, from the uniform state (the noise makes it a random one); the bounds of the 16-bit forms."""
    monkeypatch.setattr(inputs, "perturbed_density", lambda *a, **k: None)
    assert 65535 * 8193 >= 2 ** 29
    assert _block_check(D2Q9, (1, 65535, 8193), 2, 20, seed=8, tau=tau, storage="f16", bits=11) <= 1e-6


@pytest.mark.parametrize("nx,ny", [(7724, 7722), (7725, 7724)])
@pytest.mark.parametrize("schedule", [1, 3])
@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_replicas_below_and_above_4_gb_match_a_lone_box(nx, ny, schedule, tau):
    """A replica whose 2 * 9 * N floats stay just below 2^32 bytes (32-bit offsets reach its last word) and one just
    above, beside a small replica: sampled sites, the last ones among them, as a lone context has them (the bound of
    the batch tests)."""
    assert (2 * 9 * nx * ny * 4 < 2 ** 32) == (nx == 7724)
    small = dict(nx=70, ny=33, tau_a=tau, tau_b=1.0, kT=1e-4, G=0.9, seed=3)
    reps = [small, dict(small, nx=nx, ny=ny, seed=9), small]
    sites = np.concatenate([np.arange(4), nx * ny - 1 - np.arange(40), np.random.default_rng(2).integers(0, nx * ny, 40)])
    b = Batch(D2Q9, reps, schedule=schedule)
    b.init()
    b.step(3)
    got = [b.replicas[1].site_populations(sites), b.replicas[2].site_populations(np.arange(70 * 33))]
    b.close()
    for r, g, s in ((reps[1], got[0], sites), (reps[2], got[1], np.arange(70 * 33))):
        lone = Lattice(D2Q9, r["nx"], r["ny"], 1, tau, 1.0, 1e-4, 0.9, r["seed"])
        lone.init()
        lone.step(3)
        ref = lone.site_populations(s)
        lone.close()
        assert np.max(np.abs(g - ref)) <= 2e-6 * np.max(np.abs(ref))
