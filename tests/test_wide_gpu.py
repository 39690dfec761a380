"""Boxes of 2^29 sites and more, whose arrays pass the reach of the step kernels' 32-bit byte offsets."""
import pytest

from paper_1410_5584_gb300 import D2Q9
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
