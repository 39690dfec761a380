"""The thread-block options read back the shape that the launches take (host
logic only; no GPU)."""
import ctypes

import pytest

from paper_1410_5584_gb300 import flbm as F


def _fewest_lanes(nx, ny):
    """128 x 1, 64 x 2 or 32 x 4 (x cut at nx rounded up to 32): the fewest lanes over a plane, the wider on a tie unless
    a short row leaves its block at 64 lanes or fewer."""
    wx = -(-nx // 32) * 32
    best = None
    for x in (128, 64, 32):
        bx, by = min(x, wx), 128 // x
        lanes = -(-nx // bx) * -(-ny // by) * bx * by
        if best is None or lanes < best[0] or (lanes == best[0] and best[1] <= 64 and bx * by > best[1]):
            best = (lanes, bx * by, x, by)
    return best[2:]


@pytest.mark.parametrize("nx,ny", [(256, 256), (161, 150), (130, 130), (200, 200), (97, 97), (33, 20), (32, 128), (64, 2),
                                   (64, 3000), (100, 512), (2, 2), (5, 3), (128, 1000)])
@pytest.mark.parametrize("species", [2, 3])
def test_block_options_read_the_shape_in_effect(nx, ny, species):
    lib, v = F.lib(), ctypes.c_double()
    if species == 2:
        h = F.flbm_create(F.D3Q19, nx, ny, 4, 1.0, 1.0, 1e-4, 0.0, 1)
        get, put, destroy = lib.flbm_get_option, lib.flbm_set_option, lib.flbm_destroy
    else:
        h = ctypes.c_void_p()
        arr = lambda x: (ctypes.c_double * len(x))(*x)
        assert lib.flbm_mcreate(1, 3, nx, ny, 4, arr([1.0] * 3), 1e-4, arr([0.0] * 9), 1, ctypes.byref(h)) == F.OK
        get, put, destroy = lib.flbm_mget_option, lib.flbm_mset_option, lib.flbm_mdestroy

    def shape():
        out = []
        for key in (F.OPT_BLOCK_X, F.OPT_BLOCK_Y):
            assert get(h, key, ctypes.byref(v)) == F.OK
            out.append(v.value)
        return tuple(out)

    try:
        want = _fewest_lanes(nx, ny)
        assert shape() == want
        # what was read can be set, the shape then being the caller's
        for key, value in zip((F.OPT_BLOCK_X, F.OPT_BLOCK_Y), want):
            assert put(h, key, value) == F.OK
        assert shape() == want
        assert put(h, F.OPT_BLOCK_Y, 1) == F.OK and put(h, F.OPT_BLOCK_X, 128) == F.OK
        assert shape() == (128, 1)
    finally:
        destroy(h)
