"""Pixel sampling bit for bit with the oracle where the warp's selection can go
wrong: counts around the 32 lanes and the 256 pixels of a tile, ragged tiles,
draws of one kind and of all three, error maps with no weight, equal weights
and weights 2^39 apart, and many tiles of one map.

The error-proportional draw orders by fp32 quotients and, where the taken and
the others are not apart by their error bounds, those in doubt by exact keys.
At the 34th of 256 quotients neighbours differ by about 1 part in 34 and the
bounds span about 3e-5 of a quotient, so one tile in a thousand takes the exact
path: a map of 8487 tiles has about nine."""
import numpy as np
import pytest

from paper_2606_15924_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2606_15924_gb300 import binding
    binding.device_check()
    return binding


def _err(kind, W, H):
    if kind == "none":
        return np.zeros((H, W), np.uint16)
    if kind == "equal":
        return np.full((H, W), 0x3C00, np.uint16)
    if kind == "wide":                                  # the smallest and the largest weights, and values that weigh 0
        rng = np.random.default_rng(W)
        return rng.choice(np.array([0, 1, 2, 0x03FF, 0x0400, 0x3C00, 0x7BFF, 0x7C00, 0x7E00, 0x8001], np.uint16),
                          size=(H, W))
    return scenes.error_map(W, H, seed=W + H)


@pytest.mark.parametrize("W,H,kind,n_pix,sampling", [
    (200, 130, "none", 85, (400, 300, 400, 300)),
    (200, 130, "equal", 85, (400, 300, 400, 300)),
    (200, 130, "wide", 85, (1000, 0, 1000, 0)),
    (200, 130, "wide", 255, (400, 300, 1000, 0)),
    (250, 187, "map", 1, (400, 300, 1000, 0)),
    (250, 187, "map", 31, (400, 300, 400, 300)),
    (250, 187, "map", 32, (400, 300, 0, 1000)),
    (250, 187, "map", 33, (400, 300, 0, 0)),
    (250, 187, "wide", 128, (400, 300, 500, 500)),
    (250, 187, "map", 255, (400, 300, 400, 300)),
    (250, 187, "map", 256, (400, 300, 400, 300)),
    (1957, 1091, "map", 85, (400, 300, 400, 300)),
    (1957, 1091, "wide", 64, (400, 300, 1000, 0)),
])
def test_pixel_sampling_bit_exact(B, orc, W, H, kind, n_pix, sampling):
    from gpu_util import select_dev, select_host
    err = _err(kind, W, H)
    age = scenes.age_map(W, H, seed=H, max_age=30)
    n_sel = ((W + 15) // 16) * ((H + 15) // 16)
    got = select_host(select_dev(B, err, age, W, H, n_sel, n_pix, seed=77, it=3, view=1, sampling=sampling))
    want = orc.select(err, age, W, H, n_select=n_sel, n_pix=n_pix, tile_hard_pm=sampling[0],
                      tile_stable_pm=sampling[1], pix_hard_pm=sampling[2], pix_stable_pm=sampling[3], seed=77, it=3,
                      view=1)
    np.testing.assert_array_equal(got["pix_off"], want["pix_off"])
    np.testing.assert_array_equal(got["pix_idx"], want["pix_idx"])
