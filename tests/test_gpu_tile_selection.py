"""Tile selection bit for bit with the oracle where the block's selection can
go wrong: tile counts at the edges of its items per thread, one tile chosen and
all but one, keys that one pass over 1024 buckets does not separate (tiles
without any error, whose keys lie 2^900 above the others), ages that are all
equal (ties in index order), few and many distinct."""
import numpy as np
import pytest

from paper_2606_15924_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2606_15924_gb300 import binding
    binding.device_check()
    return binding


@pytest.mark.parametrize("tx,ty,kind,ages", [
    (1, 2, "map", 5), (31, 33, "map", 1), (32, 32, "half", 5), (41, 25, "none", 4000), (33, 32, "half", 1),
    (64, 64, "map", 4000), (241, 17, "half", 5), (128, 64, "none", 1), (91, 91, "map", 5), (128, 128, "half", 4000)])
def test_tile_selection_bit_exact(B, orc, tx, ty, kind, ages):
    from gpu_util import select_dev, select_host
    W, H, T = 16 * tx, 16 * ty - 5, tx * ty
    err = scenes.error_map(W, H, seed=T)
    if kind == "half":                                   # every other column of tiles without error
        err[:, (np.arange(W) // 16) % 2 == 0] = 0
    if kind == "none":
        err[:] = 0
    age = scenes.age_map(W, H, seed=H, max_age=ages) if ages > 1 else np.full((H, W), 7, np.uint16)
    for n_sel, sampling in ((1, (1000, 0)), (T - 1, (400, 300)), (max(1, T // 2), (0, 1000)),
                            (max(1, T // 3), (400, 300)))[3 if T > 9000 else 0:]:
        sm = sampling + (400, 300)
        got = select_host(select_dev(B, err, age, W, H, n_sel, 1, seed=9, it=4, view=3, sampling=sm))
        want = orc.select(err, age, W, H, n_select=n_sel, n_pix=1, tile_hard_pm=sm[0], tile_stable_pm=sm[1],
                          pix_hard_pm=sm[2], pix_stable_pm=sm[3], seed=9, it=4, view=3)
        assert got["n_active"] == want["n_active"]
        for k in ("active_tiles", "tile_rank", "pix_off"):
            np.testing.assert_array_equal(got[k], want[k])


@pytest.mark.parametrize("W,H", [(16, 16), (17, 15), (250, 187), (256, 256), (64, 16), (16, 64), (1957, 1091), (4099, 1031)])
@pytest.mark.parametrize("n_pix", [1, 85, 200, 256])
def test_every_tile_bit_exact(B, orc, W, H, n_pix):
    """Every tile selected (by itself and with a larger n_select): ragged last
    rows and columns with fewer pixels than n_pix, one row, one column, more
    tiles than the one-block selection takes."""
    from gpu_util import select_dev, select_host
    T = ((W + 15) // 16) * ((H + 15) // 16)
    rng = np.random.default_rng(T)
    err = rng.random((H, W)).astype(np.float16).view(np.uint16)
    age = rng.integers(0, 9, (H, W)).astype(np.uint16)
    for n_sel in (T, T + 5):
        got = select_host(select_dev(B, err, age, W, H, n_sel, n_pix, seed=2, it=1, view=0))
        assert got["n_active"] == T
        np.testing.assert_array_equal(got["active_tiles"], np.arange(T))
        np.testing.assert_array_equal(got["tile_rank"], np.arange(T))
        w = np.minimum(16, W - 16 * np.arange((W + 15) // 16))
        h = np.minimum(16, H - 16 * np.arange((H + 15) // 16))
        n = np.minimum(n_pix, (h[:, None] * w[None, :]).reshape(-1))
        np.testing.assert_array_equal(got["pix_off"], np.concatenate([[0], np.cumsum(n)]))
        if T < 3000:
            want = orc.select(err, age, W, H, n_select=n_sel, n_pix=n_pix, tile_hard_pm=400, tile_stable_pm=300,
                              pix_hard_pm=400, pix_stable_pm=300, seed=2, it=1, view=0)
            np.testing.assert_array_equal(got["pix_idx"], want["pix_idx"])
