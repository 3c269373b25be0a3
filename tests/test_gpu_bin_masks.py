"""Binning over some of the tiles, where a lane gathers the active tiles of its
Gaussian's rectangle as one word: rectangles of 1 to 40 tiles in every shape
(one row, one column, 32 tiles in a word, more than a word holds), at the image's
corners and edges, tile counts at the edges of the bit table's words, all but
one tile active and one tile alone - bit for bit with the oracle."""
import numpy as np
import pytest

from paper_2606_15924_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2606_15924_gb300 import binding
    binding.device_check()
    return binding


@pytest.mark.parametrize("tx,ty", [(1, 33), (33, 1), (8, 4), (31, 3), (40, 40), (64, 11)])
@pytest.mark.parametrize("which", ["one", "tenth", "half", "all but one"])
def test_masked_rectangles_bit_exact(B, orc, tx, ty, which):
    from gpu_util import bin_dev, dev, projected_dev
    W, H, T = 16 * tx - 3, 16 * ty - 7, tx * ty
    rng = np.random.default_rng(T)
    # a centre in every part of the image and beyond its edges, spans of 1 to 41 tiles an axis
    n = 3000
    pr = scenes.projected(n, W, H, seed=T)
    pr["xy"] = (rng.uniform(-0.1, 1.1, size=(n, 2)) * [W, H]).astype(np.float32)
    pr["radius"] = np.where(rng.random(n) < 0.1, 0, (2.0 ** rng.uniform(0.0, 8.4, n)).astype(np.int32)).astype(np.int32)
    act = {"one": np.arange(T) == T // 2, "tenth": rng.random(T) < 0.1, "half": rng.random(T) < 0.5,
           "all but one": np.arange(T) != T - 1}[which]
    act[0] |= not act.any()
    rank = np.where(act, np.cumsum(act) - 1, -1).astype(np.int32)
    keys_w, vals_w, _ = orc.bin_tiles(pr["xy"], pr["radius"], pr["depth"], W, H, rank)
    cam = dict(viewmat=np.eye(4), fx=100.0, fy=100.0, cx=W / 2, cy=H / 2, width=W, height=H, znear=0.2)
    out = bin_dev(B, projected_dev(pr), n, cam, dev(rank), int(act.sum()), capacity=len(vals_w) + 5)
    I = int(out["n_isect"].item())
    assert I == len(vals_w)
    np.testing.assert_array_equal(out["vals"][:I].cpu().numpy(), vals_w)
    np.testing.assert_array_equal(out["keys"][:I].cpu().numpy().view(np.uint64), keys_w)
