"""The paired-splat forward at the sizes where its division changes (pixel
counts around the warps' edges, one and two pixels a lane, list lengths around
the 32-position chunks), and an infinite colour, which stays with the pixels
that blend its splat."""
import numpy as np
import pytest
import torch

from paper_2606_15924_gb300 import scenes

pytestmark = pytest.mark.gpu
W, H = 96, 80


@pytest.fixture(scope="module")
def B():
    from paper_2606_15924_gb300 import binding
    return binding


def _render(B, pd, binned, sel, n_pix, cam, n_active_max):
    P = sel["n_sel"] * n_pix
    o = dict(rgb=torch.zeros(P, 3, device="cuda"), T=torch.zeros(P, device="cuda"),
             n_last=torch.zeros(P, dtype=torch.int32, device="cuda"))
    B.render_sampled(pd, binned["ranges"], binned["vals"], sel["active_tiles"], sel["n_active"], n_active_max,
                     sel["pix_off"], sel["pix_idx"], n_pix, cam, (0.1, 0.2, 0.3), o["rgb"], o["T"], o["n_last"])
    return o


@pytest.mark.parametrize("n_pix", [1, 32, 33, 65, 128, 129, 192, 193, 255, 256])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 900])
def test_sizes_against_oracle(B, orc, n, n_pix):
    from gpu_util import bin_dev, projected_dev, select_dev, select_host
    p = scenes.projected(n, W, H, seed=n, radius_max=90 if n < 100 else 18)
    if n < 100:
        p["xy"] = np.clip(p["xy"], 30.0, 60.0)       # every splat in the middle tiles
        p["radius"][:] = 30
    p["opac"][::5] = 0.999                            # capped alphas, early stops
    cam = scenes.look_at((0.0, 0.0, -4.0), width=W, height=H)
    sel = select_dev(B, scenes.error_map(W, H), scenes.age_map(W, H), W, H, 30, n_pix, seed=4)
    pd = projected_dev(p)
    binned = bin_dev(B, pd, n, cam, sel["tile_rank"], sel["n_sel"], capacity=60000)
    one = _render(B, pd, binned, sel, n_pix, cam, sel["n_sel"])      # few warps: one pixel a lane
    many = _render(B, pd, binned, sel, n_pix, cam, 4000)             # an upper bound with many
    if n_pix > 32:                                                   # (else two threads per pixel against one)
        for k in one:
            assert torch.equal(one[k], many[k]), k
    sh = select_host(sel)
    pix = orc.pixel_coords(sh["active_tiles"], sh["pix_off"], sh["pix_idx"], W)
    want = {k: np.asarray(v, np.float64) for k, v in p.items() if k != "radius"}
    want["radius"] = p["radius"]
    ref = orc.render_pixels(want, W, H, pix, bg=(0.1, 0.2, 0.3))
    sure = ref["margin"] > 1e-4
    for o in (one, many):
        np.testing.assert_array_equal(o["n_last"][:len(pix)].cpu().numpy()[sure], ref["n_last"][sure])
        assert np.abs(o["rgb"][:len(pix)].cpu().numpy()[sure] - ref["rgb"][sure]).max(initial=0.0) <= 1e-4


@pytest.mark.parametrize("n_active_max", [30, 4000])
def test_infinite_colour_stays_local(B, n_active_max):
    from gpu_util import bin_dev, projected_dev, select_dev
    n, n_pix = 600, 256
    p = scenes.projected(n, W, H, seed=8, radius_max=18)
    cam = scenes.look_at((0.0, 0.0, -4.0), width=W, height=H)
    sel = select_dev(B, scenes.error_map(W, H), scenes.age_map(W, H), W, H, 30, n_pix, seed=4)
    pd = projected_dev(p)
    binned = bin_dev(B, pd, n, cam, sel["tile_rank"], sel["n_sel"], capacity=60000)
    clean = _render(B, pd, binned, sel, n_pix, cam, n_active_max)
    front = int(binned["vals"][int(binned["ranges"][10, 0])])        # the first splat of some tile
    marked = {k: v.clone() for k, v in pd.items()}
    marked["rgb"].zero_()
    marked["rgb"][front] = 1.0
    seen = _render(B, marked, binned, sel, n_pix, cam, n_active_max)
    hit = (seen["rgb"][:, 0] - seen["T"] * 0.1) > 1e-6               # the pixels that blend it
    bad = {k: v.clone() for k, v in pd.items()}
    bad["rgb"][front, 1] = float("inf")
    got = _render(B, bad, binned, sel, n_pix, cam, n_active_max)
    assert hit.any() and not hit.all()
    assert torch.isinf(got["rgb"][hit, 1]).all()
    assert torch.equal(got["rgb"][~hit], clean["rgb"][~hit])
    assert torch.equal(got["T"], clean["T"]) and torch.equal(got["n_last"], clean["n_last"])
