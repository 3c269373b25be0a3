"""The loss by one warp per tile where it can go wrong: pixels a tile at the
edges of the lanes' rows (32, 64, 96, 128, 129, 255), ragged tiles with fewer,
one pixel, more tiles than the launched warps (each takes several), no active
tile, fewer active tiles than the maximum, and without maps.  Tolerances are
those of the loss's parity test: sums of up to 256 fp32 terms in another order
differ by a few 2^-24."""
import numpy as np
import pytest
import torch

from paper_2606_15924_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2606_15924_gb300 import binding
    binding.device_check()
    return binding


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30))


@pytest.mark.parametrize("structure", ["ncc", "ssim"])
@pytest.mark.parametrize("W,H,n_select,n_pix", [(250, 187, 192, 1), (250, 187, 192, 32), (250, 187, 100, 33),
                                                (250, 187, 192, 64), (250, 187, 50, 65), (250, 187, 192, 96),
                                                (250, 187, 192, 97), (250, 187, 3, 128), (250, 187, 192, 129),
                                                (250, 187, 192, 255), (1280, 720, 3600, 25), (1957, 1091, 8487, 256),
                                                (250, 187, 0, 85)])
@pytest.mark.parametrize("maps", [True, False])
def test_loss_by_warps(B, orc, W, H, n_select, n_pix, structure, maps):
    from gpu_util import dev, select_dev, select_host
    err, age = scenes.error_map(W, H, seed=W), scenes.age_map(W, H, seed=W, max_age=65535)
    target = scenes.smooth_image(W, H, seed=W + 1)
    sel = select_dev(B, err, age, W, H, n_select, n_pix, seed=9)
    sh = select_host(sel)
    P, A = int(sh["pix_off"][-1]), sh["n_active"]
    rgb = np.random.default_rng(4).uniform(0, 1, (max(P, 1), 3)).astype(np.float32)
    if P:
        xy = orc.pixel_coords(sh["active_tiles"], sh["pix_off"], sh["pix_idx"], W)
        rgb[:P] = 0.7 * target[xy[:, 1], xy[:, 0]] + 0.3 * rgb[:P]
    n_max = sel["n_sel"] + 7                                # more than are active
    tiles = torch.cat([sel["active_tiles"], torch.zeros(8, dtype=torch.int32, device="cuda")])
    off = torch.cat([sel["pix_off"], torch.zeros(8, dtype=torch.int32, device="cuda")])
    err_d, age_d = dev(err), dev(age)
    dL = torch.full((max(P, 1) + 5, 3), 9.0, device="cuda")
    lam = torch.full((n_max,), 9.0, device="cuda")
    e = torch.full((max(P, 1) + 5,), 9.0, device="cuda")
    loss = torch.full((1,), 3.0, dtype=torch.float64, device="cuda")
    B.loss_sparse_ncc(dev(rgb), dev(target), W, H, tiles, sel["n_active"], n_max, off, sel["pix_idx"], n_pix,
                      (1e-3, 1e-8, 0.4), err_d if maps else None, age_d if maps else None, dL, lam, e, loss,
                      structure=structure)
    assert bool((dL[P:] == 9.0).all()) and bool((lam[A:] == 9.0).all()) and bool((e[P:] == 9.0).all())
    if A == 0:
        assert float(loss.item()) == 0.0
        return
    oloss = orc.loss if structure == "ncc" else orc.loss_ssim
    want = oloss(W, H, sh, rgb[:P].astype(np.float64), target.astype(np.float64), err_f16_bits=err, age=age)
    assert float(loss.item()) == pytest.approx(want["loss"], rel=1e-5)
    np.testing.assert_allclose(lam[:A].cpu().numpy(), want["lam"], rtol=1e-4, atol=1e-7)
    np.testing.assert_allclose(e[:P].cpu().numpy(), want["err"], atol=1e-6)
    assert rel_l2(dL[:P].cpu().numpy(), want["dL_drgb"]) <= 1e-4
    if not maps:
        np.testing.assert_array_equal(age_d.cpu().numpy(), age)
        return
    np.testing.assert_array_equal(age_d.cpu().numpy(), want["age_map"])
    got_e = err_d.cpu().numpy().view(np.float16).astype(np.float64)
    want_e = want["err_map"].view(np.float16).astype(np.float64)
    ulp = np.spacing(np.abs(want_e).astype(np.float16)).astype(np.float64)
    assert np.all(np.abs(got_e - want_e) <= ulp)
