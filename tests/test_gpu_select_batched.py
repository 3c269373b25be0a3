"""Tile and pixel selection of several views in shared launches against one
selection per view, bit for bit: views of different sizes, tile counts on both
sides of the kernels' items per thread and past the one-block selection, no
tile, every tile and more than every tile chosen, different pixel counts, seeds
and view ids, the iteration from the host and from the device, one view and
sixteen."""
import functools

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
SIZES = [(256, 256, 64, 85), (250, 187, 192, 25), (333, 187, 0, 10), (1280, 720, 720, 84), (64, 48, 5, 256),
         (1957, 1091, 3000, 33), (40, 40, 99, 1), (4096, 1040, 1664, 25), (16, 16, 1, 200)]


@pytest.fixture(scope="module")
def B():
    from paper_2606_15924_gb300 import binding
    binding.device_check()
    return binding


@functools.lru_cache(maxsize=None)
def _maps(W, H):
    rng = np.random.default_rng(W)
    err, age = rng.random((H, W)).astype(np.float16), rng.integers(0, 40, (H, W)).astype(np.int16)
    return torch.from_numpy(err.view(np.int16)).cuda(), torch.from_numpy(age).cuda()


def _view(B, k, W, H, n_select, n_pix):
    T = ((W + 15) // 16) * ((H + 15) // 16)
    n = min(n_select, T)
    err, age = _maps(W, H)
    return dict(err_map=err, age_map=age, width=W, height=H, n_select=n_select, n_pix=n_pix, seed=11 * k, view=k,
                workspace=torch.empty(B.select_tiles_workspace_size(W, H), dtype=torch.uint8, device="cuda"),
                active_tiles=torch.full((max(n, 1),), -7, dtype=torch.int32, device="cuda"),
                n_active=torch.full((1,), -7, dtype=torch.int32, device="cuda"),
                tile_rank=torch.full((T,), -7, dtype=torch.int32, device="cuda"),
                pix_off=torch.full((n + 1,), -7, dtype=torch.int32, device="cuda"),
                pix_idx=torch.full((max(n * n_pix, 1),), 77, dtype=torch.uint8, device="cuda"))


@pytest.mark.parametrize("ids", [[0], [1, 3], [2, 8], list(range(9)), [0, 1, 2, 3, 4, 5, 6, 7, 8, 0, 1, 3, 4, 5, 6, 8]])
@pytest.mark.parametrize("on_device", [False, True])
def test_views_together_are_bit_exact(B, ids, on_device):
    sampling, it = (400, 300, 400, 300), 5
    it_dev = torch.full((1,), it, dtype=torch.int64, device="cuda") if on_device else None
    views = [_view(B, k + 1, *SIZES[i]) for k, i in enumerate(ids)]
    B.select_tiles_batched(views, sampling, 0 if on_device else it, iter_dev=it_dev)
    for k, i in enumerate(ids):
        w = _view(B, k + 1, *SIZES[i])
        B.select_tiles(w["err_map"], w["age_map"], w["width"], w["height"], w["n_select"], w["n_pix"], sampling, w["seed"],
                       0 if on_device else it, w["view"], w["workspace"], w["active_tiles"], w["n_active"], w["tile_rank"],
                       w["pix_off"], w["pix_idx"], iter_dev=it_dev)
        for name in ("active_tiles", "n_active", "tile_rank", "pix_off", "pix_idx"):
            assert torch.equal(views[k][name], w[name]), (k, name)


def test_refusals(B):
    v = [_view(B, 1, 64, 48, 4, 10)]
    for bad in ([], v * 17, [dict(v[0], n_pix=0)], [dict(v[0], n_pix=257)], v + [dict(v[0], n_select=-1)],
                [dict(v[0], workspace=v[0]["workspace"][:16])]):
        with pytest.raises(Exception):
            B.select_tiles_batched(bad, (400, 300, 400, 300), 0)
    with pytest.raises(Exception):
        B.select_tiles_batched(v, (1001, 0, 0, 0), 0)
