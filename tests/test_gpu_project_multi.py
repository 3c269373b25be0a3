"""The projection of several views in one pass against one projection per view,
bit for bit: one view (which takes the single-view kernel), a few and sixteen,
of different sizes and poses, numbers of Gaussians at the edges of a block,
every SH degree, packed arrays and rows, tile masks (no mask, some tiles, none:
a Gaussian that no view sees), Gaussians behind every camera, and warps with up
to 16, 17 and 32 visible Gaussians (the single-view kernel stages sixteen SH
rows a round)."""
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


@pytest.mark.parametrize("n,K,degree,rows", [(1, 2, 3, False), (255, 16, 0, True), (257, 3, 1, False), (5000, 1, 3, True),
                                             (5000, 5, 2, True), (20000, 8, 3, False), (16, 4, 3, True),
                                             (17, 4, 2, False), (33, 4, 3, False), (31, 4, 1, True)])
def test_views_in_one_pass_are_bit_exact(B, n, K, degree, rows):
    from gpu_util import empty_projected, gaussians_dev
    from paper_2606_15924_gb300.pipeline import as_geo_rows
    g = scenes.gaussians(n, seed=n)
    if n > 1000:
        g["means"][::7] *= 40.0                        # far off, and behind some of the cameras
        g["quats"][5] *= 3.0                             # not of unit length
    p = gaussians_dev(g)
    if rows:
        p = as_geo_rows(p)
    rng = np.random.default_rng(n)
    cams, ranks = [], []
    for k in range(K):
        W, H = (256, 256) if k % 2 == 0 else (333, 187)
        a = 2 * np.pi * k / K
        cams.append(scenes.look_at((4.0 * np.sin(a), 0.3, -4.0 * np.cos(a)), width=W, height=H))
        T = ((W + 15) // 16) * ((H + 15) // 16)
        share = (None, 0.1, 0.0, 1.0)[k % 4]
        ranks.append(None if share is None else
                     torch.from_numpy(np.where(rng.random(T) < share, np.arange(T), -1).astype(np.int32)).cuda())
    got = [empty_projected(n) for _ in range(K)]
    for o in got:
        for v in o.values():
            v.fill_(7)                                     # every value is written
    B.project_gaussians_multi(p, cams, ranks, got, sh_degree=degree)
    seen = 0
    for k in range(K):
        want = empty_projected(n)
        B.project_gaussians(p, cams[k], ranks[k], want, sh_degree=degree)
        seen += int((want["radius"] > 0).sum())
        for name in want:
            assert torch.equal(got[k][name], want[name]), (k, name)
    assert n == 1 or seen > 0


def test_invalid_views_are_rejected(B):
    from gpu_util import empty_projected, gaussians_dev
    p = gaussians_dev(scenes.gaussians(64, seed=1))
    cam = scenes.look_at((0.0, 0.0, -4.0), width=64, height=64)
    for K in (0, 17):
        with pytest.raises(Exception):
            B.project_gaussians_multi(p, [cam] * K, [None] * K, [empty_projected(64)] * K)
    with pytest.raises(ValueError):
        B.project_gaussians_multi(p, [cam, cam], [None], [empty_projected(64)] * 2)
