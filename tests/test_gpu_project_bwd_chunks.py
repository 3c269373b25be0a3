"""The one-view projection adjoint by chunks against the pass that sums several
views (run with one view), whose arithmetic per Gaussian is the same: numbers of
Gaussians at the edges of a block and on both sides of the rule that picks the
chunk, no, few and all Gaussians with a gradient, packed arrays and rows, the
gradients of the others zeroed or left, and a second view added to the first.

Both kernels take the same operations per Gaussian in fp32 in different
instruction orders; a sum of k terms differs by at most k 2^-24 of the sum of
their magnitudes, and the longest chain here is below 100 terms, so values agree
to 100 2^-24 = 6e-6 of the largest term; 2e-5 of the array's largest value is
asked, and zeros are exact."""
import numpy as np
import pytest
import torch

from paper_2606_15924_gb300 import scenes

pytestmark = pytest.mark.gpu
FIELDS = ("means", "log_scales", "quats", "opacity_logits", "sh")


@pytest.fixture(scope="module")
def B():
    from paper_2606_15924_gb300 import binding
    binding.device_check()
    return binding


def _grads(p, rows, fill):
    from paper_2606_15924_gb300.pipeline import as_geo_rows
    g = {k: torch.full_like(v, fill) for k, v in p.items()}
    return as_geo_rows(g) if rows else g


@pytest.mark.parametrize("n,share,rows,write", [(1, 1.0, False, True), (127, 0.1, True, True), (129, 0.0, False, True),
                                                (1000, 1.0, False, False), (5000, 0.05, False, True),
                                                (160001, 0.1, False, True), (160001, 1.0, True, True),
                                                (160511, 0.0, True, True)])
def test_chunked_adjoint(B, n, share, rows, write):
    from gpu_util import empty_projected, gaussians_dev
    from paper_2606_15924_gb300.pipeline import as_geo_rows
    p = gaussians_dev(scenes.gaussians(n, seed=n))
    pp = as_geo_rows(p) if rows else p
    cams = [scenes.look_at((0.0, 0.3, -4.0), width=320, height=200), scenes.look_at((3.0, 0.3, 2.0), width=320, height=200)]
    rng = np.random.default_rng(n)
    ws = torch.empty(B.project_backward_multi_workspace_size(n), dtype=torch.uint8, device="cuda")
    got = _grads(p, rows, 7.0)
    hit = torch.zeros(n, dtype=torch.uint8, device="cuda")
    total, either = None, torch.zeros(n, dtype=torch.bool, device="cuda")
    for k, cam in enumerate(cams):
        proj = empty_projected(n)
        B.project_gaussians(pp, cam, None, proj)
        g2 = torch.from_numpy((rng.normal(size=(n, 12)) * (rng.random((n, 1)) < share)).astype(np.float32)).cuda()
        g2[:, 9:] = 0
        want = _grads(p, rows, 7.0)
        touched = torch.zeros(n, dtype=torch.uint8, device="cuda")
        B.project_backward_multi(pp, B.MultiAdjoint([B.camera(cam)], [proj["radius"]], [g2]), want, touched,
                                 write_untouched=True, workspace=ws)
        total = {f: want[f].clone() if total is None else total[f] + want[f] for f in FIELDS}
        either |= touched.bool()
        B.project_backward(pp, cam, proj, g2, got, hit, write_untouched=write, accumulate=k > 0)
        if k == 0:
            assert torch.equal(hit.bool(), touched.bool())
        on = hit.bool()
        assert torch.equal(on, either)
        for f in FIELDS:
            if write:
                off = got[f][~either]
                assert k > 0 or not off.any()              # zeroed
            else:
                assert bool((got[f][~either] == 7.0).all())  # left
            if on.any():
                scale = float(total[f][on].abs().max())
                assert float((got[f][on] - total[f][on]).abs().max()) <= 2e-5 * scale, f
