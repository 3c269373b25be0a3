"""The differentiable render's buffers: the gradient taken as it comes (dense,
expanded, strided, with its sign pending) or copied, pixel lists longer than
the sampled pixels, and lists that outgrow the capacity between two passes -
against the same render from a fresh raster with room for everything."""
import copy

import numpy as np
import pytest
import torch

from paper_2606_15924_gb300 import scenes

pytestmark = pytest.mark.gpu
W, H, N = 250, 187, 3000
FIELDS = ("means", "log_scales", "quats", "opacity_logits", "sh")


@pytest.fixture(scope="module")
def AG():
    from paper_2606_15924_gb300 import autograd, binding
    binding.device_check()
    return autograd


def _leaves(scale=0.0):
    g = scenes.gaussians(N, seed=11)
    g["log_scales"] = g["log_scales"] + scale
    return {k: torch.from_numpy(np.ascontiguousarray(v).astype(np.float32)).cuda().requires_grad_(True)
            for k, v in g.items()}


def _raster(AG, pad=0, **kw):
    cam = scenes.look_at((0.0, 0.0, -4.0), width=W, height=H)
    r = AG.SampledRaster.from_tiles(cam, N, range(20, 90), **kw)
    if not pad:
        return r
    return AG.SampledRaster(cam, N, r.active_tiles, r.n_active, r.tile_rank, r.pix_off,
                            torch.cat([r.pix_idx, r.pix_idx[:pad]]), 256, **kw)


def _grads(AG, raster, leaves, grad_of):
    rgb = AG.render_sampled(leaves, raster)
    gr = torch.autograd.grad(rgb, [leaves[k] for k in FIELDS], grad_outputs=grad_of(rgb))
    return rgb.detach(), gr


def _weights(rgb):
    g = torch.Generator(device="cuda").manual_seed(3)
    return torch.rand(rgb.shape, device="cuda", generator=g)


@pytest.mark.parametrize("pad", [0, 37])
@pytest.mark.parametrize("kind", ["dense", "strided", "expanded", "negated"])
def test_gradients_as_they_come(AG, kind, pad):
    leaves = _leaves()
    make = dict(dense=_weights, strided=lambda rgb: torch.stack([_weights(rgb)] * 2, -1)[..., 0],
                expanded=lambda rgb: torch.full((1, 1), 0.5, device="cuda").expand_as(rgb),
                negated=lambda rgb: torch._neg_view(_weights(rgb)))[kind]       # the sign not yet applied
    want_rgb, want = _grads(AG, _raster(AG), leaves, lambda rgb: make(rgb).clone(memory_format=torch.contiguous_format))
    raster = _raster(AG, pad=pad)
    for _ in range(2):                                       # the second pass reuses every buffer
        rgb, got = _grads(AG, raster, leaves, make)
        assert rgb.shape == want_rgb.shape and torch.equal(rgb, want_rgb)
        for f, a, b in zip(FIELDS, got, want):
            # atomics in another order: a few 2^-24 of sums of some hundred terms
            assert float((a - b).abs().max()) <= 1e-4 * float(b.abs().max()), f


def test_copy_of_a_used_raster(AG):
    leaves = _leaves()
    raster = _raster(AG)
    want_rgb, want = _grads(AG, raster, leaves, _weights)
    twin = copy.deepcopy(raster)
    for r in (twin, raster):
        rgb, got = _grads(AG, r, leaves, _weights)
        assert torch.equal(rgb, want_rgb)
        for f, a, b in zip(FIELDS, got, want):
            assert float((a - b).abs().max()) <= 1e-4 * float(b.abs().max()), f


def test_lists_that_outgrow_the_capacity(AG):
    small, large = _leaves(), _leaves(1.2)
    raster = _raster(AG)
    _grads(AG, raster, small, _weights)
    before = raster.capacity
    rgb, got = _grads(AG, raster, large, _weights)
    assert raster.capacity > before
    want_rgb, want = _grads(AG, _raster(AG, capacity=4 * raster.capacity), large, _weights)
    assert torch.equal(rgb, want_rgb)
    for f, a, b in zip(FIELDS, got, want):
        assert float((a - b).abs().max()) <= 1e-4 * float(b.abs().max()), f


def test_lists_that_outgrow_the_capacity_on_another_stream(AG, monkeypatch):
    """The old lists are given back while the first render may still read them:
    not before that stream is done with them."""
    small, large = _leaves(), _leaves(1.2)
    raster = _raster(AG)
    _grads(AG, raster, small, _weights)
    old, kept = raster.vals, []
    record = torch.Tensor.record_stream
    monkeypatch.setattr(torch.Tensor, "record_stream", lambda t, s: (kept.append((t.data_ptr(), s)), record(t, s))[1])
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side), torch.no_grad():
        rgb = raster.forward_buffers(large)
    torch.cuda.current_stream().wait_stream(side)
    assert raster.vals is not old and (old.data_ptr(), side) in kept
    want = _raster(AG, capacity=4 * raster.capacity).forward_buffers({k: v.detach() for k, v in large.items()})
    assert torch.equal(rgb, want)


def test_capture_is_refused_as_before(AG):
    """The pair count is read on the host, so a pass cannot be captured."""
    leaves = _leaves()
    raster = _raster(AG)
    AG.render_sampled(leaves, raster)
    torch.cuda.synchronize()
    with pytest.raises(Exception):
        with torch.cuda.graph(torch.cuda.CUDAGraph()):
            AG.render_sampled(leaves, raster)
    torch.cuda.synchronize()
