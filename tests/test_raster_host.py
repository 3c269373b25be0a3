"""A pixel set described on the host: a SampledRaster of CPU tensors needs no
GPU until it renders."""
import copy

import torch

from paper_2606_15924_gb300 import scenes
from paper_2606_15924_gb300.autograd import SampledRaster


def test_raster_of_cpu_tensors():
    W, H = 50, 40
    r = SampledRaster.from_tiles(scenes.look_at((0.0, 0.0, -4.0), width=W, height=H), 7, [11, 0], device="cpu")
    xy = r.pixel_coords()
    assert r.P == xy.shape[0] == 256 + 2 * 8            # tile 11 is the 2 x 8 corner
    assert xy[0].tolist() == [0, 0] and xy[-1].tolist() == [W - 1, H - 1]
    assert torch.equal(copy.deepcopy(r).pixel_coords(), xy)
