"""Binning at a capacity of many pairs, where a launch of its own takes the
tiles' starts and clears the keys before the scatter, bit for bit against the
same scene at the capacity it needs: an odd and an even number of pairs, one
pair, none, tile masks and no mask, and more pairs than the capacity (the
lists before the cut are whole, the count is of all).  And the first call of
a process at tables that take just under the shared memory of a block that has
not asked for more."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2606_15924_gb300 import scenes

pytestmark = pytest.mark.gpu
MANY = 6 << 20


@pytest.fixture(scope="module")
def B():
    from paper_2606_15924_gb300 import binding
    binding.device_check()
    return binding


def _cam(W, H):
    return dict(viewmat=np.eye(4), fx=100.0, fy=100.0, cx=W / 2, cy=H / 2, width=W, height=H, znear=0.2)


@pytest.mark.parametrize("n,W,H,share", [(1, 64, 48, None), (1, 64, 48, 0.0), (3000, 250, 187, 0.3), (3001, 250, 187, None),
                                         (40000, 1957, 1091, 0.2), (40000, 1957, 1091, None)])
def test_starts_launch_is_bit_exact(B, n, W, H, share):
    from gpu_util import bin_dev, projected_dev
    T = ((W + 15) // 16) * ((H + 15) // 16)
    pd = projected_dev(scenes.projected(n, W, H, seed=n))
    rank, R = None, T
    if share is not None:
        on = np.random.default_rng(n).random(T) < share
        R = max(1, int(on.sum()))
        rank = torch.from_numpy(np.where(on, np.cumsum(on) - 1, -1).astype(np.int32)).cuda()
    few = bin_dev(B, pd, n, _cam(W, H), rank, R, capacity=2 * 10 ** 6)
    I = int(few["n_isect"].item())
    assert I < 2 * 10 ** 6 and (I > 0 or share == 0.0)
    many = bin_dev(B, pd, n, _cam(W, H), rank, R, capacity=MANY)
    for k in ("n_isect", "ranges"):
        assert torch.equal(few[k], many[k]), k
    for k in ("vals", "keys"):
        assert torch.equal(few[k][:I], many[k][:I]), k


@pytest.mark.parametrize("capacity", [10 ** 6, MANY])
def test_workspace_at_any_eight_bytes(B, capacity):
    from gpu_util import bin_dev, projected_dev
    n, W, H, T = 3001, 250, 187, 192
    pd, cam = projected_dev(scenes.projected(n, W, H, seed=5)), _cam(W, H)
    want = bin_dev(B, pd, n, cam, None, T, capacity=10 ** 6)
    I = int(want["n_isect"].item())
    need = B.bin_tiles_workspace_size(n, capacity, T)
    ws = torch.empty(need + 24, dtype=torch.uint8, device="cuda")
    vals = torch.zeros(capacity, dtype=torch.int32, device="cuda")
    ranges = torch.zeros(T, 2, dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    for at in (0, 8, 16, 24):
        vals.zero_()
        assert (ws.data_ptr() + at) % 8 == 0
        B.bin_tiles(pd, n, cam, None, T, ws[at:at + need], capacity, vals, None, ranges, count)
        assert torch.equal(vals[:I], want["vals"][:I]) and torch.equal(ranges, want["ranges"]) and int(count.item()) == I


def test_more_pairs_than_the_capacity(B):
    from gpu_util import bin_dev, projected_dev
    n, W, H, T = 1800, 1280, 720, 3600
    pr = scenes.projected(n, W, H, seed=3)
    pr["radius"] = np.full(n, 3000, np.int32)                # every tile
    pd = projected_dev(pr)
    out = bin_dev(B, pd, n, _cam(W, H), None, T, capacity=MANY)
    assert int(out["n_isect"].item()) == n * T > MANY
    ends = np.minimum(np.arange(T + 1) * n, MANY)
    np.testing.assert_array_equal(out["ranges"].cpu().numpy(), np.stack([ends[:-1], ends[1:]], 1))
    order = np.lexsort((np.arange(n), pr["depth"]))          # one list, the same in every tile
    whole = MANY // n
    got = out["vals"][:whole * n].view(whole, n).cpu().numpy()
    np.testing.assert_array_equal(got, np.broadcast_to(order, (whole, n)))


FIRST_CALL = """
import sys, torch
sys.path[:0] = sys.argv[3:]
from gpu_util import bin_dev, projected_dev
from paper_2606_15924_gb300 import binding as B, scenes
W, H, n, R = 1920, 1080, 4000, int(sys.argv[1])
T = 8160
cam = dict(viewmat=[1.0 * (k % 5 == 0) for k in range(16)], fx=100.0, fy=100.0, cx=W / 2, cy=H / 2, width=W, height=H, znear=0.2)
pd = projected_dev(scenes.projected(n, W, H, seed=1))
rank = torch.where(torch.arange(T) < R, torch.arange(T), -1).to(torch.int32).cuda()
got = bin_dev(B, pd, n, cam, rank, R, capacity=int(sys.argv[2]))
want = bin_dev(B, pd, n, cam, None, T, capacity=10 ** 6)
I = int(got["n_isect"].item())
assert I == int(want["ranges"][R - 1, 1].item()) and 0 < I < 10 ** 6
assert torch.equal(got["ranges"], want["ranges"][:R])
for k in ("vals", "keys"):
    assert torch.equal(got[k][:I], want[k][:I]), k
"""


@pytest.mark.parametrize("R,capacity", [(8160, 10 ** 6), (8160, MANY), (7900, 10 ** 6), (7952, 10 ** 6)])
def test_first_call_of_a_process(B, R, capacity):
    """Counters and the rank table of a view of 1920x1080: 48960 bytes with every
    tile active, 48944 and 49152 of two shares of them, where a block has 49152
    for these and the kernel's own arrays before the library asks for more."""
    here = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, "-c", FIRST_CALL, str(R), str(capacity), os.path.dirname(here), here],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
