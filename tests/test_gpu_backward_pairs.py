"""The paired-splat backward at the sizes where its division into items
changes: pixel counts around the lanes' and groups' edges, with and without
checkpoints, few and many tiles, opacities at the cap on alpha; and infinite
or NaN gradients and colours, which stay with the pixels and splats they
belong to."""
import numpy as np
import pytest
import torch

from paper_2606_15924_gb300 import scenes

pytestmark = pytest.mark.gpu
W, H, N = 96, 80, 700


@pytest.fixture(scope="module")
def B():
    from paper_2606_15924_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def _case(B, n_pix, slots, n_select, seed=11):
    from gpu_util import bin_dev, projected_dev, select_dev
    p = scenes.projected(N, W, H, seed=seed, radius_max=18)
    p["opac"][::7] = 0.995                       # capped alphas near the centre
    p["opac"][3::7] = 0.02                       # barely above the threshold
    cam = scenes.look_at((0.0, 0.0, -4.0), width=W, height=H)
    sel = select_dev(B, scenes.error_map(W, H), scenes.age_map(W, H), W, H, n_select, n_pix, seed=4)
    pd = projected_dev(p)
    binned = bin_dev(B, pd, N, cam, sel["tile_rank"], sel["n_sel"], capacity=40000)
    P = sel["n_sel"] * n_pix
    out = dict(rgb=torch.zeros(P, 3, device="cuda"), T=torch.zeros(P, device="cuda"),
               n_last=torch.zeros(P, dtype=torch.int32, device="cuda"))
    ck = None
    if slots:
        data = torch.full((B.checkpoint_bytes(sel["n_sel"], n_pix, slots) // 4,), float("nan"), device="cuda")
        last = torch.zeros(sel["n_sel"], dtype=torch.int32, device="cuda")
        ck = B.checkpoints(data, slots, P, out["rgb"], last)
        out["keep"] = (data, last)
    out["ck"] = ck
    bg = (0.3, 0.1, 0.6)
    B.render_sampled(pd, binned["ranges"], binned["vals"], sel["active_tiles"], sel["n_active"], sel["n_sel"],
                     sel["pix_off"], sel["pix_idx"], n_pix, cam, bg, out["rgb"], out["T"], out["n_last"], ckpt=ck)

    def backward(dL, proj=pd):
        g2 = torch.full((N, 12), 7.0, device="cuda")
        B.render_backward_sampled(proj, binned["ranges"], binned["vals"], sel["active_tiles"], sel["n_active"],
                                  sel["n_sel"], sel["pix_off"], sel["pix_idx"], n_pix, cam, bg, out["T"],
                                  out["n_last"], dL, g2, ckpt=ck)
        return g2
    return p, sel, binned, out, bg, backward, P, pd


@pytest.mark.parametrize("slots", [0, 3, 64])
@pytest.mark.parametrize("n_pix", [1, 31, 33, 64, 65, 96, 97, 128, 129, 193, 256])
def test_pixel_counts_against_oracle(B, orc, n_pix, slots):
    from gpu_util import select_host
    for n_select in (2, 30):
        p, sel, binned, out, bg, backward, P, pd = _case(B, n_pix, slots, n_select)
        sh = select_host(sel)
        pix = orc.pixel_coords(sh["active_tiles"], sh["pix_off"], sh["pix_idx"], W)
        dL = torch.zeros(P, 3, device="cuda")
        dL[:len(pix)] = torch.randn(len(pix), 3, generator=torch.Generator().manual_seed(5)).cuda()
        # pixels whose decisions sit at a threshold are left out of the loss
        want = {k: np.asarray(v, np.float64) for k, v in p.items() if k != "radius"}
        want["radius"] = p["radius"]
        ref = orc.render_pixels(want, W, H, pix, bg=bg)
        amb = torch.from_numpy(ref["margin"] <= 1e-4).cuda()
        dL[:len(pix)][amb] = 0.0
        g2 = backward(dL).cpu().numpy().astype(np.float64)
        w2 = orc.render_backward(want, W, H, pix, dL[:len(pix)].cpu().numpy().astype(np.float64), bg=bg)
        w2 = w2["grad2d"] if isinstance(w2, dict) else w2
        k = w2.shape[1]
        assert np.linalg.norm(g2[:, :k] - w2) <= 1e-3 * np.linalg.norm(w2) + 1e-12
        assert np.all(g2[:, 9:] == 0.0)


@pytest.mark.parametrize("n_pix,span", [(25, 1), (85, 2), (25, 4)])
def test_lists_that_end_with_the_array(B, n_pix, span):
    """Pieces of 32 span positions against whole lists (no checkpoints), where
    the last tile's list ends where the array of entries does: lists of every
    length about the pieces' chunks, and one cut off by the capacity."""
    from gpu_util import bin_dev, projected_dev, select_dev
    tiles = {1: 1, 2: 500, 4: 2600}[span]          # as many as make the pieces that long
    tx = min(tiles, 64)
    W2, H2 = 16 * tx, 16 * ((tiles + tx - 1) // tx)
    T = (W2 // 16) * (H2 // 16)
    cam = scenes.look_at((0.0, 0.0, -4.0), width=W2, height=H2)
    sel = select_dev(B, scenes.error_map(W2, H2), scenes.age_map(W2, H2), W2, H2, T, n_pix, seed=4)
    for L in (1, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 161):
        p = scenes.projected(L, W2, H2, seed=L, radius_max=5)
        rng = np.random.default_rng(L)
        p["xy"] = (np.array([W2 - 8.0, H2 - 8.0]) + rng.uniform(-2, 2, (L, 2))).astype(np.float32)   # the last tile
        p["radius"][:] = 5
        p["opac"] = rng.uniform(0.02, 0.06, L)
        pd = projected_dev(p)
        for cap in (L, L - 1):
            if cap == 0:
                continue
            b = bin_dev(B, pd, L, cam, sel["tile_rank"], T, capacity=cap)
            assert b["vals"].shape[0] == cap and int(b["ranges"][T - 1, 1]) == cap and int(b["n_isect"].item()) == L
            P = T * n_pix
            g = []
            for slots in (0, 64):
                rgb, Tf = torch.zeros(P, 3, device="cuda"), torch.zeros(P, device="cuda")
                last = torch.zeros(P, dtype=torch.int32, device="cuda")
                data = torch.full((B.checkpoint_bytes(T, n_pix, 64) // 4,), float("nan"), device="cuda")
                longest = torch.zeros(T, dtype=torch.int32, device="cuda")
                ck = B.checkpoints(data, 64, P, rgb, longest) if slots else None
                a = (pd, b["ranges"], b["vals"], sel["active_tiles"], sel["n_active"], T, sel["pix_off"], sel["pix_idx"],
                     n_pix, cam, (0.3, 0.1, 0.6))
                B.render_sampled(*a, rgb, Tf, last, ckpt=ck)
                dL = torch.randn(P, 3, generator=torch.Generator().manual_seed(5)).cuda()
                g2 = torch.zeros(L, 12, device="cuda")
                B.render_backward_sampled(*a, Tf, last, dL, g2, ckpt=ck)
                g.append(g2)
            assert float(g[0].abs().max()) > 0
            # sums of the same terms, T recovered from another end: some 2^-24 a position
            assert float((g[0] - g[1]).norm()) <= 1e-4 * float(g[0].norm()), (L, cap)


@pytest.mark.parametrize("slots", [0, 64])
def test_nonfinite_values_stay_local(B, slots):
    """One pixel with an infinite and one with a NaN gradient poison the splats
    they blend and no others; an infinite colour poisons only its own pixels'
    splats."""
    n_pix = 85
    p, sel, binned, out, bg, backward, P, pd = _case(B, n_pix, slots, 20)
    A = int(sel["n_active"].item())
    Pn = int(sel["pix_off"][A].item())
    dL = torch.randn(P, 3, generator=torch.Generator().manual_seed(6)).cuda()
    dL[Pn:] = 0.0
    clean = backward(dL)
    bad = [5, Pn // 2]
    only = torch.zeros_like(dL)
    only[bad] = 1.0
    hit = (backward(only) != 0).any(1)            # the splats those pixels blend
    assert hit.any() and not hit.all()
    d2 = dL.clone()
    d2[bad[0], 1] = float("inf")
    d2[bad[1], 0] = float("nan")
    got = backward(d2)
    assert not torch.isfinite(got[hit][:, :9]).all(1).any()
    assert torch.isfinite(got[~hit]).all()
    rest = ~hit
    err = (got[rest] - clean[rest]).norm() / clean[rest].norm()
    assert float(err) <= 1e-5
    # an infinite colour of one blended splat
    i = int(torch.nonzero(hit)[0])
    q = dict(pd)
    q["rgb"] = pd["rgb"].clone()
    q["rgb"][i, 2] = float("inf")
    got = backward(dL, proj=q)
    assert not bool(torch.isfinite(got[i, :9]).all())
    assert bool(torch.isfinite(got).all(1).sum() > 0.5 * N)


@pytest.mark.parametrize("batched", [False, True])
def test_statistics_without_checkpoints_are_the_walks(B, batched):
    """One tile, so that every splat's row takes one sum: the bits of
    error_stats_sampled, whose T are the forward's products."""
    n_pix = 32
    p, sel, binned, out, bg, backward, P, pd = _case(B, n_pix, 0, 1)
    cam = scenes.look_at((0.0, 0.0, -4.0), width=W, height=H)
    err = torch.rand(P, generator=torch.Generator().manual_seed(7)).cuda()
    dL = torch.randn(P, 3, generator=torch.Generator().manual_seed(5)).cuda()
    a = (pd, binned["ranges"], binned["vals"], sel["active_tiles"], sel["n_active"], 1, sel["pix_off"], sel["pix_idx"],
         n_pix, cam)
    want = torch.zeros(N, 4, device="cuda")
    B.error_stats_sampled(*a, out["n_last"], err, want)
    g2, got = torch.zeros(N, 12, device="cuda"), torch.zeros(N, 4, device="cuda")
    if batched:
        vb = B.view_batch([dict(proj=pd, tile_ranges=binned["ranges"], vals=binned["vals"],
                                active_tiles=sel["active_tiles"], n_active=sel["n_active"], n_active_max=1,
                                pix_off=sel["pix_off"], pix_idx=sel["pix_idx"], n_pix_max=n_pix, cam=cam, bg=bg,
                                rgb=out["rgb"], T_final=out["T"], n_last=out["n_last"], ckpt=None, dL_drgb=dL,
                                grad2d=g2)])
        B.render_backward_batched_stats(vb, 4, torch.zeros(1, dtype=torch.int32, device="cuda"), [err], got)
    else:
        B.render_backward_sampled_stats(*a, bg, out["T"], out["n_last"], dL, g2, err, got)
    assert int((want[:, 1] > 0).sum()) > 20
    assert torch.equal(got, want)
    plain = backward(dL)
    assert float((g2 - plain).norm()) <= 1e-6 * float(plain.norm())


def _one_splat_a_tile(B, opac):
    """A splat and a sampled pixel in each of 4096 tiles: every output row is one
    term.  Returns a call of the backward with checkpoints for a given gradient
    and error: (grad2d, statistics), the separate walk's statistics for the
    error, and the forward's outputs."""
    from gpu_util import bin_dev, projected_dev, select_dev
    n = T = 4096
    W1 = H1 = 1024
    rng = np.random.default_rng(9)
    p = scenes.projected(n, W1, H1, seed=9)
    t = np.arange(n)
    p["xy"] = (16.0 * np.stack([t % 64, t // 64], 1) + rng.uniform(2.0, 14.0, (n, 2))).astype(np.float32)
    p["radius"][:] = 1
    p["conic"] = np.stack([rng.uniform(0.01, 0.05, n), rng.uniform(-0.005, 0.005, n), rng.uniform(0.01, 0.05, n)],
                          1).astype(np.float32)
    p["opac"] = opac(rng, n).astype(np.float32)
    p["rgb"] = np.tile(np.float32([1.0, 0.0, 0.0]), (n, 1))
    cam = scenes.look_at((0.0, 0.0, -4.0), width=W1, height=H1)
    sel = select_dev(B, scenes.error_map(W1, H1), scenes.age_map(W1, H1), W1, H1, T, 1, seed=4)
    pd = projected_dev(p)
    b = bin_dev(B, pd, n, cam, sel["tile_rank"], T, capacity=n)
    rgb, Tf, last = torch.zeros(T, 3, device="cuda"), torch.zeros(T, device="cuda"), torch.zeros(T, dtype=torch.int32, device="cuda")
    data, longest = torch.zeros(T * 4, device="cuda"), torch.zeros(T, dtype=torch.int32, device="cuda")
    ck = B.checkpoints(data, 1, T, rgb, longest)
    a = (pd, b["ranges"], b["vals"], sel["active_tiles"], sel["n_active"], T, sel["pix_off"], sel["pix_idx"], 1, cam)
    bg = (0.0, 0.0, 0.0)
    B.render_sampled(*a, bg, rgb, Tf, last, ckpt=ck)

    def backward(dL, err):
        keep = data, longest
        g2, st, walk = (torch.zeros(n, w, device="cuda") for w in (12, 4, 4))
        B.render_backward_sampled_stats(*a, bg, Tf, last, dL, g2, err, st, ckpt=ck)
        B.error_stats_sampled(*a, last, err, walk)
        return g2, st, walk
    return p, rgb, backward


def test_statistics_take_the_rounded_square_root(B):
    """D is an IEEE square root in the replay as in the walk: where both have the
    same bits of w (T recovered as exactly 1), D w has the same bits too."""
    p, rgb, backward = _one_splat_a_tile(B, lambda rng, n: rng.uniform(0.2, 0.9, n))
    one = torch.ones(4096, device="cuda")
    _, st, walk = backward(torch.zeros(4096, 3, device="cuda"), one)
    same = (st[:, 1] == walk[:, 1]) & (walk[:, 1] > 0)
    assert int(same.sum()) > 1000
    assert torch.equal(st[same, 2], walk[same, 2])


def test_opacity_gradient_takes_the_rounded_reciprocal(B):
    """With colour (1, 0, 0), that gradient and no background, the sums of one
    splat and pixel are dL/dred = alpha T and dL/do = (alpha T) / o: the same
    bits times 1 / o rounded, over opacities of every mantissa."""
    p, rgb, backward = _one_splat_a_tile(B, lambda rng, n: rng.uniform(0.1, 0.98, n))
    dL = torch.zeros(4096, 3, device="cuda")
    dL[:, 0] = 1.0
    g2, _, _ = backward(dL, torch.zeros(4096, device="cuda"))
    g2 = g2.cpu().numpy()
    hit = g2[:, 6] > 0
    assert hit.sum() > 3000
    np.testing.assert_array_equal(g2[hit, 5], g2[hit, 6] * (np.float32(1.0) / p["opac"][hit]))


def test_skipped_splats_leave_the_transmittance_alone(B):
    """A pixel that blends the first and the last splat of a list and none of
    the thousands between, which other pixels of its group blend: its gradients
    have the bits of the list of those two."""
    from gpu_util import bin_dev, dev, projected_dev
    n, side = 6002, 16
    cam = scenes.look_at((0.0, 0.0, -4.0), width=side, height=side)
    rng = np.random.default_rng(2)
    p = scenes.projected(n, side, side, seed=2)
    ends = [0, n - 1]
    p["xy"] = np.stack([rng.uniform(11.0, 15.0, n), rng.uniform(0.0, 2.0, n)], 1).astype(np.float32)
    p["conic"] = np.tile(np.float32([1.0, 0.1, 1.0]), (n, 1))            # 10 pixels away: exp(-50)
    p["xy"][ends], p["conic"][ends] = [[1.0, 1.2], [1.5, 0.9]], [[0.05, 0.01, 0.06], [0.04, 0.0, 0.05]]
    p["radius"][:] = 4
    p["opac"] = rng.uniform(0.02, 0.6, n).astype(np.float32)
    p["depth"] = np.linspace(1.0, 9.0, n).astype(np.float32)
    sel = dict(active_tiles=dev(np.int32([0])), n_active=dev(np.int32([1])), tile_rank=dev(np.int32([0])),
               pix_off=dev(np.int32([0, 32])), pix_idx=dev(np.arange(32, dtype=np.uint8)))
    rows = []
    for keep in (np.arange(n), np.array(ends)):
        q = {k: v[keep] for k, v in p.items()}
        pd, m = projected_dev(q), len(keep)
        b = bin_dev(B, pd, m, cam, sel["tile_rank"], 1, capacity=n)
        rgb, Tf = torch.zeros(32, 3, device="cuda"), torch.zeros(32, device="cuda")
        last, g2 = torch.zeros(32, dtype=torch.int32, device="cuda"), torch.zeros(m, 12, device="cuda")
        a = (pd, b["ranges"], b["vals"], sel["active_tiles"], sel["n_active"], 1, sel["pix_off"], sel["pix_idx"], 32, cam,
             (0.3, 0.1, 0.6))
        B.set_forward_split(1)               # the sequential walk: no composition of half lists
        B.render_sampled(*a, rgb, Tf, last)
        B.set_forward_split(0)
        dL = torch.zeros(32, 3, device="cuda")
        dL[0] = torch.tensor([0.7, -0.4, 0.9])
        B.render_backward_sampled(*a, Tf, last, dL, g2)
        assert int(last[0]) == m and int((g2 != 0).any(1).sum()) == 2
        rows.append((g2[[0, m - 1]], rgb[0], Tf[0]))
    for x, y in zip(*rows):
        assert torch.equal(x, y)


@pytest.mark.parametrize("slots", [0, 3, 7, 64])
@pytest.mark.parametrize("grid", [64, 2])
def test_batched_warps_share_few_items(B, grid, slots):
    """The queue's counter after the launch: a claim for each tile and every
    piece of the first quarter, and a last one of every block."""
    n_pix, tiles = 32, 24
    p, sel, binned, out, bg, backward, P, pd = _case(B, n_pix, slots, tiles)
    cam = scenes.look_at((0.0, 0.0, -4.0), width=W, height=H)
    dL = torch.randn(P, 3, generator=torch.Generator().manual_seed(5)).cuda()
    g2 = torch.zeros(N, 12, device="cuda")
    vb = B.view_batch([dict(proj=pd, tile_ranges=binned["ranges"], vals=binned["vals"], active_tiles=sel["active_tiles"],
                            n_active=sel["n_active"], n_active_max=tiles, pix_off=sel["pix_off"], pix_idx=sel["pix_idx"],
                            n_pix_max=n_pix, cam=cam, bg=bg, rgb=out["rgb"], T_final=out["T"], n_last=out["n_last"],
                            ckpt=out["ck"], dL_drgb=dL, grad2d=g2)])
    counter = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.render_backward_batched(vb, grid, counter)
    assert int(counter.item()) == tiles * ((slots + 1 + 3) // 4) + grid      # short lists: a piece a slot, and the rest
    plain = backward(dL)
    assert float((g2 - plain).norm()) <= 1e-6 * float(plain.norm())
