"""Frames taken in depth slabs (2^26 pairs, or 2^24 of large boxes) against the same frames taken in one, and the lists of those."""
import dataclasses

import numpy as np
import pytest

from synth import scenes

pytestmark = pytest.mark.gpu


def _scene(n, spread):
    """n copies of asset 0, turned and scaled differently, around the origin."""
    rng = np.random.Generator(np.random.PCG64(n))
    return scenes.Instances(np.zeros(n, np.uint32), scenes.random_rotations(rng, n), rng.uniform(-spread, spread, (n, 3)),
                            rng.uniform(0.7, 1.4, n))


def _in_slabs(stats, at_least):
    return stats["pairs"] >= max(at_least, 1 << 24) and (stats["pairs"] >= 1 << 26 or stats["pairs"] >= 16 * stats["visible"])


@pytest.mark.parametrize("n,spread,width,height,fov,views,graphs,at_least", [
    (12, 0.5, 1920, 1080, 70.0, 1, 0, 1 << 24),    # a pile next to the camera: large boxes, early stops: two slabs
    (12, 0.5, 1001, 563, 40.0, 3, 0, 1 << 24),     # ragged images, several views
    (12, 0.5, 1001, 563, 40.0, 3, 1, 1 << 24),     # the same, captured
    (40, 3.0, 1601, 901, 50.0, 4, 0, 1 << 26),     # two slabs, small boxes
    (40, 3.0, 1601, 901, 50.0, 8, 0, 1 << 27),     # four slabs
])
def test_slabs_change_nothing(tiny_asset, n, spread, width, height, fov, views, graphs, at_least):
    """Blend variant 1 keeps its frames in one slab and gives the same image bit for bit; the sorted lists that the
    read-backs return are those of the whole frame either way."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    from paper_2505_06523_gb300._native import V3DG_OPT_BLEND_MODE, V3DG_OPT_GRAPHS
    inst = _scene(n, spread)
    cams = [scenes.look_at((0.3 * v, -2.0 - spread, 0.5), (0.0, 0.0, 0.0), width, height, fov) for v in range(views)]
    got = []
    with Context(0) as ctx:
        ctx.set_option(V3DG_OPT_GRAPHS, graphs)
        ctx.load_hierarchy(tiny_asset)
        ctx.set_instances(inst)
        for mode in (1, 0):
            ctx.set_option(V3DG_OPT_BLEND_MODE, mode)
            for _ in range(2):   # (the second frame knows the first one's size)
                ctx.select_views(cams, 0.25)
                rgb, T = ctx.render(want_T=True)
            got.append({"rgb": rgb.cpu().numpy(), "T": T.cpu().numpy(),
                        **{"proj_" + k: v for k, v in ctx.get_projected().items()}, "ranges": ctx.tile_ranges(),
                        **{"pair_" + k: v for k, v in ctx.get_pairs().items()}, "stats": ctx.frame_stats()})
            again = ctx.render(want_T=True)   # the lists were made again in between
            assert (again[0].cpu().numpy() == got[-1]["rgb"]).all()
    one, slabs = got
    assert _in_slabs(one["stats"], at_least), one["stats"]
    assert one["stats"] == {**slabs["stats"]}
    assert float(np.abs(one["rgb"]).sum()) > 0 and (one["T"] < 1e-3).any()
    for k in one:
        if k != "stats":
            assert one[k].shape == slabs[k].shape and (one[k] == slabs[k]).all(), k


def test_slabs_with_depths_in_one_bin(tiny_asset):
    """Every Gaussian in a narrow depth range (fewer histogram bins than slabs): the empty slabs change nothing."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    from paper_2505_06523_gb300._native import V3DG_OPT_BLEND_MODE
    flat = dataclasses.replace(tiny_asset, means=(tiny_asset.means * np.array([1.0, 1e-3, 1.0], np.float32)))
    n = 24
    inst = scenes.Instances(np.zeros(n, np.uint32), np.repeat(np.eye(3)[None], n, 0), np.zeros((n, 3)), np.ones(n))
    cam = scenes.look_at((0.0, -1.31, 0.0), (0.0, 0.0, 0.0), 1600, 900, 80.0)
    imgs = []
    with Context(0) as ctx:
        ctx.load_hierarchy(flat)
        ctx.set_instances(inst)
        for mode in (1, 0):
            ctx.set_option(V3DG_OPT_BLEND_MODE, mode)
            for _ in range(2):
                ctx.select(cam, 0.25)
                rgb, T = ctx.render(want_T=True)
            imgs.append((rgb.cpu().numpy(), T.cpu().numpy()))
        assert _in_slabs(ctx.frame_stats(), 1 << 24)
    assert (imgs[0][0] == imgs[1][0]).all() and (imgs[0][1] == imgs[1][1]).all()


def test_most_slabs(tiny_asset):
    """The most slabs (2^29 pairs: sixteen views of a pile): images and transmittances as in one slab, bit for bit."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    from paper_2505_06523_gb300._native import V3DG_OPT_BLEND_MODE
    inst = _scene(30, 0.6)
    cams = [scenes.look_at((0.2 * v, -2.6, 0.1 * v), (0.0, 0.0, 0.0), 1920, 1080, 70.0) for v in range(16)]
    imgs = []
    with Context(0) as ctx:
        ctx.load_hierarchy(tiny_asset)
        ctx.set_instances(inst)
        for mode in (1, 0):
            ctx.set_option(V3DG_OPT_BLEND_MODE, mode)
            for _ in range(2):
                ctx.select_views(cams, 0.25)
                rgb, T = ctx.render(want_T=True)
            imgs.append((rgb.clone(), T.clone()))
        assert _in_slabs(ctx.frame_stats(), 1 << 29), ctx.frame_stats()
    assert bool((imgs[0][0] == imgs[1][0]).all()) and bool((imgs[0][1] == imgs[1][1]).all())


@pytest.mark.parametrize("n,distance,away,tau", [
    (1, 3.0, True, 0.25),     # nothing visible
    (1, 400.0, False, 64.0),  # one node: a fraction of one sort tile
    (1, 1.2, False, 1.0),     # part of one asset, many slots outside the image
    (3, 2.5, False, 0.25),    # several sort tiles
    (9, 30.0, False, 2.0),
])
def test_one_slab_lists(tiny_asset, n, distance, away, tau):
    """The pair list of a one-slab frame, whose depth sort reads the render list's slots itself, against a stable sort on
    the host of the projected Gaussians' tiles by (tile, depth), Gaussians in slot order."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    target = (0.0, -2.0 * distance, 0.0) if away else (0.0, 0.0, 0.0)
    with Context(0) as ctx:
        ctx.load_hierarchy(tiny_asset)
        ctx.set_instances(_scene(n, 0.5))
        ctx.select(scenes.look_at((0.0, -distance, 0.3), target, 333, 217, 50.0), tau)
        ctx.render()
        proj, pairs, stats = ctx.get_projected(), ctx.get_pairs(), ctx.frame_stats()
    assert stats["pairs"] < 1 << 24 and (stats["visible"] == 0) == away
    assert len(proj["local"]) == stats["visible"] and len(pairs["tile"]) == stats["pairs"]
    tiles_x = (333 + 15) // 16
    r = proj["rect"].astype(np.int64)   # tiles x0, x1, y0, y1 (inclusive)
    w, h = r[:, 1] - r[:, 0] + 1, r[:, 3] - r[:, 2] + 1
    g = np.repeat(np.arange(len(r)), w * h)
    k = np.arange(len(g)) - np.repeat(np.cumsum(w * h) - w * h, w * h)
    tile = (r[g, 2] + k // w[g]) * tiles_x + r[g, 0] + k % w[g]
    order = np.lexsort((g, proj["depth_key"][g], tile))
    assert (tile[order] == pairs["tile"]).all()
    for name in ("depth_key", "inst", "local"):
        assert (proj[name][g[order]] == pairs[name]).all(), name
