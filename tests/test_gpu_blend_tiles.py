"""The blend where its work items (8x4 pixels of a 16x16 tile, two 4x4 halves each) meet the image's edges."""
import numpy as np
import pytest

from synth import scenes
from v3dg_cases import assert_image_matches_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height", [(1, 1), (4, 4), (5, 3), (8, 4), (9, 5), (16, 16), (17, 33), (31, 20)])
def test_ragged_images(small_asset, width, height):
    """Sizes around the edges of halves, sub-tiles and tiles, lists of 1 to a few thousand records: against the oracle
    (its image bounds), and bit for bit against the block-per-tile variant."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    from paper_2505_06523_gb300._native import V3DG_OPT_BLEND_MODE
    inst = scenes.single_instance()
    cam = scenes.look_at((0.0, -2.6, 0.4), (0.0, 0.0, 0.0), width, height, 60.0)
    out = []
    with Context(0) as ctx:
        ctx.load_hierarchy(small_asset)
        ctx.set_instances(inst)
        for mode in (0, 1):
            ctx.set_option(V3DG_OPT_BLEND_MODE, mode)
            ctx.select(cam, 1.0)
            rgb, T = ctx.render(want_T=True)
            out.append((rgb.cpu().numpy(), T.cpu().numpy()))
    assert_image_matches_oracle(*out[0], [small_asset], inst, cam, 1.0)
    assert (out[0][0] == out[1][0]).all() and (out[0][1] == out[1][1]).all()


def test_empty_and_infinite_records(small_asset):
    """An image that no Gaussian reaches is 0 with T = 1; a Gaussian whose projected covariance overflows to
    infinity (its conic is not a number) covers every tile and adds nothing, as before."""
    import dataclasses

    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    ls = small_asset.log_scales.copy()
    ls[7] = 46.0
    huge = dataclasses.replace(small_asset, log_scales=ls)
    inst = scenes.single_instance()
    cam = scenes.look_at((0.0, -2.6, 0.4), (0.0, 0.0, 0.0), 40, 24, 60.0)
    away = scenes.look_at((0.0, -9.0, 0.4), (0.0, -20.0, 0.4), 40, 24, 60.0)
    imgs = []
    for asset in (small_asset, huge):
        with Context(0) as ctx:
            ctx.load_hierarchy(asset)
            ctx.set_instances(inst)
            ctx.select(cam, 0.25)
            imgs.append([x.cpu().numpy() for x in ctx.render(want_T=True)])
            if asset is small_asset:
                ctx.select(away, 0.25)
                rgb, T = ctx.render(want_T=True)
                assert (rgb == 0).all() and (T == 1).all()
    assert np.isfinite(imgs[1][0]).all()
    err = np.abs(imgs[0][0] - imgs[1][0])
    # at most Gaussian 7 itself is missing: one of thousands, of a few pixels
    assert (err.max(-1) > 0).mean() < 0.05


@pytest.mark.parametrize("n,aside", [(1, 0), (95, 0), (97, 0), (1000, 0), (4100, 0), (1000, 190), (1500, 234), (2000, 300), (1500, 575)])
def test_long_lists(n, aside):
    """One tile with n faint Gaussians on top of each other (only the longest stack stops a pixel): lists below and above the length
    from which a block blends them together, rounds that end within a batch; against the block-per-tile variant bit
    for bit, and against the closed form T = (1 - alpha)^k at the centre pixel (n roundings of 2^-24 each).
    aside: as many more in front, small and in a corner of the same tile, so that the centre's sub-tile meets a sparse
    stretch of the list before the dense one."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    from paper_2505_06523_gb300._native import V3DG_OPT_BLEND_MODE
    from synth.assets import Asset
    rng = np.random.default_rng(n)
    stack, n = n, n + aside
    nodes = (n + 63) // 64
    o = np.float32(max(0.005, min(0.5, 2.0 / stack)))
    means = np.concatenate([rng.uniform(-1e-4, 1e-4, (n, 2)), rng.uniform(-0.01, 0.01, (n, 1))], 1).astype(np.float32)
    means[:, :2] = 0.0
    scales = np.full((n, 3), -2.0, np.float32)
    means[stack:], scales[stack:] = (0.9625, 0.175, -0.5), -4.0   # 11 and 2 px from the centre pixel, 0.2 px wide
    sh = np.zeros((n, 16, 3), np.float32)
    sh[:, 0] = rng.uniform(-1, 1, (n, 3))
    count = np.minimum(64, n - 64 * np.arange(nodes)).astype(np.uint32)
    first = (64 * np.arange(nodes)).astype(np.uint32)
    if nodes > 1:   # a root above the leaves: one more Gaussian, never selected
        means, sh, scales = (np.concatenate([x, x[:1]]) for x in (means, sh, scales))
        count, first = np.append(count, 1).astype(np.uint32), np.append(first, n).astype(np.uint32)
    level = np.array([0] * nodes + [1] * (nodes > 1), np.uint8)
    parent = np.array([nodes if nodes > 1 else -1] * nodes + [-1] * (nodes > 1), np.int32)
    m = len(means)
    asset = Asset(means=means, log_scales=scales, quats=np.tile(np.float32([1, 0, 0, 0]), (m, 1)),
                  opacity=np.full(m, o, np.float32), sh=sh, node_first=first, node_count=count, node_level=level,
                  node_parent=parent, own_sphere=np.tile(np.float32([0, 0, 0, 1]), (len(count), 1)))
    inst = scenes.single_instance()
    cam = scenes.Camera(np.array([[1.0, 0, 0, 0], [0, 1.0, 0, 0], [0, 0, 1.0, 4.0]]), 40.0, 40.0, 20.5, 12.5, 41, 25)
    out = []
    with Context(0) as ctx:
        ctx.load_hierarchy(asset)
        ctx.set_instances(inst)
        for mode in (0, 1):
            ctx.set_option(V3DG_OPT_BLEND_MODE, mode)
            ctx.select(cam, 0.0)
            rgb, T = ctx.render(want_T=True)
            out.append((rgb.cpu().numpy(), T.cpu().numpy()))
        assert ctx.frame_stats()["visible"] == n
    assert (out[0][0] == out[1][0]).all() and (out[0][1] == out[1][1]).all()
    # the centre pixel's alpha is the opacity (2^(log2 o), a few ulp); it stops before T < 1e-4
    want = (1.0 - float(o)) ** min(stack, int(np.log(1e-4) / np.log(1.0 - float(o))))
    assert abs(float(out[0][1][12, 20]) / want - 1.0) <= 1e-5 + 4 * n * 2.0 ** -24 * (1 + float(o) / (1 - float(o)))


def test_records_that_are_not_numbers_in_both_variants(small_asset):
    """A Gaussian whose covariance overflows (log alpha is not a number) adds nothing in either variant: the images are the
    same bit for bit, and not hidden behind it."""
    import dataclasses

    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    from paper_2505_06523_gb300._native import V3DG_OPT_BLEND_MODE
    ls = small_asset.log_scales.copy()
    ls[7] = 46.0
    huge = dataclasses.replace(small_asset, log_scales=ls)
    cam = scenes.look_at((0.0, -2.6, 0.4), (0.0, 0.0, 0.0), 40, 24, 60.0)
    imgs = []
    with Context(0) as ctx:
        ctx.load_hierarchy(huge)
        ctx.set_instances(scenes.single_instance())
        for mode in (0, 1):
            ctx.set_option(V3DG_OPT_BLEND_MODE, mode)
            ctx.select(cam, 0.25)
            imgs.append([x.cpu().numpy() for x in ctx.render(want_T=True)])
        proj = ctx.get_projected()
    assert not np.isfinite(proj["conic"][proj["local"] == 7]).any() and (proj["local"] == 7).sum() == 1
    assert (imgs[0][0] == imgs[1][0]).all() and (imgs[0][1] == imgs[1][1]).all()


def test_lists_on_both_sides_of_the_block_threshold(tiny_asset, small_asset):
    """A crowd with lists that a block blends together beside lists that single warps do, in many tiles: bit for bit the
    image of the block-per-tile variant."""
    import torch

    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    from paper_2505_06523_gb300._native import V3DG_OPT_BLEND_MODE
    inst = scenes.crowd_instances(200, n_assets=2, half_extent=70.0)
    cam = scenes.crowd_camera(40, 640, 360)
    out = []
    with Context(0) as ctx:
        for a in (tiny_asset, small_asset):
            ctx.load_hierarchy(a)
        ctx.set_instances(inst)
        for mode in (1, 0):
            ctx.set_option(V3DG_OPT_BLEND_MODE, mode)
            ctx.select(cam, 1.0)
            out.append([x.cpu().numpy() for x in ctx.render(want_T=True)])
        r = ctx.tile_ranges().astype(np.int64)
        pairs = ctx.frame_stats()["pairs"]
    # long: the octaves of at least a warp's share of the pairs, each key read by eight warps, and of at least 256 (five
    # blocks of four warps per SM)
    n, warps = r[:, 1] - r[:, 0], 4 * 5 * torch.cuda.get_device_properties(0).multi_processor_count
    octave = 1 << int(np.ceil(np.log2(max(pairs // (warps // 8), 256))))
    assert (n >= octave).sum() >= 8 and ((n > 0) & (n < octave)).sum() >= 8, (octave, np.sort(n)[-16:])
    assert float(np.abs(out[0][0]).sum()) > 0
    assert (out[0][0] == out[1][0]).all() and (out[0][1] == out[1][1]).all()
