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
