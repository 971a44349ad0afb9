"""The blend autotuner's times against those of the frame's own blend."""
import numpy as np
import pytest

from synth import scenes
from synth.assets import Asset

pytestmark = pytest.mark.gpu


def _stacks(n):
    """n faint Gaussians on top of each other in the middle of each tile of a 64x64 image: 16 lists, each blended by blocks."""
    px = np.arange(8, 64, 16, np.float32)
    x, y = (np.repeat(a.ravel(), n) for a in np.meshgrid(px, px))
    means = np.stack([(x - 31.5) / 16, (y - 31.5) / 16, np.zeros_like(x)], 1).astype(np.float32)
    means = np.concatenate([means, means[:1]])   # the last one: a root above the leaves, never selected
    m = len(means)
    nodes = (m - 1 + 63) // 64
    count = np.append(np.minimum(64, m - 1 - 64 * np.arange(nodes)), 1).astype(np.uint32)
    asset = Asset(means=means, log_scales=np.full((m, 3), -2.0, np.float32), quats=np.tile(np.float32([1, 0, 0, 0]), (m, 1)),
                  opacity=np.full(m, 0.0045, np.float32), sh=np.zeros((m, 16, 3), np.float32),
                  node_first=np.append(64 * np.arange(nodes), m - 1).astype(np.uint32), node_count=count,
                  node_level=np.append(np.zeros(nodes), 1).astype(np.uint8),
                  node_parent=np.append(np.full(nodes, nodes), -1).astype(np.int32),
                  own_sphere=np.tile(np.float32([0, 0, 0, 4]), (nodes + 1, 1)))
    cam = scenes.Camera(np.array([[1.0, 0, 0, 0], [0, 1.0, 0, 0], [0, 0, 1.0, 4.0]]), 64.0, 64.0, 32.0, 32.0, 64, 64)
    return asset, cam


def test_times_the_whole_blend():
    """The best time is that of a blend that does all of the frame's work, lists that blocks blend together among it: on a
    frame of nothing but such lists, within a factor of two of the frame's own blend (the same two launches; a blend
    without them is one of empty tiles, a tenth and less of the time)."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    from paper_2505_06523_gb300._native import V3DG_OPT_BLEND_MODE, V3DG_OPT_STAGE_TIMING
    asset, cam = _stacks(2500)
    with Context(0) as ctx:
        ctx.load_hierarchy(asset)
        ctx.set_instances(scenes.single_instance())
        ctx.set_option(V3DG_OPT_STAGE_TIMING, 1)
        frame = {}
        for mode in (1, 0):
            ctx.set_option(V3DG_OPT_BLEND_MODE, mode)
            t = []
            for _ in range(6):
                ctx.select(cam, 0.0)
                ctx.render()
                t.append(ctx.stage_times()[0][6])
            frame[mode] = min(t[1:])
        best = ctx.autotune_blend()
    assert best["split_pairs"] == 0xFFFFFFFF
    assert 0.5 * frame[best["mode"]] <= best["ms"] <= 2.0 * frame[best["mode"]], (best, frame)


def test_candidates_are_whole_frames(tiny_asset):
    """A candidate is timed as the frame that its choice would bring, with or without depth slabs: four runs (one warms up)
    of the frame's launches for variant 0, here in two slabs, and four for each batch size of variant 1, in one.  The
    frame's stage times, image and lists stay."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    from paper_2505_06523_gb300._native import V3DG_OPT_BLEND_MODE, V3DG_OPT_STAGE_TIMING
    n, rng = 12, np.random.Generator(np.random.PCG64(12))
    inst = scenes.Instances(np.zeros(n, np.uint32), scenes.random_rotations(rng, n), rng.uniform(-0.5, 0.5, (n, 3)),
                            rng.uniform(0.7, 1.4, n))
    cam = scenes.look_at((0.0, -2.5, 0.5), (0.0, 0.0, 0.0), 1920, 1080, 70.0)
    with Context(0) as ctx:
        ctx.load_hierarchy(tiny_asset)
        ctx.set_instances(inst)
        ctx.set_option(V3DG_OPT_STAGE_TIMING, 1)
        launches = {}
        for mode in (1, 0):
            ctx.set_option(V3DG_OPT_BLEND_MODE, mode)
            for _ in range(2):
                ctx.select(cam, 0.25)
                before = ctx.launches()
                img = ctx.render()[0]
            launches[mode] = ctx.launches() - before
        assert launches[0] > launches[1]   # (slabs)
        times, ranges, proj, kept = ctx.stage_times()[0], ctx.tile_ranges(), ctx.get_projected(), img.clone()
        before = ctx.launches()
        best = ctx.autotune_blend()
        assert ctx.launches() - before == 4 * launches[0] + 12 * launches[1]
        assert ctx.stage_times()[0] == times and bool((img == kept).all())
        assert (ctx.tile_ranges() == ranges).all() and all(np.array_equal(v, proj[k]) for k, v in ctx.get_projected().items())
        ctx.select(cam, 0.25)
        assert bool((ctx.render()[0] == kept).all()) and best["ms"] > 0
