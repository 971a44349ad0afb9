"""Capacity options given between a frame and its read-backs, and between a selection and its render."""
import numpy as np
import pytest

from synth import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,pairs", [(64, 4096), (1 << 17, 1 << 27)])
def test_capacities_of_the_next_frame(tiny_asset, nodes, pairs):
    """A capacity is that of the buffers, so an option changes it when a selection next sizes them: the lists of the
    last frame (one in depth slabs: they are made again) and a render of the present selection are not touched."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context
    from paper_2505_06523_gb300._native import V3DG_OPT_BLEND_MODE, V3DG_OPT_CAP_NODES, V3DG_OPT_CAP_PAIRS
    n, rng = 12, np.random.Generator(np.random.PCG64(12))
    inst = scenes.Instances(np.zeros(n, np.uint32), scenes.random_rotations(rng, n), rng.uniform(-0.5, 0.5, (n, 3)),
                            rng.uniform(0.7, 1.4, n))
    cam = scenes.look_at((0.0, -2.5, 0.5), (0.0, 0.0, 0.0), 1920, 1080, 70.0)
    lists = lambda ctx: {**{"proj_" + k: v for k, v in ctx.get_projected().items()}, "ranges": ctx.tile_ranges(),  # noqa: E731
                         **{"pair_" + k: v for k, v in ctx.get_pairs().items()}}
    with Context(0) as ctx:
        ctx.load_hierarchy(tiny_asset)
        ctx.set_instances(inst)
        ctx.set_option(V3DG_OPT_BLEND_MODE, 1)   # one slab: its lists are the frame's own
        ctx.select(cam, 0.25)
        want = ctx.render()[0].clone()
        want_lists = lists(ctx)
        stats = ctx.frame_stats()
        assert stats["pairs"] >= max(1 << 24, 16 * stats["visible"]) and stats["render_nodes"] > 64   # (slabs, and no fit)
        ctx.set_option(V3DG_OPT_BLEND_MODE, 0)
        for _ in range(2):
            ctx.select(cam, 0.25)
            ctx.render()
        ctx.set_option(V3DG_OPT_CAP_NODES, nodes)
        ctx.set_option(V3DG_OPT_CAP_PAIRS, pairs)
        got = lists(ctx)
        for k in want_lists:
            assert want_lists[k].shape == got[k].shape and (want_lists[k] == got[k]).all(), k
        for _ in range(2):   # the new capacities (grown again where they do not do)
            ctx.select(cam, 0.25)
            ctx.set_option(V3DG_OPT_CAP_NODES, nodes)
            ctx.set_option(V3DG_OPT_CAP_PAIRS, pairs)
            assert bool((ctx.render()[0] == want).all())
        got = lists(ctx)
        for k in want_lists:
            assert want_lists[k].shape == got[k].shape and (want_lists[k] == got[k]).all(), k
        assert ctx.frame_stats() == stats
