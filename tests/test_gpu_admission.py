"""What the server admits requests for, against the device memory that their frames take."""
import math

import pytest

from synth import scenes

pytestmark = pytest.mark.gpu


def test_admitted_for_their_buffers(tiny_asset):
    """Two requests whose frame buffers together pass the budget by a byte do not run beside each other: the estimate that
    a request is admitted for covers the buffers that are sized by it."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context, _native as N
    crowd = scenes.crowd_instances(400, n_assets=1, half_extent=70.0)
    cam = scenes.crowd_camera(40, 1920, 1080)
    requests = [(crowd, 0.25), (scenes.subset(crowd, list(range(60))), 0.25), (scenes.single_instance(), 1.0)]
    held = []
    for inst, tau in requests[:2]:
        nodes = int(1250 * inst.n * math.sqrt(1.0 / tau))   # the server's estimate at 1920x1080
        with Context(0) as ctx:
            ctx.load_hierarchy(tiny_asset)
            ctx.set_option(N.V3DG_OPT_CAP_NODES, nodes)
            ctx.set_option(N.V3DG_OPT_CAP_PAIRS, int(nodes * 64 * 2.25))
            ctx.set_instances(inst)
            ctx.select(cam, tau)
            ctx.render_host()
            stats = ctx.frame_stats()
            assert stats["render_nodes"] <= nodes and stats["pairs"] <= nodes * 64 * 2.25   # (nothing has grown)
            held.append(ctx.release_buffers())
    with Context(0) as ctx:
        ctx.load_hierarchy(tiny_asset)
        ctx.server_start(2, sum(held) - 1)
        for _ in range(2):   # (the first time warms the pinned images and the pool up)
            tickets = [ctx.submit(inst, cam, tau) for inst, tau in requests]
            done = {}
            while len(done) < 3:
                for t in tickets:
                    r = ctx.poll(t, 1000) if t not in done else None
                    if r is not None:
                        done[t] = r[0]
            del r
        ctx.server_stop()
    first, second = done[tickets[0]], done[tickets[1]]
    assert second["start_ms"] >= first["done_ms"], (first, second)
