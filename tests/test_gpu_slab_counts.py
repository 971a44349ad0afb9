"""How many depth slabs a frame is taken in, seen by its launches."""
import numpy as np
import pytest

from synth import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2505_06523_gb300 import Context, _native
    return Context, _native


def _pile(n, spread):
    """n copies of asset 0, turned and scaled differently, around the origin."""
    rng = np.random.Generator(np.random.PCG64(n))
    return scenes.Instances(np.zeros(n, np.uint32), scenes.random_rotations(rng, n), rng.uniform(-spread, spread, (n, 3)),
                            rng.uniform(0.7, 1.4, n))


def _launches(ctx, frame):
    before = ctx.launches()
    frame()
    return ctx.launches() - before


NEAR = scenes.look_at((0.0, -2.5, 0.5), (0.0, 0.0, 0.0), 1920, 1080, 70.0)   # at the pile: large boxes, two slabs
SMALL = scenes.look_at((0.0, -3.0, 0.3), (0.0, 0.0, 0.0), 160, 96, 60.0)


def test_requests_of_different_sizes(api, tiny_asset):
    """A server slot that takes large and small requests in turn runs each as a context that only renders it does: the
    large one in slabs, the small one in one; with the same images."""
    Context, _ = api
    large, small = (_pile(12, 0.5), NEAR, 0.25), (scenes.single_instance(), SMALL, 1.0)
    alone, images, served = [], [], []
    for inst, cam, tau in (large, small):
        with Context(0) as ctx:
            ctx.load_hierarchy(tiny_asset)
            ctx.set_instances(inst)

            def frame():
                ctx.select(cam, tau)
                images.append(ctx.render_host()[0])
            alone.append([_launches(ctx, frame) for _ in range(3)])
    assert alone[0][1] == alone[0][2] > alone[1][2] == alone[1][1]
    with Context(0) as ctx:
        ctx.load_hierarchy(tiny_asset)
        ctx.server_start(1)

        def serve(inst, cam, tau):
            t, r = ctx.submit(inst, cam, tau), None
            while r is None:
                r = ctx.poll(t, 100_000)
            served.append(r[1])
        got = [(_launches(ctx, lambda: serve(*large)), _launches(ctx, lambda: serve(*small))) for _ in range(5)]
        ctx.server_stop()
    for k, img in enumerate(served):
        assert (img == images[3 * (k % 2)]).all()
    assert got[1:] == [(alone[0][2], alone[1][2])] * 4, (got, alone)   # (the slot's first large one grows its buffers)


def test_alternating_graph_frames(api, tiny_asset):
    """Captured frames of one size that alternate between two slab counts are captured once for each: after that a render
    call, which only replays, takes the host no more than four times as long as when the view stays (a capture of the frame's 40
    launches takes thirteen times as long).  Every image is the view's own."""
    import time

    import torch
    Context, N = api
    far = scenes.look_at((0.0, -60.0, 0.5), (0.0, 0.0, 0.0), 1920, 1080, 70.0)
    buf, flush = torch.empty((1080, 1920, 3), device="cuda"), torch.cuda.synchronize
    with Context(0) as ctx:
        ctx.set_option(N.V3DG_OPT_GRAPHS, 1)
        ctx.load_hierarchy(tiny_asset)
        ctx.set_instances(_pile(12, 0.5))

        def frame(cam):
            ctx.select(cam, 0.25)
            flush()
            t0 = time.perf_counter()
            ctx.render(buf)
            t = time.perf_counter() - t0
            flush()
            return t
        steady, images, launches = {}, {}, {}
        for cam in (NEAR, far, NEAR, far):
            for _ in range(4):
                frame(cam)
            launches[id(cam)] = _launches(ctx, lambda: frame(cam))
            images[id(cam)] = buf.clone()
        assert launches[id(NEAR)] > launches[id(far)]
        ctx.set_option(N.V3DG_OPT_SYNC_CHECK, 0)   # (a render call then only enqueues)
        for cam in (NEAR, far):
            steady[id(cam)] = np.median([frame(cam) for _ in range(20)][4:])
        alternating = {id(NEAR): [], id(far): []}
        for _ in range(20):
            for cam in (NEAR, far):
                alternating[id(cam)].append(frame(cam))
                assert bool((buf == images[id(cam)]).all())
    for k, t in alternating.items():
        assert np.median(t[4:]) <= 4.0 * max(steady.values()), (np.median(t[4:]), steady)


def _slabs(launches, launches_one, n_tiles):
    """Slabs of a frame from its launches and those of the same frame in one (blend variant 1).  A slab takes 14 launches and
    the passes of its tile sort: three that pick its Gaussians (none in one slab), the depth sort's count and four passes, two
    expansions, the tile sort's count, the ranges, and two of the blend; and what comes before the slabs is the same."""
    if launches == launches_one:
        return 1
    passes = -(-max(1, (n_tiles - 1).bit_length()) // 8)
    k, rest = divmod(launches - launches_one + 11 + passes, 14 + passes)
    assert rest == 0
    return k


@pytest.mark.parametrize("n,spread,width,height,fov,views,fp16,host,graphs,slabs", [
    (1, 0.0, 320, 180, 50.0, 1, [0], False, 0, 1),
    (12, 0.5, 1920, 1080, 70.0, 1, [1], True, 0, 2),       # large boxes, FP16 colour, a host image
    (40, 3.0, 1601, 901, 50.0, 3, [0], False, 0, 2),       # small ones
    (40, 3.0, 1601, 901, 50.0, 4, [0, 1], True, 0, 4),     # FP32 and FP16 colour in one frame
    (40, 3.0, 1601, 901, 50.0, 8, [1], False, 1, 4),
    (120, 3.0, 1601, 901, 50.0, 12, [0], False, 0, 6),
])
def test_frames_run_in_slabs(api, tiny_asset, n, spread, width, height, fov, views, fp16, host, graphs, slabs):
    """A frame that follows one like it runs in the slabs that its size asks for, with the image and transmittance that it
    has in one, bit for bit; so does a frame whose slabs overflow the pair capacity first."""
    Context, N = api
    inst = _pile(n, spread)
    inst.asset[:] = np.arange(n) % len(fp16)
    cams = [scenes.look_at((0.3 * v, -2.0 - spread, 0.5), (0.0, 0.0, 0.0), width, height, fov) for v in range(views)]
    out, launches = [], []
    with Context(0) as ctx:
        ctx.set_option(N.V3DG_OPT_GRAPHS, graphs)
        for half in fp16:
            ctx.set_option(N.V3DG_OPT_ATTR_FP16, half)
            ctx.load_hierarchy(tiny_asset)
        ctx.set_instances(inst)

        def frame():
            ctx.select_views(cams, 0.25)
            if host:
                out.append(ctx.render_host(want_T=True))
            else:
                out.append([x.cpu().numpy() for x in ctx.render(want_T=True)])
        for mode in (1, 0):
            ctx.set_option(N.V3DG_OPT_BLEND_MODE, mode)
            frame()
            launches.append(_launches(ctx, frame))
        assert _slabs(launches[1], launches[0], views * -(-width // 16) * -(-height // 16)) == slabs, ctx.frame_stats()["pairs"]
        ctx.set_option(N.V3DG_OPT_CAP_PAIRS, 4096)
        assert _launches(ctx, frame) > launches[1]   # (it overflows and runs again)
        assert _launches(ctx, frame) == launches[1]
    assert float(np.abs(out[0][0]).sum()) > 0
    for rgb, T in out[1:]:
        assert (rgb == out[0][0]).all() and (T == out[0][1]).all()


def test_stage_times_are_of_the_last_timed_frame(api, tiny_asset):
    """Frames rendered with stage timing off, whatever their slabs, leave the stage times of the last timed one."""
    Context, N = api
    with Context(0) as ctx:
        ctx.load_hierarchy(tiny_asset)
        ctx.set_instances(_pile(12, 0.5))

        def frame():
            ctx.select(NEAR, 0.25)
            ctx.render()
        ctx.set_option(N.V3DG_OPT_STAGE_TIMING, 1)
        ctx.set_option(N.V3DG_OPT_BLEND_MODE, 1)
        frame()   # (one slab)
        one = ctx.stage_times()[0]
        ctx.set_option(N.V3DG_OPT_STAGE_TIMING, 0)
        ctx.set_option(N.V3DG_OPT_BLEND_MODE, 0)
        assert _launches(ctx, frame) > 30   # (two slabs)
        ctx.set_option(N.V3DG_OPT_STAGE_TIMING, 1)
        assert ctx.stage_times()[0] == one and min(one) > 0
        frame()
        assert ctx.stage_times()[0] != one
