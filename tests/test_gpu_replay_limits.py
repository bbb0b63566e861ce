"""Replay mode (every path traced once, replayed by each render) at the edges of what it takes."""
import numpy as np
import pytest

import workloads
from test_gpu_replay import _bind, _box_light_wall, _gi, _light, _t, _two_lights, _walls

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    from paper_2211_17263_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def _grad(ctx, wl, step=3, **kw):
    scene = ctx.upload_scene(wl.scene, wl.bindings)
    target = _t(np.random.default_rng(1).uniform(size=(wl.height, wl.width, 4)))
    g, L = scene.smoothed_grad(_t(wl.theta0), _t(wl.sigma), target, scene.grad_opts(wl, step=step, **kw))
    torch.cuda.synchronize()
    return g.cpu().numpy(), L.cpu().numpy()


def _count(ctx, wl, **kw):
    ctx.counters_enable(True)
    _grad(ctx, wl, **kw)
    n = np.array(ctx.counters_read())
    ctx.counters_enable(False)
    return n


@pytest.mark.parametrize("pairs", [3, 5, 6, 9, 12])
def test_shadow_rays_are_counted_once_per_render(ctx, pairs):
    """The renders of a job, and the same renders one pair at a time, trace the same shadow rays
    (6, 10, 12, 18 and 24 renders leave lanes of a warp without a render)."""
    wl = _light(width=19, height=11, spp=5, pairs=pairs)
    whole = _count(ctx, wl)
    one = [_count(ctx, workloads.scaled(wl, pairs=1), pair_begin=p) for p in range(pairs)]
    assert whole[5] == sum(n[5] for n in one) > 0


def _closed_walls(**kw):
    """The box with its camera inside and a front wall: no path leaves it."""
    wl = _walls(**kw)
    sc = wl.scene
    lo, hi = sc.prim_geom[:5, :3].min(0), sc.prim_geom[:5, :3].max(0)
    side = int(np.argmax(np.abs(sc.camera[3:6] - sc.camera[:3])))  # the open side faces the camera
    outside = sc.camera[side] < (lo[side] + hi[side]) / 2
    front = (lo + hi) / 2
    front[side] = lo[side] - 0.5 if outside else hi[side] + 0.5
    u, v = 20 * np.eye(3)[(side + 1) % 3], 20 * np.eye(3)[(side + 2) % 3]
    geom = np.concatenate([sc.prim_geom, [np.concatenate([front, u, v])]]).astype(np.float32)
    camera = sc.camera.copy()
    camera[side] = front[side] + (0.3 if outside else -0.3)
    wl.scene = workloads.Scene(np.append(sc.prim_type, 1).astype(np.int32), np.append(sc.prim_mat, 0).astype(np.int32),
                               geom, sc.mat_type, sc.mat_param, camera, sc.background)
    return wl


def test_work_is_counted_once_where_the_pool_runs_out(ctx):
    """Paths that did not fit their batch's pool are traced again in the next one; their rays and
    vertices count once. Without roulette every render's paths are the shared ones."""
    wl = _closed_walls(width=16, height=12, spp=32, pairs=4, depth=64, rr_start=-1)
    shared, alone = _count(ctx, wl, block_pixels=8), _count(ctx, wl, block_pixels=8, no_path_sharing=1, render_groups=-1)
    for k in (3, 4, 5, 6):
        assert shared[k] * 8 == alone[k] > 0, k
    assert shared[6] > 16 * 12 * 32 * 20  # long paths: 32 of them exceed the pool's 512 granules


def _eq9(**kw):
    return workloads.scaled(workloads.config_gi_albedo(), **kw)


@pytest.mark.parametrize("block_pixels", [0, 32])
@pytest.mark.parametrize("room", ["whole blocks", "small blocks' losses", "parts' sums"])
def test_pathwise_gradient_within_the_budget_of_whole_blocks(gpu_lib, block_pixels, room):
    """Eq. 9 under memory budgets that hold the partials of whole blocks, but not those of smaller
    blocks or the sums of blocks in parts beside them: neither may take the gradient partials' room."""
    from paper_2211_17263_gb300 import api
    wl = _eq9(width=120, height=100, spp=64, pairs=32)
    R, D, tiles, pixels = 64, 6, 15 * 25, 120 * 100  # blocks of 32 pixels, at most one part a pixel
    losses, grads, sums = 8 * R * tiles, 8 * R * tiles * D, 8 * R * tiles * 32 * (1 + D)
    extra = {"whole blocks": losses + grads, "small blocks' losses": 8 * R * pixels + grads // 2,
             "parts' sums": losses + sums + grads // 2}[room]
    ctx = api.Context(0)
    try:
        want, _ = _grad(ctx, wl, block_pixels=32)
    finally:
        ctx.close()
    # everything else a call allocates: control words, scene, instances, weights, losses, gradients
    ctx = api.Context(0, hbm_budget_bytes=1 << 30)
    try:
        _grad(ctx, _eq9(width=8, height=4, spp=1, pairs=32), block_pixels=32)
        budget = ctx.memory_used() + extra + 4096
    finally:
        ctx.close()
    ctx = api.Context(0, hbm_budget_bytes=budget)
    try:
        for _ in range(2):
            got, _ = _grad(ctx, wl, block_pixels=block_pixels)
            assert ctx.memory_used() <= budget
            # blocks of another size group the FP64 partial sums differently
            assert np.allclose(got, want, rtol=1e-6, atol=1e-6 * np.abs(want).max())
    finally:
        ctx.close()


def test_optional_sums_make_room(gpu_lib):
    """The part sums of one call do not keep a later call, job or render from the budget."""
    from paper_2211_17263_gb300 import api
    wl = _gi(width=120, height=100, spp=64, pairs=32)
    ctx = api.Context(0, hbm_budget_bytes=64 << 20)
    try:
        want, _ = _grad(ctx, wl, block_pixels=32)
        used = ctx.memory_used()
    finally:
        ctx.close()
    big = _light(width=512, height=512, spp=1, pairs=2)
    sums = 8 * 64 * (1 << 13)  # at least 8192 parts of 64 renders
    ctx = api.Context(0, hbm_budget_bytes=used + 16 * 512 * 512 - sums)
    try:
        assert np.array_equal(_grad(ctx, wl, block_pixels=32)[0], want)
        job = api.Job(ctx.upload_scene(big.scene, big.bindings), big, None, use_tuned=False)
        job.step()
        job.read()
        job.release()
        assert np.array_equal(_grad(ctx, wl, block_pixels=32)[0], want)
    finally:
        ctx.close()


def test_parts_on_a_side_stream(gpu_lib):
    """The first call of a context on a stream that does not wait for the legacy default stream:
    the counters of finished parts are zero before it."""
    from paper_2211_17263_gb300 import api
    wl = _walls(width=64, height=48, spp=16, pairs=4)
    want = None
    for _ in range(6):
        ctx = api.Context(0)
        try:
            side = torch.cuda.Stream()
            with torch.cuda.stream(side):
                got = [_grad(ctx, wl, block_pixels=32) for _ in range(2)]
        finally:
            ctx.close()
        want = want or got[0]
        for g, L in got:
            assert np.array_equal(g, want[0]) and np.array_equal(L, want[1])


def test_more_work_items_than_numbers_stay_refused(ctx):
    """512 renders of 8192^2 pixels in 8-pixel blocks: (render, block) pairs beyond 32-bit numbers,
    refused as a job and as a gradient, with or without sharing, before anything is allocated."""
    from paper_2211_17263_gb300 import capi
    wl = _walls()  # two bound materials: 512 renders' rows fit
    scene = ctx.upload_scene(wl.scene, wl.bindings)
    small, dev = np.zeros(16, np.float32), _t(np.zeros(16))
    for kw in ({}, dict(no_path_sharing=1)):
        opts = scene.grad_opts(wl, pairs=256, block_pixels=8, **kw)
        opts.width = opts.height = 8192
        desc = capi.prdpt_job_desc(grad=opts, theta0_host=small.ctypes.data, sigma0_host=small.ctypes.data,
                                   target_host=small.ctypes.data, lr=0.01, beta1=0.9, beta2=0.999, eps=1e-8,
                                   sigma_min=0.01, anneal=0, total_steps=1)
        before = ctx.memory_used()
        with pytest.raises(capi.PrdptError, match="work items"):
            capi.prdpt_job_create(ctx.handle, scene.id, desc)
        with pytest.raises(capi.PrdptError, match="work items"):
            scene.smoothed_grad(dev[:6], dev[:6], dev, opts)
        assert ctx.memory_used() == before


def _moving_and_fixed_light(**kw):  # one emitter moves, the other is fixed: no render parts from a path
    wl = _two_lights(**kw)
    return _bind(wl, wl.bindings[:3], wl.theta0[:3], wl.sigma[:3])


def _box_moves(**kw):  # the occlusion task: a box moves under a fixed light
    return workloads.scaled(workloads.config_occlusion(), **kw)


def _box_and_walls(**kw):  # a grey box and two walls' albedos under a fixed light
    wl = _box_light_wall(**kw)
    keep = [0, 1, 2, 6, 7]
    return _bind(wl, wl.bindings[keep], wl.theta0[keep], wl.sigma[keep])


@pytest.mark.parametrize("make,pairs,spp,grouped", [
    (_box_light_wall, 1, 40, True), (_box_light_wall, 1, 2, True), (_box_light_wall, 3, 16, True), (_box_light_wall, 13, 16, True),
    (_box_light_wall, 3, 2, False), (_box_light_wall, 13, 2, False), (_two_lights, 5, 16, True),
    (_moving_and_fixed_light, 1, 8, True), (_moving_and_fixed_light, 2, 8, True), (_moving_and_fixed_light, 3, 8, False),
    (_gi, 1, 16, True), (_gi, 1, 8, False), (_light, 1, 32, False), (_box_moves, 1, 65, False), (_box_moves, 8, 65, False),
    (_box_and_walls, 3, 65, True), (_box_and_walls, 4, 65, False), (_box_and_walls, 10, 65, False)])
def test_routes_where_replay_is_slower(ctx, make, pairs, spp, grouped):
    """Jobs whose renders part from the paths, and few renders beside fixed emitters, run in groups,
    which count every render's paths; where replay pays it counts each path once (beyond 64 samples
    also where path sharing would). Same results."""
    wl = make(width=96, height=60, spp=spp, pairs=pairs)
    paths = wl.width * wl.height * wl.spp * (2 * pairs if grouped else 1)
    assert _count(ctx, wl, block_pixels=8)[3] == paths
    (g, L), (g0, L0) = (_grad(ctx, wl, block_pixels=8, **kw) for kw in ({}, dict(no_path_sharing=1, render_groups=-1)))
    assert np.array_equal(L, L0) and np.array_equal(g, g0)


@pytest.mark.parametrize("make", [_gi, _walls, _light, _eq9])
@pytest.mark.parametrize("width,height,spp,pairs", [(1, 1, 1, 1), (24, 24, 1, 1), (5, 3, 3, 24), (40, 33, 3, 5),
                                                    (64, 47, 1, 16), (96, 60, 32, 1), (76, 41, 32, 3)])
def test_items_down_to_one_pixel(ctx, make, width, height, spp, pairs):
    """Small images in items of one pixel, and items of one full batch each. In parts of 8-pixel
    blocks the losses are the per-render kernel's bit for bit (Eq. 9's too); with automatic blocks its
    FP64 partial sums are grouped differently, and an FP32 loss may differ in its last bit."""
    wl = make(width=width, height=height, spp=spp, pairs=pairs)
    want = _grad(ctx, wl, block_pixels=8, no_path_sharing=1, render_groups=-1)[1]
    assert np.array_equal(_grad(ctx, wl, block_pixels=8)[1], want)
    assert np.allclose(_grad(ctx, wl)[1], want, rtol=2.0**-22, atol=0.0)


@pytest.mark.parametrize("pairs", [1, 2, 3, 5, 6, 15, 16, 17])
def test_sample_groups_side_by_side(ctx, pairs):
    """1 to 16 sample groups in a warp, powers of two and others, summed by halves."""
    wl = _light(width=45, height=23, spp=37, pairs=pairs)
    (g, L), (g0, L0) = (_grad(ctx, wl, block_pixels=16, **kw) for kw in ({}, dict(no_path_sharing=1, render_groups=-1)))
    assert np.array_equal(L, L0) and np.array_equal(g, g0)
