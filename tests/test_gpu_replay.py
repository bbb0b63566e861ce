"""Replay mode (every path traced once, replayed by each render) against tracing every render's
paths on their own: losses and the Eq. 10 gradient must be equal bit for bit at the sizes where the
kernel can go wrong -- render counts around the lane groups and halves, samples around a batch of
32, block sizes from 8 to 32 (split into parts on small images), ragged images, paths longer than
the pool holds for a whole batch, albedos that clamp to 0 and 1, emitters and objects that move
(black ones end a render's path, others part it), and fixed emitters beside moving ones."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    from paper_2211_17263_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a, np.float32), device="cuda")


def _bind(wl, rows, theta, sigma):
    wl.bindings = np.array(rows, np.int32)
    wl.theta0 = np.asarray(theta, np.float32)
    wl.sigma = np.asarray(sigma, np.float32)
    return wl


def _gi(**kw):  # light position and two walls' albedos
    return workloads.scaled(workloads.config_gi_box(), **kw)


def _walls(**kw):  # albedos only: a fixed emitter, the same visibility in every render
    return workloads.scaled(workloads.config_gi_albedo(), estimator=0, sampler=0, **kw)


def _light(**kw):  # the light only, and no Russian roulette
    wl = _gi(**kw)
    return _bind(wl, wl.bindings[:3], wl.theta0[:3], wl.sigma[:3])


def _box_light_wall(**kw):  # a grey box moves beside the light: its renders part from the path
    wl = _gi(**kw)
    box = wl.scene.prim_geom[5, :3]
    rows = [[workloads.BIND_PRIM_POS, 5, k] for k in range(3)] + wl.bindings[:3].tolist() + wl.bindings[3:5].tolist()
    wl.parting = True
    return _bind(wl, rows, np.concatenate([box + 0.02, wl.theta0[:5]]), np.full(8, 0.08))


def _two_lights(**kw):  # one emitter moves, the other is fixed and can be hidden by a moving ball
    wl = workloads.scaled(workloads.config_caustic(), **kw)
    b = workloads.SceneBuilder()
    floor = b.material(workloads.MAT_DIFFUSE, (0.8, 0.7, 0.6))
    ball = b.material(workloads.MAT_DIFFUSE, (0.3, 0.8, 0.4))
    lamp = b.material(workloads.MAT_DIFFUSE, (0.0, 0.0, 0.0), emission=(40.0, 40.0, 40.0))
    b.quad((0, 0, 0), (10, 0, 0), (0, 10, 0), floor)
    s = b.sphere((0.1, 0.2, 0.9), 0.4, ball)
    b.quad((0.6, 0.4, 2.6), (0.5, 0, 0), (0, -0.5, 0), lamp)
    moving = b.quad((-0.7, 0.1, 2.4), (0.4, 0, 0), (0, -0.4, 0), lamp)
    b.background = np.array([0.05, 0.06, 0.07], np.float32)
    b.look_at((0, -4.0, 1.6), (0, 0, 0.5), (0, 0, 1), 40.0)
    wl.scene = b.build()
    rows = [[workloads.BIND_PRIM_POS, moving, k] for k in range(3)] + [[workloads.BIND_PRIM_POS, s, 0]]
    rows += [[workloads.BIND_SPHERE_RADIUS, s, 0]]
    wl.parting = True
    return _bind(wl, rows, [-0.7, 0.1, 2.4, 0.1, 0.4], [0.1, 0.1, 0.1, 0.1, 0.05])


def _clamped(**kw):  # albedos around 0 and 1: renders whose throughput ends, black bound materials
    wl = _walls(**kw)
    return _bind(wl, wl.bindings, [0.02, 0.0, 0.98, -0.05, -0.1, -0.08], np.full(6, 0.05))


def _compare(ctx, wl, block_pixels, step=3):
    scene = ctx.upload_scene(wl.scene, wl.bindings)
    target = _t(np.random.default_rng(1).uniform(size=(wl.height, wl.width, 4)))
    out = []
    for kw in ({}, dict(no_path_sharing=1, render_groups=-1)):
        g, L = scene.smoothed_grad(_t(wl.theta0), _t(wl.sigma), target,
                                   scene.grad_opts(wl, step=step, block_pixels=block_pixels, **kw))
        torch.cuda.synchronize()
        out.append((g.cpu().numpy(), L.cpu().numpy()))
    ctx.counters_enable(True)
    scene.smoothed_grad(_t(wl.theta0), _t(wl.sigma), target, scene.grad_opts(wl, step=step, block_pixels=block_pixels))
    torch.cuda.synchronize()
    paths = ctx.counters_read()[3]
    ctx.counters_enable(False)
    # each path traced once; where renders part from the path, groups of 4 or more trace it per render
    per_path = 2 * wl.pairs if getattr(wl, "parting", False) and wl.pairs % 2 == 0 else 1
    assert paths == wl.width * wl.height * wl.spp * per_path
    return out


@pytest.mark.parametrize("make", [_gi, _walls, _light, _box_light_wall, _two_lights, _clamped])
@pytest.mark.parametrize("pairs,spp,block_pixels", [(1, 1, 8), (5, 13, 16), (8, 33, 8), (12, 20, 32), (16, 4, 32),
                                                    (17, 5, 8), (32, 3, 16)])
def test_replay_is_bit_identical(ctx, make, pairs, spp, block_pixels):
    wl = make(width=37, height=21, spp=spp, pairs=pairs)
    (g, L), (g0, L0) = _compare(ctx, wl, block_pixels)
    assert np.array_equal(L, L0) and np.array_equal(g, g0)


@pytest.mark.parametrize("make", [_gi, _walls, _box_light_wall])
@pytest.mark.parametrize("pairs,block_pixels", [(33, 8), (40, 32), (70, 0)])
def test_more_than_64_renders_in_chunks(ctx, make, pairs, block_pixels):
    """Jobs with bound materials replay 64 renders at a time (chunks of 64 and the rest)."""
    wl = make(width=29, height=13, spp=5, pairs=pairs)
    scene = ctx.upload_scene(wl.scene, wl.bindings)
    target = _t(np.random.default_rng(1).uniform(size=(wl.height, wl.width, 4)))
    out = []
    for kw in ({}, dict(no_path_sharing=1, render_groups=-1)):
        g, L = scene.smoothed_grad(_t(wl.theta0), _t(wl.sigma), target,
                                   scene.grad_opts(wl, step=3, block_pixels=block_pixels or 8, **kw))
        torch.cuda.synchronize()
        out.append((g.cpu().numpy(), L.cpu().numpy()))
    assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][0], out[1][0])
    # packed with a job of few renders: each as alone
    from paper_2211_17263_gb300 import api
    small = make(width=29, height=13, spp=5, pairs=3)
    state = []
    for packed in (False, True):
        jobs = [api.Job(ctx.upload_scene(w.scene, w.bindings), w, target.cpu().numpy()) for w in (wl, small)]
        if packed:
            api.step_batch(ctx, jobs)
        else:
            for j in jobs:
                j.step()
        state.append([j.read() for j in jobs])
        for j in jobs:
            j.release()
    for a, b in zip(*state):
        assert all(np.array_equal(a[k], b[k]) for k in ("theta", "grad", "losses"))


@pytest.mark.parametrize("make", [_gi, _walls, _light, _two_lights])
@pytest.mark.parametrize("spp,block_pixels", [(64, 0), (65, 8), (32, 0), (16, 16)])
def test_items_of_one_two_and_four_pixels(ctx, make, spp, block_pixels):
    """Small images with many samples: blocks, or parts of blocks, of 1, 2 and 4 pixels. With
    block_pixels = 0 the blocks differ from the per-render kernel's, so its FP64 partial sums are
    grouped differently: the FP32 losses may then differ in their last bit."""
    wl = make(width=23, height=9, spp=spp, pairs=3)
    (g, L), (g0, L0) = _compare(ctx, wl, block_pixels)
    if block_pixels:
        assert np.array_equal(L, L0) and np.array_equal(g, g0)
    else:
        assert np.allclose(L, L0, rtol=2.0**-22, atol=0.0)


@pytest.mark.parametrize("make", [_gi, _walls, _box_light_wall])
def test_long_paths_fill_the_pool(ctx, make):
    """Depth 64 without roulette: a batch's paths do not fit the pool and are taken in smaller batches."""
    wl = make(width=16, height=12, spp=32, pairs=4, depth=64, rr_start=-1)
    (g, L), (g0, L0) = _compare(ctx, wl, 8)
    assert np.array_equal(L, L0) and np.array_equal(g, g0)


@pytest.mark.parametrize("slots,pairs,spp", [(2, 4, 5), (3, 16, 33), (6, 17, 4), (8, 5, 7)])
def test_pathwise_replay(ctx, slots, pairs, spp):
    """Eq. 9 with 2 to 8 albedo parameters (3, 6 and 12 tangent slots): the losses are the per-render
    kernel's bit for bit; the tangents are the same products rounded in another order, at most three
    roundings (2^-24) a vertex over 8 vertices, with a factor of 8 for cancellation in the sum."""
    wl = workloads.scaled(workloads.config_gi_albedo(), width=33, height=18, spp=spp, pairs=pairs)
    rows = (wl.bindings.tolist() + [[workloads.BIND_MAT_ALBEDO, 0, 1], [workloads.BIND_MAT_ALBEDO, 5, 1]])[:slots]
    _bind(wl, rows, (wl.theta0.tolist() + [0.5, 0.7])[:slots], np.full(slots, 0.1))
    (g, L), (g0, L0) = _compare(ctx, wl, 8)
    assert np.array_equal(L, L0)
    assert np.linalg.norm(g - g0) <= 3 * 8 * 2.0**-24 * 8 * np.linalg.norm(g0)


def test_whole_blocks_where_the_budget_refuses_small_ones(gpu_lib):
    """A small image's one-pixel blocks have up to 32 times the partials; a call that the memory
    budget would then refuse takes the per-render kernel's blocks instead, as a job and as a gradient."""
    from paper_2211_17263_gb300 import api
    wl = _gi(width=120, height=100, spp=64, pairs=32)
    target = _t(np.random.default_rng(1).uniform(size=(wl.height, wl.width, 4)))

    def run(ctx, job):
        scene = ctx.upload_scene(wl.scene, wl.bindings)
        if job:
            j = api.Job(scene, wl, target.cpu().numpy(), use_tuned=False)
            j.step()
            return j.read()["grad"]
        g, _ = scene.smoothed_grad(_t(wl.theta0), _t(wl.sigma), target, scene.grad_opts(wl))
        torch.cuda.synchronize()
        return g.cpu().numpy()

    for job in (True, False):
        ctx = api.Context(0, hbm_budget_bytes=200 << 20)
        try:
            grad = run(ctx, job)
            used = ctx.memory_used()
        finally:
            ctx.close()
        # one-pixel blocks: 12000 x 64 FP64 partials, 6.1 MB; the per-render kernel's hold 8 to 32 pixels
        ctx = api.Context(0, hbm_budget_bytes=used - (3 << 20))
        try:
            small = run(ctx, job)
            assert ctx.memory_used() <= used - (3 << 20)
        finally:
            ctx.close()
        # differences of losses that are rounded to FP64 sums in another order
        assert np.allclose(small, grad, rtol=1e-6, atol=1e-6 * np.abs(grad).max())


def test_packed_step_of_every_class(ctx):
    """Replay jobs of all variants (renders per lane, chunks, bound albedos, moving emitters, parting
    renders), in mixed order, in one packed step: each equals the job stepped alone, bit for bit."""
    from paper_2211_17263_gb300 import api
    shapes = [(_gi, 3, 33, 18), (_walls, 20, 24, 11), (_light, 24, 16, 9), (_gi, 40, 13, 8), (_box_light_wall, 5, 21, 10),
              (_gi, 2, 40, 6), (_two_lights, 17, 12, 12), (_walls, 4, 9, 9), (_light, 8, 31, 7)]
    wls = [make(width=w, height=h, spp=6, pairs=p) for make, p, w, h in shapes]
    scenes = [ctx.upload_scene(wl.scene, wl.bindings) for wl in wls]
    rng = np.random.default_rng(5)
    targets = [rng.uniform(size=(wl.height, wl.width, 4)).astype(np.float32) for wl in wls]
    make = lambda: [api.Job(s, wl, t, use_tuned=False, block_pixels=8) for s, wl, t in zip(scenes, wls, targets)]
    alone, packed = make(), make()
    for _ in range(2):
        for j in alone:
            j.step()
        api.step_batch(ctx, packed)
    for a, b in zip(alone, packed):
        x, y = a.read(), b.read()
        assert x["steps"] == y["steps"] == 2
        for k in ("theta", "grad", "losses"):
            assert np.array_equal(x[k], y[k])
        a.release()
        b.release()


@pytest.mark.parametrize("make", [_gi, _walls, _two_lights])
@pytest.mark.parametrize("pairs,spp,width,height", [(39, 3, 86, 86), (20, 1, 33, 7), (3, 8, 29, 31), (35, 2, 5, 3)])
def test_few_samples_on_small_images(ctx, make, pairs, spp, width, height):
    """Fewer work items than warps: blocks go down to 8 paths, less than a batch. The per-render
    kernel's blocks are larger, so FP64 partial sums are grouped differently: an FP32 loss may differ
    in its last bit."""
    wl = make(width=width, height=height, spp=spp, pairs=pairs)
    scene = ctx.upload_scene(wl.scene, wl.bindings)
    target = _t(np.random.default_rng(2).uniform(size=(height, width, 4)))
    L = []
    for kw in ({}, dict(no_path_sharing=1, render_groups=-1)):
        L.append(scene.smoothed_grad(_t(wl.theta0), _t(wl.sigma), target, scene.grad_opts(wl, step=1, **kw))[1].cpu().numpy())
    assert np.allclose(L[0], L[1], rtol=2.0**-22, atol=0.0)
