"""Prefix sharing (each path traced once up to the first ray that could meet a moving object that is
not black, then by every render) against tracing every render's paths on their own: losses and
gradient equal bit for bit, for render counts around the lane groups and halves, samples around a
batch of 32, every block size, ragged images and a radius that changes an emitter's area."""
import numpy as np
import pytest

import workloads
from test_gpu_replay import _bind, _light, _t

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    from paper_2211_17263_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def _box_and_light(**kw):  # a grey box moves beside the only light: diffuse walls, roulette
    wl = _light(**kw)
    box = wl.scene.prim_geom[5, :3]
    rows = [[workloads.BIND_PRIM_POS, 5, k] for k in range(3)] + wl.bindings.tolist()
    return _bind(wl, rows, np.concatenate([box + 0.02, wl.theta0]), np.full(6, 0.08))


def _glass_and_light(**kw):  # a glass ball moves beside the light: specular chains, long prefixes
    wl = workloads.scaled(workloads.config_caustic(), **kw)
    s = int(np.nonzero(wl.scene.prim_type == workloads.PRIM_SPHERE)[0][0])
    rows = [[workloads.BIND_PRIM_POS, s, 0], [workloads.BIND_SPHERE_RADIUS, s, 0]] + wl.bindings.tolist()
    theta = np.concatenate([[wl.scene.prim_geom[s, 0], wl.scene.prim_geom[s, 3]], wl.theta0])
    return _bind(wl, rows, theta, np.full(5, 0.05))


def _lamp_and_mirror(**kw):  # a sphere lamp's radius and a mirror ball move under a background
    wl = workloads.scaled(workloads.config_caustic(), **kw)
    b = workloads.SceneBuilder()
    floor = b.material(workloads.MAT_DIFFUSE, (0.8, 0.7, 0.6))
    mirror = b.material(workloads.MAT_MIRROR, (0.9, 0.9, 0.9))
    lamp = b.material(workloads.MAT_DIFFUSE, (0.0, 0.0, 0.0), emission=(9.0, 8.0, 7.0))
    b.quad((0, 0, 0), (10, 0, 0), (0, 10, 0), floor)
    s = b.sphere((0.1, 0.2, 0.7), 0.4, mirror)
    p = b.sphere((-0.6, 0.1, 2.2), 0.2, lamp)
    b.background = np.array([0.05, 0.06, 0.07], np.float32)
    b.look_at((0, -4.0, 1.6), (0, 0, 0.5), (0, 0, 1), 40.0)
    wl.scene = b.build()
    rows = [[workloads.BIND_PRIM_POS, s, 0], [workloads.BIND_SPHERE_RADIUS, p, 0]]
    return _bind(wl, rows, [0.1, 0.2], [0.1, 0.05])


def _grad(ctx, wl, block_pixels, **kw):
    scene = ctx.upload_scene(wl.scene, wl.bindings)
    target = _t(np.random.default_rng(1).uniform(size=(wl.height, wl.width, 4)))
    g, L = scene.smoothed_grad(_t(wl.theta0), _t(wl.sigma), target,
                               scene.grad_opts(wl, step=3, block_pixels=block_pixels, **kw))
    torch.cuda.synchronize()
    return g.cpu().numpy(), L.cpu().numpy()


@pytest.mark.parametrize("make", [_box_and_light, _glass_and_light, _lamp_and_mirror])
@pytest.mark.parametrize("pairs,spp,block_pixels", [(1, 1, 8), (5, 13, 16), (8, 33, 8), (12, 20, 32), (16, 4, 32),
                                                    (17, 5, 8), (32, 3, 16)])
def test_prefix_sharing_is_bit_identical(ctx, make, pairs, spp, block_pixels):
    wl = make(width=37, height=21, spp=spp, pairs=pairs)
    (g, L), (g0, L0) = (_grad(ctx, wl, block_pixels, **kw) for kw in ({}, dict(no_path_sharing=1, render_groups=-1)))
    assert np.array_equal(L, L0) and np.array_equal(g, g0)


def test_packed_with_other_kinds(ctx):
    """Prefix-sharing jobs beside replayed, grouped and path-sharing ones in one packed step: each
    equals the job stepped alone, bit for bit."""
    from paper_2211_17263_gb300 import api
    wls = [_glass_and_light(width=33, height=18, spp=6, pairs=3), _light(width=24, height=11, spp=6, pairs=5),
           _box_and_light(width=21, height=10, spp=6, pairs=8),
           workloads.scaled(workloads.config_occlusion(), width=30, height=17, spp=4, pairs=4),
           _lamp_and_mirror(width=13, height=8, spp=40, pairs=20)]
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
        for k in ("theta", "grad", "losses"):
            assert np.array_equal(x[k], y[k])
        a.release()
        b.release()
