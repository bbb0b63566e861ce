"""Quads at the limits of FP32: emitters so small that the square of u x v is subnormal, and rays
that are parallel to an axis-aligned quad within the intersection test's bound."""
import numpy as np
import pytest

import oracle
import workloads
from gpu_helpers import assert_image_parity

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    from paper_2211_17263_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def _render(ctx, sc, binds, theta, W, H, spp, depth):
    img = ctx.upload_scene(sc, binds).render_batch(torch.as_tensor(theta, device="cuda"), W, H, spp, depth, seed=5)
    torch.cuda.synchronize()
    return img.cpu().numpy()[..., :3]


@pytest.mark.parametrize("eu,ev,tilt", [(2e-10, 2e-10, 0.0), (1e-12, 5e-8, 0.0), (3e-10, 1e-10, 0.4), (2e-9, 2e-9, 0.0)])
def test_tiny_quad_emitter_lights_the_floor(ctx, eu, ev, tilt):
    """|u x v|^2 is between 1e-40 and 2e-35 here, subnormal below 1.2e-38. Its FP32 value is off by at
    most 2^-150 / 1e-40 = 7e-6, its root (normal and area) by half of that each: 2.1e-5 of a
    radiance below 2 with the shading's own roundings, within the image parity's 1e-4."""
    s = workloads.SceneBuilder()
    grey = s.material(workloads.MAT_DIFFUSE, (0.7, 0.5, 0.3))
    e = 4.0 / (eu * ev)  # 4 W/sr at 1 unit
    lamp = s.material(workloads.MAT_DIFFUSE, (0.0, 0.0, 0.0), emission=(e, 0.8 * e, 0.6 * e))
    s.quad((0, 0, 0), (4, 0, 0), (0, 4, 0), grey)
    s.sphere((0.4, 0.1, 0.2), 0.2, grey)
    i = s.quad((0.1, -0.2, 1.2), (eu * np.cos(tilt), 0, eu * np.sin(tilt)), (0, -ev, 0), lamp)
    s.look_at((0, -2.5, 1.5), (0, 0, 0), (0, 0, 1), 45.0)
    sc, binds = s.build(), np.array([[workloads.BIND_PRIM_POS, i, k] for k in range(3)], np.int32)
    theta = sc.prim_geom[i, :3].astype(np.float32)[None]
    img = _render(ctx, sc, binds, theta, 40, 30, 8, 3)
    ref = np.asarray(oracle.render(sc, binds, theta, 40, 30, 8, 3, seed=5))[..., :3]
    assert 0.1 < ref.max() < 2.0
    assert_image_parity(img, ref)


def _axis_or_general(ctx, quads, albedo, camera, general, W, H, spp, depth):
    """The scene's quads with plain material `albedo`, or with a 1 x 1 texture of that albedo: the
    texture's second and later quads take the general test."""
    s = workloads.SceneBuilder()
    grey = s.material(workloads.MAT_DIFFUSE, albedo)
    lamp = s.material(workloads.MAT_DIFFUSE, (0.0, 0.0, 0.0), emission=(9.0, 8.0, 7.0))
    s.quad((900, 900, 900), (1, 0, 0), (0, 1, 0), grey)  # the texture's first quad, out of sight
    for c, u, v in quads:
        s.quad(c, u, v, grey)
    s.sphere((1.5, -1.2, 2.2), 0.4, lamp)
    s.background = np.array([0.2, 0.3, 0.4], np.float32)
    s.look_at(*camera)
    binds = [[workloads.BIND_TEXTURE, grey, 1]] if general else [[workloads.BIND_MAT_ALBEDO, grey, k] for k in range(3)]
    return _render(ctx, s.build(), np.array(binds, np.int32), np.array([albedo], np.float32), W, H, spp, depth)


@pytest.mark.parametrize("seed", range(4))
def test_axis_aligned_test_is_the_general_one_bit_for_bit(ctx, seed):
    """Boxes of quads of every axis, facing and edge order, seen directly and after bounces."""
    rng = np.random.default_rng(seed)
    quads = []
    for _ in range(9):
        a, b, c = np.roll(np.eye(3), rng.integers(3), axis=0) * rng.choice([-1.0, 1.0], size=(3, 1))
        eu, ev = rng.choice([0.25, 0.5, 1.0, 3.0], 2) if rng.random() < 0.5 else rng.uniform(0.05, 3.0, 2)
        quads.append((rng.choice([-1.0, -0.5, 0.0, 0.25, 1.0], 3) if rng.random() < 0.5 else rng.uniform(-1, 1, 3),
                      eu * b, ev * c))
    camera = ((0.3, -3.0, 1.1), (0, 0, 0), (0, 0, 1), 60.0)
    args = (ctx, quads, (0.75, 0.5, 0.25), camera)
    axis, general = (_axis_or_general(*args, g, 96, 64, 32, 4) for g in (False, True))
    assert np.unique(general).size > 1000
    assert np.array_equal(axis, general)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("vfov", [2e-11, 3e-10, 1e-6])
def test_rays_along_an_axis_aligned_quad(ctx, axis, vfov):
    """A camera a hair above a quad's plane that looks along it: rays whose cosine with the normal is
    below 1e-12 miss the quad, as in the general test."""
    f, up = np.eye(3)[(axis + 1) % 3], np.eye(3)[axis]
    eye = -f + 1e-14 * up
    camera = (eye, eye + f, up, vfov)
    quads = [(np.zeros(3), 4 * f, 4 * np.cross(up, f))]
    args = (ctx, quads, (0.75, 0.5, 0.25), camera)
    plain, general = (_axis_or_general(*args, g, 16, 16, 4, 2) for g in (False, True))
    assert np.array_equal(plain, general)
    if vfov == 2e-11:  # every ray's cosine is below 2e-13
        assert np.array_equal(plain, np.broadcast_to(np.float32([0.2, 0.3, 0.4]), plain.shape))
