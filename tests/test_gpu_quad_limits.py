"""Quads at the limits of FP32: emitters so small that the square of u x v is subnormal."""
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
