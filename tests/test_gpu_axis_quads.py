"""Axis-aligned quads take a short intersection test: images of scenes made of them (a wall, a
floating occluder, a light) equal the FP64 oracle's for every axis, facing, edge order and edge
sign, for square, oblong, tiny and large quads and for edge lengths whose unit normal rounds off 1
(which take the general test), beside a tilted quad. Tolerance: the image parity of the other
parity tests (FP32 against FP64 branch decisions)."""
import numpy as np
import pytest

import oracle
import workloads
from gpu_helpers import assert_image_parity

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _scene(axis, sign, swap, eu, ev):
    a, b, c = np.eye(3)[axis] * sign, np.eye(3)[(axis + 1) % 3], np.eye(3)[(axis + 2) % 3]
    if swap:
        b, c = -c, b
    s = workloads.SceneBuilder()
    grey = s.material(workloads.MAT_DIFFUSE, (0.7, 0.5, 0.3))
    red = s.material(workloads.MAT_DIFFUSE, (0.8, 0.2, 0.2))
    lamp = s.material(workloads.MAT_DIFFUSE, (0.0, 0.0, 0.0), emission=(9.0, 8.0, 7.0))
    o = np.array([0.13, -0.21, 0.08])
    size = max(eu, ev)
    s.quad(o, eu * b, ev * c, grey)                                             # the wall
    occ = s.quad(o + 0.3 * size * a + 0.1 * eu * b, 0.25 * eu * c, -0.3 * ev * b, red)  # a floating occluder
    s.quad(o + 0.2 * size * a - 0.2 * ev * c, 0.2 * size * (b + 0.3 * a), 0.2 * size * c, red)  # a tilted one
    lu, lv = 0.4 * size * b, 0.3 * size * c
    if np.dot(np.cross(lu, lv), a) > 0:
        lu = -lu
    s.quad(o + 1.5 * size * a, lu, lv, lamp)                                    # faces the wall
    eye = o + size * (1.4 * a + 0.5 * b + 0.1 * c)
    s.look_at(eye, o, c, 50.0)
    return s.build(), np.array([[workloads.BIND_PRIM_POS, occ, k] for k in range(3)], np.int32)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("sign,swap", [(1, False), (-1, True), (1, True)])
@pytest.mark.parametrize("eu,ev", [(2.0, 2.0), (1.0, 0.37), (0.013, 0.031), (61.0, 17.3)])
def test_axis_quads_match_oracle(gpu_lib, axis, sign, swap, eu, ev):
    from paper_2211_17263_gb300 import api
    sc, binds = _scene(axis, sign, swap, eu, ev)
    W, H, spp, depth = 40, 30, 8, 3
    ctx = api.Context(0)
    try:
        scene = ctx.upload_scene(sc, binds)
        theta = sc.prim_geom[1, :3].astype(np.float32)[None]
        img = scene.render_batch(torch.as_tensor(theta, device="cuda"), W, H, spp, depth, seed=5)
        torch.cuda.synchronize()
        ref = oracle.render(sc, binds, theta, W, H, spp, depth, seed=5)
        assert ref[..., :3].max() > 1e-3  # the wall is lit
        assert_image_parity(img.cpu().numpy()[..., :3], np.asarray(ref)[..., :3], what=f"axis {axis}")
    finally:
        ctx.close()
