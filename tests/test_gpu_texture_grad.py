"""Gradient of a texture scene (k_hd_grad) against the definition, over pair counts around the
kernel's batches of eight, odd parameter counts and both estimator forms: with the draws' weights
w and the losses L of the same call, g = (1/2P) sum_p w_2p (L_2p - L_2p+1) (antithetic) or
(1/2P) sum_r w_r L_r. The call sums FP64 losses and returns them rounded to FP32, so the two
differ by at most mean_r |w_r| 2^-24 L_r (with both losses of a pair: twice that), and the final
rounding of g."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("pairs", [1, 7, 8, 9, 17])
@pytest.mark.parametrize("antithetic", [1, 0])
@pytest.mark.parametrize("res", [5, 12])
def test_gradient_is_the_weighted_sum_of_losses(gpu_lib, pairs, antithetic, res):
    from paper_2211_17263_gb300 import api
    wl = workloads.config_texture(res=res)
    wl.pairs, wl.spp, wl.antithetic = pairs, 1, antithetic
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.float32), device="cuda")  # noqa: E731
    ctx = api.Context(0)
    try:
        scene = ctx.upload_scene(wl.scene, wl.bindings)
        target = t(np.random.default_rng(3).uniform(size=(wl.height, wl.width, 4)))
        g, L = scene.smoothed_grad(t(wl.theta0), t(wl.sigma), target, scene.grad_opts(wl, step=2))
        _, w = ctx.sample_perturbations(t(wl.sigma), pairs, sampler=wl.sampler, antithetic=antithetic, seed=wl.seed,
                                        step=2)
        torch.cuda.synchronize()
        g, L, w = (x.cpu().numpy().astype(np.float64) for x in (g, L, w))
    finally:
        ctx.close()
    assert np.all(L > 0.0)
    ref = (w[0::2] * (L[0::2] - L[1::2])[:, None]).sum(0) / (2 * pairs) if antithetic else (w * L[:, None]).mean(0)
    tol = (np.abs(w) * L[:, None]).mean(0) * 2.0**-24 * (1 + antithetic) + np.abs(ref) * 2.0**-23 + 1e-30
    assert np.all(np.abs(g - ref) <= tol)
