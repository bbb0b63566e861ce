"""The autotuner's cache key (no GPU): a cached launch shape is taken up only by jobs that run the
same kernels, under the routing rules it was tuned for."""
import numpy as np

import workloads
from paper_2211_17263_gb300 import autotune


def _key_without_routes(wl):
    """The key of caches written before the routes were part of it."""
    sc = wl.scene
    counts = [int((sc.prim_type == t).sum()) for t in range(3)]
    mats = sorted(set(int(m) for m in sc.mat_type))
    return (f"W{wl.width}xH{wl.height}_spp{wl.spp}_d{wl.depth}_rr{wl.rr_start}_R{wl.renders}_D{wl.D}"
            f"_prims{counts[0]}-{counts[1]}-{counts[2]}_mats{'-'.join(map(str, mats))}")


def test_entries_tuned_for_other_routes_are_ignored(tmp_path):
    path = str(tmp_path / "tune.json")
    wl = workloads.config_gi_albedo()
    entry = {"block_pixels": 16, "ctas_per_sm": 2, "render_groups": -1, "no_path_sharing": 1, "ms": 31.4}
    autotune._store(path, {_key_without_routes(wl): entry})
    assert autotune.cached_shape(wl, path) is None
    autotune._store(path, {autotune.shape_key(wl): entry})
    assert autotune.cached_shape(wl, path) == entry


def test_estimator_streams_and_bindings_are_part_of_the_key():
    wl = workloads.config_gi_albedo()
    other = [workloads.scaled(wl, estimator=1 - wl.estimator), workloads.scaled(wl, crn=1 - wl.crn)]
    moved = workloads.scaled(wl)
    moved.bindings = wl.bindings.copy()
    moved.bindings[-1] = [workloads.BIND_PRIM_POS, 5, 0]
    keys = {autotune.shape_key(w) for w in [wl, moved, *other]}
    assert len(keys) == 4
    same = workloads.scaled(wl)
    same.theta0 = wl.theta0 + np.float32(0.1)
    assert autotune.shape_key(same) == autotune.shape_key(wl)
    assert len({autotune.shape_key(workloads.config_texture(res=r)) for r in (16, 32)}) == 2
