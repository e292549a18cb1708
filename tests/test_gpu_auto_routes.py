"""AUTO on full hemisphere and environment sets around every size and density at
which it changes its walk: the values are those of the per-ray binary walk, up
to the order of the factors (h <= 1024) and the snap at T_min."""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("scene,n,k", [
    ("object", 700, 16), ("object", 700, 17), ("object", 3000, 8), ("object", 3000, 9), ("object", 3000, 17),
    ("object", 1023, 16), ("object", 1025, 16), ("uniform", 1500, 32), ("uniform", 1500, 33), ("uniform", 4096, 32),
    ("uniform", 4096, 33), ("uniform", 4100, 32), ("uniform", 9000, 32), ("uniform", 17_000, 16),
    ("object", 32_768, 8), ("object", 32_769, 8), ("object", 131_073, 2), ("object", 131_073, 1)])
@pytest.mark.parametrize("kind", ["hemi", "env"])
def test_full_sets(scene, n, k, kind):
    from paper_2311_16043_gb300 import rt
    sc = scenes.object_scene(n, 3) if scene == "object" else scenes.uniform_scene(n, 3)
    bvh = rt.rt_build_bvh(*(_dev(sc[x]) for x in ("mean", "scale", "quat", "opacity")))
    env = None
    if kind == "hemi":
        nrm = scenes.shortest_axis_normals(sc["scale"], sc["quat"])
        rs = rt.rayspec(rt.RT_RAYS_HEMI, dirs=_dev(scenes.fibonacci_hemisphere(k)), normals=_dev(nrm))
    else:
        m = scenes.envmap(399)
        env = rt.rt_envmap_create(m["radiance"], m["solid_angle"], m["corners"])
        rs = rt.rayspec(rt.RT_RAYS_ENV, env=env, n_samples=k, seed=3)
    a, b = (rt.rt_trace_visibility(bvh, rs, opts=rt.trace_opts(kernel=x)).double() for x in (1, 0))
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    tol = 2 * 1024 * 2.0 ** -24
    assert bool((((b - a).abs() <= tol * a) | (torch.maximum(a, b) <= 1e-4 * (1 + tol))).all())
    if env is not None:
        env.destroy()


@pytest.mark.parametrize("n,k", [(3000, 8), (20_000, 16), (60_000, 16)])
def test_a_list_and_the_full_set_agree(n, k):
    """The same ray in a full set and in an id list: AUTO may take different
    walks, whose factors come in another order, so the last bits may differ."""
    from paper_2311_16043_gb300 import rt
    sc = scenes.object_scene(n, 3)
    bvh = rt.rt_build_bvh(*(_dev(sc[x]) for x in ("mean", "scale", "quat", "opacity")))
    nrm = scenes.shortest_axis_normals(sc["scale"], sc["quat"])
    kw = dict(dirs=_dev(scenes.fibonacci_hemisphere(k)), normals=_dev(nrm))
    ids = _dev(scenes.sample_ray_ids(n * k, 9000, 5))
    a = rt.rt_trace_visibility(bvh, rt.rayspec(rt.RT_RAYS_HEMI, **kw)).double()[ids]
    b = rt.rt_trace_visibility(bvh, rt.rayspec(rt.RT_RAYS_HEMI, ray_ids=ids, **kw)).double()
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    tol = 2 * 1024 * 2.0 ** -24
    assert bool((((b - a).abs() <= tol * a) | (torch.maximum(a, b) <= 1e-4 * (1 + tol))).all())
