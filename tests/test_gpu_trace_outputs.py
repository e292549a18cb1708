"""What a trace writes besides T, whichever walk AUTO takes."""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _rays(rt, kind, sc, n, k):
    if kind == "list":
        ids = _dev(scenes.sample_ray_ids(n * k, n * k // 3, 3))
        return rt.rayspec(rt.RT_RAYS_DIRS, dirs=_dev(scenes.fibonacci_sphere(k)), ray_ids=ids)
    if kind == "dirs":
        return rt.rayspec(rt.RT_RAYS_DIRS, dirs=_dev(scenes.fibonacci_sphere(k)))
    nrm = scenes.shortest_axis_normals(sc["scale"], sc["quat"])
    return rt.rayspec(rt.RT_RAYS_HEMI, dirs=_dev(scenes.fibonacci_hemisphere(k)), normals=_dev(nrm))


@pytest.mark.parametrize("kind,n,k", [("dirs", 3000, 8), ("dirs", 3000, 32), ("hemi", 3000, 8), ("hemi", 3000, 64),
                                      ("hemi", 20000, 64), ("list", 3000, 32)])
def test_hit_count_without_a_log(kind, n, k):
    """Without hit_ids every count is written, as 0."""
    from paper_2311_16043_gb300 import rt
    sc = scenes.uniform_scene(n, 7)
    bvh = rt.rt_build_bvh(*(_dev(sc[x]) for x in ("mean", "scale", "quat", "opacity")))
    rs = _rays(rt, kind, sc, n, k)
    for kernel in range(7):
        cnt = torch.full((rt.rt_rayspec_count(bvh, rs),), -1, dtype=torch.int32, device="cuda")
        rt.rt_trace_visibility(bvh, rs, opts=rt.trace_opts(kernel=kernel, hit_count=cnt))
        torch.cuda.synchronize()
        assert rt.rt_status_last() == 0
        assert int(cnt.min()) == 0 and int(cnt.max()) == 0, kernel
