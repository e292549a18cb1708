"""RT_KERNEL_WARP_RAY gives a ray the same T bit for bit in a full set and in a
list of any length, and so does the surrogate's fallback, which is traced with
it."""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu
N, K = 12_000, 32


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.fixture(scope="module")
def scene():
    from paper_2311_16043_gb300 import rt
    sc = scenes.object_scene(N, 3)
    bvh = rt.rt_build_bvh(*(_dev(sc[x]) for x in ("mean", "scale", "quat", "opacity")))
    dirs = _dev(scenes.fibonacci_sphere(K))
    full = rt.rt_trace_visibility_dirs(bvh, dirs, opts=rt.trace_opts(kernel=rt.RT_KERNEL_WARP_RAY)).view(-1)
    return bvh, dirs, full


@pytest.mark.parametrize("m", [1, 8192, 8193, 65_537, 262_145])
def test_lists_of_any_length(scene, m):
    from paper_2311_16043_gb300 import rt
    bvh, dirs, full = scene
    ids = _dev(scenes.sample_ray_ids(N * K, m, 5))
    T = rt.rt_trace_visibility(bvh, rt.rayspec(rt.RT_RAYS_DIRS, dirs=dirs, ray_ids=ids),
                               opts=rt.trace_opts(kernel=rt.RT_KERNEL_WARP_RAY))
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    assert torch.equal(T, full[ids])


@pytest.mark.parametrize("m", [9000, 70_000, 300_000])
def test_fallback_of_a_list(scene, m):
    from paper_2311_16043_gb300 import rt
    bvh, dirs, full = scene
    s = rt.rt_surrogate_create(rt.mlp_cfg(batch=16384), seed=5)
    rt.rt_surrogate_train(s, bvh, rt.rayspec(rt.RT_RAYS_DIRS, dirs=dirs), full, steps=20, seed=5)
    ids = _dev(scenes.sample_ray_ids(N * K, m, 6))
    rs = rt.rayspec(rt.RT_RAYS_DIRS, dirs=dirs, ray_ids=ids)
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    got = rt.rt_surrogate_infer(s, bvh, rs, band=0.3, n_fallback=count)
    o, d, _ = rt.rt_materialize_rays(bvh, rs, ids)
    fell = (rt.rt_surrogate_forward(s, o, d) - 0.5).abs() < 0.3
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    assert int(count) == int(fell.sum()) > 0
    assert torch.equal(got[fell], full[ids][fell])
    s.destroy()
