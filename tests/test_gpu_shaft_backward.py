"""The adjoint of a full direction set in shaft packets against the per-ray
adjoint over the same rays as an explicit list.

Both find the accepted set with the same arithmetic.  A Gaussian's gradient is
a sum of terms of about 20 float32 roundings each; the packets add up to 64 of
them in float32 before the atomics, so the two differ by at most (20 + 64) 2^-24
= 5e-6 of the sum of the terms' sizes; terms of both signs may halve the sum, so
the relative norm of the difference stays below 1e-5.
"""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu
TOL = 1e-5


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _compare(sc, dirs, seed=0, pays=True, sparse=False, **kw):
    from paper_2311_16043_gb300 import rt
    args = tuple(_dev(sc[k]) for k in ("mean", "scale", "quat", "opacity"))
    bvh = rt.rt_build_bvh(*args, rt.params(**kw))
    rs = rt.rayspec(rt.RT_RAYS_DIRS, dirs=_dev(dirs))
    if pays is not None:
        assert rt.rt_backward_wants_log(bvh, rs) == (not pays)  # what autograd follows
    R = len(sc["mean"]) * len(dirs)
    rng = np.random.default_rng(seed)
    w = rng.uniform(-1, 1, R).astype(np.float32)
    if sparse:  # most rays without a gradient
        w[rng.uniform(size=R) < 0.9] = 0.0
    T = rt.rt_trace_visibility(bvh, rs)
    o, d, s = rt.rt_materialize_rays(bvh, rs, torch.arange(R, dtype=torch.int64, device="cuda"))
    ex = rt.rayspec(rt.RT_RAYS_EXPLICIT, ray_o=o, ray_d=d, ray_src=s)
    g = rt.rt_trace_visibility_backward(bvh, rs, *args, T, _dev(w))
    g2 = rt.rt_trace_visibility_backward(bvh, rs, *args, T, _dev(w))
    ray_o = torch.empty(R, 3, device="cuda")
    want = rt.rt_trace_visibility_backward(bvh, ex, *args, T, _dev(w), d_ray_o=ray_o)
    got_o = torch.full((R, 3), 7.0, device="cuda")
    rt.rt_trace_visibility_backward(bvh, rs, *args, T, _dev(w), d_ray_o=got_o)
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    # an explicit ray's origin is not the mean of its Gaussian
    want["mean"] = want["mean"] + ray_o.view(-1, len(dirs), 3).double().sum(1).float()
    for k in ("mean", "scale", "quat", "opacity"):
        a, b = g[k].double(), want[k].double()
        assert float((a - b).norm()) <= TOL * float(b.norm()) + 1e-30, k
        if kw.get("deterministic"):
            assert torch.equal(g[k], g2[k]), k
    assert float((got_o - ray_o).double().norm()) <= TOL * float(ray_o.double().norm()) + 1e-30


@pytest.mark.parametrize("deterministic", [False, True])
@pytest.mark.parametrize("t_min", [0.0, 1e-4])
def test_object_scene(t_min, deterministic):
    _compare(scenes.object_scene(20_001, 3), scenes.fibonacci_sphere(13), pays=None, t_min=t_min,
             deterministic=deterministic)


@pytest.mark.parametrize("n", [31, 64, 65, 129, 1000])
def test_sizes(n):
    sc = {k: v[:n] for k, v in scenes.uniform_scene(1000, 11, lo=-0.2, hi=0.2).items()}
    _compare(sc, scenes.fibonacci_sphere(7), pays=None, t_min=0.0)


def test_dense_scene_fills_lists():
    """Hundreds of Gaussians in every shaft, most pairs accepted."""
    sc = scenes.uniform_scene(3000, 4, lo=-0.2, hi=0.2)
    sc["opacity"] = (0.05 * sc["opacity"]).astype(np.float32)
    _compare(sc, scenes.fibonacci_sphere(5), t_min=0.0)
    _compare(sc, scenes.fibonacci_sphere(5), t_min=0.0, sparse=True)


def test_few_rays_a_group_keep_the_log():
    _compare(scenes.object_scene(4000, 5), scenes.fibonacci_sphere(5), pays=False, t_min=0.0)


def test_coincident_and_overflowing():
    sc = scenes.uniform_scene(700, 8, lo=-0.2, hi=0.2)
    sc["scale"][::7] = 1e-20  # squares of the inverse scales overflow
    sc["mean"][::5] = sc["mean"][0]
    _compare(sc, scenes.fibonacci_sphere(6), pays=None, t_min=0.0)
