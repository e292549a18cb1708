"""The autotuner's choices are kept per process for scenes alike in what decides
between the strategies; a call that finds one leaves its scratch as it is."""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def test_scenes_of_another_density_are_measured():
    from paper_2311_16043_gb300 import rt
    n, k = 4096, 29  # a number of directions no other test tunes
    rs = rt.rayspec(rt.RT_RAYS_DIRS, dirs=_dev(scenes.fibonacci_sphere(k)))
    measured = []
    for sc in (scenes.object_scene(n, 3), scenes.uniform_scene(n, 3), scenes.object_scene(n, 4), scenes.uniform_scene(n, 4)):
        bvh = rt.rt_build_bvh(*(_dev(sc[x]) for x in ("mean", "scale", "quat", "opacity")))
        T = torch.full((n * k,), -1.0, device="cuda")
        o = rt.rt_trace_autotune(bvh, rs, T)
        torch.cuda.synchronize()
        measured.append(bool((T >= 0).any()))
        a = rt.rt_trace_visibility(bvh, rs, opts=o).double()
        b = rt.rt_trace_visibility(bvh, rs, opts=rt.trace_opts(kernel=1)).double()
        assert (a - b).abs().max().item() <= 1e-6
    assert measured == [True, True, False, False]


@pytest.mark.parametrize("n", [1, 2, 3])
def test_smallest_trees(n):
    from paper_2311_16043_gb300 import rt
    sc = scenes.uniform_scene(3, 5, log_scale_mean=np.log(0.3))
    bvh = rt.rt_build_bvh(*(_dev(sc[x][:n]) for x in ("mean", "scale", "quat", "opacity")))
    rs = rt.rayspec(rt.RT_RAYS_DIRS, dirs=_dev(scenes.fibonacci_sphere(7)))
    T = torch.empty(n * 7, device="cuda")
    o = rt.rt_trace_autotune(bvh, rs, T)
    a, b = (rt.rt_trace_visibility(bvh, rs, opts=x) for x in (o, rt.trace_opts(kernel=1)))
    assert (a - b).abs().max().item() <= 1e-6
