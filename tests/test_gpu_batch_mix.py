"""Batches of every mixture of shaft, item and lane-refill jobs: the launches
of the captured graph differ with it, the values do not."""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# dense: a direction set in shaft packets; small: one that joins the item jobs
# when there are others; items: one thread per ray; env: lane refill
@pytest.mark.parametrize("mix", [("dense",), ("items",), ("env",), ("dense", "env"), ("dense", "items"), ("items", "env"),
                                 ("dense", "items", "env", "env"), ("items", "items", "env"), ("empty", "env", "items")])
@pytest.mark.parametrize("autotune", [True, False])
def test_mixtures_equal_single_launches(mix, autotune):
    from paper_2311_16043_gb300 import rt
    env = scenes.envmap(399)
    E = rt.rt_envmap_create(env["radiance"], env["solid_angle"], env["corners"])
    jobs = []
    for j, what in enumerate(mix):
        n, k = {"dense": (25_000, 8), "items": (1500, 5), "env": (900, 7), "empty": (0, 4)}[what]
        sc = scenes.uniform_scene(max(n, 1), 20 + j)
        bvh = rt.rt_build_bvh(*(_dev(sc[x][:n]) for x in ("mean", "scale", "quat", "opacity")))
        rs = (rt.rayspec(rt.RT_RAYS_ENV, env=E, n_samples=k, seed=j) if what == "env"
              else rt.rayspec(rt.RT_RAYS_DIRS, dirs=_dev(scenes.fibonacci_sphere(k))))
        jobs.append((bvh, rs, torch.full((n * k,), -1.0, device="cuda")))
    batch = rt.rt_batch_create(jobs, autotune=autotune)
    kernels = batch.info()["kernel"]
    if not autotune:
        assert kernels == [{"dense": 3, "items": 4, "env": 5, "empty": 2}[w] for w in mix]
    refs = [rt.rt_trace_visibility(b, rs, opts=rt.trace_opts(kernel=k)) for (b, rs, _), k in zip(jobs, kernels)]
    for _ in range(2):
        for _, _, T in jobs:
            T.fill_(-1.0)
        batch.run()
        torch.cuda.synchronize()
        assert rt.rt_status_last() == 0
        for (_, _, T), ref in zip(jobs, refs):
            assert torch.equal(T, ref)
    batch.destroy()
    E.destroy()


def test_small_shaft_jobs_join_the_others():
    """Fewer than 2^17 direction rays beside other jobs are not given a launch of
    their own, whatever tuning preferred."""
    from paper_2311_16043_gb300 import rt
    env = scenes.envmap(399)
    E = rt.rt_envmap_create(env["radiance"], env["solid_angle"], env["corners"])
    sc = scenes.uniform_scene(22_000, 4)
    bvh = rt.rt_build_bvh(*(_dev(sc[x]) for x in ("mean", "scale", "quat", "opacity")))
    kernels = []
    for k in (5, 6):  # 110 and 132 thousand rays
        dirs = rt.rayspec(rt.RT_RAYS_DIRS, dirs=_dev(scenes.fibonacci_sphere(k)))
        rays = rt.rayspec(rt.RT_RAYS_ENV, env=E, n_samples=4, seed=1)
        T = [torch.empty(22_000 * k, device="cuda"), torch.empty(88_000, device="cuda")]
        batch = rt.rt_batch_create([(bvh, dirs, T[0]), (bvh, rays, T[1])], autotune=False)
        kernels.append(batch.info()["kernel"])
        batch.run()
        torch.cuda.synchronize()
        ref = rt.rt_trace_visibility(bvh, dirs, opts=rt.trace_opts(kernel=kernels[-1][0]))
        assert torch.equal(T[0], ref)
        batch.destroy()
    assert kernels == [[rt.RT_KERNEL_RAY_WIDE, rt.RT_KERNEL_RAY_REFILL], [rt.RT_KERNEL_WIDE, rt.RT_KERNEL_RAY_REFILL]]
    E.destroy()
