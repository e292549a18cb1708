"""Kernel 6 (a group of lanes per ray): the lane count follows the length of the
list, so every list length around a change of it is compared with the
one-thread-per-ray walk (kernel 4).  Both accept the same Gaussians; the factors
are multiplied in another order, so a ray of H hits may differ by 2 H 2^-24
relative, and by whether the last bits put it under t_min (then 0)."""
import numpy as np
import pytest

import torch

import scenes

pytestmark = pytest.mark.gpu

MAX_HITS = 2349  # of a ray with T >= t_min: ln 1e-4 / ln(1 - 1/255)


def build(sc):
    from paper_2311_16043_gb300 import rt
    return rt.rt_build_bvh(*(torch.from_numpy(np.ascontiguousarray(sc[k])).cuda()
                             for k in ("mean", "scale", "quat", "opacity")), rt.params())


def scene(kind):
    if kind == "two":
        return scenes.uniform_scene(2, 3, log_scale_mean=np.log(0.3))
    sc = scenes.uniform_scene(3000, 7)
    if kind == "coincident":  # a deep tree: equal Morton codes
        sc["mean"][200:] = sc["mean"][200]
        sc["opacity"][:] = 0.02
    return sc


@pytest.mark.parametrize("kind", ["spread", "coincident", "two"])
@pytest.mark.parametrize("m", [1, 33, 8192, 8193, 65536, 65537, 262144, 262145])
def test_lane_groups_match_single_thread(kind, m):
    from paper_2311_16043_gb300 import rt
    sc = scene(kind)
    bvh = build(sc)
    rng = np.random.default_rng(m)
    ro = torch.as_tensor(rng.uniform(-1, 1, (m, 3)).astype(np.float32)).cuda()
    rd = rng.normal(size=(m, 3)).astype(np.float32)
    rd = torch.as_tensor(rd / np.linalg.norm(rd, axis=1, keepdims=True)).cuda()
    rs = rt.rayspec(rt.RT_RAYS_EXPLICIT, ray_o=ro, ray_d=rd)
    ref = rt.rt_trace_visibility(bvh, rs, opts=rt.trace_opts(kernel=4)).double()
    tol = 2.0 * MAX_HITS * 2.0 ** -24
    t_min = 1e-4
    for kernel in (0, 6):
        got = rt.rt_trace_visibility(bvh, rs, opts=rt.trace_opts(kernel=kernel)).double()
        torch.cuda.synchronize()
        off = (got - ref).abs() > tol * ref
        near = torch.maximum(got, ref) <= t_min * (1 + tol)
        assert not bool((off & ~near).any())


@pytest.mark.parametrize("n", [0, 1])
@pytest.mark.parametrize("m", [5, 8193])
def test_lane_groups_without_a_tree(n, m):
    from paper_2311_16043_gb300 import rt
    sc = scenes.uniform_scene(1, 5, log_scale_mean=np.log(0.3))
    bvh = build({k: v[:n] for k, v in sc.items()})
    rng = np.random.default_rng(m)
    ro = torch.as_tensor(rng.uniform(-1, 1, (m, 3)).astype(np.float32)).cuda()
    rd = rng.normal(size=(m, 3)).astype(np.float32)
    rd = torch.as_tensor(rd / np.linalg.norm(rd, axis=1, keepdims=True)).cuda()
    rs = rt.rayspec(rt.RT_RAYS_EXPLICIT, ray_o=ro, ray_d=rd)
    out = [rt.rt_trace_visibility(bvh, rs, opts=rt.trace_opts(kernel=k)) for k in (1, 0, 6)]
    torch.cuda.synchronize()
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])


def test_auto_list_with_hit_log():
    """A hit log needs the one-thread-per-ray walk: AUTO takes it for a list."""
    from paper_2311_16043_gb300 import rt
    bvh = build(scene("spread"))
    rng = np.random.default_rng(2)
    m = 300
    ro = torch.as_tensor(rng.uniform(-1, 1, (m, 3)).astype(np.float32)).cuda()
    rd = rng.normal(size=(m, 3)).astype(np.float32)
    rd = torch.as_tensor(rd / np.linalg.norm(rd, axis=1, keepdims=True)).cuda()
    rs = rt.rayspec(rt.RT_RAYS_EXPLICIT, ray_o=ro, ray_d=rd)
    out = []
    for kernel in (4, 0):
        ids = torch.full((m, 64), -1, dtype=torch.int32, device="cuda")
        cnt = torch.full((m,), -1, dtype=torch.int32, device="cuda")
        rt.rt_trace_visibility(bvh, rs, opts=rt.trace_opts(kernel=kernel, hit_ids=ids, hit_count=cnt))
        torch.cuda.synchronize()
        out.append((ids, cnt))
    assert int(out[0][1].min()) >= 0
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("n,K", [(3000, 1), (3000, 10), (3000, 16), (3000, 17), (3000, 32), (3000, 33), (500, 16), (500, 17)])
@pytest.mark.parametrize("kind", ["dirs", "hemi"])
def test_auto_small_sets(kind, n, K):
    """Full sets around the sizes where AUTO leaves the lane groups."""
    from paper_2311_16043_gb300 import rt
    sc = scenes.uniform_scene(n, 7)
    bvh = build(sc)
    if kind == "dirs":
        rs = rt.rayspec(rt.RT_RAYS_DIRS, dirs=torch.from_numpy(scenes.fibonacci_sphere(K)).cuda())
    else:
        nrm = torch.from_numpy(scenes.shortest_axis_normals(sc["scale"], sc["quat"])).cuda()
        rs = rt.rayspec(rt.RT_RAYS_HEMI, dirs=torch.from_numpy(scenes.fibonacci_hemisphere(K)).cuda(), normals=nrm)
    ref = rt.rt_trace_visibility(bvh, rs, opts=rt.trace_opts(kernel=1)).double()
    got = rt.rt_trace_visibility(bvh, rs).double()
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    tol = 2.0 * MAX_HITS * 2.0 ** -24
    off = (got - ref).abs() > tol * ref
    assert not bool((off & (torch.maximum(got, ref) > 1e-4 * (1 + tol))).any())
