"""Shaft packets (RT_KERNEL_WIDE on a full direction set) against the per-ray
binary traversal.

Both take every accept decision with the same float32 arithmetic, so the
accepted sets are equal and only the order of the factors of T differs: a
product of h float32 factors has a relative error below h 2^-24 in any order,
so two orders differ by at most 2 h 2^-24 (h <= 512 in these scenes: 6.2e-5),
or by the snap at T_min where T lies that close to it.
"""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu
RTOL = 2 * 512 * 2.0 ** -24


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _trace(sc, dirs, kernel, order_block=0, **kw):
    from paper_2311_16043_gb300 import rt
    bvh = rt.rt_build_bvh(*(_dev(sc[k]) for k in ("mean", "scale", "quat", "opacity")), rt.params(**kw))
    T = rt.rt_trace_visibility_dirs(bvh, _dev(dirs), opts=rt.trace_opts(kernel=kernel, order_block=order_block))
    ao = rt.rt_trace_ao(bvh, rt.rayspec(rt.RT_RAYS_DIRS, dirs=_dev(dirs)), opts=rt.trace_opts(kernel=rt.RT_KERNEL_WIDE))
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    return T.cpu().numpy().astype(np.float64), ao.cpu().numpy()


def _check(sc, dirs, t_min=1e-4, **kw):
    a, _ = _trace(sc, dirs, 1, t_min=t_min, **kw)
    b, ao = _trace(sc, dirs, 3, t_min=t_min, **kw)
    err = np.abs(b - a) / np.maximum(a, 1e-30)
    snapped = (np.minimum(a, b) == 0) & (np.maximum(a, b) <= t_min * (1 + RTOL))
    assert (snapped | (err <= RTOL)).all(), err[~snapped].max()
    K = dirs.shape[0]
    np.testing.assert_allclose(ao, b.mean(1), rtol=2 * K * 2.0 ** -24, atol=1e-7)
    return a


def _cut(sc, n):
    return {k: v[:n] for k, v in sc.items()}


@pytest.mark.parametrize("n", [2, 3, 5, 31, 32, 33, 63, 64, 65, 128, 129, 1000])
def test_sizes(n):
    _check(_cut(scenes.uniform_scene(1000, 11), n), scenes.fibonacci_sphere(7))


@pytest.mark.parametrize("box_mode", [0, 1])
@pytest.mark.parametrize("t_min", [0.0, 1e-4])
def test_object_scene(t_min, box_mode):
    T = _check(scenes.object_scene(20_001, 3), scenes.fibonacci_sphere(13), t_min=t_min, box_mode=box_mode)
    assert (T > 0.5).any() and (T < 1e-3).any()


def test_dense_scene_fills_batches():
    """Hundreds of Gaussians in every shaft: batches of 64, lists in parts."""
    sc = scenes.uniform_scene(6000, 4, lo=-0.2, hi=0.2)
    _check(sc, scenes.fibonacci_sphere(9))
    sc["opacity"] = (0.05 * sc["opacity"]).astype(np.float32)  # hardly any ray ends early
    _check(sc, scenes.fibonacci_sphere(9), t_min=0.0)


def test_axis_directions_and_lengths():
    sc = scenes.object_scene(5000, 5)
    ax = np.array([[1, 0, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1], [0, 0.6, -0.8], [1e-20, 0, 1]], np.float32)
    _check(sc, ax)
    _check(sc, (scenes.fibonacci_sphere(6) * 0.25).astype(np.float32), origin_eps=4e-4)


@pytest.mark.parametrize("what", ["coincident", "line", "far", "needles", "tiny", "mixed"])
def test_degenerate_scenes(what):
    sc = scenes.uniform_scene(700, 6)
    if what == "coincident":
        sc["mean"][:] = sc["mean"][0]
    elif what == "line":
        sc["mean"][:, 1:] = 0.25
    elif what == "far":
        sc["mean"] += np.float32(100.0)
    elif what == "needles":
        sc["scale"] = (sc["scale"] * np.array([30, 0.01, 1])).astype(np.float32)
    elif what == "tiny":
        sc["scale"] = np.full_like(sc["scale"], 1e-7)
    else:
        sc["scale"][::50] *= 40
    _check(sc, scenes.fibonacci_sphere(11))


def test_order_block_and_refit():
    from paper_2311_16043_gb300 import rt
    sc = scenes.object_scene(4000, 7)
    dirs = scenes.fibonacci_sphere(10)
    np.testing.assert_array_equal(_trace(sc, dirs, 3)[0], _trace(sc, dirs, 3, order_block=37)[0])
    moved = dict(sc)
    moved["mean"] = (sc["mean"] + np.random.default_rng(0).normal(0, 0.2, sc["mean"].shape)).astype(np.float32)
    bvh = rt.rt_build_bvh(*(_dev(sc[k]) for k in ("mean", "scale", "quat", "opacity")))
    rt.rt_bvh_refit(bvh, *(_dev(moved[k]) for k in ("mean", "scale", "quat", "opacity")))  # groups of the old means
    a = rt.rt_trace_visibility_dirs(bvh, _dev(dirs), opts=rt.trace_opts(kernel=1)).cpu().numpy().astype(np.float64)
    b = rt.rt_trace_visibility_dirs(bvh, _dev(dirs), opts=rt.trace_opts(kernel=3)).cpu().numpy().astype(np.float64)
    assert ((np.abs(b - a) <= RTOL * a) | ((np.minimum(a, b) == 0) & (np.maximum(a, b) <= 1.001e-4))).all()


@pytest.mark.parametrize("n", [40, 90, 700])
def test_overflowing_inverse_scales(n):
    """Inverse scales whose squares overflow make every plane test of their
    Gaussian NaN: it is a candidate of all rays, accepted by none, and the lanes
    past a batch that starts with it add nothing."""
    sc = _cut(scenes.uniform_scene(700, 8), n)
    sc["scale"] = sc["scale"].copy()
    sc["scale"][::3] = 1e-20
    _check(sc, scenes.fibonacci_sphere(11))


def test_directions_that_are_not_finite():
    sc = scenes.uniform_scene(700, 8)
    dirs = scenes.fibonacci_sphere(6)
    dirs[1, 0], dirs[3], dirs[4, 2] = np.nan, 0.0, np.inf
    a, b = (_trace(sc, dirs, k)[0] for k in (1, 3))
    np.testing.assert_allclose(b, a, rtol=RTOL, atol=0)
    assert (b[:, [1, 3, 4]] == 1).all()
