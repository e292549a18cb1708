"""The rejection test of the shaft packets (RT_KERNEL_WIDE on a full direction
set) never drops a Gaussian that the per-ray walks accept, where its own
rounding is largest: rays that pass long needles nearly end-on, or thin discs
edge-on, just inside the limit of acceptance, from a group much narrower than
those are long.

A Gaussian accepted there multiplies T by 1 - 2e-3; two orders of the at most
2304 factors of a ray differ by 2 * 2304 * 2^-24 = 2.8e-4, and both walks take
their decisions with the same arithmetic.
"""
import numpy as np
import pytest
import torch
from scipy.spatial.transform import Rotation

import scenes

pytestmark = pytest.mark.gpu
RTOL = 2 * 2304 * 2.0 ** -24
N_SRC, N, K = 256, 2048, 8


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def grazing(aspect, what, k_sigma, alpha_min, opacity):
    """N_SRC specks at the origin cast the rays; each of N needles along an
    oblique axis (discs along it), tilted by up to 1 / aspect, is passed by the
    rays of one direction at 1 - 1e-6 to 1 - 0.03 of the limit."""
    rng = np.random.default_rng(int(aspect))
    thin = 1.0 / aspect
    off = np.minimum(np.geomspace(0.3, 30.0, K) / aspect, 0.1)
    phi = rng.uniform(0, 2 * np.pi, K)
    frame, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    frame[:, 0] *= np.linalg.det(frame)
    dirs = np.stack([np.sin(off) * np.cos(phi), np.sin(off) * np.sin(phi), np.cos(off)], 1) @ frame.T
    dirs = dirs.astype(np.float32)
    axes = np.array([thin, thin, 1.0] if what == "needles" else [thin, 1.0, 1.0])
    tilt = Rotation.from_rotvec(rng.uniform(-1, 1, (N, 3)) * thin)
    quat = (Rotation.from_matrix(frame) * tilt).as_quat()[:, [3, 0, 1, 2]].astype(np.float32)
    q = quat / np.linalg.norm(quat.astype(np.float64), axis=1, keepdims=True)
    w, x, y, z = q.T
    R = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                  2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                  2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(N, 3, 3)
    d = dirs[np.arange(N) % K].astype(np.float64)
    ud = np.einsum("nji,nj->ni", R, d) / axes
    ud /= np.linalg.norm(ud, axis=1, keepdims=True)
    u = rng.normal(size=(N, 3))
    u -= (u * ud).sum(1, keepdims=True) * ud
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    m = min(k_sigma, np.sqrt(2 * np.log(opacity / alpha_min))) * (1 - 10 ** rng.uniform(-6, -1.5, N))
    # the peak lies at t d for a t of up to two needles' lengths
    mean = rng.uniform(0.1, 2.0, (N, 1)) * d - np.einsum("nij,nj->ni", R, u * m[:, None] * axes)
    speck = 1e-3 * thin
    return dirs, {"mean": np.concatenate([rng.uniform(-speck, speck, (N_SRC, 3)), mean]),
                  "scale": np.concatenate([np.full((N_SRC, 3), speck), np.broadcast_to(axes, (N, 3))]),
                  "quat": np.concatenate([np.tile([1.0, 0, 0, 0], (N_SRC, 1)), quat]),
                  "opacity": np.concatenate([np.full(N_SRC, 0.5 * alpha_min), np.full(N, opacity)])}


@pytest.mark.parametrize("limit", ["k_sigma", "alpha_min"])
@pytest.mark.parametrize("what", ["needles", "discs"])
@pytest.mark.parametrize("aspect", [50.0, 1e3, 1e4, 1e5])
def test_accepts_what_single_rays_accept(aspect, what, limit):
    from paper_2311_16043_gb300 import rt
    k_sigma, alpha_min, opacity = (3.0, 1e-6, 2e-3 * np.exp(4.5)) if limit == "k_sigma" else (8.0, 2e-3, 0.5)
    dirs, sc = grazing(aspect, what, k_sigma, alpha_min, opacity)
    bvh = rt.rt_build_bvh(*(_dev(sc[k]) for k in ("mean", "scale", "quat", "opacity")),
                          rt.params(k_sigma=k_sigma, alpha_min=alpha_min, t_min=0.0, origin_eps=0.0))
    a, b = (rt.rt_trace_visibility_dirs(bvh, _dev(dirs), opts=rt.trace_opts(kernel=k))[:N_SRC].double()
            for k in (1, 3))
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    assert a.max().item() < 0.9  # the needles are met
    assert bool(((b - a).abs() <= RTOL * a + 1e-30).all()), ((b - a).abs() / a).max().item()


@pytest.mark.parametrize("length", [1e-21, 1e-19, 1e-12, 1e12, 1e15])
def test_directions_of_any_length(length):
    """|d|^2 may underflow or lose its digits where the per-ray walks, which
    never form it, are exact (h <= 512 factors)."""
    from paper_2311_16043_gb300 import rt
    sc = scenes.uniform_scene(1500, 6)
    sc["mean"] = (0.5 * sc["mean"]).astype(np.float32)
    dirs = scenes.fibonacci_sphere(6) * length
    bvh = rt.rt_build_bvh(*(_dev(sc[k]) for k in ("mean", "scale", "quat", "opacity")),
                          rt.params(t_min=0.0, origin_eps=0.0))
    a, b = (rt.rt_trace_visibility_dirs(bvh, _dev(dirs), opts=rt.trace_opts(kernel=k)).double() for k in (1, 3))
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    assert a.min().item() < 0.5
    assert bool(((b - a).abs() <= 2 * 512 * 2.0 ** -24 * a).all()), ((b - a).abs() / a).max().item()


@pytest.mark.parametrize("eps", [float("inf"), 3e38])
def test_origins_that_are_not_finite(eps):
    """Origins at infinity: nothing is met, and nothing is walked to find that."""
    from paper_2311_16043_gb300 import rt
    sc = scenes.uniform_scene(700, 6)
    dirs = 2.0 * scenes.fibonacci_sphere(6)
    bvh = rt.rt_build_bvh(*(_dev(sc[k]) for k in ("mean", "scale", "quat", "opacity")), rt.params(origin_eps=eps))
    a, b = (rt.rt_trace_visibility_dirs(bvh, _dev(dirs), opts=rt.trace_opts(kernel=k)) for k in (1, 3))
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    assert torch.equal(a, torch.ones_like(a)) and torch.equal(a, b)


@pytest.mark.parametrize("far", [1e27, -1e30, 3e38])
def test_rays_from_far_off_walk_no_tree(far):
    """Axis-parallel rays whose o / d overflows meet no box (at most the root's
    children are tested, 4 a node)."""
    from paper_2311_16043_gb300 import rt
    sc = scenes.uniform_scene(700, 6)
    bvh = rt.rt_build_bvh(*(_dev(sc[k]) for k in ("mean", "scale", "quat", "opacity")))
    o = np.zeros((300, 3))
    o[np.arange(300), np.arange(300) % 3] = far
    d = np.zeros((300, 3))
    d[np.arange(300), (np.arange(300) + 1) % 3] = 1.0
    d[::2] *= -1.0
    rs = rt.rayspec(rt.RT_RAYS_EXPLICIT, ray_o=_dev(o), ray_d=_dev(d))
    for kernel in (0, 4, 6):
        cnt = torch.zeros(4, dtype=torch.int64, device="cuda")
        T = rt.rt_trace_visibility(bvh, rs, opts=rt.trace_opts(kernel=kernel, counters=cnt))
        torch.cuda.synchronize()
        assert rt.rt_status_last() == 0
        assert bool((T == 1).all())
        assert int(cnt[0]) <= 4 * 300 and int(cnt[1]) == 0
