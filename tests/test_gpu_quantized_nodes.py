"""Walks of single rays over the 64-byte nodes (kernels 5 and 6) against the
binary tree (kernel 1): the quantized boxes contain the exact ones, so with
T_min = 0 every ray accepts the same Gaussians.  The factors are multiplied in
another order: 2 H 2^-24 relative for H hits (H <= 700 in these scenes), where T is a
normal number.  Scenes of 1e12 and more have no rays along an axis: there the
binary tree's plane distances overflow and it misses hits."""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu
RTOL = 2 * 700 * 2.0 ** -24


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _scene(what):
    sc = scenes.uniform_scene(2, 6, log_scale_mean=np.log(0.3)) if what == "two" else scenes.uniform_scene(700, 6)
    n = len(sc["mean"])
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
    elif what == "mixed":
        sc["scale"][::50] *= 40
    elif what in ("large", "larger"):
        f = np.float32(1e12 if what == "large" else 1e17)
        sc["mean"] *= f
        sc["scale"] *= f
    elif what == "outlier":  # more than the 64-byte nodes hold
        sc["mean"][0] = 1e24
    elif what == "small":
        sc["mean"] *= np.float32(1e-8)
        sc["scale"] *= np.float32(1e-8)
    elif what == "faint":  # empty boxes
        sc["opacity"][::2] = 1e-4
    return sc, n


@pytest.mark.parametrize("what", ["two", "plain", "coincident", "line", "far", "needles", "tiny", "mixed", "large",
                                  "larger", "outlier", "small",
                                  "faint"])
@pytest.mark.parametrize("refit", [False, True])
def test_same_hits(what, refit):
    from paper_2311_16043_gb300 import rt
    sc, n = _scene(what)
    args = [_dev(sc[k]) for k in ("mean", "scale", "quat", "opacity")]
    prm = rt.params(t_min=0.0, box_mode=1)
    if refit:  # the nodes made by the refit
        moved = [args[0].flip(0).contiguous(), *args[1:]]
        bvh = rt.rt_build_bvh(*moved, prm)
        rt.rt_bvh_refit(bvh, *args)
    else:
        bvh = rt.rt_build_bvh(*args, prm)
    rng = np.random.default_rng(1)
    nrm = rng.normal(size=(n, 3))
    axes = what not in ("large", "larger", "outlier")
    if axes:
        nrm[::3] = [0, 0, 1]  # axis directions among the hemisphere's
    nrm = (nrm / np.linalg.norm(nrm, axis=1, keepdims=True)).astype(np.float32)
    K = 12
    dirs = scenes.fibonacci_hemisphere(K)
    if axes:
        dirs[0], dirs[1] = [0, 0, 1], [1, 0, 0]
    hemi = rt.rayspec(rt.RT_RAYS_HEMI, dirs=_dev(dirs), normals=_dev(nrm))
    o, d, s = rt.rt_materialize_rays(bvh, hemi, torch.arange(n * K, dtype=torch.int64, device="cuda"))
    d = d * torch.from_numpy(10.0 ** rng.uniform(-8, 4, (n * K, 1))).float().cuda()  # any length
    ex = rt.rayspec(rt.RT_RAYS_EXPLICIT, ray_o=o, ray_d=d, ray_src=s)

    def run(rs, kernel):
        cnt = torch.zeros(4, dtype=torch.int64, device="cuda")
        T = rt.rt_trace_visibility(bvh, rs, opts=rt.trace_opts(kernel=kernel, counters=cnt))
        torch.cuda.synchronize()
        assert rt.rt_status_last() == 0
        return T.double(), cnt.cpu().numpy()

    for rs, kernel in ((hemi, 5), (ex, 6)):
        want, cw = run(rs, 1)
        got, cg = run(rs, kernel)
        assert cg[2] == cw[2] and cg[3] == cw[3]  # hits, rays
        assert cg[1] >= cw[1]  # no leaf box is missed
        normal = torch.maximum(got, want) >= 2.0 ** -126
        assert bool(((got - want).abs() <= RTOL * want)[normal].all())


def test_rays_that_are_not_finite():
    from paper_2311_16043_gb300 import rt
    sc, _ = _scene("plain")
    bvh = rt.rt_build_bvh(*(_dev(sc[k]) for k in ("mean", "scale", "quat", "opacity")))
    o = np.zeros((8, 3), np.float32)
    d = np.tile(np.array([[0, 0.6, 0.8]], np.float32), (8, 1))
    d[1, 0], d[2], d[3, 2], d[4] = np.nan, np.nan, np.inf, 0.0
    o[5, 1], o[6, 0] = np.nan, -np.inf
    ex = rt.rayspec(rt.RT_RAYS_EXPLICIT, ray_o=_dev(o), ray_d=_dev(d))
    want = rt.rt_trace_visibility(bvh, ex, opts=rt.trace_opts(kernel=1))
    got = rt.rt_trace_visibility(bvh, ex, opts=rt.trace_opts(kernel=6))
    torch.cuda.synchronize()
    assert torch.allclose(got, want, rtol=RTOL, atol=0)
