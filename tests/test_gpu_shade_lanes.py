"""PBR colour from a table over every way its terms are dealt to threads:
1, 4 and 16 lanes per Gaussian, tables of directions in several chunks, V read
one and four terms at a time, maps from 1 x 1 on; the oracle's FP64 Eq. 10,
with the bounds of the other colour tests (rtol 1e-3 for near-mirror terms in
float32, median 1e-5)."""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n,K,env_h,with_sh,offset", [
    (1, 1, 16, True, 0), (7, 64, 16, True, 0), (500, 128, 4, True, 0), (500, 130, 16, False, 0), (300, 300, 32, True, 0),
    (300, 64, 16, True, 1), (40_000, 16, 8, True, 0), (40_000, 17, 8, False, 0), (120_000, 8, 16, True, 0),
    (120_000, 9, 1, True, 0)])
def test_lanes_and_chunks(orc, n, K, env_h, with_sh, offset):
    from paper_2311_16043_gb300 import rt
    sc = scenes.uniform_scene(n, 31)
    nrm = scenes.shortest_axis_normals(sc["scale"], sc["quat"])
    hemi = scenes.fibonacci_hemisphere(K)
    m = scenes.pbr_material(n, 32, with_sh)
    env = scenes.light_envmap(33, env_h, 2 * env_h)
    V = np.random.default_rng(34).uniform(0, 1, (n, K)).astype(np.float32)
    cam = (2.5, -3.0, 4.0)
    dv = _dev(np.concatenate([np.zeros(offset, np.float32), V.ravel()]))[offset:]  # offset 1: not 16-byte aligned
    bvh = rt.rt_build_bvh(*(_dev(sc[k]) for k in ("mean", "scale", "quat", "opacity")))
    inp = rt.pbr_inputs(_dev(m["albedo"]), _dev(m["roughness"]), _dev(env), cam, sh=_dev(m["sh"]) if with_sh else None)
    rgb = rt.rt_pbr_shade(bvh, rt.rayspec(rt.RT_RAYS_HEMI, dirs=_dev(hemi), normals=_dev(nrm)), inp, V=dv)
    torch.cuda.synchronize()
    assert rt.rt_status_last() == 0
    got = rgb.cpu().numpy().astype(np.float64)
    want = orc.pbr(sc, nrm, m, hemi, V, env, np.array(cam))
    np.testing.assert_allclose(got, want, rtol=1e-3, atol=1e-6)
    rel = np.abs(got - want) / np.maximum(np.abs(want), 1e-3)
    assert np.median(rel) < 1e-5
