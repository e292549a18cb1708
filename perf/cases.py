"""The work a user has this library do, as cases that can be timed.

Each case goes through the public entry points of ``paper_2311_16043_gb300``
(``rt`` and ``autograd``), over the ranges the tests and the benchmark use:
scenes of 4 thousand to 2 million Gaussians, 16 to 128 rays per Gaussian.

  listed()             the named cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  inputs and handles a program holds before the call
  run(state)           one pass, with its whole outputs
  work(case)           bytes and operations one pass cannot do without
  exact(case, seed)    the outputs in float64 by plain torch (small cases)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_16043_gb300 import autograd, rt

DEV = "cuda"
ALPHA_MIN = float(np.float32(1.0 / 255.0))


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # The smallest precompute: a 4,096-Gaussian volume, tree and trace, as
        # an interactive editor runs it per change (launches and latency).
        {"name": "precompute_4k_k32", "op": "precompute", "scene": "uniform", "n": 4096, "k": 32},
        # The ordinary precompute of one reconstructed object: tree and all
        # 38.4M rays over the sphere of directions.
        {"name": "precompute_300k_k128", "op": "precompute", "scene": "object", "n": 300_000, "k": 128},
        # The largest scene, traced again with its tree at hand (new
        # directions): 2M Gaussians.
        {"name": "dirs_2m_k64", "op": "dirs", "scene": "object", "n": 2_000_000, "k": 64},
        # The visibility table of the hemisphere sets, Ns = 64 about each
        # normal, that the shading reads.
        {"name": "hemi_300k_k64", "op": "hemi", "scene": "object", "n": 300_000, "k": 64},
        # Shadow rays of an environment light: importance-sampled directions,
        # different for every Gaussian.
        {"name": "env_200k_s64", "op": "env", "scene": "object", "n": 200_000, "k": 64},
        # The per-iteration colour pass from the precomputed table.
        {"name": "shade_1m_k64", "op": "shade", "scene": "object", "n": 1_000_000, "k": 64, "env_h": 16, "sh": True},
        # Rays a program brings itself (origins and directions of its own):
        # shadow rays to point lights in no particular order.
        {"name": "rays_600k_of_300k", "op": "rays", "scene": "object", "n": 300_000, "rays": 600_000},
        # One differentiation step through autograd at the small parity size,
        # without early termination.
        {"name": "adjoint_4k_k32", "op": "adjoint", "scene": "uniform", "n": 4096, "k": 32, "t_min": 0.0,
         "deterministic": False},
        # The same step on an object of odd size, with early termination and
        # bit-reproducible sums.
        {"name": "adjoint_50k_k32_det", "op": "adjoint", "scene": "object", "n": 50_001, "k": 32, "t_min": 1e-4,
         "deterministic": True},
        # Several scenes of uneven size in one captured launch, directions and
        # environment samples (the multi-scene service).
        {"name": "batch_4_scenes", "op": "batch", "scene": "uniform", "n": 30_000, "n_jobs": 4, "growth": 1.9,
         "k": 32, "s": 32},
        # The learned surrogate with tracer fallback on held-out rays.
        {"name": "infer_2m_rays", "op": "infer", "scene": "object", "n": 200_000, "k": 64, "rays": 2_000_003,
         "band": 0.3},
        # One training gradient of the surrogate at its default batch.
        {"name": "mlp_grad_256k", "op": "mlp_grad", "scene": "uniform", "n": 4096, "rays": 262_144},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["precompute", "precompute", "dirs", "hemi", "env", "shade", "rays", "adjoint", "batch", "infer",
                     "mlp_grad"])
    scene = rng.choice(["uniform", "object"])
    c = {"op": op, "scene": scene}
    if op in ("precompute", "dirs"):
        c["n"] = _log_int(rng, 500, 200_000 if scene == "uniform" else 1_500_000)
        c["k"] = max(1, min(_log_int(rng, 8, 128), 40_000_000 // c["n"]))
    elif op in ("hemi", "env"):
        c["n"] = _log_int(rng, 500, 60_000 if scene == "uniform" else 500_000)
        c["k"] = max(1, min(_log_int(rng, 8, 128), 20_000_000 // c["n"]))
    elif op == "shade":
        c["n"] = _log_int(rng, 1000, 2_000_000)
        c["k"] = max(1, min(_log_int(rng, 8, 128), 64_000_000 // c["n"]))
        c["env_h"] = rng.choice([4, 8, 16, 32])
        c["sh"] = rng.random() < 0.7
    elif op == "rays":
        c["n"] = _log_int(rng, 500, 100_000 if scene == "uniform" else 1_000_000)
        c["rays"] = _log_int(rng, 1000, 3_000_000)
    elif op == "adjoint":
        c["n"] = _log_int(rng, 500, 50_000)
        c["k"] = _log_int(rng, 8, 32)
        c["t_min"] = rng.choice([0.0, 1e-4]) if c["n"] < 8000 else 1e-4
        c["deterministic"] = rng.random() < 0.3
    elif op == "batch":
        c["n"] = _log_int(rng, 2000, 30_000)
        c["n_jobs"] = rng.randint(2, 5)
        c["growth"] = round(rng.uniform(1.2, 1.8), 3)
        c["k"] = rng.randint(8, 32)
        c["s"] = rng.randint(8, 32)
    elif op == "infer":
        c["n"] = _log_int(rng, 4000, 300_000)
        c["scene"] = "object"
        c["k"] = 64
        c["rays"] = min(_log_int(rng, 1000, 4_000_000), c["n"] * 64)
        c["band"] = rng.choice([0.0, 0.2, 0.3])
    else:
        c["n"] = 4096
        c["scene"] = "uniform"
        c["rays"] = _log_int(rng, 1000, 500_000)
    return c


# ---------------------------------------------------------------------------
# Inputs (made on the GPU from the seed)
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _u(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _nrm(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _scene_dict(mean, scale, quat, opacity, **more):
    d = {"mean": mean.float().contiguous(), "scale": scale.float().contiguous(), "quat": quat.float().contiguous(),
         "opacity": opacity.float().clamp(max=1.0 - 2.0 ** -20).contiguous()}
    d.update(more)
    return d


def _uniform(n, seed, side=2.0, offset=(0.0, 0.0, 0.0)):
    """Means uniform in a box, log-scales N(log 0.02, 0.5), random rotations,
    opacity Beta(2,2) (the median of three uniforms)."""
    g = _gen(seed)
    mean = (_u(g, n, 3) - 0.5) * side + torch.tensor(offset, device=DEV, dtype=torch.float64)
    scale = torch.exp(math.log(0.02) + 0.5 * _nrm(g, n, 3))
    quat = _unit(_nrm(g, n, 4))
    opacity = _u(g, n, 3).median(dim=1).values
    return _scene_dict(mean, scale, quat, opacity)


def _object(n, seed):
    """Flattened Gaussians on the surfaces of two spheres, a torus, a box and a
    ground plane (area-proportional), jittered along the way, opacity
    Beta(5,1); the surface normals come along."""
    g = _gen(seed)
    h = np.random.default_rng(int(seed))
    ctr = torch.tensor(np.stack([h.uniform(-0.6, 0.6, 4), h.uniform(-0.6, 0.6, 4), h.uniform(-0.5, 0.3, 4)], 1),
                       device=DEV)
    r = h.uniform(0.2, 0.5, 2)
    box = h.uniform(0.3, 0.6, 3)
    areas = np.array([4 * math.pi * r[0] ** 2, 4 * math.pi * r[1] ** 2, 4 * math.pi ** 2 * 0.04,
                      2 * (box[0] * box[1] + box[1] * box[2] + box[0] * box[2]), 9.0])
    cum = torch.tensor(np.cumsum(areas / areas.sum())[:-1], device=DEV)
    kind = torch.bucketize(_u(g, n), cum)[:, None]
    a, b = _u(g, n), _u(g, n)
    sph = _unit(_nrm(g, n, 3))
    # torus (R 0.4, r 0.1): density 1 + (r/R) cos v by flipping v to v + pi
    uu, vv = 2 * math.pi * a, 2 * math.pi * b
    vv = torch.where(_u(g, n) < 0.5 * (1 + 0.25 * torch.cos(vv)), vv, vv + math.pi)
    ring = 0.4 + 0.1 * torch.cos(vv)
    tor = torch.stack([ring * torch.cos(uu), ring * torch.sin(uu), 0.1 * torch.sin(vv)], 1)
    tor_n = torch.stack([torch.cos(vv) * torch.cos(uu), torch.cos(vv) * torch.sin(uu), torch.sin(vv)], 1)
    # box: a face by area, a point on it
    fa = np.array([box[1] * box[2], box[0] * box[2], box[0] * box[1]])
    ax = torch.bucketize(_u(g, n), torch.tensor(np.cumsum(fa / fa.sum())[:-1], device=DEV))
    sign = torch.where(_u(g, n) < 0.5, 1.0, -1.0)
    half = torch.tensor(box / 2, device=DEV)
    box_n = torch.nn.functional.one_hot(ax, 3).double() * sign[:, None]
    bx = (2 * torch.stack([a, b, _u(g, n)], 1) - 1) * half
    bx = torch.where(box_n != 0, box_n * half, bx)
    pln = torch.stack([3 * a - 1.5, 3 * b - 1.5, torch.full_like(a, -1.0)], 1)
    pln_n = torch.zeros_like(pln)
    pln_n[:, 2] = 1.0
    pts = torch.where(kind == 0, ctr[0] + r[0] * sph, torch.where(kind == 1, ctr[1] + r[1] * sph, torch.where(
        kind == 2, ctr[2] + tor, torch.where(kind == 3, ctr[3] + bx, pln))))
    nv = torch.where(kind <= 1, sph, torch.where(kind == 2, tor_n, torch.where(kind == 3, box_n, pln_n)))
    mean = pts + 0.005 * _nrm(g, n, 3)
    st = torch.exp(math.log(0.01) + 0.3 * _nrm(g, n, 2))
    scale = torch.cat([st, 0.1 * (st[:, :1] * st[:, 1:]).sqrt()], 1)
    # local z onto the normal, then a random twist about it
    w = (1 + nv[:, 2]).clamp(min=1e-9)
    flip = nv[:, 2] < -0.999999
    q0 = _unit(torch.stack([w, -nv[:, 1], nv[:, 0], torch.zeros_like(w)], 1))
    q0 = torch.where(flip[:, None], torch.tensor([0.0, 1.0, 0.0, 0.0], device=DEV, dtype=torch.float64), q0)
    psi = math.pi * _u(g, n)
    cz, sz = torch.cos(psi), torch.sin(psi)
    quat = torch.stack([q0[:, 0] * cz - q0[:, 3] * sz, q0[:, 1] * cz + q0[:, 2] * sz, q0[:, 2] * cz - q0[:, 1] * sz,
                        q0[:, 0] * sz + q0[:, 3] * cz], 1)
    opacity = _u(g, n) ** 0.2
    return _scene_dict(mean, scale, quat, opacity, normal=_unit(nv).float().contiguous(), centres=ctr, radii=r)


def _scene(case, seed, n=None):
    n = case["n"] if n is None else n
    sc = _object(n, seed) if case["scene"] == "object" else _uniform(n, seed)
    if "normal" not in sc:
        sc["normal"] = _unit(_nrm(_gen(seed + 1), n, 3)).float().contiguous()
    return sc


def _sphere_dirs(k, seed):
    """The Fibonacci directions under a seeded rotation."""
    i = np.arange(k)
    z = 1 - (2 * i + 1) / k
    rr = np.sqrt(np.maximum(0, 1 - z * z))
    phi = i * math.pi * (3 - math.sqrt(5))
    d = np.stack([rr * np.cos(phi), rr * np.sin(phi), z], 1)
    q, _ = np.linalg.qr(np.random.default_rng(int(seed)).standard_normal((3, 3)))
    d = d @ q.T
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return torch.from_numpy(d.astype(np.float32)).to(DEV)


def _hemi_dirs(k):
    i = np.arange(k)
    z = 1 - (i + 0.5) / k
    rr = np.sqrt(np.maximum(0, 1 - z * z))
    phi = i * math.pi * (3 - math.sqrt(5))
    return torch.from_numpy(np.stack([rr * np.cos(phi), rr * np.sin(phi), z], 1).astype(np.float32)).to(DEV)


def _envmap(seed, h=32, w=64):
    """A log-normal (sigma 1.5) equirectangular map for importance sampling."""
    rad = np.exp(1.5 * np.random.default_rng(int(seed)).standard_normal((h, w)))
    th, ph = np.arange(h + 1) * math.pi / h, np.arange(w + 1) * 2 * math.pi / w
    st, ct = np.sin(th)[:, None], np.cos(th)[:, None]
    corners = np.stack([st * np.cos(ph), st * np.sin(ph), np.broadcast_to(ct, (h + 1, w + 1))], 2).astype(np.float32)
    z = np.cos(th)
    return rt.rt_envmap_create(rad, (z[:-1] - z[1:])[:, None] * np.full((1, w), 2 * math.pi / w), corners)


def _build(sc, prm=None):
    return rt.rt_build_bvh(sc["mean"], sc["scale"], sc["quat"], sc["opacity"], prm)


def _mlp_params(seed):
    """He-uniform weights, zero biases, in the parameter block's order."""
    g = _gen(seed)

    def mat(o, i):
        return ((2 * _u(g, o, i) - 1) * math.sqrt(6.0 / i)).flatten()

    z = torch.zeros(128, device=DEV, dtype=torch.float64)
    p = torch.cat([mat(128, 80), z, mat(128, 128), z, mat(128, 128), z, mat(128, 128), z,
                   (2 * _u(g, 128) - 1) * math.sqrt(1 / 128), z[:1]])
    return p.float().contiguous()


def _sphere_visibility(sc, dirs):
    """Whether each Gaussian's ray misses the scene's two spheres and the
    ground: a smooth stand-in for traced visibility, as training targets."""
    m, d = sc["mean"].double(), dirs.double()
    vis = torch.ones(m.shape[0], d.shape[0], device=DEV, dtype=torch.float64)
    for c, r in zip(sc["centres"][:2], sc["radii"]):
        oc = m - c
        b = oc @ d.T
        near = (oc * oc).sum(1, keepdim=True) - b * b < r * r
        vis = torch.where(near & (b < -0.05), torch.zeros_like(vis), vis)
    down = ((m[:, 2:] + 1.0) + 0.02 > 0) & (d[:, 2] < -0.05)
    return torch.where(down, torch.zeros_like(vis), vis).float().contiguous()


def prepare(case, seed):
    op = case["op"]
    s = {"case": case, "op": op}
    if op in ("precompute", "adjoint"):
        sc = _scene(case, seed)
        s.update(sc=sc, dirs=_sphere_dirs(case["k"], seed))
        if op == "adjoint":
            s["prm"] = rt.params(t_min=case["t_min"], deterministic=case["deterministic"])
            s["leaves"] = [sc[k].clone().requires_grad_(True) for k in ("mean", "scale", "quat", "opacity")]
            s["w"] = _u(_gen(seed + 2), case["n"], case["k"]).float()
    elif op in ("dirs", "hemi", "env"):
        sc = _scene(case, seed)
        s["bvh"] = _build(sc)
        if op == "dirs":
            s["dirs"] = _sphere_dirs(case["k"], seed)
        elif op == "hemi":
            s["rs"] = rt.rayspec(rt.RT_RAYS_HEMI, dirs=_hemi_dirs(case["k"]), normals=sc["normal"])
        else:
            s["rs"] = rt.rayspec(rt.RT_RAYS_ENV, env=_envmap(seed), n_samples=case["k"], seed=int(seed) + 7)
    elif op == "shade":
        s.update(_shade_inputs(case, seed))
        s["bvh"] = _build(s["sc"])
        s["rs"] = rt.rayspec(rt.RT_RAYS_HEMI, dirs=s["hemi"], normals=s["sc"]["normal"])
        s["in"] = rt.pbr_inputs(s["albedo"], s["rough"], s["env"], s["cam"], sh=s["sh"])
    elif op == "rays":
        sc = _scene(case, seed)
        s["bvh"] = _build(sc)
        o, d, src = _light_rays(case, sc, seed)
        s["rs"] = rt.rayspec(rt.RT_RAYS_EXPLICIT, ray_o=o, ray_d=d, ray_src=src)
    elif op == "batch":
        env = _envmap(seed)
        jobs, s["bvhs"], s["outs"] = [], [], []
        for j, (n, side, off) in enumerate(_batch_scenes(case, seed)):
            bvh = _build(_uniform(n, seed + 10 + j, side, off))
            for rs, m in ((rt.rayspec(rt.RT_RAYS_DIRS, dirs=_sphere_dirs(case["k"], seed + j)), case["k"]),
                          (rt.rayspec(rt.RT_RAYS_ENV, env=env, n_samples=case["s"], seed=int(seed) + j), case["s"])):
                out = torch.empty(n * m, dtype=torch.float32, device=DEV)
                jobs.append((bvh, rs, out))
                s["outs"].append(out)
            s["bvhs"].append(bvh)
        s["batch"] = rt.rt_batch_create(jobs, autotune=True)
    elif op == "infer":
        sc = _scene(case, seed)
        s["bvh"] = _build(sc)
        sur = rt.rt_surrogate_create(rt.mlp_cfg(batch=65536, pos_weight=4.0), seed=int(seed) + 3)
        dirs = _sphere_dirs(case["k"], seed)
        rt.rt_surrogate_train(sur, s["bvh"], rt.rayspec(rt.RT_RAYS_DIRS, dirs=dirs), _sphere_visibility(sc, dirs),
                              200, seed=int(seed) + 4)
        # held-out directions, one id drawn from each of `rays` equal strata
        total, m = case["n"] * case["k"], case["rays"]
        edge = torch.arange(m + 1, device=DEV, dtype=torch.int64) * total // m
        width = edge[1:] - edge[:-1]
        ids = edge[:-1] + torch.minimum((_u(_gen(seed + 5), m) * width).long(), width - 1)
        s["sur"] = sur
        s["rs"] = rt.rayspec(rt.RT_RAYS_DIRS, dirs=_sphere_dirs(case["k"], seed + 6), ray_ids=ids)
        s["count"] = torch.zeros(1, dtype=torch.int64, device=DEV)
    else:  # mlp_grad
        s["sur"] = rt.rt_surrogate_create(rt.mlp_cfg(pos_weight=4.0), seed=1)
        s["pos"], s["dir"], s["y"], params = _mlp_samples(case, seed)
        rt.rt_surrogate_set_params(s["sur"], params)
    return s


def _batch_scenes(case, seed):
    h = np.random.default_rng(int(seed))
    return [(int(case["n"] * case["growth"] ** j), h.uniform(1.5, 2.5), tuple(h.uniform(-4, 4, 3)))
            for j in range(case["n_jobs"])]


def _light_rays(case, sc, seed):
    """From random Gaussians towards four point lights, skipping the source."""
    g = _gen(seed + 3)
    src = torch.randint(0, case["n"], (case["rays"],), generator=g, device=DEV, dtype=torch.int32)
    light = _unit(_nrm(g, 4, 3)) * 3.0
    to = light[torch.randint(0, 4, (case["rays"],), generator=g, device=DEV)]
    m = sc["mean"][src.long()]
    d = _unit(to - m.double()).float().contiguous()
    return (m + 1e-4 * d).contiguous(), d, src


def _shade_inputs(case, seed):
    sc = _scene(case, seed)
    g = _gen(seed + 2)
    n, k, h = case["n"], case["k"], case["env_h"]
    sh = None
    if case["sh"]:
        sh = 0.1 * _nrm(g, n, 9, 3)
        sh[:, 0] = 0.5 * _u(g, n, 3)
        sh = sh.float().contiguous()
    # visibility of a dense surface: mostly occluded, the rest spread over (0, 1)
    V = torch.where(_u(g, n, k) < 0.7, 0.0, _u(g, n, k)).float().contiguous()
    return {"sc": sc, "hemi": _hemi_dirs(k), "albedo": _u(g, n, 3).float().contiguous(),
            "rough": _u(g, n).float().contiguous(), "sh": sh, "V": V,
            "env": torch.exp(_nrm(g, h, 2 * h, 3)).float().contiguous(), "cam": (1.0, 3.0, 2.5)}


def _mlp_samples(case, seed):
    g = _gen(seed)
    m = case["rays"]
    pos = (2 * _u(g, m, 3) - 1).float().contiguous()
    d = _unit(_nrm(g, m, 3)).float().contiguous()
    y = torch.where(_u(g, m) < 0.6, 0.0, _u(g, m)).float().contiguous()
    return pos, d, y, _mlp_params(seed + 1)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(s):
    op = s["op"]
    if op == "precompute":
        bvh = _build(s["sc"])
        T = rt.rt_trace_visibility_dirs(bvh, s["dirs"])
        bvh.destroy()
        return T
    if op == "dirs":
        return rt.rt_trace_visibility_dirs(s["bvh"], s["dirs"])
    if op in ("hemi", "env", "rays"):
        return rt.rt_trace_visibility(s["bvh"], s["rs"])
    if op == "shade":
        return rt.rt_pbr_shade(s["bvh"], s["rs"], s["in"], V=s["V"])
    if op == "adjoint":
        T = autograd.visibility(*s["leaves"], s["dirs"], s["prm"])
        return [T, *torch.autograd.grad(T, s["leaves"], s["w"])]
    if op == "batch":
        s["batch"].run()
        return s["outs"]
    if op == "infer":
        return [rt.rt_surrogate_infer(s["sur"], s["bvh"], s["rs"], s["case"]["band"], n_fallback=s["count"]),
                s["count"]]
    return rt.rt_surrogate_loss_grad(s["sur"], s["pos"], s["dir"], s["y"])


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    op, n = case["op"], case["n"]
    hit_flops = 60  # one accepted Gaussian: peak, distance, response, product
    # accepted hits per ray (measured with the library's counters, rounded)
    per_ray = 30.0 if case["scene"] == "object" else min(80.0, 4e-4 * n)
    scene = 44.0 * n
    if op in ("precompute", "dirs", "hemi", "env"):
        rays = n * case["k"]
        return {"bytes": scene + 4.0 * rays, "flops": rays * per_ray * hit_flops}
    if op == "shade":
        terms = n * case["k"]
        return {"bytes": 4.0 * terms + n * (12 + 12 + 4 + 12 + 12 + (108 if case["sh"] else 0)),
                "flops": terms * (150 if case["sh"] else 100)}
    if op == "rays":
        return {"bytes": scene + 32.0 * case["rays"], "flops": case["rays"] * per_ray * hit_flops}
    if op == "adjoint":
        rays = n * case["k"]
        return {"bytes": 2 * scene + 8.0 * rays, "flops": rays * per_ray * (hit_flops + 150)}
    if op == "batch":
        ns = [int(n * case["growth"] ** j) for j in range(case["n_jobs"])]
        rays = sum(ns) * (case["k"] + case["s"])
        return {"bytes": 44.0 * sum(ns) + 4.0 * rays,
                "flops": sum(m * (case["k"] + case["s"]) * min(80.0, 4e-4 * m) * hit_flops for m in ns)}
    if op == "infer":
        return {"bytes": 16.0 * n + 12.0 * case["rays"] + 240e3, "flops": 118_528.0 * case["rays"]}
    return {"bytes": 28.0 * case["rays"] + 480e3, "flops": 3 * 118_528.0 * case["rays"]}


# ---------------------------------------------------------------------------
# float64 values by plain torch
# ---------------------------------------------------------------------------
MAX_PAIRS = 6e9


def exact(case, seed):
    op = case["op"]
    if op in ("precompute", "dirs", "hemi"):
        if float(case["n"]) ** 2 * case["k"] > MAX_PAIRS:
            return None
        sc = _scene(case, seed)
        o, d, src = _implicit_rays(case, sc, seed)
        T = _brute(sc, o, d, src, 1e-4)
        return T if op == "hemi" else T.view(case["n"], case["k"])
    if op == "rays":
        if float(case["n"]) * case["rays"] > MAX_PAIRS:
            return None
        sc = _scene(case, seed)
        o, d, src = _light_rays(case, sc, seed)
        return _brute(sc, o.double(), d.double(), src.long(), 1e-4)
    if op == "adjoint":
        if float(case["n"]) ** 2 * case["k"] > MAX_PAIRS / 5:
            return None
        return _brute_adjoint(case, seed)
    if op == "shade":
        return _shade64(_shade_inputs(case, seed))
    if op == "mlp_grad":
        return _mlp64(case, seed)
    return None


def _implicit_rays(case, sc, seed):
    """The float32 rays of a direction or hemisphere set, as float64."""
    n, k = case["n"], case["k"]
    if case["op"] == "hemi":
        nv = sc["normal"]
        x, y, z = nv.unbind(1)
        ln = torch.sqrt(x * x + y * y + z * z)
        x, y, z = x / ln, y / ln, z / ln
        sg = torch.copysign(torch.ones_like(z), z)
        a = -1.0 / (sg + z)
        b = x * y * a
        t1 = torch.stack([1.0 + sg * x * x * a, sg * b, -(sg * x)], 1)
        t2 = torch.stack([b, sg + y * y * a, -y], 1)
        nn = torch.stack([x, y, z], 1)
        hd = _hemi_dirs(k)
        d = (hd[None, :, 0:1] * t1[:, None] + hd[None, :, 1:2] * t2[:, None]) + hd[None, :, 2:3] * nn[:, None]
    else:
        d = _sphere_dirs(k, seed)[None].expand(n, k, 3)
    o = sc["mean"][:, None] + 1e-4 * d
    src = torch.arange(n, device=DEV).repeat_interleave(k)
    return o.reshape(-1, 3).double(), d.reshape(-1, 3).double(), src


def _whitening(scale, quat):
    q = quat / quat.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    return R.transpose(1, 2) / scale[:, :, None]


def _pair_T(mean, W, opacity, o, d, src, ids):
    """prod (1 - alpha) of each ray over all Gaussians (Eq. 13-15)."""
    e = [o[:, None, c] - mean[None, :, c] for c in range(3)]
    uo = [W[None, :, k, 0] * e[0] + W[None, :, k, 1] * e[1] + W[None, :, k, 2] * e[2] for k in range(3)]
    ud = [d[:, 0:1] * W[None, :, k, 0] + d[:, 1:2] * W[None, :, k, 1] + d[:, 2:3] * W[None, :, k, 2] for k in range(3)]
    dd = ud[0] * ud[0] + ud[1] * ud[1] + ud[2] * ud[2]
    t = -(uo[0] * ud[0] + uo[1] * ud[1] + uo[2] * ud[2]) / dd
    m2 = sum((uo[k] + t * ud[k]) ** 2 for k in range(3))
    alpha = opacity[None] * torch.exp(-0.5 * m2)
    ok = (t > 0) & (m2 <= 9.0) & (alpha >= ALPHA_MIN) & (ids[None] != src[:, None])
    return torch.exp(torch.log1p(-torch.where(ok, alpha, torch.zeros_like(alpha))).sum(1))


def _brute(sc, o, d, src, t_min):
    mean, W, op = sc["mean"].double(), _whitening(sc["scale"].double(), sc["quat"].double()), sc["opacity"].double()
    ids = torch.arange(mean.shape[0], device=DEV)
    step = max(1, int(3e7 // mean.shape[0]))
    T = torch.cat([_pair_T(mean, W, op, o[i:i + step], d[i:i + step], src[i:i + step], ids)
                   for i in range(0, o.shape[0], step)])
    return torch.where(T < t_min, torch.zeros_like(T), T)


def _brute_adjoint(case, seed):
    sc = _scene(case, seed)
    n, k = case["n"], case["k"]
    leaves = [sc[x].double().requires_grad_(True) for x in ("mean", "scale", "quat", "opacity")]
    mean, scale, quat, op = leaves
    d32 = _sphere_dirs(k, seed)
    w = _u(_gen(seed + 2), n, k).float().double()
    ids = torch.arange(n, device=DEV)
    step = max(1, int(4e6 // (n * k)))
    grads = [torch.zeros_like(x) for x in leaves]
    Ts = []
    for i in range(0, n, step):
        o32 = (sc["mean"][i:i + step, None] + 1e-4 * d32[None]).double()
        mi = mean[i:i + step, None]
        o = (mi + (o32 - mi).detach()).reshape(-1, 3)
        d = d32.double()[None].expand(o32.shape).reshape(-1, 3)
        src = ids[i:i + step].repeat_interleave(k)
        T = _pair_T(mean, _whitening(scale, quat), op, o, d, src, ids)
        T = torch.where(T < case["t_min"], torch.zeros_like(T), T)
        for a, g in zip(grads, torch.autograd.grad((T * w[i:i + step].reshape(-1)).sum(), leaves)):
            a += g
        Ts.append(T.detach())
    return [torch.cat(Ts).view(n, k), *grads]


def _shade64(s):
    sc = s["sc"]
    n, k = s["V"].shape
    nn = _unit(sc["normal"].double())
    x, y, z = nn.unbind(1)
    sg = torch.copysign(torch.ones_like(z), z)
    a = -1.0 / (sg + z)
    b = x * y * a
    t1 = torch.stack([1 + sg * x * x * a, sg * b, -sg * x], 1)
    t2 = torch.stack([b, sg + y * y * a, -y], 1)
    wo = _unit(torch.tensor([s["cam"]], device=DEV, dtype=torch.float64) - sc["mean"].double())
    r = s["rough"].double().clamp(0.04, 1.0)
    a2 = r ** 4
    kk = (r + 1) ** 2 / 8
    nv = (nn * wo).sum(1).clamp(min=0)
    env = s["env"].double()
    h, w = env.shape[:2]
    acc = torch.zeros(n, 3, device=DEV, dtype=torch.float64)
    hd = s["hemi"].double()
    for j in range(k):
        wi = hd[j, 0] * t1 + hd[j, 1] * t2 + hd[j, 2] * nn
        nl = (nn * wi).sum(1).clamp(min=0)
        hv = _unit(wi + wo)
        nh, vh = (nn * hv).sum(1), (wo * hv).sum(1).clamp(min=0)
        q = torch.linalg.cross(nn, hv).square().sum(1) + nh * nh * a2
        fs = 0.25 * a2 / (math.pi * q * q) * (0.04 + 0.96 * (1 - vh) ** 5) / (nl * (1 - kk) + kk) / (nv * (1 - kk) + kk)
        vv = torch.acos(wi[:, 2].clamp(-1, 1)) / math.pi * h - 0.5
        ph = torch.atan2(wi[:, 1], wi[:, 0])
        uu = torch.where(ph < 0, ph + 2 * math.pi, ph) / (2 * math.pi) * w - 0.5
        fv, fu = vv.floor(), uu.floor()
        bv, bu = (vv - fv)[:, None], (uu - fu)[:, None]
        i0, i1 = fv.long().clamp(0, h - 1), (fv.long() + 1).clamp(0, h - 1)
        j0, j1 = fu.long() % w, (fu.long() + 1) % w
        Ld = (env[i0, j0] * (1 - bu) + env[i0, j1] * bu) * (1 - bv) + (env[i1, j0] * (1 - bu) + env[i1, j1] * bu) * bv
        Li = torch.zeros_like(Ld)
        if s["sh"] is not None:
            X, Y, Z = wi.unbind(1)
            basis = torch.stack([torch.full_like(X, 0.282094791773878), -0.488602511902920 * Y, 0.488602511902920 * Z,
                                 -0.488602511902920 * X, 1.092548430592079 * X * Y, -1.092548430592079 * Y * Z,
                                 0.315391565252520 * (2 * Z * Z - X * X - Y * Y), -1.092548430592079 * X * Z,
                                 0.546274215296040 * (X * X - Y * Y)], 1)
            Li = (s["sh"].double() * basis[:, :, None]).sum(1).clamp(min=0)
        acc += (s["albedo"].double() / math.pi + fs[:, None]) * (s["V"][:, j:j + 1].double() * Ld + Li) * nl[:, None]
    return acc * (2 * math.pi / k)


def _mlp64(case, seed):
    """The weighted loss and its gradient without the 16-bit roundings."""
    pos, d, y, p32 = _mlp_samples(case, seed)
    p = p32.double().requires_grad_(True)
    at, mats = 0, []
    for o, i in ((128, 80), (128, 128), (128, 128), (128, 128)):
        mats.append((p[at:at + o * i].view(o, i), p[at + o * i:at + o * i + o]))
        at += o * i + o
    w5, b5 = p[at:at + 128], p[at + 128]
    m, total, grad = case["rays"], 0.0, torch.zeros_like(p)
    for i in range(0, m, 65536):
        x = torch.cat([pos[i:i + 65536], d[i:i + 65536]], 1).double()
        f = []
        for c in range(6):
            f.append(x[:, c])
            for k in range(6):
                f += [torch.sin(2.0 ** k * math.pi * x[:, c]), torch.cos(2.0 ** k * math.pi * x[:, c])]
        a = torch.stack(f + [torch.zeros_like(f[0])] * 2, 1)
        for W, b in mats:
            a = torch.relu(a @ W.T + b)
        z, t = a @ w5 + b5, y[i:i + 65536].double()
        loss = (4.0 * t * torch.nn.functional.softplus(-z) + (1 - t) * torch.nn.functional.softplus(z)).sum() / m
        grad += torch.autograd.grad(loss, p)[0]
        total += float(loss.detach())
    return [torch.tensor([total], dtype=torch.float64), grad.detach()]
