"""The workloads this package is used for, as measurable cases.

Three kinds of call, each through the package's public entry points:

* ``frame``  one pinhole view: the hierarchy rebuilt for the current Gaussians
             (unless the scene is static) and ``trace_stochastic``;
* ``fit``    one differentiable rendering and its gradients: rebuild, image,
             L2 loss to a photograph, gradients of every parameter;
* ``views``  the batched form: many views of uneven size over a ground quad
             with point lights, soft shadows and a diffuse bounce.

Sizes follow the repository's own configurations: the 1,000-Gaussian cloud at
64x64, the 1M-Gaussian shell at 1080p with 1, 16 and 64 samples per pixel and
with four hits per traversal, the 3M-Gaussian reduced-precision form, the
16-view batched frame, the 500k-Gaussian fitting step at 800x800 and the
2,000-Gaussian subset its gradients are checked on."""

from __future__ import annotations

import math
import types

import numpy as np
import torch

PARAMS = ("means", "log_scales", "quats", "opacity_logits", "sh")
BG = (0.05, 0.1, 0.2)


# ------------------------------------------------------------------ the cases


def _frame(name, cloud, m, width, height, spp, n_hits=1, degree=3, sh="float32", nodes="binary",
           rebuild=True, hits=False):
    c = dict(kind="frame", cloud=cloud, m=m, width=width, height=height, spp=spp, n_hits=n_hits,
             degree=degree, sh=sh, nodes=nodes, rebuild=rebuild, hits=hits)
    return dict(c, name=name) if name else c


def _fit(name, cloud, m, width, height, spp, degree=3):
    c = dict(kind="fit", cloud=cloud, m=m, width=width, height=height, spp=spp, degree=degree)
    return dict(c, name=name) if name else c


def _views(name, m, views, min_width, min_height, max_width, max_height, spp, lights, graph,
           degree=3, sh="float32"):
    c = dict(kind="views", cloud="shell", m=m, views=views, min_width=min_width,
             min_height=min_height, max_width=max_width, max_height=max_height, spp=spp,
             lights=lights, graph=graph, degree=degree, sh=sh)
    return dict(c, name=name) if name else c


def listed():
    return [
        # an interactive thumbnail of a small moving cloud: latency and launches
        _frame("tiny-64", "tiny", 1000, 64, 64, 1, degree=0),
        # picking in a static object of the smallest reconstructed size: a ragged
        # view with every sample's hit id and depth, two hits per traversal,
        # bfloat16 colours
        _frame("pick-90k", "shell", 90_000, 411, 307, 5, n_hits=2, degree=2, sh="bfloat16",
               rebuild=False, hits=True),
        # a moving 1M-Gaussian scene at full HD: preview, ordinary and final quality
        _frame("hd-1m-spp1", "shell", 1_000_000, 1920, 1080, 1),
        _frame("hd-1m-spp16", "shell", 1_000_000, 1920, 1080, 16),
        _frame("hd-1m-spp64", "shell", 1_000_000, 1920, 1080, 64),
        # the same number of samples as four hits of sixteen traversals
        _frame("hd-1m-n4-spp16", "shell", 1_000_000, 1920, 1080, 16, n_hits=4),
        # the reduced-precision form of a large scene
        _frame("hd-3m-f16-q8", "shell", 3_000_000, 1920, 1080, 64, sh="float16",
               nodes="binary_q8"),
        # gradients of a small subset, as they are checked before a long run
        _fit("fit-2k", "shell", 2000, 96, 72, 16),
        # one view of a fitting step, at the cheap sampling rate
        _fit("fit-500k", "shell", 500_000, 800, 800, 4),
        # one full-HD view of a large fitting step
        _fit("fit-1m-hd", "shell", 1_000_000, 1920, 1080, 16),
        # a few small previews of a lit scene
        _views("views-2", 5000, 2, 96, 72, 160, 120, 4, 2, False),
        # the batched frame: 16 views up to full HD, captured once, replayed per frame
        _views("views-16", 1_000_000, 16, 256, 256, 1920, 1080, 16, 4, True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("frame", "frame", "frame", "fit", "views"))
    if kind == "frame":
        m = _log_int(rng, 1000, 3_000_000)
        return _frame(None, "tiny" if m < 5000 else "shell", m, _log_int(rng, 64, 1920),
                      _log_int(rng, 64, 1080), _log_int(rng, 1, 64),
                      n_hits=rng.choice((1, 1, 1, 2, 4)), degree=rng.choice((3, 3, 0, 1, 2)),
                      sh=rng.choice(("float32", "float32", "float16", "bfloat16")),
                      nodes=rng.choice(("binary", "binary", "binary", "binary_q8", "wide4",
                                        "wide4_q8")),
                      rebuild=rng.random() < 0.7, hits=rng.random() < 0.2)
    if kind == "fit":
        return _fit(None, "shell", _log_int(rng, 2000, 1_000_000), _log_int(rng, 96, 1920),
                    _log_int(rng, 72, 1080), _log_int(rng, 1, 16), degree=rng.choice((3, 3, 1, 0)))
    big = _log_int(rng, 120, 1080)
    return _views(None, _log_int(rng, 5000, 1_000_000), rng.randint(1, 16), 96, 72,
                  big * 16 // 9, big, _log_int(rng, 1, 16), rng.randint(1, 4), rng.random() < 0.5,
                  sh=rng.choice(("float32", "float32", "float16")))


# ------------------------------------------------------------------ inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gaussians(case, seed):
    """Raw parameters: a uniform cloud, or 64 anisotropic clusters on the unit
    sphere (the repository's tiny and shell generators, drawn on the device)."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(int(seed))

    def normal(mean, sd, *shape):
        return torch.empty(shape, device=dev).normal_(mean, sd, generator=gen)

    def uniform(lo, hi, *shape):
        return torch.empty(shape, device=dev).uniform_(lo, hi, generator=gen)

    m, k = case["m"], (case["degree"] + 1) ** 2
    p = {"quats": normal(0.0, 1.0, m, 4)}
    if case["cloud"] == "tiny":
        p["means"] = uniform(-1.0, 1.0, m, 3)
        p["log_scales"] = normal(-3.0, 0.5, m, 3)
        p["opacity_logits"] = normal(0.0, 1.5, m)
    else:
        centres = normal(0.0, 1.0, 64, 3)
        centres /= centres.norm(dim=1, keepdim=True)
        which = torch.randint(0, 64, (m,), device=dev, generator=gen)
        p["means"] = centres[which] + normal(0.0, 0.05, m, 3)
        p["log_scales"] = normal(-4.5, 0.6, m, 3)
        p["opacity_logits"] = normal(0.0, 2.0, m)
    p["sh"] = normal(0.0, 0.2, m, k, 3)
    p["sh"][:, 0] = uniform(0.0, 1.0, m, 3)
    p["sh"] = p["sh"].to(getattr(torch, case.get("sh", "float32")))
    return p


def _eye(rng, lo_deg, hi_deg):
    az, el = rng.uniform(0.0, 2 * math.pi), math.radians(rng.uniform(lo_deg, hi_deg))
    v = (3 * math.cos(el) * math.cos(az), 3 * math.sin(el), 3 * math.cos(el) * math.sin(az))
    return tuple(float(np.float32(x)) for x in v)


def _resolutions(case):
    """Uneven resolutions spread over the case's range (the same for every seed)."""
    out = []
    for i in range(case["views"]):
        u, v = (i + 0.5) * 0.6180339887 % 1.0, (i + 0.5) * 0.7548776662 % 1.0
        out.append((round(case["min_width"] + u * (max(case["max_width"], case["min_width"])
                                                   - case["min_width"])),
                    round(case["min_height"] + v * (max(case["max_height"], case["min_height"])
                                                    - case["min_height"]))))
    return out


def _cameras(case, seed):
    """Plain camera descriptions: eyes at distance 3 that look at the origin."""
    rng = np.random.default_rng(int(seed) + 1)
    sizes = _resolutions(case) if case["kind"] == "views" else [(case["width"], case["height"])]
    lo, hi = (15.0, 60.0) if case["kind"] == "views" else (-30.0, 30.0)
    cams, offset = [], 0
    for w, h in sizes:
        cams.append(dict(width=w, height=h, eye=_eye(rng, lo, hi), ray_id_offset=offset))
        offset += w * h
    return cams


def _lights(case, seed):
    """A ground quad below the cloud and point lights above it."""
    rng = np.random.default_rng(int(seed) + 2)
    lights = []
    for _ in range(case["lights"]):
        a = rng.uniform(0.0, 2 * math.pi)
        pos = (2.5 * math.cos(a), rng.uniform(2.0, 3.0), 2.5 * math.sin(a))
        lights.append((tuple(float(np.float32(x)) for x in pos), (4.0, 4.0, 4.0)))
    return types.SimpleNamespace(lights=lights, has_ground=True, ground_y=-1.3,
                                 ground_half_extent=3.0, ground_albedo=(0.5, 0.5, 0.5),
                                 bounce=True, shadow_eps=1e-4)


def _photograph(case, seed):
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(int(seed) + 3)
    return torch.rand((case["height"], case["width"], 3), device=dev, generator=gen) * 0.5


# ------------------------------------------------------------------ the calls


def prepare(case, seed):
    import paper_2504_06598_gb300 as gs

    p = _gaussians(case, seed)
    cams = [gs.Camera(**c) for c in _cameras(case, seed)]
    g = gs.Gaussians(*(p[k] for k in PARAMS), case["degree"])
    bvh = gs.build_bvh(g, node_format=case.get("nodes", "binary"))
    state = dict(gs=gs, case=case, seed=int(seed), g=g, bvh=bvh, cams=cams)
    if case["kind"] == "fit":
        state["params"] = [p[k].requires_grad_(True) for k in PARAMS]
        state["target"] = _photograph(case, seed)
    elif case["kind"] == "views":
        state["extras"] = _lights(case, seed)
        if case["graph"]:
            state["frame"] = gs.FrameGraph(bvh, g, cams, state["extras"], rebuild=True,
                                           seed=int(seed), spp=case["spp"], bg=BG)
    return state


def run(state):
    gs, case, g, bvh = state["gs"], state["case"], state["g"], state["bvh"]
    if case["kind"] == "frame":
        if case["rebuild"]:
            bvh.rebuild(g)
        return gs.trace_stochastic(bvh, g, state["cams"][0], seed=state["seed"], spp=case["spp"],
                                   n_hits=case["n_hits"], bg=BG, want_hits=case["hits"])
    if case["kind"] == "fit":
        rgb = gs.render_differentiable(*state["params"], case["degree"], state["cams"][0],
                                       bvh=bvh, seed=state["seed"], spp=case["spp"], bg=BG)
        loss = ((rgb - state["target"]) ** 2).mean()
        return [rgb.detach(), *torch.autograd.grad(loss, state["params"])]
    if case["graph"]:
        return state["frame"].replay(torch.cuda.current_stream())
    bvh.rebuild(g)
    return gs.render_views(bvh, g, state["cams"], state["extras"], seed=state["seed"],
                           spp=case["spp"], bg=BG)


def work(case):
    """Every parameter read once and every output written once; a ray descends
    the hierarchy once (two boxes a level), evaluates one Gaussian, and each
    sample takes one Philox draw and one colour."""
    m, k = case["m"], 3 * (case["degree"] + 1) ** 2
    sh_bytes = 4 if case.get("sh", "float32") == "float32" else 2
    per_ray = 2 * 24 * math.log2(m + 1) + 110
    if case["kind"] == "views":
        px = sum(w * h for w, h in _resolutions(case))
        rays, samples = px, px * case["spp"]
        return {"bytes": m * (44 + k * sh_bytes) + px * 12, "flops": rays * per_ray + samples * 150}
    px = case["width"] * case["height"]
    samples = px * case["spp"] * case.get("n_hits", 1)
    data = m * (44 + k * sh_bytes) + px * 12
    if case["kind"] == "fit":
        return {"bytes": data + px * 12 + m * (44 + k * 4),
                "flops": 2 * px * per_ray + 2 * samples * 150}
    if case["hits"]:
        data += samples * 8
    return {"bytes": data, "flops": px * per_ray + samples * 150}


# ------------------------------------------------------------------ 64 bits


def _philox(c, key):
    """Philox-4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF

    def mul(a, b):
        p0, p1 = (a & 0xFFFF) * b, (a >> 16) * b
        return (p1 + (p0 >> 16)) >> 16, (p0 + ((p1 & 0xFFFF) << 16)) & mask

    k0, k1 = key & mask, (key >> 32) & mask
    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _normalise32(v):
    n = torch.sqrt(v[..., 0] * v[..., 0] + v[..., 1] * v[..., 1] + v[..., 2] * v[..., 2])
    return v / n[..., None]


def _camera_rays(cam):
    """The float32 rays that the library defines, one rounding per operation."""
    dev = _device()
    eye = torch.tensor(cam["eye"], dtype=torch.float32, device=dev)
    up = torch.tensor((0.0, 1.0, 0.0), device=dev)

    def cross(a, b):
        return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2],
                            a[0] * b[1] - a[1] * b[0]])

    f = _normalise32(-eye)
    r = _normalise32(cross(f, up))
    u = cross(r, f)
    th = torch.tensor(math.tan(60.0 * math.pi / 360.0), dtype=torch.float32, device=dev)
    w, h = cam["width"], cam["height"]
    s = th / torch.tensor(float(h), device=dev)
    x = torch.arange(w, device=dev).repeat(h)
    y = torch.arange(h, device=dev).repeat_interleave(w)
    ux, uy = (2 * x + 1 - w).float() * s, (h - 1 - 2 * y).float() * s
    d = _normalise32((f + ux[:, None] * r) + uy[:, None] * u)
    return eye.expand(w * h, 3), d, cam["ray_id_offset"] + torch.arange(w * h, device=dev)


def _transforms(p):
    """Means, M = S^-1 R^T and opacities in 64 bits (Eq. 1)."""
    q = p["quats"].double()
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                       2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                       2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                      1).reshape(-1, 3, 3)
    mat = rot.transpose(1, 2) * torch.exp(-p["log_scales"].double())[:, :, None]
    return p["means"].double(), mat, torch.sigmoid(p["opacity_logits"].double())


def _pair(tr, o, d, gid):
    """Depth and alpha of listed (ray, Gaussian) pairs."""
    mu, mat, opacity = tr
    v = torch.einsum("pij,pj->pi", mat[gid], o - mu[gid])
    md = torch.einsum("pij,pj->pi", mat[gid], d)
    t = -(v * md).sum(1) / (md * md).sum(1)
    q = ((v + t[:, None] * md) ** 2).sum(1)
    return t, opacity[gid] * torch.exp(-0.5 * q)


def _candidates(tr, o, d, t_min=0.0, t_max=None):
    """Every (ray, Gaussian) whose 1D mean is in range and inside the bounding
    ellipsoid (q <= 8), as index lists: brute force over all pairs."""
    mu, mat, _ = tr
    m = mu.shape[0]
    at_mu = torch.einsum("mij,mj->mi", mat, mu)
    rays, gids = [], []
    step = max(1, 20_000_000 // m)
    flat = mat.reshape(3 * m, 3).T.contiguous()
    for b in range(0, o.shape[0], step):
        od, dd = o[b:b + step].double(), d[b:b + step].double()
        md = (dd @ flat).reshape(-1, m, 3)
        mv = (od @ flat).reshape(-1, m, 3) - at_mu
        aa, ab, bb = (md * md).sum(2), (mv * md).sum(2), (mv * mv).sum(2)
        t = -ab / aa
        ok = (t > t_min) & (bb - ab * ab / aa <= 8.0)
        if t_max is not None:
            ok &= t < t_max[b:b + step, None].double()
        i, j = ok.nonzero(as_tuple=True)
        rays.append(i + b)
        gids.append(j)
    return torch.cat(rays), torch.cat(gids)


def _accepted(cand, ray_id, sample, tag, seed):
    """Which candidates sample `sample` of their ray accepts (xi < alpha)."""
    ray, gid, _, alpha = cand
    rid = ray_id[ray]
    u = _philox([rid, gid, torch.full_like(rid, sample >> 2), torch.full_like(rid, tag)], seed)
    return (u[sample & 3] >> 8).double() * 2.0 ** -24 < alpha


def _closest(cand, acc, n):
    """Per ray the depth (inf if none) and the id (-1) of the closest accepted hit."""
    ray, gid, t, _ = cand
    dev = t.device
    best = torch.full((n,), math.inf, dtype=torch.float64, device=dev)
    best.scatter_reduce_(0, ray[acc], t[acc], "amin")
    win = acc & (t == best[ray])
    ids = torch.full((n,), 1 << 40, dtype=torch.int64, device=dev)
    ids.scatter_reduce_(0, ray[win], gid[win], "amin")
    return best, torch.where(ids == 1 << 40, -1, ids)


def _sh(deg, d):
    """Real spherical harmonics with the Condon-Shortley phase; the DC term is 1."""
    x, y, z = d.double().unbind(-1)
    out = [torch.ones_like(x)]
    if deg >= 1:
        c = math.sqrt(3 / (4 * math.pi))
        out += [-c * y, c * z, -c * x]
    if deg >= 2:
        c, e = math.sqrt(15 / (4 * math.pi)), math.sqrt(5 / (16 * math.pi))
        out += [c * x * y, -c * y * z, e * (3 * z * z - 1), -c * x * z, c / 2 * (x * x - y * y)]
    if deg >= 3:
        a, b = math.sqrt(35 / (32 * math.pi)), math.sqrt(105 / (4 * math.pi))
        c, e = math.sqrt(21 / (32 * math.pi)), math.sqrt(7 / (16 * math.pi))
        out += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (5 * z * z - 1),
                e * z * (5 * z * z - 3), -c * x * (5 * z * z - 1), b / 2 * z * (x * x - y * y),
                -a * x * (x * x - 3 * y * y)]
    return torch.stack(out, -1)


def _colour(p, deg, d, ids, bg):
    """Colour of hit `ids` seen along d, the background where there is none."""
    c = torch.einsum("rk,rkc->rc", _sh(deg, d), p["sh"][ids.clamp(min=0)].double()).clamp(min=0.0)
    return torch.where((ids >= 0)[:, None], c, bg)


def _all(tr, o, d, t_min=0.0, t_max=None):
    ray, gid = _candidates(tr, o, d, t_min, t_max)
    t, alpha = _pair(tr, o[ray].double(), d[ray].double(), gid)
    return ray, gid, t, alpha


def _exact_frame(case, seed, p, bg):
    o, d, rid = _camera_rays(_cameras(case, seed)[0])
    cand = _all(_transforms(p), o, d)
    rgb, depth = 0.0, []
    total = case["spp"] * case["n_hits"]
    for s in range(total):
        t, ids = _closest(cand, _accepted(cand, rid, s, 0, seed), o.shape[0])
        rgb = rgb + _colour(p, case["degree"], d, ids, bg) / total
        depth.append(t)
    rgb = rgb.reshape(case["height"], case["width"], 3)
    if not case["hits"]:
        return rgb
    return rgb, None, torch.stack(depth).reshape(case["spp"], case["n_hits"], case["height"],
                                                 case["width"])


def _exact_fit(case, seed, p, bg):
    """The estimator's gradient: dL/dc of each sample's hit k, and
    dL/dalpha_i = g . (c_i - c_k) / (1 - alpha_i) for every valid Gaussian i in
    front of it; alpha and the colours are differentiated by autograd."""
    o, d, rid = _camera_rays(_cameras(case, seed)[0])
    cand = _all(_transforms(p), o, d)
    ray, gid, t, alpha = cand
    n, spp = o.shape[0], case["spp"]
    wins, rgb = [], 0.0
    for s in range(spp):
        wins.append(_closest(cand, _accepted(cand, rid, s, 0, seed), n))
        rgb = rgb + _colour(p, case["degree"], d, wins[-1][1], bg) / spp
    g = 2.0 * (rgb - _photograph(case, seed).double().reshape(-1, 3)) / (3 * n) / spp
    c_i = _colour(p, case["degree"], d[ray], gid, bg)
    weight = torch.zeros_like(alpha)
    leaf = {k: p[k].double().requires_grad_(True) for k in PARAMS}
    total = 0.0
    for tk, ids in wins:
        c_k = _colour(p, case["degree"], d, ids, bg)
        front = t < tk[ray]
        weight += torch.where(front, (g[ray] * (c_i - c_k[ray])).sum(1), 0.0)
        total = total + (g * _colour(leaf, case["degree"], d, ids, bg)).sum()
    _, alpha_leaf = _pair(_transforms(leaf), o[ray].double(), d[ray].double(), gid)
    total = total + (weight / (1.0 - alpha) * alpha_leaf).sum()
    return [rgb.reshape(case["height"], case["width"], 3),
            *torch.autograd.grad(total, [leaf[k] for k in PARAMS])]


def _bounce_dirs(rid, s, seed):
    """normalise((0, 1, 0) + u), u uniform on the sphere by rejection, in float32."""
    u = torch.zeros((rid.shape[0], 3), device=rid.device)
    u[:, 1] = 1.0
    done = torch.zeros_like(rid, dtype=torch.bool)
    for attempt in range(16):
        w = _philox([rid, torch.full_like(rid, attempt), s, torch.full_like(rid, 16)], seed)
        v = torch.stack([2.0 * ((w[i] >> 8).float() * 2.0 ** -24) - 1.0 for i in range(3)], 1)
        r2 = v[:, 0] * v[:, 0] + v[:, 1] * v[:, 1] + v[:, 2] * v[:, 2]
        take = ~done & (r2 > 1e-8) & (r2 <= 1.0)
        u = torch.where(take[:, None], v / torch.sqrt(r2)[:, None], u)
        done |= take
    b = torch.stack([u[:, 0], 1.0 + u[:, 1], u[:, 2]], 1)
    n2 = b[:, 0] * b[:, 0] + b[:, 1] * b[:, 1] + b[:, 2] * b[:, 2]
    up = torch.tensor((0.0, 1.0, 0.0), device=rid.device)
    return torch.where((n2 > 1e-12)[:, None], b / torch.sqrt(n2)[:, None], up)


def _exact_views(case, seed, p, bg):
    ex, tr, deg, spp = _lights(case, seed), _transforms(p), case["degree"], case["spp"]
    albedo = torch.tensor(ex.ground_albedo, dtype=torch.float64, device=bg.device)
    out = []
    for cam in _cameras(case, seed):
        o, d, rid = _camera_rays(cam)
        n = o.shape[0]
        cand = _all(tr, o, d)
        tq = (torch.tensor(ex.ground_y, device=o.device) - o[:, 1]) / d[:, 1]
        pt = torch.stack([o[:, 0] + tq * d[:, 0], torch.full_like(tq, ex.ground_y),
                          o[:, 2] + tq * d[:, 2]], 1)
        ground = ((d[:, 1] != 0) & (tq > 0) & (pt[:, 0].abs() <= 3.0) & (pt[:, 2].abs() <= 3.0))
        at = ground.nonzero()[:, 0]
        shadow = []
        for pos, inten in ex.lights:
            wl = torch.tensor(pos, device=o.device) - pt[at]
            d2 = wl[:, 0] * wl[:, 0] + wl[:, 1] * wl[:, 1] + wl[:, 2] * wl[:, 2]
            dist = torch.sqrt(d2)
            om = wl / dist[:, None]
            gain = albedo / math.pi * torch.tensor(inten, dtype=torch.float64, device=o.device)
            gain = gain * (om[:, 1].double() / d2.double())[:, None]
            shadow.append((_all(tr, pt[at], om, ex.shadow_eps, dist), gain, om[:, 1] > 0))
        rgb = torch.zeros((n, 3), dtype=torch.float64, device=o.device)
        for s in range(spp):
            t, ids = _closest(cand, _accepted(cand, rid, s, 0, seed), n)
            c = _colour(p, deg, d, ids, bg)
            lit = torch.zeros((at.shape[0], 3), dtype=torch.float64, device=o.device)
            for tag, (sc, gain, facing) in enumerate(shadow):
                hit = torch.zeros(at.shape[0], dtype=torch.bool, device=o.device)
                hit[sc[0][_accepted(sc, rid[at], s, 1 + tag, seed)]] = True
                lit += torch.where((facing & ~hit)[:, None], gain, 0.0)
            db = _bounce_dirs(rid[at], torch.full_like(rid[at], s), seed)
            bc = _all(tr, pt[at], db, ex.shadow_eps)
            _, bid = _closest(bc, _accepted(bc, rid[at], s, 9, seed), at.shape[0])
            lit += albedo * _colour(p, deg, db, bid, bg)
            c[at] = torch.where((t[at] < tq[at].double())[:, None], c[at], lit)
            rgb += c / spp
        out.append(rgb)
    return torch.cat(out)


def exact(case, seed):
    if case["kind"] == "views":
        px = sum(w * h for w, h in _resolutions(case))
        pairs = px * (1 + case["lights"] + case["spp"]) * case["m"]
    else:
        pairs = case["width"] * case["height"] * case["m"]
    if pairs > 1.5e10:
        return None
    p = _gaussians(case, seed)
    bg = torch.tensor(BG, dtype=torch.float32, device=_device()).double()
    return {"frame": _exact_frame, "fit": _exact_fit, "views": _exact_views}[case["kind"]](
        case, int(seed), p, bg)
