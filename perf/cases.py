"""The workloads whose speed is measured: what programs that use this renderer have it do.

Sizes are those of this repository's scenes, tests and benchmark, or plain odd ones.  Every case goes through the
Python binding (`api.Scene`, `api.render*`, `api.TransientRender`) with the launch configuration such a program has:
the library's default for calls nobody tuned ("form": "default"), or, as the benchmark and the large-scene tests do,
the table's entry and else the wavefront form ("form": "tuned").
"""
import functools
import math

import numpy as np
import torch

from paper_2510_25660_gb300 import api, autotune, scenes


def listed():
    return [
        # a preview while a scene is being set up: one sample per pixel, a ragged frame, a host-bound call
        dict(name="cornell_preview", kind="render", scene="cornell", form="default", H=23, W=37, T=100, spp=1, depth=3),
        # the first call of the usage notes: the Cornell box as it comes
        dict(name="cornell_render", kind="render", scene="cornell", form="default", H=64, W=64, T=256, spp=16, depth=4),
        # one step of an optimisation loop on it: forward, L2 loss, backward through the autograd function
        dict(name="cornell_train", kind="train", scene="cornell", form="default", H=64, W=64, T=256, spp=16, depth=4),
        # an untuned render of a medium mesh with time-resolved materials (delays) and a Gaussian source pulse
        dict(name="terrain97k_delays", kind="render", scene="terrain97k", form="default", H=135, W=241, T=367, spp=19,
             depth=6, delays=True),
        # inverse rendering of the 97k-triangle scene: forward and path replay at its own film
        dict(name="terrain97k_train", kind="train", scene="terrain97k", form="tuned", H=256, W=256, T=512, spp=64,
             depth=8),
        # loading a large scene: upload, BVH build, first queries
        dict(name="terrain1m_load", kind="load", scene="terrain1m", rays=262144),
        # the benchmark frame of the 1.16M-triangle scene: the largest call
        dict(name="terrain1m_render", kind="render", scene="terrain1m", form="tuned", H=512, W=512, T=2048, spp=256,
             depth=8),
        # the same frame at four modulation frequencies instead of time bins (frequency space)
        dict(name="terrain1m_phasor", kind="phasor", scene="terrain1m", form="tuned", H=512, W=512, K=4, spp=256,
             depth=8),
        # transient polarization of the frame
        dict(name="terrain1m_stokes", kind="stokes", scene="terrain1m", form="tuned", H=512, W=512, T=512, spp=64,
             depth=8),
        # inverse rendering inside a heterogeneous medium: forward and path replay
        dict(name="media_train", kind="train", scene="media", form="tuned", H=256, W=256, T=1024, spp=128, depth=16),
        # a confocal NLOS capture of the relay wall
        dict(name="nlos_confocal", kind="nlos", scene="nlos", mode="confocal", nx=64, ny=64, T=4096, spp=1024),
        # an exhaustive laser x sensor capture
        dict(name="nlos_exhaustive", kind="nlos", scene="nlos", mode="exhaustive", lx=16, ly=16, nx=32, ny=32, T=4096,
             spp=1024),
    ]


def _log(rng, lo, hi):
    """A whole number spread evenly over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    k = rng.choice(["cornell", "cornell_train", "delays", "train97k", "load", "render", "phasor", "stokes", "media",
                    "confocal", "exhaustive"])
    if k in ("cornell", "cornell_train"):
        return dict(kind="render" if k == "cornell" else "train", scene="cornell", form="default",
                    H=_log(rng, 16, 128), W=_log(rng, 16, 128), T=_log(rng, 32, 512), spp=_log(rng, 1, 32),
                    depth=rng.randint(2, 6))
    if k == "delays":
        return dict(kind="render", scene="terrain97k", form="default", H=_log(rng, 48, 256), W=_log(rng, 48, 256),
                    T=_log(rng, 64, 512), spp=_log(rng, 2, 48), depth=rng.randint(3, 8), delays=rng.random() < 0.7)
    if k == "train97k":
        return dict(kind="train", scene="terrain97k", form="tuned", H=_log(rng, 64, 256), W=_log(rng, 64, 256),
                    T=_log(rng, 64, 512), spp=_log(rng, 8, 64), depth=rng.randint(3, 8))
    if k == "load":
        return dict(kind="load", scene=rng.choice(["terrain1m", "terrain97k", "nlos"]), rays=_log(rng, 1024, 1 << 20))
    if k in ("render", "phasor", "stokes"):
        c = dict(kind=k, scene="terrain1m", form="tuned", H=_log(rng, 96, 512), W=_log(rng, 96, 512),
                 spp=_log(rng, 16, 256 if k != "stokes" else 64), depth=rng.randint(4, 8))
        c["K" if k == "phasor" else "T"] = rng.randint(1, 8) if k == "phasor" else _log(
            rng, 128, 2048 if k == "render" else 512)
        return c
    if k == "media":
        return dict(kind="train", scene="media", form="tuned", H=_log(rng, 64, 256), W=_log(rng, 64, 256),
                    T=_log(rng, 128, 1024), spp=_log(rng, 8, 128), depth=rng.randint(4, 16))
    if k == "confocal":
        return dict(kind="nlos", scene="nlos", mode="confocal", nx=_log(rng, 8, 64), ny=_log(rng, 8, 64),
                    T=_log(rng, 512, 4096), spp=_log(rng, 32, 1024))
    return dict(kind="nlos", scene="nlos", mode="exhaustive", lx=_log(rng, 2, 16), ly=_log(rng, 2, 16),
                nx=_log(rng, 8, 32), ny=_log(rng, 8, 32), T=_log(rng, 512, 4096), spp=_log(rng, 64, 1024))


# --- inputs -------------------------------------------------------------------------------------------------------
_WINDOW = {  # film window (start, length in metres of optical path) of each scene's own film
    "cornell": (3.5, 2.56), "terrain97k": (15.0, 2.56), "terrain1m": (12.0, 10.24), "media": (3.5, 5.12),
    "nlos": (0.0, 12.288)}


@functools.lru_cache(maxsize=None)
def _base(name):
    return {"cornell": scenes.cornell_box, "terrain97k": scenes.diff_scene, "terrain1m": scenes.large_scene,
            "media": scenes.media_scene, "nlos": scenes.nlos_scene}[name]()


def _scene(name, seed):
    """The scene with albedos of its own for each seed (x U[0.8, 1.2], as an optimisation moves them)."""
    sc = _base(name)
    f = np.random.default_rng(seed).uniform(0.8, 1.2, (sc.n_tris, 1)).astype(np.float32)
    return scenes.Scene(sc.tris, np.clip(sc.albedo * f, 0.0, 1.0), sc.roughness, sc.mtype, sc.emitters, sc.camera,
                        sc.medium, sc.hidden, sc.wall)


def _launch(scene, sc, case, kinds):
    if case["form"] != "tuned":
        return
    spec = scenes.FilmSpec(case["H"], case["W"], case.get("T", 2048), 3, 0.0, 1.0)
    for kind in kinds:
        if autotune.apply(scene, kind, sc, spec, case["spp"], case["depth"]) is None:
            scene.set_launch(api.MT_LAUNCH_RENDER if kind == "render" else api.MT_LAUNCH_BACKWARD, 256, 1, 0, 0,
                             api.MT_OPT_WAVEFRONT)


def _target(case, seed):
    """A measured transient to fit: photon noise under an exponential decay."""
    g = torch.Generator("cuda").manual_seed(seed)
    t = torch.rand((case["H"], case["W"], case["T"], 3), device="cuda", generator=g)
    return t.mul_(torch.exp(torch.linspace(0.0, -4.0, case["T"], device="cuda"))[:, None] * 0.01)


def _rays(sc, n, seed):
    """Camera-like rays toward random points of the scene, from random points above it."""
    g = torch.Generator("cuda").manual_seed(seed)
    lo = torch.from_numpy(sc.tris.reshape(-1, 3).min(0)).cuda()
    hi = torch.from_numpy(sc.tris.reshape(-1, 3).max(0)).cuda()
    u = torch.rand((n, 6), device="cuda", generator=g)
    o = lo + (hi - lo) * (u[:, :3] * 1.5 - 0.25)
    d = lo + (hi - lo) * u[:, 3:] - o
    return torch.cat((o, d / d.norm(dim=1, keepdim=True)), 1).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    sc = _scene(case["scene"], seed)
    st = dict(case=case, seed=seed, start=_WINDOW[case["scene"]][0])
    if kind == "load":  # host arrays: what the loader of a scene file leaves behind (another pose for each seed)
        shift = np.random.default_rng(seed + 1).uniform(-0.5, 0.5, 3).astype(np.float32)
        cam = dict(sc.camera, origin=tuple(np.asarray(sc.camera["origin"]) + shift),
                   target=tuple(np.asarray(sc.camera["target"]) + shift))
        sc = scenes.Scene(sc.tris + shift, sc.albedo, sc.roughness, sc.mtype, sc.emitters, cam)
        st.update(sc=sc, rays=_rays(sc, case["rays"], seed))
        return st
    scene = api.Scene(sc)
    st["scene"] = scene
    if kind == "nlos":
        st["lasers"] = torch.from_numpy(scenes.wall_grid(case["nx"], case["ny"])).cuda()
        st["sensors"] = None
        if case["mode"] == "exhaustive":
            st["sensors"] = st["lasers"]
            st["lasers"] = torch.from_numpy(scenes.wall_grid(case["lx"], case["ly"])).cuda()
        else:
            autotune.apply(scene, "nlos", sc, None, case["spp"], 0)
        rows = st["lasers"].shape[0] * (st["sensors"].shape[0] if st["sensors"] is not None else 1)
        st["out"] = (torch.empty((rows, case["T"]), device="cuda"), torch.empty(rows, device="cuda"))
        st["width"] = _WINDOW["nlos"][1] / case["T"]
        return st
    _launch(scene, sc, case, ("render", "backward") if kind == "train" else ("render",))
    H, W = case["H"], case["W"]
    if kind == "phasor":
        st["lambdas"] = torch.tensor([0.4 / 2 ** k for k in range(case["K"])], device="cuda")
        return st
    st["width"] = _WINDOW[case["scene"]][1] / case["T"]
    if kind == "stokes":
        st["out"] = (torch.empty((H, W, case["T"], 4, 3), device="cuda"), torch.empty((H, W, 4, 3), device="cuda"))
    elif kind == "train":
        st["albedo"] = torch.from_numpy(sc.albedo).cuda().requires_grad_(True)
        st["radiance"] = torch.tensor([list(e["radiance"]) for e in sc.emitters], device="cuda", requires_grad=True)
        st["target"] = _target(case, seed)
    elif case["form"] == "tuned":
        st["out"] = api.new_film(H, W, case["T"])
    if case.get("delays"):
        g = torch.Generator("cuda").manual_seed(seed + 7)
        scene.set_delays(torch.rand(sc.n_tris, device="cuda", generator=g) * 0.05)
        scene.set_pulse(api.MT_PULSE_GAUSSIAN, 0.03, 0.01)
    return st


def run(st):
    c, seed = st["case"], st["seed"]
    kind = c["kind"]
    if kind == "load":
        scene = api.Scene(st["sc"])
        return api.probe_trace(scene, st["rays"])
    s = st["scene"]
    if kind == "nlos":
        mode = api.MT_EXHAUSTIVE if c["mode"] == "exhaustive" else api.MT_CONFOCAL
        return api.render_nlos(s, st["lasers"], st["sensors"], mode, c["T"], st["start"], st["width"], c["spp"], seed,
                               out=st["out"])
    if kind == "phasor":
        return api.render_phasor(s, c["H"], c["W"], st["lambdas"], c["spp"], seed, c["depth"])
    if kind == "stokes":
        return api.render_polarized(s, c["H"], c["W"], c["T"], st["start"], st["width"], c["spp"], seed, c["depth"],
                                    out=st["out"])
    if kind == "train":
        film, steady = api.TransientRender.apply(st["albedo"], st["radiance"], s, c["H"], c["W"], c["T"], st["start"],
                                                 st["width"], c["spp"], seed, c["depth"])
        loss = (film - st["target"]).square().sum()
        grads = torch.autograd.grad(loss, (st["albedo"], st["radiance"]))
        return film.detach(), steady.detach(), grads[0], grads[1]
    return api.render(s, c["H"], c["W"], c["T"], st["start"], st["width"], c["spp"], seed, c["depth"],
                      out=st.get("out"))


# --- the work nobody can do without -------------------------------------------------------------------------------
# flops: per ray about 40 per level of a binary tree over the triangles and 150 for the triangle tests, per path
# vertex about 300 for sampling and shading; a path has about half of its largest number of vertices, two rays each.
def work(case):
    n = _base(case["scene"]).n_tris
    ray = 40.0 * math.log2(n) + 150.0
    scene_bytes = 68.0 * n
    if case["kind"] == "load":
        return dict(bytes=(56.0 + 48 + 32) * n + 32.0 * case["rays"], flops=case["rays"] * ray + 100.0 * n * math.log2(n))
    if case["kind"] == "nlos":
        las = case["lx"] * case["ly"] if case["mode"] == "exhaustive" else case["nx"] * case["ny"]
        pairs = las * (case["nx"] * case["ny"] if case["mode"] == "exhaustive" else 1)
        return dict(bytes=scene_bytes + 4.0 * pairs * (case["T"] + 1),
                    flops=case["spp"] * (pairs * (ray + 60.0) + las * 100.0))
    px = case["H"] * case["W"]
    vertices = px * case["spp"] * max(1.0, 0.5 * case["depth"])
    film = 4.0 * px * {"phasor": 6 * case.get("K", 0) + 3, "stokes": 12 * (case.get("T", 0) + 1)}.get(
        case["kind"], 3 * (case.get("T", 0) + 1))
    flops = vertices * (2 * ray + 300.0)
    if case["kind"] == "train":  # the forward film written; film and target read; its gradient written and read
        return dict(bytes=scene_bytes + 5 * film + 24.0 * n, flops=2 * flops)
    return dict(bytes=scene_bytes + film, flops=flops)


# --- the same results in 64 bits, from the estimator's definition, by brute force over the triangles --------------
def _philox(a, b, c, d, seed):
    """Philox4x32-10 of int64 tensors of counters; four tensors of 32-bit words."""
    k0, k1, m = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF, 0xFFFFFFFF
    for r in range(10):
        p, q = 0xD2511F53 * a, 0xCD9E8D57 * c
        a, b, c, d = ((q >> 32) & m) ^ b ^ k0, q & m, ((p >> 32) & m) ^ d ^ k1, p & m
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return a, b, c, d


def _u(x):
    return (x >> 8).double() / 2 ** 24


def _dot(a, b):
    return (a * b).sum(-1)


def _unit(a):
    return a / a.norm(dim=-1, keepdim=True)


def _eps(p):
    return 1e-4 * p.abs().amax(-1, keepdim=True).clamp(min=1.0)


def _hits(v, o, d, tmax=None):
    """Closest (t, index) of rays o, d over the triangles v [n, 3, 3], by Moeller and Trumbore; occlusion with tmax."""
    e1, e2 = v[:, 1] - v[:, 0], v[:, 2] - v[:, 0]
    ts, ids = [], []
    step = max(1, 40_000_000 // len(v))
    for lo in range(0, len(o), step):
        oo, dd = o[lo:lo + step, None], d[lo:lo + step, None]
        p = torch.linalg.cross(dd, e2[None])
        det = _dot(e1, p)
        s = oo - v[:, 0]
        b1 = _dot(s, p) / det
        q = torch.linalg.cross(s, e1[None])
        b2, t = _dot(dd, q) / det, _dot(e2, q) / det
        ok = (det != 0) & (b1 >= 0) & (b2 >= 0) & (b1 + b2 <= 1) & (t > 0)
        t, k = torch.where(ok, t, math.inf).min(1)
        ts.append(t)
        ids.append(k)
    t = torch.cat(ts)
    return (t, torch.cat(ids)) if tmax is None else t < tmax


def _basis(n):
    sg = torch.where(n[:, 2] >= 0, 1.0, -1.0).double()
    a = -1.0 / (sg + n[:, 2])
    c = n[:, 0] * n[:, 1] * a
    return (torch.stack((1 + sg * n[:, 0] ** 2 * a, sg * c, -sg * n[:, 0]), -1),
            torch.stack((c, sg + n[:, 1] ** 2 * a, -n[:, 1]), -1))


def _cornell(case, seed, albedo, radiance):
    """Film and steady image of the Lambertian box: next-event estimation with the power heuristic, every
    contribution in the bin of its own optical path length (arXiv 2510.25660 Sec. 3)."""
    sc = _base("cornell")
    H, W, T, spp = case["H"], case["W"], case["T"], case["spp"]
    start, width = np.float32(_WINDOW["cornell"][0]), np.float32(_WINDOW["cornell"][1] / T)
    v = torch.from_numpy(sc.tris).cuda().double()
    cr = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    area, normal = cr.norm(dim=1) / 2, _unit(cr)
    em = sc.emitters[0]
    first, n_light = em["first_tri"], em["n_tris"]
    pick = area[first:] / area[first:].sum()
    cdf = torch.ceil(pick.cumsum(0) * 2 ** 24).long()
    cdf[-1] = 2 ** 24
    f64 = functools.partial(torch.tensor, dtype=torch.float64, device="cuda")
    o0 = f64([float(np.float32(x)) for x in sc.camera["origin"]])
    fw = _unit(f64([float(np.float32(x)) for x in sc.camera["target"]]) - o0)
    rt = _unit(torch.linalg.cross(fw, f64(sc.camera["up"])))
    up = torch.linalg.cross(rt, fw)
    th = math.tan(math.radians(sc.camera["fov_x_deg"]) / 2)
    j = torch.arange(H * W * spp, device="cuda")
    pix, smp = j // spp, j % spp
    zero = torch.zeros_like(j)
    r0, r1, _, _ = _philox(pix, smp, zero, zero, seed)
    sx = (2 * (pix % W + _u(r0)) / W - 1) * th
    sy = (1 - 2 * (pix // W + _u(r1)) / H) * th * H / W
    d = _unit(fw + rt * sx[:, None] + up * sy[:, None])
    o = o0.expand_as(d)
    opl = torch.zeros(len(j), dtype=torch.float64, device="cuda")
    beta, pdf = torch.ones_like(d), opl
    film = torch.zeros((H * W * T, 3), dtype=torch.float64, device="cuda")
    steady = torch.zeros((H * W, 3), dtype=torch.float64, device="cuda")

    def add(film, steady, pix, opl, c):
        c = c / spp
        x = (opl - float(start)) / float(width)
        ok = (x >= 0) & (x < T)
        return (film.index_add(0, (pix * T + x.clamp(0, T - 1).long())[ok], c[ok]), steady.index_add(0, pix, c))

    for depth in range(1, case["depth"] + 1):
        t, k = _hits(v, o, d)
        keep = t < math.inf
        o, d, opl, beta, pdf, pix, smp, t, k = (a[keep] for a in (o, d, opl, beta, pdf, pix, smp, t, k))
        x = o + d * t[:, None]
        opl = opl + t
        cwo = -_dot(normal[k], d)
        lit = (k >= first) & (k < first + n_light) & (cwo > 0)
        pl = (pick / area[first:])[(k - first).clamp(min=0)] * t * t / cwo
        w = torch.ones_like(t) if depth == 1 else pdf ** 2 / (pdf ** 2 + pl ** 2)
        film, steady = add(film, steady, pix[lit], opl[lit], (beta * w[:, None])[lit] * radiance[0])
        if depth == case["depth"]:
            break
        n = torch.where((cwo >= 0)[:, None], normal[k], -normal[k])
        dep = torch.full_like(pix, depth)
        rho = albedo[k]
        # next-event estimate
        r0, r1, r2, _ = _philox(pix, smp, dep, torch.zeros_like(pix), seed)
        li = torch.searchsorted(cdf, r0 >> 8, right=True).clamp(max=n_light - 1)
        su = _u(r1).sqrt()[:, None]
        b0, b1 = 1 - su, _u(r2)[:, None] * su
        lv = v[first + li]
        y = lv[:, 0] * b0 + lv[:, 1] * b1 + lv[:, 2] * (1 - b0 - b1)
        xo = x + n * _eps(x)
        dist = (y - xo).norm(dim=1)
        wi = (y - xo) / dist[:, None]
        cx, cy = _dot(n, wi), -_dot(normal[first + li], wi)
        ok = (cx > 0) & (cy > 0)
        ok[ok.clone()] = ~_hits(v, xo[ok], wi[ok], (dist - _eps(y)[:, 0])[ok])
        pa = pick[li] / area[first + li]
        pl = pa * dist ** 2 / cy
        w = pl ** 2 / (pl ** 2 + (cx / math.pi) ** 2)
        c = beta * rho / math.pi * (cx * cy / dist ** 2 / pa * w)[:, None] * radiance[0]
        film, steady = add(film, steady, pix[ok], (opl + dist)[ok], c[ok])
        # continuation: cosine sampling, weight rho
        r0, r1, _, _ = _philox(pix, smp, dep, torch.ones_like(pix), seed)
        u0, ph = _u(r0), 2 * math.pi * _u(r1)
        tb, bb = _basis(n)
        z = (1 - u0).sqrt()
        d = (tb * (u0.sqrt() * ph.cos())[:, None] + bb * (u0.sqrt() * ph.sin())[:, None] + n * z[:, None])
        o, beta, pdf = xo, beta * rho, z / math.pi
    return film.view(H, W, T, 3), steady.view(H, W, 3)


def _confocal(case, seed):
    """Confocal impulse responses (Sec. 4.5): hidden points uniform by area, one segment there and back."""
    sc = _scene("nlos", seed)
    T, spp = case["T"], case["spp"]
    first, count = sc.hidden
    v = torch.from_numpy(sc.tris).cuda().double()
    cr = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    area = cr.norm(dim=1)[first:first + count] / 2
    cdf = torch.ceil(area.cumsum(0) / area.sum() * 2 ** 24).long()
    cdf[-1] = 2 ** 24
    xs = torch.from_numpy(scenes.wall_grid(case["nx"], case["ny"])).cuda().double()
    j = torch.arange(len(xs) * spp, device="cuda")
    row = j // spp
    r0, r1, r2, _ = _philox(row, j % spp, torch.zeros_like(j), torch.zeros_like(j), seed)
    k = first + torch.searchsorted(cdf, r0 >> 8, right=True).clamp(max=count - 1)
    su = _u(r1).sqrt()[:, None]
    b0, b1 = 1 - su, _u(r2)[:, None] * su
    y = v[k, 0] * b0 + v[k, 1] * b1 + v[k, 2] * (1 - b0 - b1)
    nw = torch.tensor(sc.wall["normal"], dtype=torch.float64, device="cuda")
    x = xs[row]
    d1 = (y - x).norm(dim=1)
    w1 = (y - x) / d1[:, None]
    cl, cy = _dot(w1, nw), _dot(_unit(cr[k]), w1).abs()
    xo = x + nw * _eps(x)
    l1 = (y - xo).norm(dim=1)
    ok = (cl > 0) & (cy > 0)
    ok[ok.clone()] = ~_hits(v, xo[ok], ((y - xo) / l1[:, None])[ok], (l1 - _eps(y)[:, 0])[ok])
    fh = torch.from_numpy(sc.albedo).cuda().double()[k].mean(1) / math.pi
    fw = sc.wall["albedo"] / math.pi
    h = torch.where(ok, (fw * cl * cy / d1 ** 2) ** 2 * fh * area.sum(), 0.0) / spp
    b = 2 * d1 / float(np.float32(_WINDOW["nlos"][1] / T))
    inside = ok & (b < T)
    film = torch.zeros(len(xs) * T, dtype=torch.float64, device="cuda")
    film.index_add_(0, (row * T + b.clamp(max=T - 1).long())[inside], h[inside])
    return film.view(len(xs), T), torch.zeros(len(xs), dtype=torch.float64, device="cuda").index_add_(0, row, h)


def exact(case, seed):
    if case["scene"] == "cornell":
        sc = _scene("cornell", seed)
        albedo = torch.from_numpy(sc.albedo).cuda().double()
        radiance = torch.tensor([list(e["radiance"]) for e in sc.emitters], dtype=torch.float64, device="cuda")
        if case["kind"] == "render":
            return _cornell(case, seed, albedo, radiance)
        albedo.requires_grad_(True)
        radiance.requires_grad_(True)
        film, steady = _cornell(case, seed, albedo, radiance)
        grads = torch.autograd.grad((film - _target(case, seed).double()).square().sum(), (albedo, radiance))
        return film.detach(), steady.detach(), grads[0], grads[1]
    if case["scene"] == "nlos" and case.get("mode") == "confocal" and case["nx"] * case["ny"] * case["spp"] <= 300_000:
        return _confocal(case, seed)
    return None  # brute force over 49k triangles and more would take minutes, and the medium's walks longer
