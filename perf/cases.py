"""The work a user of the differentiable path tracer has it do, as a list of measurable cases.

A case is a plain dict: a mesh, a set of views, the lights and the options of one call sequence.
Five kinds of call sequence are listed:

* ``step``: one iteration of the reconstruction loop (the paper's Sec. 3.2): new vertex positions
  and materials in, images and both gradients out, through the autograd wrapper ``st.render``;
* ``material``: the same with the geometry held (Sec. 3.3): new materials, images, their gradient;
* ``render``: the images of new vertex positions, without a gradient (targets, previews);
* ``trace``: closest-hit queries of the caller's own rays after a vertex update;
* ``rebuild``: a full rebuild of the hierarchy at moved vertices, then such queries.

Vertices, materials, lights, environments and targets come from the seed alone; meshes, view
layouts and sizes are those of this repository's workloads, tests and benchmark or generic.
``exact`` restates the forward estimator and its interior gradient in 64 bits with plain torch
(brute-force intersection), for the cases small enough for that.
"""
import functools
import math

import numpy as np
import torch

from paper_2012_03939_gb300 import scenes as S
from paper_2012_03939_gb300 import st

DEFAULTS = dict(kind="step", mesh="icosphere", m1=2, m2=0, views=1, width=64, height=64, uneven=False, spp=4,
                bounces=2, lights=0, view_lights=False, env_w=0, env_h=0, edge=0, color_res=0, rgb=False,
                smooth=False, fresnel=0, brdf="ggx", rays=0)
# a ray query and the vertex it finds: one watertight test, one BRDF value and pdf, one sample
FLOPS_PER_VERTEX = 400
EXACT_PAIRS = 2e10   # ray/triangle pairs a 64-bit brute force does in well under 20 seconds


def _case(name, **kw):
    return dict(DEFAULTS, name=name, **kw)


def listed():
    return [
        # the smallest iteration: a coarse initial mesh, one small view; launches and latency are its cost
        _case("step_320f_1view", mesh="icosphere", m1=2, width=64, height=64, spp=4, bounces=2, lights=1, edge=1),
        # an open scene with interreflection between three walls, a few small views
        _case("step_planes_4views", mesh="planes", m1=8, views=4, width=64, height=64, spp=16, bounces=3, lights=1,
              edge=1),
        # a smooth object under scene lights with silhouette edges: the ordinary iteration
        _case("step_5120f_16views", mesh="icosphere", m1=4, views=16, width=128, height=128, spp=16, bounces=3,
              lights=3, edge=1),
        # the paper's captures: 32 cameras of 128x128, each lit from the camera and beside it, with the primary
        # and the point-light shadow edges
        _case("step_captures_32views", mesh="icosphere", m1=5, views=32, width=128, height=128, spp=4, bounces=2,
              view_lights=True, edge=5),
        # a concave object under an environment, many medium views, interior gradient
        _case("step_knot_32views", mesh="knot", m1=500, m2=50, views=32, width=256, height=256, spp=4, bounces=4,
              env_w=256, env_h=128),
        # the same object with primary and secondary silhouettes
        _case("step_knot_secondary", mesh="knot", m1=500, m2=50, views=8, width=256, height=256, spp=4, bounces=4,
              env_w=256, env_h=128, edge=3),
        # many views of uneven size and sample count on a fine mesh
        _case("step_200kf_64views", mesh="uv_sphere", m1=500, m2=201, views=64, width=512, height=512, uneven=True,
              spp=16, bounces=3, env_w=512, env_h=256, edge=1),
        # the largest iteration: a rough mesh of a million faces, an 8-view minibatch
        _case("step_1mf_8views", mesh="fractal", m1=1000, m2=501, views=8, width=512, height=512, spp=16, bounces=5,
              lights=2, env_w=1024, env_h=512, edge=1),
        # material estimation on fixed geometry: mesh colors, RGB specular, interpolated normals, ragged views
        _case("material_1280f_16views", kind="material", mesh="icosphere", m1=3, views=16, width=129, height=97, spp=4,
              bounces=2, lights=2, color_res=2, rgb=True, smooth=True, fresnel=1, brdf="beckmann"),
        # previews of the current mesh
        _case("render_200kf_2views", kind="render", mesh="uv_sphere", m1=500, m2=201, views=2, width=640, height=480,
              spp=16, bounces=3, lights=2, env_w=512, env_h=256),
        # the caller's own rays against a deforming mesh
        _case("trace_5120f", kind="trace", mesh="icosphere", m1=4, rays=262144),
        # a rebuild after the vertices moved far
        _case("rebuild_50kf", kind="rebuild", mesh="knot", m1=500, m2=50, rays=65536),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["material", "render", "trace", "rebuild"])
    c = dict(DEFAULTS, kind=kind, mesh=rng.choice(["icosphere", "uv_sphere", "fractal", "knot", "planes"]))
    if c["mesh"] == "icosphere":
        c["m1"] = rng.randint(2, 5)
    elif c["mesh"] == "planes":
        c["m1"] = _log_int(rng, 4, 64)
    else:
        c["m1"] = _log_int(rng, 24, 500)
        c["m2"] = max(8, c["m1"] // rng.choice([2, 3, 5]))
    if kind in ("trace", "rebuild"):
        c["rays"] = _log_int(rng, 1000, 1000000)
        return c
    c["width"], c["height"] = _log_int(rng, 48, 512), _log_int(rng, 48, 512)
    c["spp"] = rng.choice([1, 2, 4, 4, 8, 16])
    c["bounces"] = rng.randint(1, 5)
    # at most half the camera samples of the largest listed case
    most = 16e6 / (c["width"] * c["height"] * c["spp"])
    c["views"] = max(1, min(64, _log_int(rng, 1, max(1.0, min(64.0, most)))))
    if rng.random() < 0.5:
        c["env_w"], c["env_h"] = rng.choice([(64, 32), (256, 128), (512, 256)])
    if not c["env_w"] or rng.random() < 0.4:
        c["lights"] = rng.randint(1, 3)
    c["view_lights"] = rng.random() < 0.2
    c["smooth"] = rng.random() < 0.2
    c["fresnel"] = int(rng.random() < 0.2)
    c["brdf"] = rng.choice(["ggx", "ggx", "ggx", "beckmann"])
    if kind == "material":
        c["color_res"], c["rgb"] = rng.randint(0, 3), rng.random() < 0.5
    elif kind == "step":
        c["edge"] = rng.choice([0, 1, 1, 1, 3, 5])
    return c


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _base_mesh(mesh, m1, m2):
    """Vertices [V, 3] and faces [F, 3] of the undeformed mesh."""
    if mesh == "icosphere":
        return S.icosphere(m1)
    if mesh == "uv_sphere":
        return S.uv_sphere(m1, m2)
    if mesh == "fractal":
        V, F = S.uv_sphere(m1, m2)
        return S.fractal_displace(V, np.random.default_rng(7)), F
    if mesh == "knot":
        return S.torus_knot(2, 3, m1, m2)
    sc = S.color_bleed(n=m1)
    return sc.vertices.astype(np.float64), sc.faces


def _views(case, rng):
    n, w, h = case["views"], case["width"], case["height"]
    if case["mesh"] == "planes":
        eyes = [(3.6, 2.2, 3.0), (3.0, 2.2, 3.6), (3.4, 2.2, 3.4), (4.0, 2.2, 2.6)]
        vs = [S.View(tuple(x * (1.0 + 0.1 * (i // 4)) for x in eyes[i % 4]), (0.6, 0.5, 0.6), (0.0, 1.0, 0.0), 45.0, w,
                     h, case["spp"]) for i in range(n)]
        off = 0
        for v in vs:
            v.pixel_offset = off
            off += v.width * v.height
    elif case["uneven"]:
        ws, hs = rng.choice([w // 8, w // 4, w // 2, w], size=n), rng.choice([h // 8, h // 4, h // 2, h], size=n)
        vs = S.fibonacci_views(n, ws, hs, rng.choice([1, 4, case["spp"]], size=n))
    elif case["lights"] and not case["env_w"]:
        vs = S.ring_views(n, w, case["spp"])
        off = 0
        for v in vs:
            v.height, v.pixel_offset = h, off
            off += w * h
    else:
        vs = S.fibonacci_views(n, [w] * n, [h] * n, [case["spp"]] * n)
    return S.with_view_lights(vs) if case["view_lights"] else vs


def _scene(case, seed):
    """The scene of a case: a host description whose arrays are a function of (case, seed)."""
    rng = np.random.default_rng(seed)
    V, F = _base_mesh(case["mesh"], case["m1"], case["m2"])
    if case["mesh"] == "planes":
        V = V * rng.uniform(0.97, 1.03, size=3)
    else:   # a smooth radial field of the seed on the base mesh
        V = V * np.linalg.norm(S.sinusoid_displace(V, rng), axis=1, keepdims=True)
    tex = (case["color_res"] + 1) * (case["color_res"] + 2) // 2
    P = S.random_face_params(rng, len(F) * tex)
    if case["rgb"]:
        P = np.concatenate([P[:, :3], rng.uniform(0.02, 0.3, size=(len(P), 3)).astype(np.float32), P[:, 4:]], 1)
    lp, li = np.zeros((0, 3), np.float32), np.zeros((0, 3), np.float32)
    if case["lights"]:
        d = rng.normal(size=(case["lights"], 3))
        d[:, 1] = np.abs(d[:, 1])
        d /= np.linalg.norm(d, axis=1, keepdims=True)
        lp = (np.abs(d) * 0.8 + 0.6 if case["mesh"] == "planes" else 3.0 * d).astype(np.float32)
        li = np.full((case["lights"], 3), 4.0 if case["mesh"] == "planes" else 6.0, np.float32)
    env = S.lognormal_env(rng, case["env_w"], case["env_h"]) if case["env_w"] else None
    # sizes of uneven views belong to the case, not to the seed
    views = _views(case, np.random.default_rng(S.BASE_SEED))
    return S.Scene("case", np.ascontiguousarray(V, np.float32), np.ascontiguousarray(F, np.int32), P, case["brdf"],
                   light_pos=lp, light_intensity=li, env=env, views=views, max_bounces=case["bounces"], seed=seed,
                   color_res=case["color_res"], smooth_normals=case["smooth"], fresnel=case["fresnel"])


def _target(sc, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.rand((sc.n_pixels, 3), generator=g)


def _rays(case, seed):
    """[n, 8] rays from a shell around the mesh toward points inside its bounds."""
    g = torch.Generator().manual_seed(seed)
    o = torch.nn.functional.normalize(torch.randn((case["rays"], 3), generator=g), dim=1) * 3.0
    to = torch.rand((case["rays"], 3), generator=g) * 2.0 - 1.0
    d = torch.nn.functional.normalize(to - o, dim=1)
    r = torch.zeros((case["rays"], 8))
    r[:, :3], r[:, 4:7], r[:, 7] = o, d, math.inf
    return r


def prepare(case, seed):
    sc = _scene(case, seed)
    state = {"case": case, "sc": sc, "seed": seed + 1, "scene": st.Scene.from_scene(sc),
             "V": torch.from_numpy(sc.vertices).cuda(), "P": torch.from_numpy(sc.face_params).cuda()}
    if case["kind"] in ("trace", "rebuild"):
        state["rays"] = _rays(case, seed).cuda()
    elif case["kind"] != "render":
        state["target"] = _target(sc, seed).cuda()
        state["P"].requires_grad_()
        if case["kind"] == "step":
            state["V"].requires_grad_()
            state["bopts"] = st.make_opts(edge_term=case["edge"])
    return state


# ---------------------------------------------------------------- one pass
def run(s):
    case, scene, sc, V, P = s["case"], s["scene"], s["sc"], s["V"], s["P"]
    if case["kind"] == "step":
        V.grad = P.grad = None
        img = st.render(V, P, scene, sc.views, sc.max_bounces, s["seed"], bwd_opts=s["bopts"])
        torch.nn.functional.mse_loss(img, s["target"]).backward()
        return {"image": img.detach(), "d_vertices": V.grad, "d_params": P.grad}
    if case["kind"] == "material":
        scene.set_face_params(P)
        img = scene.render(sc.views, sc.max_bounces, s["seed"])
        dLdI = (img - s["target"]) * (2.0 / img.numel())
        _, dP = scene.backward(sc.views, sc.max_bounces, s["seed"], dLdI, want_vertices=False)
        return {"image": img, "d_params": dP}
    if case["kind"] == "render":
        scene.refit(V)
        return {"image": scene.render(sc.views, sc.max_bounces, s["seed"])}
    (scene.refit if case["kind"] == "trace" else scene.rebuild)(V)
    face, t = scene.trace_closest(s["rays"])
    return {"face": face, "t": t}


def _sizes(case):
    """(vertices, faces, texels) of the case's mesh."""
    V, F = _base_mesh(case["mesh"], case["m1"], case["m2"])
    return len(V), len(F), len(F) * (case["color_res"] + 1) * (case["color_res"] + 2) // 2


def work(case):
    nv, nf, nt = _sizes(case)
    mesh = 12 * (nv + nf)
    if case["kind"] in ("trace", "rebuild"):
        return {"bytes": mesh + 40 * case["rays"], "flops": 60 * case["rays"]}
    vs = _views(case, np.random.default_rng(S.BASE_SEED))
    pixels = sum(v.width * v.height for v in vs)
    paths = sum(v.width * v.height * v.spp for v in vs)
    params = 4 * nt * (7 if case["rgb"] else 5)
    b = mesh + params + 16 * case["env_w"] * case["env_h"] + 12 * pixels
    flops = FLOPS_PER_VERTEX * paths
    if case["kind"] in ("step", "material"):   # target in, gradients out; the paths are traced again, edges twice
        b += 12 * pixels + params + (12 * nv if case["kind"] == "step" else 0)
        flops *= 2 + (2 if case["edge"] & 1 else 0)
    return {"bytes": b, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits
def exact(case, seed):
    sc = _scene(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] in ("trace", "rebuild"):
        if case["rays"] * len(sc.faces) > EXACT_PAIRS:
            return None
        r = _rays(case, seed).to(dev).double()
        tri = torch.from_numpy(sc.vertices).to(dev).double()[torch.from_numpy(sc.faces).to(dev).long()]
        none = torch.full((len(r),), -1, device=dev)
        _, t = _closest(tri, r[:, :3], r[:, 4:7], none)
        return {"face": None, "t": t}
    paths = sum(v.width * v.height * v.spp for v in sc.views)
    lights = len(sc.light_pos) + 2 * case["view_lights"] + (sc.env is not None)
    if paths * sc.max_bounces * (1 + lights) * len(sc.faces) > EXACT_PAIRS:
        return None
    V = torch.from_numpy(sc.vertices).to(dev).double()
    P = torch.from_numpy(sc.face_params).to(dev).double()
    if case["kind"] == "render":
        with torch.no_grad():
            return {"image": _Tracer(sc, V, P).image(seed + 1)}
    P.requires_grad_()
    if case["kind"] == "step":
        V.requires_grad_()
    img = _Tracer(sc, V, P).image(seed + 1)
    torch.nn.functional.mse_loss(img, _target(sc, seed).to(dev).double()).backward()
    out = {"image": img.detach(), "d_params": P.grad}
    if case["kind"] == "step":   # the edge terms are not restated here: they add to the vertices' gradient alone
        out["d_vertices"] = None if case["edge"] else V.grad
    return out


def _dot(a, b):
    return (a * b).sum(-1)


def _unit(a):
    return a / a.norm(dim=-1, keepdim=True)


def _closest(tri, o, d, exclude, tmax=None):
    """Nearest (face, t) of each ray with t > 1e-5 (and < tmax), its excluded face skipped; (-1, inf) on a miss."""
    v0, e1, e2 = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    n = torch.cross(e1, e2, dim=1)
    faces, ts = [exclude.new_zeros(0)], [o.new_zeros(0)]
    for a in range(0, len(o), max(1, (1 << 24) // len(tri))):
        b = min(len(o), a + max(1, (1 << 24) // len(tri)))
        oo, dd = o[a:b], d[a:b]
        # solve o + t d = v0 + u e1 + v e2: with m = (o - v0) x d, every term is a product of per-ray and
        # per-face vectors, so the pairs need matrix products only
        od = torch.cross(oo, dd, dim=1)
        det = -dd @ n.T
        vd1, vd2 = dd @ torch.cross(v0, e1, dim=1).T, dd @ torch.cross(v0, e2, dim=1).T
        u = (od @ e2.T + vd2) / det
        v = -(od @ e1.T + vd1) / det
        t = (oo @ n.T - _dot(v0, n)) / det
        ok = (u >= 0) & (v >= 0) & (u + v <= 1) & (t > 1e-5)
        if tmax is not None:
            ok &= t < tmax[a:b, None]
        ok &= torch.arange(len(tri), device=o.device)[None] != exclude[a:b, None]
        t = torch.where(ok, t, math.inf)
        t, f = t.min(dim=1)
        ts.append(t)
        faces.append(torch.where(torch.isinf(t), -1, f))
    return torch.cat(faces), torch.cat(ts)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 of Salmon et al. (SC'11) on int64 tensors holding 32-bit words."""
    M = 0xFFFFFFFF

    def mul(a, x):
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        mid = hi + (lo >> 16)
        return mid >> 16, ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)

    c0, c1, c2, c3 = (torch.as_tensor(c, device=c0.device).expand_as(c0) & M for c in (c0, c1, c2, c3))
    k0, k1 = seed & M, (seed >> 32) & M
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c0, c1, c2, c3


def _unif(w):
    return (w >> 8).double() / 16777216.0


def _alias_table(weights):
    """Vose's alias table over flat weights: stacks seeded in index order, the accept threshold a float32."""
    n, q = len(weights), (weights * len(weights) / weights.sum()).tolist()
    prob, alias = [1.0] * n, list(range(n))
    small, large = [i for i in range(n) if q[i] < 1.0], [i for i in range(n) if q[i] >= 1.0]
    while small and large:
        a, b = small.pop(), large[-1]
        prob[a], alias[a] = q[a], b
        q[b] = (q[b] + q[a]) - 1.0
        if q[b] < 1.0:
            small.append(large.pop())
    return np.float32(prob).astype(np.float64), np.array(alias)


class _Tracer:
    """The forward estimator on 64-bit tensors; autograd through it is the interior gradient (sampled
    directions, pdfs and MIS weights held constant, hit points moving along their rays)."""

    def __init__(self, sc, V, P):
        self.sc, self.V, self.P, self.dev = sc, V, P, V.device
        self.F = torch.from_numpy(sc.faces).to(self.dev).long()
        self.rgb = P.shape[1] == 7
        if sc.smooth_normals:
            v = V[self.F]
            m = torch.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0], dim=1)
            M = torch.zeros_like(V)
            for k in range(3):
                M = M.index_add(0, self.F[:, k], m)
            self.N = _unit(M)
        if sc.env is not None:
            h, w, _ = sc.env.shape
            e = sc.env.astype(np.float64)
            lum = e @ np.array([0.2126, 0.7152, 0.0722])
            wt = (lum * np.sin(np.pi * (np.arange(h) + 0.5) / h)[:, None]).reshape(-1)
            prob, alias = _alias_table(wt)
            self.env = torch.from_numpy(e.reshape(-1, 3)).to(self.dev)
            self.pmf = torch.from_numpy(wt / wt.sum()).to(self.dev)
            self.prob, self.alias = torch.from_numpy(prob).to(self.dev), torch.from_numpy(alias).to(self.dev)

    def image(self, seed):
        out = [self.view(v, seed) for v in self.sc.views]
        return torch.cat(out)

    # -- material
    def _D(self, c, a):
        if self.sc.brdf == "ggx":
            return a * a / (math.pi * (c * c * (a * a - 1.0) + 1.0) ** 2)
        c2 = c * c
        return torch.exp(-(1.0 - c2) / c2 / (a * a)) / (math.pi * a * a * c2 * c2)

    def _G1(self, c, a):
        if self.sc.brdf == "ggx":
            return 2.0 * c / (c + torch.sqrt(a * a + (1.0 - a * a) * c * c))
        s2 = 1.0 - c * c
        x = c / (a * torch.sqrt(s2.clamp_min(1e-300)))
        g = 2.0 / (1.0 + torch.erf(x) + torch.exp(-x * x) / (x * math.sqrt(math.pi)))
        return torch.where(s2 > 0, g, 1.0)

    def _value(self, m, n, wi, wo):
        """f(wi, wo) cos(n, wi), RGB; the caller keeps both cosines positive."""
        kd, ks, a = m
        ci, co = _dot(n, wi), _dot(n, wo)
        h = _unit(wi + wo)
        spec = self._D(_dot(n, h), a) * self._G1(ci, a) * self._G1(co, a) / (4.0 * co)
        x5 = (1.0 - _dot(wi, h)) ** 5 if self.sc.fresnel else torch.zeros_like(ci)
        return kd * (ci / math.pi)[:, None] + (ks + (1.0 - ks) * x5[:, None]) * spec[:, None]

    @staticmethod
    def _lobe(m):
        ks, kd = m[1].mean(1), m[0].mean(1)
        return (ks / (ks + kd)).clamp(0.05, 0.95)

    def _pdf(self, m, n, wi, wo):
        h = _unit(wi + wo)
        ch, ps = _dot(n, h), self._lobe(m)
        return (1.0 - ps) * _dot(n, wi) / math.pi + ps * self._D(ch, m[2]) * ch / (4.0 * _dot(wo, h).abs())

    def _sample(self, m, n, wo, ul, u1, u2):
        h = torch.tensor([0.4375, 0.5625, 0.6875], device=self.dev, dtype=torch.float64)
        t = _unit(torch.cross(h.expand_as(n), n, dim=1))
        b = torch.cross(n, t, dim=1)
        a2 = m[2] ** 2
        tan2 = a2 * u1 / (1.0 - u1) if self.sc.brdf == "ggx" else -a2 * torch.log(1.0 - u1)
        ch = 1.0 / torch.sqrt(1.0 + tan2)
        sh = torch.sqrt((1.0 - ch * ch).clamp_min(0))
        ph = 2.0 * math.pi * u2
        hv = t * (sh * torch.cos(ph))[:, None] + b * (sh * torch.sin(ph))[:, None] + n * ch[:, None]
        ws = hv * (2.0 * _dot(wo, hv))[:, None] - wo
        a, c = 2.0 * u1 - 1.0, 2.0 * u2 - 1.0
        wide = a.abs() > c.abs()
        r = torch.where(wide, a, c)
        safe = torch.where(r == 0, 1.0, r)
        ph = torch.where(wide, math.pi / 4 * (c / safe), math.pi / 2 - math.pi / 4 * (a / safe))
        x, y = r * torch.cos(ph), r * torch.sin(ph)
        z = torch.sqrt((1.0 - x * x - y * y).clamp_min(0))
        wd = t * x[:, None] + b * y[:, None] + n * z[:, None]
        return torch.where((ul < self._lobe(m))[:, None], ws, wd)

    def _texel(self, d):
        h, w, _ = self.sc.env.shape
        col = ((torch.atan2(d[:, 0], -d[:, 2]) + math.pi) / (2 * math.pi) * w).long().clamp(0, w - 1)
        row = (torch.acos(d[:, 1].clamp(-1, 1)) / math.pi * h).long().clamp(0, h - 1)
        return row * w + col, torch.sqrt((1.0 - d[:, 1] ** 2).clamp_min(0))

    def _env_pdf(self, tex, sin):
        return self.pmf[tex] * len(self.pmf) / (2 * math.pi ** 2) / sin

    # -- one view: every sample of every pixel as one batch of paths
    def view(self, v, seed):
        sc, dev, B = self.sc, self.dev, self.sc.max_bounces
        f64 = dict(device=dev, dtype=torch.float64)
        eye, at, up = (torch.tensor(np.float32(x).astype(np.float64), **f64) for x in (v.eye, v.target, v.up))
        fwd = _unit(at - eye)
        right = _unit(torch.linalg.cross(fwd, up))
        upv = torch.linalg.cross(right, fwd)
        th = math.tan(float(np.float32(v.fov_y_deg)) * math.pi / 360.0)
        n = v.width * v.height * v.spp
        job = torch.arange(n, device=dev)
        pixel, smp = job // v.spp, job % v.spp
        c0 = pixel + v.pixel_offset
        u = _philox(c0, smp, torch.zeros_like(c0), torch.zeros_like(c0), seed)
        sx = 2.0 * ((pixel % v.width) + _unif(u[0])) / v.width - 1.0
        sy = 1.0 - 2.0 * ((pixel // v.width) + _unif(u[1])) / v.height
        d = _unit(fwd + right * (sx * th * v.width / v.height)[:, None] + upv * (sy * th)[:, None])
        lights = [(np.asarray(p, np.float32), np.asarray(i, np.float32))
                  for p, i in list(zip(sc.light_pos, sc.light_intensity)) + list(v.lights)]
        lights = [(torch.tensor(p.astype(np.float64), **f64), torch.tensor(i.astype(np.float64), **f64))
                  for p, i in lights]
        total = torch.zeros((n, 3), **f64)
        idx, o, T = job, eye.expand(n, 3), torch.ones((n, 3), **f64)
        origin, last = torch.full((n,), -1, device=dev), None
        tri = self.V[self.F]
        flat = tri.detach()
        for b in range(B + 1):
            with torch.no_grad():
                face, _ = _closest(flat, o.detach(), d, origin)
            miss = face < 0
            if sc.env is not None and miss.any():
                with torch.no_grad():
                    tex, sin = self._texel(d[miss])
                    w = torch.ones_like(sin)
                    if b > 0:
                        pe = self._env_pdf(tex, sin)
                        w = last[miss] ** 2 / (last[miss] ** 2 + pe ** 2)
                    add = self.env[tex] * w[:, None]
                total = total.index_add(0, idx[miss], T[miss] * add)
            if b == B or bool(miss.all()):
                break
            k = ~miss
            idx, o, d, T, face = idx[k], o[k], d[k], T[k], face[k]
            v0, e1, e2 = tri[face, 0], tri[face, 1] - tri[face, 0], tri[face, 2] - tri[face, 0]
            m = torch.cross(e1, e2, dim=1)
            p = o + d * (_dot(v0 - o, m) / _dot(d, m))[:, None]
            wo = -d
            sgn = torch.where(_dot(m, wo) < 0, -1.0, 1.0).detach()[:, None]
            ng = _unit(m) * sgn
            q, mm = p - v0, _dot(m, m)
            b1, b2 = _dot(torch.cross(q, e2, dim=1), m) / mm, _dot(torch.cross(e1, q, dim=1), m) / mm
            ns = ng
            if sc.smooth_normals:
                nv = self.N[self.F[face]]
                ns = _unit(nv[:, 0] * (1 - b1 - b2)[:, None] + nv[:, 1] * b1[:, None] + nv[:, 2] * b2[:, None]) * sgn
            tex = face
            if sc.color_res:
                r = sc.color_res
                i = (r * b1.detach()).floor().long().clamp(0, r)
                j = torch.minimum((r * b2.detach()).floor().long().clamp_min(0), r - i)
                tex = face * ((r + 1) * (r + 2) // 2) + (i * (2 * r - i + 3)) // 2 + j
            mp = self.P[tex]
            mat = (mp[:, :3], mp[:, 3:6] if self.rgb else mp[:, 3:4].expand(-1, 3), mp[:, -1])
            held = tuple(x.detach() for x in mat)
            pd, nd, nsd = p.detach(), ng.detach(), ns.detach()

            def lit(wi, tmax, scale):
                """T f cos scale along wi where the direction counts and nothing blocks it."""
                with torch.no_grad():
                    wd = wi.detach()
                    ok = (_dot(nd, wd) > 0) & (_dot(nsd, wd) > 0) & (_dot(nsd, wo) > 0)
                    j = ok.nonzero()[:, 0]
                    blocked, _ = _closest(flat, pd[j], wd[j], face[j], tmax[j])
                    j = j[blocked < 0]
                val = self._value(tuple(x[j] for x in mat), ns[j], wi[j], wo[j])
                return idx[j], T[j] * val * scale[j]

            for lp, li in lights:
                dv = lp - p
                dist = dv.norm(dim=1)
                at_, add = lit(dv / dist[:, None], dist.detach() - 1e-5, li / (dist * dist)[:, None])
                total = total.index_add(0, at_, add)
            if sc.env is not None:
                h, w, _ = sc.env.shape
                with torch.no_grad():
                    u = _philox(c0[idx], smp[idx], torch.full_like(idx, (b << 4) | 1), torch.zeros_like(idx), seed)
                    bin_ = ((u[0] >> 8) * (w * h)) >> 24
                    te = torch.where(_unif(u[1]) < self.prob[bin_], bin_, self.alias[bin_])
                    ph = 2 * math.pi * ((te % w) + _unif(u[2])) / w
                    tt = math.pi * (torch.div(te, w, rounding_mode="floor") + _unif(u[3])) / h
                    wi = torch.stack([-tt.sin() * ph.sin(), tt.cos(), tt.sin() * ph.cos()], 1)
                    pe = self._env_pdf(te, tt.sin())
                    wt = torch.ones_like(pe)
                    if b < B - 1:
                        up_ = (_dot(nsd, wi) > 0) & (_dot(nsd, wo) > 0)
                        pb = torch.where(up_, self._pdf(held, nsd, wi, wo), 0.0)
                        wt = pe ** 2 / (pe ** 2 + pb ** 2)
                at_, add = lit(wi, torch.full_like(pe, math.inf), self.env[te] * (wt / pe)[:, None])
                total = total.index_add(0, at_, add)
            if b == B - 1:
                break
            with torch.no_grad():
                u = _philox(c0[idx], smp[idx], torch.full_like(idx, (b << 4) | 2), torch.zeros_like(idx), seed)
                wi = self._sample(held, nsd, wo, _unif(u[0]), _unif(u[1]), _unif(u[2]))
                ok = (_dot(nsd, wi) > 0) & (_dot(nsd, wo) > 0) & (_dot(nd, wi) > 0)
                pdf = self._pdf(held, nsd, wi, wo)
                ok &= pdf > 0
            if not bool(ok.any()):
                break
            T = T[ok] * self._value(tuple(x[ok] for x in mat), ns[ok], wi[ok], wo[ok]) / pdf[ok][:, None]
            idx, o, d, origin, last = idx[ok], p[ok], wi[ok], face[ok], pdf[ok]
        return torch.zeros((v.width * v.height, 3), **f64).index_add(0, pixel, total) / v.spp
