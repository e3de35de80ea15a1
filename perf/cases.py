"""Performance cases: the calls a user of this framework makes, over the range of sizes they use.

Each case is a dict of plain values whose "kind" names the call; `prepare` makes the inputs and the
handles a program keeps between calls (scene, BVH, renderer, guide), `run` is one pass through the
public entry points of `paper_2406_09733_gb300.ugp`, and `exact` gives the same outputs in 64 bits
with plain torch where that is affordable. Scenes follow the generators of
`paper_2406_09733_gb300.scenes` (the random scene in the unit cube and the room of surface splats
and aggregate clusters), drawn on the GPU so that millions of primitives take milliseconds.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2406_09733_gb300 import scenes, ugp

DEV = "cuda"
CUTOFF_EPS = 0.01
FAR = 8.0  # beyond every scene, seen from its camera


def listed():
    return [
        # the smallest calls: a probe of a scene of a thousand primitives with a few thousand rays
        # (interactive picking, a host application's visibility test)
        dict(name="query_small", kind="query", scene="tiny", prims=1000, rays=2048),
        # free flights at the size of one bounce of a 1024 x 1024 frame in a 1M-primitive room
        dict(name="free_flight_room", kind="free_flight", scene="room", prims=1_000_000, rays=1_048_576),
        # light-sample transmittances of such a bounce, an odd number of them
        dict(name="transmittance_room", kind="transmittance", scene="room", prims=1_000_000, rays=1_000_003),
        # the small plain configuration: 1,000 primitives, 128 x 128, 4 samples, depth 4
        dict(name="render_tiny", kind="render", scene="tiny", prims=1000, width=128, height=128, spp=4, depth=4,
             disney=0.0),
        # one sample per pixel of the paper-scale frame
        dict(name="render_large", kind="render", scene="room", prims=5_500_000, width=1920, height=1080, spp=1,
             depth=12, disney=0.0),
        # an edited scene: rebuild the BVH, then a few probe rays
        dict(name="rebuild_large", kind="rebuild", scene="room", prims=5_500_000, rays=16_384),
        # an online-training frame of the learned guide in a room lit by small emitters, with
        # light sampling of the emitters and Disney materials
        dict(name="guided_training", kind="guided", scene="room_b", prims=300_000, width=480, height=270, depth=8,
             minibatch=16384, disney=0.2),
        # the guide alone: proposals for a frame's vertices, and one optimiser step of a minibatch
        dict(name="guide_forward", kind="guide_forward", rows=1_000_000),
        dict(name="guide_step", kind="guide_step", rows=65_536),
        # uneven render requests over several scenes, served as one batch
        dict(name="serving", kind="serving", prims=300_000, scenes=4, requests=12, size=384, spp=8, depth=8,
             pool_log2=18),
        # a deterministic radiance-field view (1280 x 720 camera rays)
        dict(name="radiance_field", kind="radiance", scene="room", prims=1_000_000, rays=921_600),
        # compressing a scene to codebook records and reading it back
        dict(name="codebook", kind="codebook", prims=1_000_000, iters=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "free_flight", "transmittance", "render", "rebuild", "guided", "guide_forward",
                       "guide_step", "serving", "radiance", "codebook"])
    scene = "tiny" if rng.random() < 0.2 else "room"
    prims = _log(rng, 500, 5000) if scene == "tiny" else _log(rng, 20_000, 3_000_000)
    if kind == "query":
        return dict(kind=kind, scene=scene, prims=min(prims, 60_000), rays=_log(rng, 1, 8192))
    if kind in ("free_flight", "transmittance", "radiance"):
        return dict(kind=kind, scene=scene, prims=prims, rays=_log(rng, 4000, 1_500_000))
    if kind == "render":
        w = _log(rng, 32, 1200)
        h = max(16, int(w * rng.uniform(0.5, 1.0)))
        spp = max(1, min(8, 400_000 // (w * h)))
        return dict(kind=kind, scene=scene, prims=prims, width=w, height=h, spp=spp, depth=rng.randint(1, 12),
                    disney=rng.choice([0.0, 0.0, 0.3]))
    if kind == "rebuild":
        return dict(kind=kind, scene="room", prims=_log(rng, 10_000, 5_000_000), rays=_log(rng, 256, 16_384))
    if kind == "guided":
        w = _log(rng, 64, 480)
        return dict(kind=kind, scene="room_b", prims=_log(rng, 20_000, 500_000), width=w,
                    height=max(16, int(w * rng.uniform(0.5, 0.7))), depth=rng.randint(2, 8),
                    minibatch=rng.choice([4096, 16384, 65536]), disney=rng.choice([0.0, 0.3]))
    if kind == "guide_forward":
        return dict(kind=kind, rows=_log(rng, 100, 1_000_000))
    if kind == "guide_step":
        return dict(kind=kind, rows=_log(rng, 1000, 1_000_000))
    if kind == "serving":
        return dict(kind=kind, prims=_log(rng, 20_000, 300_000), scenes=rng.randint(1, 4),
                    requests=rng.randint(2, 12), size=rng.choice([96, 150, 256, 320]), spp=rng.randint(1, 8),
                    depth=rng.randint(3, 8), pool_log2=rng.choice([16, 18, 20]))
    return dict(kind=kind, prims=_log(rng, 10_000, 1_000_000), iters=rng.randint(2, 8))


# ------------------------------------------------------------------ scenes on the GPU
class _Gen:
    """Seeded draws on the GPU, in float64 (rounded to float32 once the scene is made)."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed))

    def rand(self, *shape):
        return torch.rand(shape, generator=self.g, device=DEV, dtype=torch.float64)

    def uniform(self, lo, hi, *shape):
        return lo + (hi - lo) * self.rand(*shape)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device=DEV, dtype=torch.float64)

    def integers(self, n, *shape):
        return torch.randint(0, n, shape, generator=self.g, device=DEV)

    def unit(self, n):
        v = self.normal(n, 3)
        return v / v.norm(dim=1, keepdim=True)

    def uniforms24(self, n):
        return (torch.randint(0, 1 << 24, (n,), generator=self.g, device=DEV).double() * 2.0 ** -24).float()

    def quaternions(self, n):
        q = self.normal(n, 4)
        return q / q.norm(dim=1, keepdim=True)


def _quat_of_frame(t1, t2, nrm):
    """Quaternions (w, x, y, z) of the rotations whose columns are (t1, t2, nrm)."""
    m = torch.stack([t1, t2, nrm], 2)
    d = torch.diagonal(m, dim1=1, dim2=2)
    tr = d.sum(1)
    # the four candidates scaled by their own largest component; the best-conditioned one is taken
    a = torch.stack([1 + tr, 1 + 2 * d[:, 0] - tr, 1 + 2 * d[:, 1] - tr, 1 + 2 * d[:, 2] - tr], 1)
    wx, wy, wz = m[:, 2, 1] - m[:, 1, 2], m[:, 0, 2] - m[:, 2, 0], m[:, 1, 0] - m[:, 0, 1]
    xy, xz, yz = m[:, 0, 1] + m[:, 1, 0], m[:, 0, 2] + m[:, 2, 0], m[:, 1, 2] + m[:, 2, 1]
    cand = torch.stack([torch.stack([a[:, 0], wx, wy, wz], 1), torch.stack([wx, a[:, 1], xy, xz], 1),
                        torch.stack([wy, xy, a[:, 2], yz], 1), torch.stack([wz, xz, yz, a[:, 3]], 1)], 1)
    q = cand.gather(1, a.argmax(1).view(-1, 1, 1).expand(-1, 1, 4)).squeeze(1)
    return q / q.norm(dim=1, keepdim=True)


def _f32(d):
    return {k: (v if v is None or v.dtype == torch.uint8 else v.float()).contiguous() if v is not None else None
            for k, v in d.items()}


def _tiny(n, seed):
    """Random Gaussians in the unit cube; primitive 0 is an emitter. The sizes keep the optical
    depth of the thousand-primitive scene whatever n."""
    g = _Gen(seed)
    f = (1000.0 / n) ** (1.0 / 3.0)
    scale = f * torch.exp(g.uniform(math.log(0.01), math.log(0.05), n, 3))
    rho = g.uniform(0.5, 5.0, n)
    mtype = torch.full((n,), scenes.MAT_DIFFUSE, dtype=torch.uint8, device=DEV)
    mtype[0] = scenes.MAT_EMISSIVE
    emission = torch.zeros(n, 3, dtype=torch.float64, device=DEV)
    emission[0] = 10.0
    sggx = torch.tensor([1.0, 1, 1, 0, 0, 0], dtype=torch.float64, device=DEV).repeat(n, 1)
    return _f32(dict(mean=g.rand(n, 3), quat=g.quaternions(n), scale=scale,
                     magnitude=rho * (2 * math.pi) ** 1.5 * scale.prod(1), sggx=sggx, mtype=mtype,
                     albedo=g.uniform(0.2, 0.8, n, 3), roughness=torch.full((n,), 0.3, dtype=torch.float64, device=DEV),
                     emission=emission, disney=None))


def _room(n, seed, emitters=False, disney=0.0):
    """The room: 70 % surface splats on five planes, 12 spheres and 8 boxes, 30 % isotropic
    primitives in Gaussian clusters; mixed materials, a tenth of the surfaces near-specular."""
    g = _Gen(seed)
    rng = np.random.Generator(np.random.Philox(int(seed)))
    n_surf = int(round(0.7 * n))
    n_aggr = n - n_surf
    t = lambda v: torch.tensor(v, dtype=torch.float64, device=DEV)
    X, Y, Z, o = (t(v) for v in ([1.0, 0, 0], [0.0, 1, 0], [0.0, 0, 1], [0.0, 0, 0]))
    shapes = [("plane", (o, Z, X), 1.0), ("plane", (Y, X, Z), 1.0), ("plane", (Z, X, Y), 1.0),
              ("plane", (o, Y, Z), 1.0), ("plane", (X, Z, Y), 1.0)]
    for _ in range(12):
        r = rng.uniform(0.05, 0.15)
        shapes.append(("sphere", (t(rng.uniform(0.2, 0.8, 3)), r), 4 * math.pi * r * r))
    for _ in range(8):
        e = rng.uniform(0.05, 0.2)
        lo = rng.uniform(0.05, 0.95 - e, 3)
        lo[1] = 0.0
        shapes.append(("box", (t(lo), e), 6 * e * e))
    area = np.array([s[2] for s in shapes])
    counts = np.floor(n_surf * area / area.sum()).astype(np.int64)
    counts[0] += n_surf - counts.sum()
    P, N = [], []
    for (kind, prm, _), m in zip(shapes, counts):
        m = int(m)
        if kind == "plane":
            c, e1, e2 = prm
            uv = g.rand(m, 2)
            P.append(c + uv[:, :1] * e1 + uv[:, 1:] * e2)
            N.append(torch.linalg.cross(e1, e2).expand(m, 3))
        elif kind == "sphere":
            nv = g.unit(m)
            P.append(prm[0] + prm[1] * nv)
            N.append(nv)
        else:
            lo, e = prm
            face = g.integers(6, m)
            p = g.rand(m, 3) * e
            side = (face % 2).double()
            hot = torch.nn.functional.one_hot(face // 2, 3).double()
            P.append(lo + p * (1 - hot) + hot * (side * e)[:, None])
            N.append(hot * (2 * side - 1)[:, None])
    p, nrm = torch.cat(P), torch.cat(N)
    sid = torch.repeat_interleave(torch.arange(len(shapes), device=DEV), torch.from_numpy(counts).to(DEV))
    a = g.normal(n_surf, 3)
    t1 = a - (a * nrm).sum(1, keepdim=True) * nrm
    t1 = t1 / t1.norm(dim=1, keepdim=True)
    t2 = torch.linalg.cross(nrm, t1)
    s_t = torch.sqrt(0.16 * t(area) / t(np.maximum(counts, 1).astype(float)))[sid]
    S = nrm[:, :, None] * nrm[:, None] + 1e-4 * (t1[:, :, None] * t1[:, None] + t2[:, :, None] * t2[:, None])
    sggx = torch.stack([S[:, 0, 0], S[:, 1, 1], S[:, 2, 2], S[:, 0, 1], S[:, 0, 2], S[:, 1, 2]], 1)
    # clusters keep the density of 300 per million primitives
    n_cl = max(1, int(round(300 * n / 1e6)))
    cl = g.integers(n_cl, n_aggr)
    ap = g.uniform(0.1, 0.9, n_cl, 3)[cl] + 0.03 * g.normal(n_aggr, 3)
    s_a = torch.exp(g.uniform(math.log(0.003), math.log(0.01), n_aggr))

    def kinds(m, rough_lo):
        u = g.rand(m)
        ty = torch.where(u < 0.5, scenes.MAT_DIFFUSE, torch.where(u < 0.9, scenes.MAT_GGX, scenes.MAT_EMISSIVE))
        return (ty, g.uniform(0.2, 0.8, m, 3), g.uniform(rough_lo, 0.5, m),
                g.uniform(0.5, 5.0, m, 1) * g.uniform(0.3, 1.0, m, 3))

    ty_s, al_s, ro_s, em_s = kinds(len(shapes), 0.05)
    ty_s[:5] = torch.where(g.rand(5) < 0.7, scenes.MAT_DIFFUSE, scenes.MAT_GGX)
    near = g.rand(len(shapes)) < 0.1
    ty_s[near] = scenes.MAT_GGX
    ro_s[near] = 0.02
    ty_c, al_c, ro_c, em_c = kinds(n_cl, 0.05)
    mtype = torch.cat([ty_s[sid], ty_c[cl]]).to(torch.uint8)
    emission = torch.cat([em_s[sid], em_c[cl]])
    emission[mtype != scenes.MAT_EMISSIVE] = 0.0
    if emitters:  # small emissive aggregates: the density of 12,000 per million primitives
        k = max(1, int(0.012 * n))
        pick = n_surf + torch.randperm(n_aggr, generator=g.g, device=DEV)[:k]
        mtype[pick] = scenes.MAT_EMISSIVE
        emission[pick] = g.uniform(2.0, 20.0, k, 1) * g.uniform(0.5, 1.0, k, 3)
    dis = None
    if disney > 0:
        pick = (mtype != scenes.MAT_EMISSIVE) & (g.rand(n) < disney)
        mtype[pick] = scenes.MAT_DISNEY
        dis = g.rand(n, 9)
        dis[:, 4] = g.uniform(0.3, 0.9, n)
        dis[:, 7] *= (g.rand(n) < 0.5).double()
        dis[~pick] = 0.0
    iso = torch.tensor([1.0, 1, 1, 0, 0, 0], dtype=torch.float64, device=DEV).repeat(n_aggr, 1)
    return _f32(dict(mean=torch.cat([p, ap]), quat=torch.cat([_quat_of_frame(t1, t2, nrm), g.quaternions(n_aggr)]),
                     scale=torch.cat([torch.stack([s_t, s_t, 0.01 * s_t], 1), s_a[:, None].expand(-1, 3)]),
                     magnitude=torch.cat([6 * math.pi * s_t * s_t,
                                          4 * math.pi * g.uniform(0.05, 0.5, n_aggr) * s_a * s_a]),
                     sggx=torch.cat([sggx, iso]), mtype=mtype, albedo=torch.cat([al_s[sid], al_c[cl]]),
                     roughness=torch.cat([ro_s[sid], ro_c[cl]]), emission=emission, disney=dis))


def _scene(case, seed):
    if case.get("scene") == "tiny":
        return _tiny(case["prims"], seed)
    return _room(case["prims"], seed, emitters=case.get("scene") == "room_b", disney=case.get("disney", 0.0))


def _bvh(s):
    return ugp.build_bvh(s["mean"], s["quat"], s["scale"], s["magnitude"], CUTOFF_EPS)


def _materials(s):
    return ugp.Materials(s["sggx"], s["mtype"], s["albedo"], s["roughness"], s["emission"], s["disney"])


def _camera(case, w, h):
    if case.get("scene") == "tiny":
        return ugp.camera_struct((0.5, 0.5, -1.5), (0.5, 0.5, 0.5), (0.0, 1.0, 0.0), 40.0, w, h)
    return ugp.camera_struct((0.5, 0.5, -0.8), (0.5, 0.5, 0.5), (0.0, 1.0, 0.0), 45.0, w, h)


def _lights(case):
    if case.get("scene") == "room_b":
        return ugp.lights_struct()
    if case.get("scene") == "tiny":
        return ugp.lights_struct(bg=(0.2, 0.2, 0.2))
    return ugp.lights_struct(True, (0.35, 0.98, 0.35), (0.3, 0, 0), (0, 0, 0.3), (20, 20, 20), (0.2, 0.2, 0.2))


def _unit32(v):
    v = v.float()
    return (v.double() / v.double().norm(dim=1, keepdim=True)).float().contiguous()


def _camera_rays(case, g, n):
    """Pinhole rays through random points of the case's image."""
    tiny = case["scene"] == "tiny"
    eye = torch.tensor([0.5, 0.5, -1.5 if tiny else -0.8], dtype=torch.float64, device=DEV)
    th = math.tan(math.radians(20.0 if tiny else 22.5))
    # image order: rays of neighbouring pixels are neighbours, as a renderer's are
    w = max(1, int(math.sqrt(n * 16 / 9)))
    i = torch.arange(n, device=DEV)
    h = (n + w - 1) // w
    x = (2 * ((i % w).double() + g.rand(n)) / w - 1) * th * w / h
    y = (1 - 2 * ((i // w).double() + g.rand(n)) / h) * th
    d = torch.stack([-x, y, torch.ones_like(x)], 1)
    return eye.expand(n, 3).float().contiguous(), _unit32(d)


def _bounce_rays(s, g, n):
    """Rays that leave primitives in random directions (a path's later vertices), with the primitive
    they leave."""
    k = g.integers(s["mean"].shape[0], n)
    return s["mean"][k].contiguous(), _unit32(g.unit(n)), k.int()


def _query_rays(case, s, g):
    """Half camera rays, half bounce rays, a quarter of them ending inside the scene."""
    n = case["rays"]
    m = n // 2
    o1, d1 = _camera_rays(case, g, n - m)
    o2, d2, k = _bounce_rays(s, g, m)
    ex = torch.cat([torch.full((n - m,), -1, dtype=torch.int32, device=DEV), k])
    t1 = torch.full((n,), FAR, dtype=torch.float32, device=DEV)
    cut = g.rand(n) < 0.25
    t1 = torch.where(cut, g.uniform(0.2, 2.0, n).float(), t1)
    return dict(o=torch.cat([o1, o2]).contiguous(), d=torch.cat([d1, d2]).contiguous(),
                t0=torch.zeros(n, dtype=torch.float32, device=DEV), t1=t1.contiguous(), ex=ex.contiguous(),
                u=g.uniforms24(n), u2=g.uniforms24(n))


def _shadow_rays(case, s, g):
    """From primitives to points of the light below the ceiling, skipping the primitive left."""
    n = case["rays"]
    o, _, k = _bounce_rays(s, g, n)
    y = torch.stack([g.uniform(0.35, 0.65, n), torch.full((n,), 0.98, dtype=torch.float64, device=DEV),
                     g.uniform(0.35, 0.65, n)], 1)
    v = y - o.double()
    r = v.norm(dim=1, keepdim=True).clamp_min(1e-3)
    return dict(o=o, d=_unit32(v / r), t0=torch.zeros(n, dtype=torch.float32, device=DEV),
                t1=r[:, 0].float().contiguous(), ex=k)


def _rays_of(case, s, seed):
    g = _Gen(int(seed) + 7777)
    if case["kind"] in ("transmittance", "rebuild"):
        return _shadow_rays(case, s, g)
    if case["kind"] == "radiance":
        n = case["rays"]
        o, d = _camera_rays(case, g, n)
        return dict(o=o, d=d, t0=torch.zeros(n, dtype=torch.float32, device=DEV),
                    t1=torch.full((n,), FAR, dtype=torch.float32, device=DEV))
    return _query_rays(case, s, g)


def _radiance_colours(case, seed):
    """Per-primitive colours of a radiance field, and the background."""
    g = _Gen(int(seed) + 99)
    return g.rand(case["prims"], 3).float().contiguous(), (0.1, 0.2, 0.3)


def _vertices(rows, seed, weights):
    g = _Gen(int(seed) + 5)
    x = g.uniform(-0.05, 1.05, rows, 3).float().contiguous()
    out = dict(x=x, wo=_unit32(g.unit(rows)))
    if weights:
        w = 10.0 ** g.uniform(-2, 2, rows)
        w[g.rand(rows) < 0.1] = 0.0
        out.update(wi=_unit32(g.unit(rows)), w=w.float().contiguous())
    return out


def _requests(case, seed):
    """(scene, width, height, spp, depth, seed) of every request, uneven in all but the seeds."""
    rng = np.random.Generator(np.random.Philox(31))
    out = []
    for i in range(case["requests"]):
        w = int(case["size"] * rng.choice([0.5, 1.0, 1.0, 1.5]))
        h = int(w * rng.uniform(0.6, 1.0))
        out.append((int(rng.integers(0, case["scenes"])), w, h, int(rng.integers(1, case["spp"] + 1)),
                    int(rng.integers(min(3, case["depth"]), case["depth"] + 1)), 1000 * int(seed) + i))
    return out


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, case=case)
    if kind in ("guide_forward", "guide_step"):
        st["v"] = _vertices(case["rows"], seed, kind == "guide_step")
        st["guide"] = ugp.Guide(scenes.guide_init_params(int(seed), 0.1), device=DEV)
        return st
    if kind == "serving":
        sizes = [max(1000, int(case["prims"] * f)) for f in (1.0, 0.4, 0.15, 0.05)][:case["scenes"]]
        st["scenes"] = []
        for k, n in enumerate(sizes):
            s = _room(n, 10 * int(seed) + k, emitters=k % 2 == 1)
            st["scenes"].append((s, _bvh(s), _materials(s)))
        st["specs"] = _requests(case, seed)
        st["server"] = ugp.BatchRenderer(case["requests"], pool_log2=case["pool_log2"], device=DEV)
        return st
    s = _room(case["prims"], seed, disney=0.3) if kind == "codebook" else _scene(case, seed)
    st["s"] = s
    if kind == "codebook":
        st["mats"] = _materials(s)
        return st
    if kind == "rebuild":
        st["r"] = _rays_of(case, s, seed)
        st["ws"] = torch.empty(ugp.build_bvh_workspace_size(case["prims"]), dtype=torch.uint8, device=DEV)
        return st
    st["bvh"] = _bvh(s)
    if kind in ("render", "guided"):
        w, h = case["width"], case["height"]
        st["mats"] = _materials(s)
        st["cam"], st["lights"] = _camera(case, w, h), _lights(case)
        st["renderer"] = ugp.Renderer(w, h, device=DEV)
        st["seed"] = int(seed)
        if kind == "guided":
            st["guide"] = ugp.Guide(scenes.guide_init_params(int(seed)), device=DEV)
            st["emitters"] = ugp.build_emitter_table(st["bvh"], st["mats"])
        return st
    st["r"] = _rays_of(case, s, seed)
    if kind == "radiance":
        st["colours"], st["bg"] = _radiance_colours(case, seed)
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "query":
        r = st["r"]
        T, Ts = ugp.trace_transmittance(st["bvh"], r["o"], r["d"], r["t0"], r["t1"], exclude=r["ex"])
        p, tu, tsp, fs = ugp.sample_free_flight(st["bvh"], r["o"], r["d"], r["t0"], r["t1"], r["u"], r["u2"],
                                                exclude=r["ex"])
        return dict(T=T, T_status=Ts, prim=p, t_u=tu, t_spawn=tsp, status=fs)
    if kind == "free_flight":
        r = st["r"]
        p, tu, tsp, fs = ugp.sample_free_flight(st["bvh"], r["o"], r["d"], r["t0"], r["t1"], r["u"], r["u2"],
                                                exclude=r["ex"])
        return dict(prim=p, t_u=tu, t_spawn=tsp, status=fs)
    if kind == "transmittance":
        r = st["r"]
        T, s = ugp.trace_transmittance(st["bvh"], r["o"], r["d"], r["t0"], r["t1"], exclude=r["ex"])
        return dict(T=T, status=s)
    if kind == "radiance":
        r = st["r"]
        rgb, s = ugp.render_radiance_field(st["bvh"], r["o"], r["d"], r["t0"], r["t1"], st["colours"], st["bg"])
        return dict(rgb=rgb, status=s)
    if kind == "rebuild":
        s, r = st["s"], st["r"]
        bvh = ugp.build_bvh(s["mean"], s["quat"], s["scale"], s["magnitude"], CUTOFF_EPS, workspace=st["ws"])
        T, ts = ugp.trace_transmittance(bvh, r["o"], r["d"], r["t0"], r["t1"], exclude=r["ex"])
        return dict(T=T, status=ts)
    if kind == "render":
        acc, acc2 = st["renderer"].render(st["bvh"], st["mats"], st["cam"], st["lights"], case["spp"], case["depth"],
                                          seed=st["seed"])
        return dict(accum=acc, accum_sq=acc2)
    if kind == "guided":
        acc, acc2 = st["renderer"].render(st["bvh"], st["mats"], st["cam"], st["lights"], 1, case["depth"],
                                          seed=st["seed"], guide=st["guide"], guide_log=True,
                                          emitters=st["emitters"])
        n, loss = st["guide"].train_from(st["renderer"], minibatch=case["minibatch"])
        return dict(accum=acc, accum_sq=acc2, samples=n, loss=loss, params=st["guide"].params)
    if kind == "guide_forward":
        Y, M = st["guide"].forward(st["v"]["x"], st["v"]["wo"])
        return dict(head=Y, mixture=M)
    if kind == "guide_step":
        v = st["v"]
        g, loss = st["guide"].grad(v["x"], v["wo"], v["wi"], v["w"])
        st["guide"].adam_step(g)
        return dict(grad=g, loss=loss, params=st["guide"].params)
    if kind == "serving":
        reqs = []
        for sc, w, h, spp, depth, seed in st["specs"]:
            _, bvh, mats = st["scenes"][sc]
            lit = dict(scene="room_b" if sc % 2 else "room")
            reqs.append(ugp.Request(bvh, mats, _camera(lit, w, h), _lights(lit), spp, depth, seed=seed, device=DEV))
        st["server"].render(reqs)
        return [q.accum for q in reqs] + [q.accum_sq for q in reqs]
    s = st["s"]
    book, rec = ugp.codebook_encode(s["mean"], s["quat"], s["scale"], s["magnitude"], st["mats"], iters=case["iters"])
    out = ugp.codebook_decode(rec, book)
    return dict(book=book, records=rec, decoded=out)


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Bytes: the caller's arrays read once and the results written once. Operations: about 60 per
    interval of a ray (the ellipsoid test and its share of the integral), with the intervals a ray
    of these scenes meets (20 in the random scene, 60 in the room), and the arithmetic of the
    network or of the assignment to codebook entries."""
    kind = case["kind"]
    n, rays = case.get("prims", 0), case.get("rays", 0)
    per_ray = 60 * (20 if case.get("scene") == "tiny" else 60)
    prim_b, mat_b = 44, 61
    if kind == "query":
        return dict(bytes=44 * n + rays * (44 + 18), flops=2 * rays * per_ray)
    if kind == "free_flight":
        return dict(bytes=44 * n + rays * (44 + 13), flops=rays * per_ray)
    if kind == "transmittance":
        return dict(bytes=44 * n + rays * (36 + 5), flops=rays * per_ray)
    if kind == "radiance":
        return dict(bytes=56 * n + rays * (32 + 13), flops=rays * per_ray)
    if kind == "rebuild":
        return dict(bytes=44 * n + rays * (36 + 5), flops=200 * n + rays * per_ray)
    if kind in ("render", "guided"):
        px = case["width"] * case["height"] * case.get("spp", 1)
        q = px * (2 if case["scene"] == "tiny" else min(7, 2 + case["depth"]))
        b = dict(bytes=(prim_b + mat_b) * n + 24 * px, flops=q * (per_ray + 300))
        if kind == "guided":
            b["flops"] += q // 2 * (37_888 + 105_472)
        return b
    if kind == "guide_forward":
        return dict(bytes=case["rows"] * (24 + 320) + 4 * 19240, flops=37_888 * case["rows"])
    if kind == "guide_step":
        return dict(bytes=case["rows"] * 40 + 4 * 19240 * 8, flops=105_472 * case["rows"])
    if kind == "serving":
        px = int(case["requests"] * case["size"] ** 2 * 0.8)
        q = int(px * 0.5 * (case["spp"] + 1)) * min(7, 2 + case["depth"])
        return dict(bytes=(prim_b + mat_b) * n + 24 * px, flops=q * (per_ray + 300))
    # every point against the 4096 entries of four codebooks (29 values), iters + 1 times
    return dict(bytes=n * (44 + 97 - 44 + 24 + 24 + 97), flops=2 * 29 * 4096 * n * (case["iters"] + 1))


# ------------------------------------------------------------------ the same results in 64 bits
def exact(case, seed):
    kind = case["kind"]
    if kind in ("query", "free_flight", "transmittance", "radiance", "rebuild"):
        pairs = case["rays"] * case["prims"] * (1 if kind in ("transmittance", "rebuild") else 40)
        if pairs > 4e9:
            return None
        s = _scene(case, seed)
        r = _rays_of(case, s, seed)
        if kind in ("transmittance", "rebuild"):
            return dict(T=_exact_rays(case, s, r, want="T")["T"], status=None)
        if kind == "query":
            e = _exact_rays(case, s, r, want="T t_u")
            return dict(T=e["T"], T_status=None, prim=None, t_u=e["t_u"], t_spawn=None, status=None)
        if kind == "free_flight":
            e = _exact_rays(case, s, r, want="t_u")
            return dict(prim=None, t_u=e["t_u"], t_spawn=None, status=None)
        col, bg = _radiance_colours(case, seed)
        e = _exact_rays(case, s, r, want="rgb", colours=col.double(), bg=bg)
        return dict(rgb=e["rgb"], status=None)
    if kind == "guide_forward":
        return _exact_guide_forward(case, seed)
    if kind == "guide_step":
        return _exact_guide_step(case, seed)
    if kind == "codebook":
        return _exact_codebook(case, seed)
    return None


def _exact_rays(case, s, r, want, colours=None, bg=None):
    """Every ray against every primitive (Eq. 1, 4, 6, 7 and 8)."""
    k2 = -2.0 * math.log(CUTOFF_EPS)
    q = s["quat"].double()
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    sc = s["scale"].double()
    W = R.transpose(1, 2) / sc[:, :, None]
    g0 = s["magnitude"].double() / ((2 * math.pi) ** 1.5 * sc.prod(1))
    wm = torch.einsum("nij,nj->ni", W, s["mean"].double())
    n, N = r["o"].shape[0], W.shape[0]
    ids = torch.arange(N, device=DEV)
    out = {k: [] for k in ("T", "t_u", "rgb")}
    step = max(1, int(2e7) // N)
    sq = math.sqrt(math.pi)
    for i in range(0, n, step):
        o, d = r["o"][i:i + step].double(), r["d"][i:i + step].double()
        t0, t1 = r["t0"][i:i + step].double()[:, None], r["t1"][i:i + step].double()[:, None]
        wo = torch.einsum("nij,rj->rni", W, o) - wm
        wd = torch.einsum("nij,rj->rni", W, d)
        A = (wd * wd).sum(2)
        tc = -(wo * wd).sum(2) / A
        c = wo + tc[:, :, None] * wd
        d2 = (c * c).sum(2)
        half = torch.sqrt(((k2 - d2) / A).clamp_min(0))
        a, b = torch.maximum(t0, tc - half), torch.minimum(t1, tc + half)
        hit = (d2 < k2) & (a < b)
        if "ex" in r:
            hit &= ids[None] != r["ex"][i:i + step][:, None]
        # the pairs that meet, in ray order
        ri, pi = hit.nonzero(as_tuple=True)
        a, b, tc, ss = a[hit], b[hit], tc[hit], torch.sqrt(0.5 * A[hit])
        amp = g0[pi] * torch.exp(-0.5 * d2[hit]) * (0.25 * sq) / ss
        ea = torch.erf(ss * (a - tc))
        m = o.shape[0]

        def F(t):
            y = torch.minimum(b, t[ri])
            v = torch.where(y > a, amp * (torch.erf(ss * (y - tc)) - ea), torch.zeros_like(a))
            return v, torch.zeros(m, dtype=torch.float64, device=DEV).index_add_(0, ri, v)

        end = t1[:, 0].contiguous()
        _, Fe = F(end)
        out["T"].append((1 - Fe).clamp_min(0))
        if "t_u" in want or "rgb" in want:
            u = r["u"][i:i + step].double() if "t_u" in want else torch.ones(m, dtype=torch.float64, device=DEV)
            last = torch.zeros(m, dtype=torch.float64, device=DEV).scatter_reduce(0, ri, b, "amax")
            lo, hi = t0[:, 0].clone(), torch.maximum(last, t0[:, 0])
            for _ in range(60):
                mid = 0.5 * (lo + hi)
                over = F(mid)[1] > u
                lo, hi = torch.where(over, lo, mid), torch.where(over, mid, hi)
            tu = torch.where(Fe > u, 0.5 * (lo + hi), end)
            out["t_u"].append(tu)
            if "rgb" in want:
                v, _ = F(tu)
                rgb = torch.zeros(m, 3, dtype=torch.float64, device=DEV).index_add_(0, ri, v[:, None] * colours[pi])
                rest = torch.where(Fe <= 1, 1 - Fe, torch.zeros_like(Fe))
                out["rgb"].append(rgb + rest[:, None] * torch.tensor(bg, dtype=torch.float64, device=DEV))
    return {k: torch.cat(v) for k, v in out.items() if v}


def _net(params, x, wo):
    """Head outputs of the guide's network, 64 bits."""
    xn = x.double().clamp(0, 1)
    w = wo.double()
    th, ph = torch.acos(w[:, 2].clamp(-1, 1)), torch.atan2(w[:, 1], w[:, 0])
    f = []
    for v, top, base in ((xn[:, 0], 6, math.pi), (xn[:, 1], 6, math.pi), (xn[:, 2], 6, math.pi), (th, 4, 1.0),
                         (ph, 4, 1.0)):
        for l in range(top):
            f += [torch.sin(base * 2 ** l * v), torch.cos(base * 2 ** l * v)]
    f += [xn[:, 0], xn[:, 1], xn[:, 2], th / math.pi, ph / (2 * math.pi) + 0.5]
    h = torch.stack(f + [torch.zeros_like(th)] * (64 - len(f)), 1)
    for l, (ws, bs) in enumerate(scenes.guide_param_slices()):
        o, i = scenes.GUIDE_SHAPES[l]
        h = h @ params[ws].view(o, i).T + params[bs]
        if l < scenes.GUIDE_LAYERS:
            h = torch.relu(h)
    return h


def _lobes(Y):
    L = Y.view(-1, scenes.GUIDE_LOBES, 5)
    mu = L[:, :, :3] / L[:, :, :3].norm(dim=2, keepdim=True)
    kappa = (0.1 + torch.nn.functional.softplus(L[:, :, 3])).clamp_max(1e4)
    return mu, kappa, torch.softmax(L[:, :, 4], 1)


def _exact_guide_forward(case, seed):
    v = _vertices(case["rows"], seed, False)
    p = torch.from_numpy(scenes.guide_init_params(int(seed), 0.1)).to(DEV).double()
    with torch.no_grad():
        Y = _net(p, v["x"], v["wo"])
        mu, kappa, pi = _lobes(Y)
        M = torch.cat([mu, kappa[:, :, None], pi[:, :, None]], 2).reshape(-1, 40)
    return dict(head=Y, mixture=M)


def _exact_guide_step(case, seed):
    v = _vertices(case["rows"], seed, True)
    p = torch.from_numpy(scenes.guide_init_params(int(seed), 0.1)).to(DEV).double().requires_grad_(True)
    loss = 0.0
    for i in range(0, case["rows"], 1 << 17):
        j = slice(i, i + (1 << 17))
        mu, kappa, pi = _lobes(_net(p, v["x"][j], v["wo"][j]))
        cw = (mu * v["wi"][j].double()[:, None]).sum(2)
        lq = torch.logsumexp(torch.log(pi) + torch.log(kappa) - math.log(2 * math.pi)
                             - torch.log(-torch.expm1(-2 * kappa)) + kappa * (cw - 1), 1)
        part = -(v["w"][j].double() * lq).sum() / case["rows"]
        part.backward()
        loss += float(part.detach())
    g = p.grad
    new = p.detach() - 1e-3 * g / (g.abs() + 1e-8)  # the first step of Adam
    return dict(grad=g, loss=torch.tensor([loss], dtype=torch.float64, device=DEV), params=new)


def _exact_codebook(case, seed):
    s = _room(case["prims"], seed, disney=0.3)
    n, K = case["prims"], 4096
    q = s["quat"].double()
    q = torch.where(q[:, :1] < 0, -q, q) / q.norm(dim=1, keepdim=True)
    parts = [torch.log(s["scale"].double()), q, s["sggx"].double(),
             torch.cat([s["albedo"], s["roughness"][:, None], s["emission"], s["disney"]], 1).double()]
    start = (torch.arange(K, device=DEV) * n) // K
    books, near = [], []
    for X in parts:
        B = X[start].clone()
        for it in range(case["iters"] + 1):
            code = torch.empty(n, dtype=torch.long, device=DEV)
            for i in range(0, n, 1 << 16):
                x = X[i:i + (1 << 16)]
                code[i:i + (1 << 16)] = ((B * B).sum(1)[None] - 2 * x @ B.T).argmin(1)
            if it == case["iters"]:
                break
            cnt = torch.bincount(code, minlength=K)
            m = torch.zeros_like(B).index_add_(0, code, X) / cnt.clamp_min(1)[:, None]
            B = torch.where((cnt > 0)[:, None], m, B)
        books.append(B)
        near.append(B[code])
    r = near[3]
    dec = dict(mean=s["mean"].double(), quat=near[1] / near[1].norm(dim=1, keepdim=True), scale=torch.exp(near[0]),
               magnitude=s["magnitude"].double(), sggx=near[2], mtype=None, albedo=r[:, :3].contiguous(),
               roughness=r[:, 3].contiguous(), emission=r[:, 4:7].contiguous(), disney=r[:, 7:].contiguous())
    return dict(book=torch.cat(books, 1), records=None, decoded=dec)
