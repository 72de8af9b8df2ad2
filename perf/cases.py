"""The calls whose speed this framework is measured by, at sizes its users meet.

Each kind of case is one call (or the pair of calls a program always makes
together) of `paper_2510_07729_gb300.sop`:

  bake     every texel of a probe set traced through a Gaussian cloud
  query    shading points against baked probes (SHADE on the object, SHADOW on the receiver)
  relight  importance-sampled directions of a new octahedral environment, then the shading with them
  grad     the differentiable query, forward and backward
  gbuffer  camera rays and the multi-target trace of a surfel scene
  rebake   the learned rebake after an edit
  place    probe placement on a surface cloud

The scenes stand in for captured ones: Gaussians and surfels area-uniform on a
union of random ellipsoids (the object), on a ground plane with clutter (the
scene), or in a spherical shell, with the sizes of the repository's workloads.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_07729_gb300 import sop

DEV = "cuda"
F64 = torch.float64
DTYPES = {"f32": sop.SOP_F32, "bf16": sop.SOP_BF16, "f16": sop.SOP_F16}
TORCH_DT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
QUANT = 1048576.0  # probe positions are compared in units of 2^-20
ALPHA_MIN, ALPHA_MAX, T_STOP = 1.0 / 255.0, 0.99, 1e-4


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the quick-start scene: a call whose launches and host time count
        dict(name="bake_tiny", kind="bake", scene="shell", gauss=2000, probes=64, R=8, dtype="f32"),
        # a reconstructed object's probes, baked before it is relit
        dict(name="bake_object", kind="bake", scene="object", gauss=200_000, probes=4096, R=16, dtype="f32"),
        # the shadow probes of the ground it is put on, baked against it, in the 16-bit form a renderer keeps
        dict(name="bake_ground", kind="bake", scene="ground", gauss=200_000, probes=4096, R=16, dtype="f16"),
        # a few thousand points, as an editor's preview or a light probe would ask; neighbours returned too
        dict(name="query_tiny", kind="query", scene="sphere", mode="shade", points=4096, probes=64, R=8, K=4, S=64,
             dtype="f32", env=16, radius=0.0, nbrs=True),
        # the object's pixels of an 800x800 view
        dict(name="query_object", kind="query", scene="object", mode="shade", points=418_111, probes=4096, R=16, K=8,
             S=128, dtype="f32", env=256, radius=0.0, nbrs=False),
        # the receiver's pixels of a 1920x1080 frame
        dict(name="query_frame_shadow", kind="query", scene="ground", mode="shadow", points=2_051_693, probes=4096,
             R=16, K=8, S=64, dtype="f16", env=256, radius=0.0, nbrs=False),
        # a new light on the same object: directions drawn from the estimated environment, then the frame
        dict(name="relight", kind="relight", scene="object", points=250_007, probes=4096, R=16, K=8, S=64, dtype="f16",
             H=512),
        # one optimisation batch of random pixels
        dict(name="grad_batch", kind="grad", points=8191, probes=4096, R=16, K=8, S=128, env=256, batch=True),
        # one optimisation step over a whole view
        dict(name="grad_view", kind="grad", points=418_111, probes=4096, R=16, K=8, S=128, env=256, batch=False),
        # the scene's G-buffer of a 1920x1080 frame
        dict(name="gbuffer_scene", kind="gbuffer", scene="ground", gauss=1_000_000, W=1920, H=1080),
        # an object moved: its probes rebaked by the network
        dict(name="rebake", kind="rebake", gauss=200_000, probes=4096, R=16),
        # probes placed on the fused depth of several views
        dict(name="place", kind="place", points=750_710, probes=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bake", "query", "query", "relight", "grad", "gbuffer", "rebake", "place"])
    if kind == "bake":
        return dict(kind=kind, scene=rng.choice(["shell", "object", "ground"]), gauss=_log(rng, 2000, 200_000),
                    probes=_log(rng, 64, 4096), R=rng.choice([8, 11, 16, 16]), dtype=rng.choice(["f32", "f16", "bf16"]))
    if kind == "query":
        mode = rng.choice(["shade", "shadow"])
        S = rng.choice([32, 64, 100, 128]) if mode == "shade" else rng.choice([32, 50, 64])
        return dict(kind=kind, scene="object" if mode == "shade" else "ground", mode=mode,
                    points=_log(rng, 1000, 418_111 if mode == "shade" else 2_051_693), probes=_log(rng, 64, 4096),
                    R=rng.choice([8, 11, 16, 16]), K=rng.choice([4, 6, 8, 8]), S=S,
                    dtype=rng.choice(["f32", "f16", "bf16"]), env=rng.choice([16, 64, 256]),
                    radius=rng.choice([0.0, 0.0, 0.1]), nbrs=rng.random() < 0.25)
    if kind == "relight":
        return dict(kind=kind, scene="object", points=_log(rng, 1000, 250_007), probes=_log(rng, 64, 4096),
                    R=rng.choice([8, 16]), K=rng.choice([4, 8]), S=rng.choice([32, 64]),
                    dtype=rng.choice(["f32", "f16"]), H=rng.choice([32, 128, 256, 512]))
    if kind == "grad":
        return dict(kind=kind, points=_log(rng, 500, 418_111), probes=_log(rng, 64, 4096), R=rng.choice([8, 11, 16]),
                    K=rng.choice([4, 8]), S=rng.choice([32, 64, 100, 128]), env=rng.choice([16, 64, 256]),
                    batch=rng.random() < 0.5)
    if kind == "gbuffer":
        h = _log(rng, 90, 1080)
        return dict(kind=kind, scene=rng.choice(["object", "ground"]), gauss=_log(rng, 20_000, 1_000_000),
                    W=(h * 16) // 9, H=h)
    if kind == "rebake":
        return dict(kind=kind, gauss=_log(rng, 10_000, 200_000), probes=_log(rng, 64, 4096), R=rng.choice([8, 16]))
    n = _log(rng, 4096, 750_710)
    return dict(kind=kind, points=n, probes=min(n, _log(rng, 64, 4096)))


# ---------------------------------------------------------------------------
# inputs, made on the GPU from the seed
# ---------------------------------------------------------------------------
class _Rand:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed))
        self.np = np.random.default_rng(int(seed))

    def u(self, lo, hi, *shape, dtype=F64):
        return torch.rand(shape, generator=self.g, device=DEV, dtype=dtype) * (hi - lo) + lo

    def normal(self, *shape, dtype=F64):
        return torch.randn(shape, generator=self.g, device=DEV, dtype=dtype)

    def unit(self, n):
        v = self.normal(n, 3)
        return v / v.norm(dim=1, keepdim=True)


def _f32(t):
    return t.to(torch.float32).contiguous()


class _Ellipsoids:
    """Union of oriented ellipsoids: centres c, semi-axes a, rotations R (columns: local axes)."""

    def __init__(self, c, a, R):
        self.c, self.a, self.R = (torch.as_tensor(v, dtype=F64, device=DEV) for v in (c, a, R))
        self.n = len(c)

    def sample(self, r, n):
        """n area-uniform points of the union's surface, with outward normals."""
        pts, nrm, got = [], [], 0
        wmax = (self.a.prod(1) / self.a.min(1).values).max()
        while got < n:
            m = max(4 * (n - got), 8192)
            e = torch.randint(0, self.n, (m,), generator=r.g, device=DEV)
            u = r.unit(m)
            keep = r.u(0.0, 1.0, m) * wmax < self.a[e].prod(1) * (u / self.a[e]).norm(dim=1)
            e, u = e[keep], u[keep]
            loc = u * self.a[e]
            x = self.c[e] + torch.einsum("nij,nj->ni", self.R[e], loc)
            g = torch.einsum("nij,nj->ni", self.R[e], loc / self.a[e] ** 2)
            ok = torch.ones(len(x), dtype=torch.bool, device=DEV)
            for k in range(self.n):
                q = ((x - self.c[k]) @ self.R[k] / self.a[k]).square().sum(1)
                ok &= (q >= 1.0 - 1e-9) | (e == k)
            pts.append(x[ok])
            nrm.append(g[ok] / g[ok].norm(dim=1, keepdim=True))
            got += len(pts[-1])
        return torch.cat(pts)[:n], torch.cat(nrm)[:n]

    def hit(self, o, d):
        """First hit of the rays o + t d: t (inf where missed) and the normal there."""
        best = torch.full((len(d),), math.inf, dtype=F64, device=DEV)
        nrm = torch.zeros_like(d)
        for k in range(self.n):
            M = self.R[k] / self.a[k]
            lo, ld = (o - self.c[k]) @ M, d @ M
            A, B, C = ld.square().sum(1), ld @ lo, lo.square().sum() - 1.0
            disc = B * B - A * C
            t = (-B - disc.clamp_min(0.0).sqrt()) / A
            ok = (disc > 0) & (t > 1e-9) & (t < best)
            g = ((lo + t[:, None] * ld) / self.a[k]) @ self.R[k].T
            best = torch.where(ok, t, best)
            nrm = torch.where(ok[:, None], g / g.norm(dim=1, keepdim=True), nrm)
        return best, nrm


def _rotations(r, n):
    q, t = np.linalg.qr(r.np.standard_normal((n, 3, 3)))
    q = q * np.sign(np.diagonal(t, axis1=1, axis2=2))[:, None, :]
    q[:, :, 0] *= np.sign(np.linalg.det(q))[:, None]
    return q


def _object(r):
    return _Ellipsoids(r.np.uniform(-0.6, 0.6, (5, 3)), r.np.uniform(0.2, 0.6, (5, 3)), _rotations(r, 5))


class _Ground:
    """The plane under an object, six times its size, with 30 small ellipsoids standing on it away from it."""

    def __init__(self, r, ells):
        s, _ = ells.sample(r, 8192)
        lo, hi = s.min(0).values.cpu().numpy(), s.max(0).values.cpu().numpy()
        self.size, self.z, self.c = float((hi - lo).max()), float(lo[2]), 0.5 * (lo[:2] + hi[:2])
        self.half, self.diag = 3.0 * self.size, float(np.linalg.norm(hi - lo))
        ax, cc = r.np.uniform(0.05, 0.15, (30, 3)), []
        while len(cc) < 30:
            p = self.c + r.np.uniform(-self.half, self.half, 2)
            if np.linalg.norm(p - self.c) > 0.75 * self.size:
                cc.append(p)
        cc = np.concatenate([np.array(cc), self.z + ax[:, 2:]], axis=1)
        self.clutter = _Ellipsoids(cc, ax, np.repeat(np.eye(3)[None], 30, axis=0))

    def sample(self, r, n, z):
        xy = r.u(-self.half, self.half, n, 2) + torch.as_tensor(self.c, device=DEV)
        return torch.cat([xy, torch.full((n, 1), z, dtype=F64, device=DEV)], dim=1)

    def camera(self, r):
        az, el, dist = r.np.uniform(0, 2 * np.pi), np.deg2rad(35.0), 2.2 * self.size / np.tan(np.deg2rad(25.0))
        at = np.array([self.c[0], self.c[1], self.z + 0.3 * self.size])
        return at + dist * np.array([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)]), at, 50.0


def _gaussians(r, mean):
    n = len(mean)
    q = r.normal(n, 4)
    return dict(mean=_f32(mean), scale=_f32(torch.exp(r.u(math.log(0.002), math.log(0.02), n, 3))),
                quat=_f32(q / q.norm(dim=1, keepdim=True)), opacity=_f32(r.u(0.2, 1.0, n)),
                rgb=_f32(r.u(0.0, 1.0, n, 3)))


def _surfels(r, mean, nrm):
    """Gaussians flattened along their normal: the third scale is a tenth of the smaller tangent one."""
    n = len(mean)
    g = _gaussians(r, mean)
    st = torch.exp(r.u(math.log(0.002), math.log(0.02), n, 2))
    g["scale"] = _f32(torch.cat([st, 0.1 * st.min(1, keepdim=True).values], dim=1))
    # shortest rotation that takes z to the normal, after a random spin about z
    half = 0.5 * r.u(0.0, 2 * math.pi, n)
    w, x, y = 1.0 + nrm[:, 2], -nrm[:, 1], nrm[:, 0]
    flip = w < 1e-6
    w, x, y = torch.where(flip, 0.0, w), torch.where(flip, 1.0, x), torch.where(flip, 0.0, y)
    c, s = half.cos(), half.sin()
    q = torch.stack([w * c, x * c + y * s, y * c - x * s, w * s], dim=1)
    g["quat"] = _f32(q / q.norm(dim=1, keepdim=True))
    return g


def _spread(pts, k, start=0):
    """Indices of k of the points, each the farthest from those before it."""
    out = torch.empty(k, dtype=torch.int64, device=DEV)
    cur = torch.full((1,), start, dtype=torch.int64, device=DEV)
    far = torch.full((len(pts),), math.inf, dtype=pts.dtype, device=DEV)
    for i in range(k):
        out[i] = cur[0]
        far = torch.minimum(far, (pts - pts[cur]).square().sum(1))
        cur = far.argmax().reshape(1)
    return out


def _probes(r, pts, nrm, k, offset):
    sel = _spread(pts, k) if k < len(pts) else torch.arange(k, device=DEV)
    return _f32(pts[sel] + offset * nrm[sel]), _f32(nrm[sel])


def _scene(case, r):
    """Gaussians to bake against and the probes' positions and normals."""
    n, P = case.get("gauss", 0), case["probes"]
    if case["scene"] in ("shell", "sphere"):
        rad = r.u(0.8 ** 3, 1.0, max(n, 1)) ** (1.0 / 3.0)
        g = _gaussians(r, r.unit(max(n, 1)) * rad[:, None])
        s = torch.exp(r.u(math.log(0.005), math.log(0.03), max(n, 1)))
        g["scale"] = _f32(s[:, None].expand(-1, 3))
        i = torch.arange(P, device=DEV, dtype=F64) + 0.5
        z, ph = 1.0 - 2.0 * i / P, i * math.pi * (3.0 - math.sqrt(5.0))
        x = torch.stack([(1 - z * z).sqrt() * ph.cos(), (1 - z * z).sqrt() * ph.sin(), z], dim=1)
        return g, _f32(x), _f32(x), None, None
    ells = _object(r)
    ground = _Ground(r, ells)
    g = _gaussians(r, ells.sample(r, n)[0]) if n else None
    if case["scene"] == "object":
        pts, nrm = ells.sample(r, max(16_384, P))
    else:
        pts = ground.sample(r, max(16_384, P), ground.z)
        nrm = torch.tensor([0.0, 0.0, 1.0], dtype=F64, device=DEV).expand(len(pts), 3)
    pos, pn = _probes(r, pts, nrm, P, 0.01 * ground.diag)
    return g, pos, pn, ells, ground


def _rays(eye, at, fov, W, H):
    """Unit directions of a W x H pinhole view, row by row."""
    f = torch.as_tensor(np.asarray(at, float) - eye, dtype=F64, device=DEV)
    f = f / f.norm()
    right = torch.linalg.cross(f, torch.tensor([0.0, 0.0, 1.0], dtype=F64, device=DEV))
    right = right / right.norm()
    up = torch.linalg.cross(right, f)
    th = math.tan(math.radians(fov) * 0.5)
    sx = ((torch.arange(W, device=DEV, dtype=F64) + 0.5) / W * 2 - 1) * th * W / H
    sy = (1 - (torch.arange(H, device=DEV, dtype=F64) + 0.5) / H * 2) * th
    d = f + sx[None, :, None] * right + sy[:, None, None] * up
    d = d.reshape(-1, 3)
    return d / d.norm(dim=1, keepdim=True)


def _view(case, r, ells, ground):
    """The first `points` shading points of a view, in pixel order."""
    M = case["points"]
    if ells is None:
        x = r.unit(M)
        return x, x, x
    if case.get("scene", "object") == "object":
        v = r.np.standard_normal(3) * np.array([1.0, 1.0, 0.6])
        eye, at, fov, wide = 3.0 * v / np.linalg.norm(v), np.zeros(3), 28.0, 1.0
    else:
        eye, at, fov = ground.camera(r)
        wide = 16.0 / 9.0
    o = torch.as_tensor(eye, dtype=F64, device=DEV)

    def shoot(h):
        d = _rays(eye, at, fov, int(h * wide), h)
        t, n = ells.hit(o, d)
        if case.get("scene", "object") == "object":
            return d, t, n, t.isfinite()
        tc, nc = ground.clutter.hit(o, d)
        tg = torch.where(d[:, 2] < 0, (ground.z - o[2]) / d[:, 2], math.inf)
        up = torch.tensor([0.0, 0.0, 1.0], dtype=F64, device=DEV)
        ts, ns = torch.minimum(tc, tg), torch.where((tc < tg)[:, None], nc, up)
        return d, ts, ns, ts.isfinite() & ~(t < ts)

    share = max(float(shoot(128)[3].double().mean()), 0.02)
    h = int(math.sqrt(1.03 * M / (share * wide))) + 2
    while True:
        d, t, n, ok = shoot(h)
        pix = ok.nonzero()[:, 0]
        if len(pix) >= M:
            break
        h = int(h * 1.05) + 1
    pix = pix[:M]
    return o + t[pix, None] * d[pix], n[pix], -d[pix]


def _materials(r, m):
    return _f32(r.u(0.0, 1.0, m, 3)), _f32(r.u(0.1, 1.0, m)), _f32(r.u(0.0, 1.0, m))


def _maps(r, P, R):
    """Probe maps [P, R, R, 4] (radiance, occlusion): a smooth wave per probe and channel, with texel noise."""
    k = torch.arange(R, device=DEV, dtype=F64) * (2 * math.pi / R)
    ph = r.u(0.0, 2 * math.pi, P, 4, 2)
    wave = (k + ph[:, :, 0, None]).sin()[:, :, None, :] * (k + ph[:, :, 1, None]).cos()[:, :, :, None]
    amp = torch.tensor([0.15, 0.15, 0.15, 0.3], dtype=F64, device=DEV)
    mid = torch.tensor([0.25, 0.25, 0.25, 0.5], dtype=F64, device=DEV)
    return _f32(mid + amp * wave.permute(0, 2, 3, 1) + r.u(-0.1, 0.1, P, R, R, 4))


def _env(r, h, w):
    """High-dynamic-range environment: log-normal texels."""
    return _f32(torch.exp(1.5 * r.normal(h, w, 3)))


def _query_inputs(case, seed):
    r = _Rand(seed)
    _, pos, _, ells, ground = _scene(dict(case, gauss=0, scene=case.get("scene", "object")), r)
    x, n, wo = _view(case, r, ells, ground)
    M = case["points"]
    if case.get("batch"):  # the batch is random pixels of the view
        p = torch.randperm(M, generator=r.g, device=DEV)
        x, n, wo = x[p], n[p], wo[p]
    alb, rough, metal = _materials(r, M)
    env = _env(r, case["H"], case["H"]) if case["kind"] == "relight" else _env(r, case["env"], 2 * case["env"])
    return dict(pts=(_f32(x), _f32(n), _f32(wo), alb, rough, metal), pos=pos, maps=_maps(r, case["probes"], case["R"]),
                env=env, go=_f32(r.normal(M, 3)) / M)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "bake":
        g, pos, nrm, _, _ = _scene(case, _Rand(seed))
        dt = DTYPES[case["dtype"]]
        return dict(kind=kind, gauss=g, atlas=sop.make_atlas(pos, case["R"], dt, dt, nrm))
    if kind in ("query", "relight"):
        s = _query_inputs(case, seed)
        m = s["maps"]
        atlas = sop.make_atlas(s["pos"], case["R"], DTYPES[case["dtype"]], with_depth=False)
        sop.atlas_pack(m[..., :3].contiguous(), m[..., 3].contiguous(), None, atlas)
        return dict(case, pts=s["pts"], atlas=atlas, envmap=s["env"])
    if kind == "grad":
        return dict(case, **_query_inputs(case, seed))
    if kind == "gbuffer":
        r = _Rand(seed)
        ells = _object(r)
        ground = _Ground(r, ells)
        if case["scene"] == "object":
            x, n = ells.sample(r, case["gauss"])
        else:  # 7 in 10 surfels on the (slightly uneven) ground, the others on the clutter
            k = int(0.7 * case["gauss"])
            x = ground.sample(r, k, ground.z)
            x[:, 2] += 5e-3 * ground.size * r.normal(k)
            c, cn = ground.clutter.sample(r, case["gauss"] - k)
            up = torch.tensor([0.0, 0.0, 1.0], dtype=F64, device=DEV).expand(k, 3)
            x, n = torch.cat([x, c]), torch.cat([up, cn])
        g = _surfels(r, x, n)
        mats = dict(zip(("albedo", "rough", "metal"), _materials(r, len(x))))
        eye, at, fov = ground.camera(r)
        return dict(kind=kind, W=case["W"], H=case["H"], tracer=sop.GbufferTracer(g, mats), eye=eye, at=at, fov=fov,
                    origin=_f32(torch.as_tensor(eye, device=DEV).reshape(1, 3)), gauss=g, mats=mats)
    if kind == "rebake":
        g, pos, nrm, _, ground = _scene(dict(case, scene="object"), _Rand(seed))
        net = sop.Surrogate(device=DEV, seed=seed)
        atlas = sop.make_atlas(pos, case["R"], probe_nrm=nrm, depth_scale=ground.diag)
        return dict(kind=kind, gauss=g, atlas=atlas, net=net, seed=seed)
    if kind == "place":
        r = _Rand(seed)
        ells = _object(r)
        x, n = ells.sample(r, case["points"])
        return dict(kind=kind, pts=_f32(x), nrm=_f32(n), k=case["probes"])
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "bake":
        a = sop.bake(s["gauss"], s["atlas"])
        return a.rgbo, a.depth
    if kind == "query":
        mode = sop.MODE_SHADE if s["mode"] == "shade" else sop.MODE_SHADOW
        return sop.query_shade(*s["pts"], s["atlas"], s["envmap"], s["K"], s["S"], mode, radius=s["radius"],
                               return_idx=s["nbrs"])
    if kind == "relight":
        d = sop.env_importance_dirs(s["envmap"], s["S"])
        return d, sop.query_shade(*s["pts"], s["atlas"], s["envmap"], s["K"], s["S"], dirs_world=d,
                                  env_layout=sop.ENV_OCTAHEDRAL)
    if kind == "grad":
        x, n, wo, alb, rough, metal = s["pts"]
        leaf = [t.detach().requires_grad_() for t in (n, alb, rough, metal, s["maps"], s["env"])]
        c = sop.SopQueryShade.apply(x, leaf[0], wo, leaf[1], leaf[2], leaf[3], leaf[4], leaf[5], s["pos"], s["K"],
                                    s["S"])
        return [c.detach(), *torch.autograd.grad(c, leaf, s["go"])]
    if kind == "gbuffer":
        return s["tracer"].trace(s["origin"], sop.pinhole_dirs(s["W"], s["H"], s["eye"], s["at"], s["fov"]))
    if kind == "rebake":
        # the network keeps its initial weights, so the check of its result may never ask for the traced bake
        err, fell = s["net"].rebake(s["gauss"], s["atlas"], tau=1e6, seed=s["seed"])
        return s["atlas"].rgbo, s["atlas"].depth, err, fell
    return sop.place_probes(s["pts"], s["k"], s["nrm"], offset=0.02)


def work(case):
    """Bytes of the inputs and outputs; operations of the method itself (texel fetches and blends, shading, one
    response per Gaussian that a ray meets), not of any way to find what a ray or a point needs."""
    kind, P, R = case["kind"], case.get("probes", 0), case.get("R", 0)
    tex = 16 if case.get("dtype", "f32") == "f32" else 8
    if kind == "bake":
        d = tex // 4
        return dict(bytes=56 * case["gauss"] + 24 * P + P * (R + 2) ** 2 * (tex + d), flops=P * R * R * 40.0 * 108)
    if kind in ("query", "relight"):
        e = 12 * (case["H"] ** 2 if kind == "relight" else 2 * case["env"] ** 2)
        shade = kind == "relight" or case["mode"] == "shade"
        pd = case["points"] * case["S"]
        pt = 12 * 4 + 8 + 12 + (8 * case["K"] if case.get("nbrs") else 0)
        return dict(bytes=case["points"] * pt + P * (R + 2) ** 2 * tex + e + 12 * P,
                    flops=pd * (case["K"] * (32.0 if shade else 8.0) + (170 if shade else 60)))
    if kind == "grad":
        pd = case["points"] * case["S"]
        e = 24 * case["env"] ** 2
        return dict(bytes=case["points"] * (12 * 4 + 8 + 12 + 12 + 32) + 2 * P * R * R * 16 + 2 * e + 12 * P,
                    flops=pd * (case["K"] * 96.0 + 600))
    if kind == "gbuffer":
        n = case["W"] * case["H"]
        return dict(bytes=76 * case["gauss"] + n * 64, flops=n * 20.0 * 130)
    if kind == "rebake":
        n = P * R * R
        return dict(bytes=56 * case["gauss"] + 24 * P + P * (R + 2) ** 2 * 20, flops=n * (19_300.0 + 60 * 100))
    return dict(bytes=24 * case["points"] + 20 * P, flops=8.0 * case["points"])


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def _wrap(R):
    """Compact texel index [R+2, R+2] of every texel of a bordered map."""
    idx = np.empty((R + 2, R + 2), np.int64)
    for j in range(-1, R + 1):
        for i in range(-1, R + 1):
            a, b = i, j
            oi, oj = not 0 <= i < R, not 0 <= j < R
            if oi and oj:
                a, b = (R - 1 if i < 0 else 0), (R - 1 if j < 0 else 0)
            elif oi:
                a, b = (0 if i < 0 else R - 1), R - 1 - j
            elif oj:
                a, b = R - 1 - i, (0 if j < 0 else R - 1)
            idx[j + 1, i + 1] = b * R + a
    return torch.from_numpy(idx.reshape(-1)).to(DEV)


def _oct(w):
    p = w[..., :2] / w.abs().sum(-1, keepdim=True)
    s = torch.where(p >= 0, 1.0, -1.0)
    p = torch.where(w[..., 2:] < 0, (1.0 - p.abs().flip(-1)) * s, p)
    return 0.5 * (p + 1.0)


def _texel_dirs(R):
    u = (torch.arange(R, device=DEV, dtype=F64) + 0.5) / R * 2 - 1
    px, py = u[None, :].expand(R, R), u[:, None].expand(R, R)
    z = 1 - px.abs() - py.abs()
    sx, sy = torch.where(px >= 0, 1.0, -1.0), torch.where(py >= 0, 1.0, -1.0)
    qx, qy = torch.where(z < 0, (1 - py.abs()) * sx, px), torch.where(z < 0, (1 - px.abs()) * sy, py)
    d = torch.stack([qx, qy, z], dim=-1).reshape(-1, 3)
    return d / d.norm(dim=1, keepdim=True)


def _bilinear(s, t):
    fs, ft = s.detach().floor(), t.detach().floor()
    a, b = s - fs, t - ft
    return fs.long(), ft.long(), torch.stack([(1 - a) * (1 - b), a * (1 - b), (1 - a) * b, a * b], dim=-1)


def _neighbours(x, pos, K, radius):
    """K nearest probes by the integer distance; -1 beyond the radius. And the nearest one's distance."""
    q, p = (torch.round(t.double() * QUANT).long() for t in (x, pos))
    d = q[:, None, 0] - p[:, 0]
    key = d * d
    for a in (1, 2):
        d = q[:, None, a] - p[:, a]
        key += d * d
    key, idx = torch.topk(key, K, dim=1, largest=False, sorted=True)
    if radius > 0:
        idx = torch.where(key <= math.floor((float(np.float32(radius)) * QUANT) ** 2), idx, -1)
    return idx, key[:, 0]


def _weights(x, n, pos, idx, near):
    d = pos[idx.clamp_min(0)] - x[:, None]
    dl = d.norm(dim=-1)
    found = idx >= 0
    w = torch.where(found, (0.5 * (1 + (d * n[:, None]).sum(-1) / dl) + 0.01) / dl, 0.0)
    w = w / w.sum(1, keepdim=True).clamp_min(1e-300)
    snap = ((near <= 1) & found[:, 0])[:, None]
    return torch.where(snap, torch.nn.functional.one_hot(torch.zeros_like(near), idx.shape[1]).double(), w)


def _shade64(x, n_raw, wo, alb, rough, metal, idx, near, pos, maps, wrap, env, case, world):
    """Shading of some points; maps [P, R*R, 4] and env [texels, 3] in 64 bits, differentiable."""
    R, S, shadow = case["R"], case["S"], case.get("mode") == "shadow"
    RS = R + 2
    n = n_raw / n_raw.norm(dim=1, keepdim=True)
    W = _weights(x, n, pos, idx, near)
    if world is None:
        i = torch.arange(S, device=DEV)
        z = (i.double() + 0.5) / S
        ri = sum((((i >> b) & 1).double() * 0.5 ** (b + 1)) for b in range(13))
        lx, ly = (1 - z * z).sqrt() * (2 * math.pi * ri).cos(), (1 - z * z).sqrt() * (2 * math.pi * ri).sin()
        sg = torch.where(n[:, 2] >= 0, 1.0, -1.0)
        a = -1.0 / (sg + n[:, 2])
        c = n[:, 0] * n[:, 1] * a
        tt = torch.stack([1 + sg * n[:, 0] ** 2 * a, sg * c, -sg * n[:, 0]], dim=1)
        bb = torch.stack([c, sg + n[:, 1] ** 2 * a, -n[:, 1]], dim=1)
        w = lx[:, None] * tt[:, None] + ly[:, None] * bb[:, None] + z[:, None] * n[:, None]
        cosl, wt = z.expand(len(x), S), 2 * math.pi / S
    else:
        w = world[:, :3].expand(len(x), S, 3)
        cosl = (n[:, None] * w).sum(-1)
        wt = torch.where(cosl > 0, 1.0 / world[:, 3], 0.0) / S
    # probes: the footprint lies at the same place of every probe's map
    uv = _oct(w)
    i0, j0, q = _bilinear(uv[..., 0] * R - 0.5, uv[..., 1] * R - 0.5)
    i0, j0 = (i0 + 1).clamp(0, R), (j0 + 1).clamp(0, R)
    off = torch.stack([wrap[(j0 + b) * RS + i0 + a] for b in (0, 1) for a in (0, 1)], dim=-1)
    at = (idx.clamp_min(0) * (R * R))[:, None, :, None] + off[:, :, None, :]
    tex = maps.index_select(0, at.reshape(-1)).reshape(*at.shape, 4)
    pr = torch.einsum("msq,mk,mskqc->msc", q, W, tex)
    # environment
    if case["kind"] == "relight":
        H = case["H"]
        s, t, e = _bilinear(uv[..., 0] * H - 0.5, uv[..., 1] * H - 0.5)
        ew = _wrap(H)
        cols = [ew[(t + 1 + b).clamp(0, H + 1) * (H + 2) + (s + 1 + a).clamp(0, H + 1)] for b in (0, 1) for a in (0, 1)]
    else:
        He, We = case["env"], 2 * case["env"]
        th = torch.atan2((w[..., 0] ** 2 + w[..., 1] ** 2).sqrt(), w[..., 2])
        ph = torch.atan2(w[..., 1], w[..., 0])
        s, t, e = _bilinear((ph + math.pi) / (2 * math.pi) * We - 0.5, th / math.pi * He - 0.5)
        cols = [(t + b).clamp(0, He - 1) * We + (s + a) % We for b in (0, 1) for a in (0, 1)]
    L = sum(e[..., k:k + 1] * env.index_select(0, cols[k].reshape(-1)).reshape(*cols[k].shape, 3) for k in range(4))
    vis = 1 - pr[..., 3:]
    cw = (cosl * wt)[..., None]
    if shadow:
        den = (L * cw).sum(1)
        return torch.where(den < 1e-20, 1.0, (L * vis * cw).sum(1) / den.clamp_min(1e-300))
    h = w + wo[:, None]
    h = h / h.norm(dim=-1, keepdim=True)
    ndv = (n * wo).sum(-1).clamp_min(1e-4)[:, None]
    ndh, vdh = (h * n[:, None]).sum(-1), (h * wo[:, None]).sum(-1)
    sin2 = torch.linalg.cross(n[:, None].expand_as(h), h).square().sum(-1)
    a2, k = (rough ** 4)[:, None], ((rough + 1) ** 2 / 8)[:, None]
    D = a2 / (math.pi * (ndh * ndh * a2 + sin2) ** 2)
    cl = torch.where(cosl > 0, cosl, 1.0)
    G = (cl / (cl * (1 - k) + k)) * (ndv / (ndv * (1 - k) + k))
    spec = (D * G / (4 * cl * ndv))[..., None]
    F0 = (0.08 * 0.5 * (1 - metal)[:, None] + alb * metal[:, None])[:, None]
    F = F0 + (1 - F0) * ((1 - vdh) ** 5)[..., None]
    f = ((1 - metal)[:, None] * alb / math.pi)[:, None] + spec * F
    return (f * (vis * L + pr[..., :3]) * cw).sum(1)


def _importance64(env, S):
    """Directions and densities by exact integer intervals over the texels' intensities."""
    H = env.shape[0]
    I = (env[..., 0] + env[..., 1] + env[..., 2]).reshape(-1)
    q = (I.double() / I.max().double() * QUANT).floor().long().clamp_min(1)
    c = q.cumsum(0)
    Q = int(c[-1])
    at = torch.searchsorted(c, (2 * torch.arange(S, device=DEV) + 1) * Q // (2 * S), right=True)
    d = _texel_dirs(H)[at]
    return torch.cat([d, (H * H * q[at].double() / (4 * math.pi * Q))[:, None]], dim=1)


def _exact_query(case, seed):
    s = _query_inputs(case, seed)
    R, P, K, M, kind = case["R"], case["probes"], case["K"], case["points"], case["kind"]
    grad = kind == "grad"
    maps = s["maps"].to(TORCH_DT[case.get("dtype", "f32")]).double().reshape(P * R * R, 4)
    env, pos = s["env"].double().reshape(-1, 3), s["pos"].double()
    world = _importance64(s["env"], case["S"]) if kind == "relight" else None
    # the shading takes the directions as they are returned, in 32 bits
    world_in = None if world is None else world.float().double()
    wrap = _wrap(R)
    pts = [t.double() for t in s["pts"]]
    outs, nbr, wts, per = [], [], [], [[], [], [], []]
    if grad:
        maps, env = maps.requires_grad_(), env.requires_grad_()
        gm, ge = torch.zeros_like(maps), torch.zeros_like(env)
    chunk = max(1, min((1 << 19) // case["S"], (1 << 27) // P))
    for m in range(0, M, chunk):
        x, n, wo, alb, rough, metal = (t[m:m + chunk] for t in pts)
        idx, near = _neighbours(s["pts"][0][m:m + chunk], s["pos"], K, case.get("radius", 0.0))
        if grad:
            leaf = [t.detach().requires_grad_() for t in (n, alb, rough, metal)]
            c = _shade64(x, leaf[0], wo, *leaf[1:], idx, near, pos, maps, wrap, env, case, None)
            *g, dm, de = torch.autograd.grad(c, [*leaf, maps, env], s["go"][m:m + chunk].double())
            gm += dm
            ge += de
            for a, b in zip(per, g):
                a.append(b)
            outs.append(c.detach())
            continue
        outs.append(_shade64(x, n, wo, alb, rough, metal, idx, near, pos, maps, wrap, env, case, world_in))
        if case.get("nbrs"):
            nbr.append(idx.to(torch.int32))
            wts.append(_weights(x, n / n.norm(dim=1, keepdim=True), pos, idx, near))
    out = torch.cat(outs)
    if grad:
        return [out, *[torch.cat(p) for p in per], gm.reshape(P, R, R, 4), ge.reshape(s["env"].shape)]
    if kind == "relight":
        return world, out
    return (out, torch.cat(nbr), torch.cat(wts)) if case.get("nbrs") else out


def _hits64(g, o, d):
    """(ray, Gaussian, t, alpha) of all hits of the rays, ordered along each ray."""
    q = g["quat"].double()
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).T
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                       2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                       2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], dim=1).reshape(-1, 3, 3)
    M = rot.transpose(1, 2) / g["scale"].double()[:, :, None]
    mu, op = g["mean"].double(), g["opacity"].double()
    found = []
    step = max(1, (1 << 23) // len(mu))
    for r in range(0, len(d), step):
        oo, dd = o[r:r + step], d[r:r + step]
        v = torch.einsum("nij,rj->rni", M, dd)
        u = torch.einsum("nij,rnj->rni", M, oo[:, None] - mu)
        t = -(v * u).sum(-1) / v.square().sum(-1)
        a = op * torch.exp(-0.5 * (u + t[..., None] * v).square().sum(-1))
        i, k = ((a >= ALPHA_MIN) & (t > 0)).nonzero(as_tuple=True)
        found.append((i + r, k, t[i, k], a[i, k].clamp_max(ALPHA_MAX)))
    i, k, t, a = (torch.cat(c) for c in zip(*found))
    at = t.argsort(stable=True)
    at = at[i[at].argsort(stable=True)]
    return i[at], k[at], t[at], a[at], rot


def _composite64(i, a, rays):
    """Weight of every hit, and each ray's transmittance, with the early stop."""
    lg = torch.log1p(-a)
    cum = lg.cumsum(0)
    first = torch.searchsorted(i, torch.arange(rays, device=DEV))
    base = torch.cat([torch.zeros(1, dtype=F64, device=DEV), cum])[first]
    before = torch.exp(cum - lg - base[i])
    use = before >= T_STOP
    left = torch.zeros(rays, dtype=F64, device=DEV).index_add_(0, i[use], lg[use])
    return torch.where(use, before * a, 0.0), torch.exp(left)


def _sum(i, v, rays):
    return torch.zeros((rays, *v.shape[1:]), dtype=F64, device=DEV).index_add_(0, i, v)


def _exact_bake(case, seed):
    g, pos, _, _, _ = _scene(case, _Rand(seed))
    P, R = case["probes"], case["R"]
    d = _texel_dirs(R).repeat(P, 1)
    i, k, t, a, _ = _hits64(g, pos.double().repeat_interleave(R * R, 0), d)
    w, T = _composite64(i, a, P * R * R)
    L = _sum(i, w[:, None] * g["rgb"].double()[k], P * R * R)
    W, D = _sum(i, w, P * R * R), _sum(i, w * t, P * R * R)
    wrap = _wrap(R)
    rgbo = torch.cat([L, 1 - T[:, None]], dim=1).reshape(P, R * R, 4)[:, wrap].reshape(P, R + 2, R + 2, 4)
    depth = torch.where(W > 1e-8, D / W.clamp_min(1e-300), 0.0).reshape(P, R * R)[:, wrap]
    return rgbo, depth.reshape(P, R + 2, R + 2)


def _exact_gbuffer(case, seed):
    s = prepare(case, seed)
    g, n = s["gauss"], case["W"] * case["H"]
    d = _rays(s["eye"], s["at"], s["fov"], case["W"], case["H"])
    i, k, t, a, rot = _hits64(g, s["origin"].double().expand(n, 3), d)
    w, _ = _composite64(i, a, n)
    nrm = rot[torch.arange(len(rot), device=DEV), :, g["scale"].argmin(1)][k]
    nrm = torch.where(((nrm * d[i]).sum(1) > 0)[:, None], -nrm, nrm)
    m = s["mats"]
    v = torch.cat([g["rgb"].double()[k], torch.ones_like(t)[:, None], nrm, t[:, None], m["albedo"].double()[k],
                   m["rough"].double()[k, None], m["metal"].double()[k, None], torch.zeros(len(k), 3, device=DEV)], 1)
    return _sum(i, w[:, None] * v, n)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("query", "relight", "grad"):
        return _exact_query(case, seed)
    pairs = case.get("gauss", 0) * (case["W"] * case["H"] if kind == "gbuffer" else
                                    case["probes"] * case.get("R", 1) ** 2)
    if kind == "bake":
        return _exact_bake(case, seed) if pairs <= 4e9 else None
    if kind == "gbuffer":
        return _exact_gbuffer(case, seed) if pairs <= 4e9 else None
    if kind == "place":
        s = prepare(case, seed)
        q = torch.round(s["pts"].double() * QUANT)
        idx = _spread(q, case["probes"])
        return idx, s["pts"].double()[idx] + float(np.float32(0.02)) * s["nrm"].double()[idx]
    return None
