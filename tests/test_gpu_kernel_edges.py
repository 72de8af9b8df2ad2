"""Kernels at the sizes where their launch shape changes: the edges of tiles
and of dispatch rules, remainders, the smallest and largest of a range;
against the oracle, through the C ABI."""
import numpy as np
import pytest
import torch

from tests.tolerance import assert_close

pytestmark = pytest.mark.gpu
F = np.float32


@pytest.fixture(scope="module")
def sop():
    from paper_2510_07729_gb300 import sop as S
    S.load()
    return S


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n,k,scale", [
    (2, 2, 1.0), (513, 100, 1.0),                    # one CTA
    (4096, 300, 1.0), (4097, 300, 1.0),              # one CTA / several
    (155_648, 40, 1.0), (155_649, 40, 1.0),          # 2 / 4 points a thread on 152 SMs
    (311_297, 40, 1.0), (622_593, 40, 1.0),          # 8, 10
    (778_241, 30, 1.0), (1_245_185, 30, 1.0),        # 16, keys in the workspace
    (5000, 50, 1500.0), (1_300_000, 20, 1500.0),     # differences beyond 2^31 quantised units
])
def test_fps_point_counts(sop, orc, n, k, scale):
    """Whole-number results: the indices equal the oracle's at every split of
    the points over threads and CTAs."""
    rng = np.random.default_rng(n)
    pts = (rng.uniform(-1, 1, (n, 3)) * scale).astype(F)
    pts[n // 3: n // 3 + 20] = pts[0]  # equal points: ties, keys of zero
    start = n - 1
    idx, pos = sop.place_probes(cuda(pts), k, start=start)
    oi, _ = orc.fps(pts, k, start=start)
    assert np.array_equal(idx.cpu().numpy(), oi)
    assert np.array_equal(pos.cpu().numpy(), pts[oi])


@pytest.mark.parametrize("H,S", [(2, 1), (3, 7), (45, 33), (46, 4096), (91, 64), (512, 9)])
@pytest.mark.parametrize("values", ["lognormal", "wide", "flat", "zero", "one"])
def test_importance_texels(sop, orc, H, S, values):
    """The texel of every sample (an exact integer decision) over tiles of
    2,048 texels and their remainders, for intensities from denormal to huge."""
    rng = np.random.default_rng(H + S)
    env = {"lognormal": lambda: np.exp(rng.normal(0, 1.5, (H, H, 3))),
           "wide": lambda: np.exp(rng.uniform(-100, 85, (H, H, 3))),
           "flat": lambda: np.full((H, H, 3), 0.37),
           "zero": lambda: np.zeros((H, H, 3)),
           "one": lambda: (np.arange(H * H * 3).reshape(H, H, 3) == 3 * (H * H // 2)) * 1e-42}[values]().astype(F)
    got = sop.env_importance_dirs(cuda(env), S).cpu().numpy().astype(np.float64)
    want = orc.env_importance_dirs(env, S)
    assert np.max(np.abs(got[:, :3] - want[:, :3])) < 2e-7  # one float32 rounding of a unit vector
    np.testing.assert_allclose(got[:, 3], want[:, 3], rtol=2e-7)


def _query_workload(P, R, M, He, seed):
    """Points above a bumpy sheet of probes, iid maps, a smooth environment
    (so that FP32 direction rounding stays far below the tolerance)."""
    rng = np.random.default_rng(seed)
    pp = np.concatenate([rng.uniform(-1, 1, (P, 2)), 0.1 * rng.standard_normal((P, 1))], axis=1).astype(F)
    x = np.concatenate([rng.uniform(-1.2, 1.2, (M, 2)), 0.1 * rng.standard_normal((M, 1))], axis=1).astype(F)
    n = rng.standard_normal((M, 3))
    wo = rng.standard_normal((M, 3))
    wo *= np.sign(np.sum(wo * n, axis=1, keepdims=True))  # seen from above the surface
    n, wo = (v / np.linalg.norm(v, axis=1, keepdims=True) for v in (n, wo))
    th = (np.arange(He) + 0.5) / He * np.pi
    ph = (np.arange(2 * He) + 0.5) / He * np.pi
    env = (1.0 + 0.5 * np.sin(th)[:, None, None] * np.cos(ph[None, :, None] + np.arange(3))).astype(F)
    return dict(pp=pp, x=x, n=n.astype(F), wo=wo.astype(F), albedo=rng.uniform(0, 1, (M, 3)).astype(F),
                rough=rng.uniform(0.3, 1, M).astype(F), metal=rng.uniform(0, 1, M).astype(F), env=env,
                rgb=rng.uniform(0, 0.5, (P, R, R, 3)).astype(F), occ=rng.uniform(0, 1, (P, R, R)).astype(F))


PTS = ("x", "n", "wo", "albedo", "rough", "metal")


@pytest.mark.parametrize("M,P,R,K,S", [
    (1, 8, 2, 8, 5), (7, 40, 3, 1, 33), (9, 40, 16, 8, 128), (64, 64, 16, 8, 100), (333, 200, 16, 4, 129),
    (65, 100, 11, 16, 64), (33, 100, 8, 32, 96), (40, 50, 24, 8, 256), (5, 8, 64, 4, 40),
])
@pytest.mark.parametrize("caller_dirs", [False, True])
def test_shade_and_adjoint_shapes(sop, orc, M, P, R, K, S, caller_dirs):
    """SHADE and its adjoint over remainders of the warp (32 directions) and
    of the eight points of a CTA, one to 32 probes, maps from 2x2 to 64x64,
    the library's directions or the caller's. Tolerances as for the oracle
    tests of either: 1e-5 of the output plus its sensitivity to 2e-6 rad;
    gradients 1e-4 plus 2e-4 of the terms' magnitudes."""
    c = _query_workload(P, R, M, 16, 100 * M + R)
    rng = np.random.default_rng(S)
    dirs = None
    if caller_dirs:
        d = rng.standard_normal((S, 3))
        d[:, 2] = np.abs(d[:, 2]) + 0.2
        dirs = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(F)
    at = sop.make_atlas(cuda(c["pp"]), R, with_depth=False)
    sop.atlas_pack(cuda(c["rgb"]), cuda(c["occ"]), None, at)
    pts = [cuda(c[k]) for k in PTS]
    gd = None if dirs is None else cuda(dirs)
    out = sop.query_shade(*pts, at, cuda(c["env"]), K, S, dirs_local=gd).cpu().numpy()
    args = [c[k] for k in PTS] + [c["pp"], c["rgb"], c["occ"], c["env"], K, S]
    kw = dict(dirs=None if dirs is None else dirs.astype(np.float64))
    want, _, _ = orc.query_shade(*args, **kw)
    sens = orc.query_shade_sensitivity(*args, **kw)
    assert np.all(np.abs(out - want) <= 1e-5 * np.maximum(np.abs(want), 1e-3 * np.abs(want).mean()) + sens)
    go = rng.standard_normal((M, 3)).astype(F)
    g = sop.query_shade_backward(*pts, at, cuda(c["env"]), K, S, cuda(go), dirs_local=gd)
    w = orc.query_shade_grad(*args, go, **kw)
    for key in ("albedo", "rough", "metal", "normal"):
        d = np.abs(g[key].cpu().numpy() - w[key])
        terms = w["abs_" + key][:, None] if key == "normal" else w["abs_" + key]
        assert np.all(d <= 1e-4 * np.abs(w[key]) + 2e-4 * terms + 1e-12), key
    for got, ref in ((g["env"], w["env"]), (g["maps"][..., :3], w["maps_rgb"]), (g["maps"][..., 3], w["maps_occ"])):
        d = np.abs(got.cpu().numpy() - ref)
        assert np.all(d <= 1e-4 * np.abs(ref) + 2e-5 * np.abs(ref).max() + 1e-12)


@pytest.mark.parametrize("M,P,K,radius", [
    (1, 1, 1, 0.0), (33, 3, 3, 0.0), (100, 256, 8, 0.0), (100, 257, 8, 0.0), (2000, 4096, 32, 0.0), (500, 1000, 8, 0.05),
    (24_576, 300, 5, 0.0), (24_577, 300, 5, 0.0), (24_577, 20, 16, 0.3), (3000, 9000, 8, 0.0), (40_000, 30_000, 8, 0.0),
])
@pytest.mark.parametrize("layout", ["volume", "sheet", "point"])
def test_nearest_probes_exact(sop, orc, M, P, K, radius, layout):
    """Probe indices bit-exact on both sides of every rule: all probes
    without a grid (up to 256), a warp or a thread a point (24,576 points),
    grids in shared memory or in the workspace (8,192 cells), flat and
    degenerate probe sets, ties (every tenth probe twice), points outside."""
    rng = np.random.default_rng(P + K)
    pp = rng.uniform(-1, 1, (P, 3))
    if layout == "sheet":
        pp[:, 2] = 0.25
    elif layout == "point":
        pp[:] = pp[:1] + 1e-6 * rng.integers(0, 2, (P, 3))
    pp[9::10] = pp[8::10][:len(pp[9::10])]
    pp = pp.astype(F)
    x = rng.uniform(-1.5, 1.5, (M, 3)).astype(F)
    x[::7] = pp[rng.integers(0, P, len(x[::7]))]  # on a probe
    n = rng.standard_normal((M, 3))
    n = (n / np.linalg.norm(n, axis=1, keepdims=True)).astype(F)
    z1, z3 = np.full(M, 0.5, F), np.full((M, 3), 0.5, F)
    at = sop.make_atlas(cuda(pp), 2, with_depth=False)
    sop.atlas_pack(cuda(np.zeros((P, 2, 2, 3), F)), cuda(np.zeros((P, 2, 2), F)), None, at)
    env = np.ones((2, 4, 3), F)
    _, idx, w = sop.query_shade(cuda(x), cuda(n), cuda(n), cuda(z3), cuda(z1), cuda(z1), at, cuda(env), K, 1,
                                mode=sop.MODE_SHADOW, return_idx=True, radius=radius)
    _, oi, ow = orc.query_shade(x, n, n, z3, z1, z1, pp, np.zeros((P, 2, 2, 3), F), np.zeros((P, 2, 2), F), env, K, 1,
                                mode=orc.MODE_SHADOW, radius=radius)
    assert np.array_equal(idx.cpu().numpy(), oi)
    near = np.abs(w.cpu().numpy() - ow) <= 1e-5 * np.abs(ow).max(initial=1e-3)
    # (probes within a few ulp of a point: 1/d itself is not resolved in float32)
    d = np.linalg.norm(pp[np.clip(oi[:, 0], 0, None)].astype(np.float64) - x, axis=1)
    assert near[d > 1e-3].all()


@pytest.mark.parametrize("M", [262_143, 262_144, 262_175])
@pytest.mark.parametrize("dtype", [0, 1, 2])
@pytest.mark.parametrize("K,S", [(8, 64), (4, 33), (12, 128)])
def test_shadow_shared_integrals(sop, orc, M, dtype, K, S):
    """SHADOW on both sides of the size from which warps on one normal share
    their probes' integrals; warps with one normal, with two, and with more
    distinct probes than a warp keeps. A sample against the oracle: 1e-5 plus
    the sensitivity, on maps that are exact in 16 bits."""
    P, R = 600, 8
    rng = np.random.default_rng(S)
    pp = np.concatenate([rng.uniform(-1, 1, (P, 2)), np.full((P, 1), 0.02)], axis=1).astype(F)
    x = np.zeros((M, 3), F)
    x[:, 0] = np.linspace(-1.1, 1.1, M)
    x[:, 1] = 0.3 * np.sin(5 * x[:, 0])
    x[M // 2: M // 2 + 4096] = rng.uniform(-1, 1, (4096, 3)) * [1, 1, 0]  # scattered: many probes a warp
    n = np.tile(np.array([0.0, 0.0, 1.0], F), (M, 1))
    n[5000:5040:3] = np.array([0.6, 0.0, 0.8], F)  # mixed normals in two warps
    occ = (rng.integers(0, 65, (P, R, R)) / 64).astype(F)
    rgb = np.zeros((P, R, R, 3), F)
    env = np.exp(0.3 * np.sin(np.arange(16 * 32 * 3).reshape(16, 32, 3) / 50.0)).astype(F)
    one = np.full(M, 0.5, F)
    at = sop.make_atlas(cuda(pp), R, dtype, with_depth=False)
    sop.atlas_pack(cuda(rgb), cuda(occ), None, at)
    dev = [cuda(v) for v in (x, n, n, np.full((M, 3), 0.5, F), one, one)]
    out = sop.query_shade(*dev, at, cuda(env), K, S, mode=sop.MODE_SHADOW).cpu().numpy()
    sel = np.unique(np.concatenate([rng.integers(0, M, 300), np.arange(4990, 5045), np.arange(M // 2, M // 2 + 200),
                                    np.arange(M - 70, M)]))
    args = [x[sel], n[sel], n[sel], np.full((len(sel), 3), 0.5, F), one[sel], one[sel], pp, rgb, occ, env, K, S]
    want, _, _ = orc.query_shade(*args, mode=orc.MODE_SHADOW)
    sens = orc.query_shade_sensitivity(*args, mode=orc.MODE_SHADOW)
    assert np.all(np.abs(out[sel] - want) <= 1e-5 * np.maximum(np.abs(want), 1e-3 * np.abs(want).mean()) + sens)


def _cloud(rng, n, needles):
    s = np.exp(rng.uniform(np.log(0.002), np.log(0.01), (n, 3)))
    if needles:
        s[:, 0] = 0.3
    q = rng.standard_normal((n, 4))
    g = dict(mean=rng.uniform(-1, 1, (n, 3)), scale=s, quat=q / np.linalg.norm(q, axis=1, keepdims=True).clip(1e-9),
             opacity=rng.uniform(0.1, 0.9, n), rgb=rng.uniform(0, 1, (n, 3)))
    return {k: v.astype(F) for k, v in g.items()}


@pytest.mark.parametrize("n", [0, 1, 33, 4096, 4097, 70_000])
def test_bake_binning_sizes(sop, orc, n):
    """Binning by one CTA (up to 4,096 Gaussians) and by many: the traced maps
    against the oracle on rays whose hits are not within rounding of a
    decision."""
    rng = np.random.default_rng(n)
    g, pp, R = _cloud(rng, n, False), rng.uniform(-1.2, 1.2, (3, 3)).astype(F), 4
    at = sop.make_atlas(cuda(pp), R)
    sop.bake({k: cuda(v) for k, v in g.items()}, at)
    sop.device_status()
    rgb, occ, dep = (t.cpu().numpy() for t in at.interior())
    o_rgb, o_occ, o_dep, fl, sens = orc.bake(g, pp, R, with_sens=True)
    ok = fl == 0
    if ok.any():  # the FP32 bound, plus the rounding of the texel directions
        assert_close(occ[ok], o_occ[ok], what="O", absolute=sens[..., 3][ok])
        assert_close(rgb[ok], o_rgb[ok], what="L_in", absolute=sens[..., :3][ok])


@pytest.mark.parametrize("n,needles", [(1000, False), (4096, False), (4096, True)])
def test_bake_binning_paths_agree(sop, n, needles):
    """The same Gaussians binned by one CTA and, with invisible ones added to
    pass 4,096, by many: the same bits. Needles' boxes span so many cells that
    their lists overflow the workspace and a coarser grid is taken (the status
    word says so), in both."""
    rng = np.random.default_rng(n)
    g, pp = _cloud(rng, n, needles), rng.uniform(-1.2, 1.2, (5, 3)).astype(F)
    extra = _cloud(rng, 4097 - n + 700, False)
    extra["opacity"][:] = 1e-3
    both = {k: np.concatenate([g[k], extra[k]]) for k in g}
    out = []
    for c in (g, both):
        at = sop.make_atlas(cuda(pp), 8)
        sop.bake({k: cuda(v) for k, v in c.items()}, at)
        assert bool(sop.device_status() & sop.DEVSTAT_GRID_COARSENED) == needles
        out.append((at.rgbo.cpu().numpy(), at.depth.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])

