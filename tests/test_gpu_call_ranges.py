"""Calls at the ends of their ranges: parameters, types and set sizes far from
the workloads the kernels were tuned on; against the oracle, through the C ABI."""
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


@pytest.mark.parametrize("rough", [1e-3, 4e-4, 2e-4, 5e-5])
def test_adjoint_at_the_mirror_direction(sop, orc, rough):
    """A direction set with the pole and a view along the normal: h = n, and
    the lobe's denominator is r^4, whose inverse square is still a float32 but
    whose inverse cube is not. Normals along the axes, so that h = n exactly
    and the oracle has the same lobe. Tolerances of the adjoint's other tests."""
    rng = np.random.default_rng(7)
    n = np.array([[0, 0, 1], [1, 0, 0], [0, 1, 0], [0, 0, -1]], F)
    M, P, R, K, S = len(n), 12, 8, 4, 40
    d = rng.standard_normal((S, 3))
    d[:, 2] = np.abs(d[:, 2]) + 0.2
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    d[S // 2] = [0, 0, 1]
    dirs = d.astype(F)
    pp, x = rng.uniform(-1, 1, (P, 3)).astype(F), rng.uniform(-0.5, 0.5, (M, 3)).astype(F)
    rgb, occ = rng.uniform(0, 0.5, (P, R, R, 3)).astype(F), rng.uniform(0, 1, (P, R, R)).astype(F)
    env = rng.uniform(0.5, 1.5, (8, 16, 3)).astype(F)
    alb, met, go = rng.uniform(0, 1, (M, 3)).astype(F), rng.uniform(0, 1, M).astype(F), rng.standard_normal((M, 3)).astype(F)
    pts = (x, n, n, alb, np.full(M, rough, F), met)
    at = sop.make_atlas(cuda(pp), R, with_depth=False)
    sop.atlas_pack(cuda(rgb), cuda(occ), None, at)
    g = sop.query_shade_backward(*[cuda(v) for v in pts], at, cuda(env), K, S, cuda(go), dirs_local=cuda(dirs))
    w = orc.query_shade_grad(*pts, pp, rgb, occ, env, K, S, go, dirs=dirs.astype(np.float64))
    for key in ("albedo", "rough", "metal", "normal"):
        got = g[key].cpu().numpy().astype(np.float64)
        assert np.all(np.isfinite(got)), key
        terms = w["abs_" + key][:, None] if key == "normal" else w["abs_" + key]
        assert np.all(np.abs(got - w[key]) <= 1e-4 * np.abs(w[key]) + 2e-4 * terms + 1e-12), key
    for got, ref in ((g["env"], w["env"]), (g["maps"][..., :3], w["maps_rgb"]), (g["maps"][..., 3], w["maps_occ"])):
        d = np.abs(got.cpu().numpy() - ref)
        assert np.all(d <= 1e-4 * np.abs(ref) + 2e-5 * np.abs(ref).max() + 1e-12)


def _rods(n, length, width, diagonal, seed):
    """Gaussians of one long and two short axes; along the space diagonals their
    boxes are cubes of nearly the rods' length."""
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((n, 3))
    if diagonal:
        u = np.sign(u) + 0.05 * rng.standard_normal((n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True).clip(1e-9)
    q = np.stack([1 + u[:, 0], 0 * u[:, 0], -u[:, 2], u[:, 1]], axis=1)  # x to u
    g = dict(mean=rng.uniform(-1, 1, (n, 3)), scale=np.tile([length, width, width], (n, 1)),
             quat=q / np.linalg.norm(q, axis=1, keepdims=True).clip(1e-9), opacity=rng.uniform(0.05, 0.3, n),
             rgb=rng.uniform(0, 1, (n, 3)))
    return {k: v.astype(F) for k, v in g.items()}


@pytest.mark.parametrize("n,length,width,two,extra", [
    (0, 0.1, 0.01, False, 1 << 22),             # nothing to bin, in a workspace with room
    (4096, 0.4, 0.01, False, 0), (4096, 3.0, 0.02, True, 0),         # one CTA
    (4096, 0.4, 0.01, False, 1 << 24),                               # room for the first grid's lists: many CTAs
    (5000, 3.0, 0.02, True, 0), (30_000, 0.15, 0.004, False, 0),     # many CTAs
    (190_000, 0.05, 0.004, False, 0), (190_000, 0.15, 0.002, True, 0),  # more than 8,192 coarse cells
])
def test_coarsened_bakes(sop, orc, n, length, width, two, extra):
    """Sets whose cell lists overflow the workspace, binned by one CTA and by
    many into the grid of 1/16 of the cells and into the one of two (`two`:
    diagonal rods, which overflow the former too): the traced maps against the
    oracle (the bakes' bound: 1e-5 and the rounding of the texel directions;
    occlusion alone where two hits are within rounding of each other)."""
    g, R = _rods(n, length, width, two, n), 4
    far = 1.5 + (3.6 * length if n < 10_000 else 0.6)  # outside every box: no hits with one entry point
    out = np.concatenate([np.eye(3), -np.eye(3)]) * far + 0.1
    pp = (out if two else np.array([[0.1, 0.2, -0.1], [0.4, -0.3, 0.2]])).astype(F)
    ws = sop.BakeWorkspace(n, "cuda", extra_bytes=extra)
    at = sop.make_atlas(cuda(pp), R)
    sop.device_status()
    sop.bake({k: cuda(v) for k, v in g.items()}, at, t_stop=0.0, workspace=ws)
    assert bool(sop.device_status() & sop.DEVSTAT_GRID_COARSENED) == (n > 0 and extra == 0)
    rgb, occ, dep = (t.cpu().numpy() for t in at.interior())
    if n == 0:
        assert not occ.any() and not rgb.any()
        return
    o_rgb, o_occ, o_dep, fl, sens = orc.bake(g, pp, R, t_stop=0.0, with_sens=True)
    decided = (fl & (orc.FLAG_ALPHA_MIN | orc.FLAG_TNEAR | orc.FLAG_TSTOP)) == 0
    assert (decided & (o_occ > 0.1)).sum() >= 6  # enough rays through many Gaussians
    assert_close(occ[decided], o_occ[decided], what="O", absolute=sens[..., 3][decided])
    ok = decided & ((fl & orc.FLAG_ORDER) == 0)
    assert_close(rgb[ok], o_rgb[ok], what="L_in", absolute=sens[..., :3][ok])


def test_bakes_on_two_streams(sop):
    """Bakes of equally many Gaussians side by side on two streams, each with
    its stream's own scratch: the maps of single bakes, bit for bit."""
    pp = cuda(np.random.default_rng(1).uniform(-1, 1, (256, 3)).astype(F))
    sets = [{k: cuda(v) for k, v in _rods(20_000, 0.02, 0.01, False, seed).items()} for seed in (3, 4)]
    want = [sop.make_atlas(pp, 8) for _ in sets]
    for g, at in zip(sets, want):
        sop.bake(g, at)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in sets]
    got = [[sop.make_atlas(pp, 8) for _ in range(10)] for _ in sets]
    torch.cuda.synchronize()
    for i in range(10):
        for s, st in enumerate(streams):
            with torch.cuda.stream(st):
                sop.bake(sets[s], got[s][i])
    torch.cuda.synchronize()
    for s in range(2):
        for at in got[s]:
            assert torch.equal(at.rgbo, want[s].rgbo) and torch.equal(at.depth, want[s].depth)


def test_queries_of_several_threads(sop):
    """Host threads with maps and direction sets of different sizes, whose
    launches want different amounts of shared memory of the same kernels:
    every call is accepted, and returns what it returns alone."""
    import threading
    rng = np.random.default_rng(5)
    M, K = 48, 8
    x, n = rng.uniform(-1, 1, (M, 3)).astype(F), rng.standard_normal((M, 3))
    n = (n / np.linalg.norm(n, axis=1, keepdims=True)).astype(F)
    pts = [cuda(v) for v in (x, n, n, rng.uniform(0, 1, (M, 3)).astype(F), np.full(M, 0.5, F), np.full(M, 0.5, F))]
    env, go = cuda(rng.uniform(0.5, 1, (8, 16, 3)).astype(F)), cuda(rng.standard_normal((M, 3)).astype(F))
    jobs = []
    for R, S in ((16, 128), (24, 128), (18, 700), (8, 4096)):
        P = 16
        at = sop.make_atlas(cuda(rng.uniform(-1, 1, (P, 3)).astype(F)), R, with_depth=False)
        sop.atlas_pack(cuda(rng.uniform(0, 0.5, (P, R, R, 3)).astype(F)), cuda(rng.uniform(0, 1, (P, R, R)).astype(F)), None, at)

        def job(at=at, S=S):
            out = sop.query_shade(*pts, at, env, K, S)
            return [out] + [sop.query_shade_backward(*pts, at, env, K, S, go)[k] for k in ("albedo", "rough", "normal")]
        jobs.append((job, [t.clone() for t in job()]))
    torch.cuda.synchronize()
    failed = []

    def work(job, want):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(300):
                    got = job()
                torch.cuda.current_stream().synchronize()
                if not all(torch.equal(a, b) for a, b in zip(got, want)):
                    failed.append("other results")
        except Exception as e:  # a refused launch
            failed.append(repr(e))
    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


@pytest.mark.parametrize("dtype", [0, 1, 2])
def test_shadow_of_a_hidden_sun(sop, orc, dtype):
    """A large SHADOW call on one plane whose only bright light is hidden by
    its probe: what is left is a small sum, not the difference of two large
    ones. One probe a point (its weight is exactly 1). Bound: 1e-5 and the
    sensitivity to the rounding of the directions."""
    M, P, R, S, He = 262_144, 40, 8, 64, 16
    rng = np.random.default_rng(11)
    pp = np.concatenate([rng.uniform(-1, 1, (P, 2)), np.full((P, 1), 0.05)], axis=1).astype(F)
    x = np.concatenate([rng.uniform(-1, 1, (M, 2)), np.zeros((M, 1))], axis=1).astype(F)
    n = np.tile(np.array([0.0, 0.0, 1.0], F), (M, 1))
    env = rng.uniform(0.005, 0.015, (He, 2 * He, 3)).astype(F)
    r, c = 4, 9  # a sun half way up
    env[r:r + 2, c:c + 2] = 2e4
    th, ph = (r + 1) / He * np.pi, (c + 1) / He * np.pi - np.pi
    sun = np.array([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)])
    u = (np.arange(R) + 0.5) / R * 2 - 1
    px, py = np.meshgrid(u, u, indexing="xy")
    z = 1 - np.abs(px) - np.abs(py)
    fx, fy = (np.where(z < 0, (1 - np.abs(b)) * np.where(a >= 0, 1, -1), a) for a, b in ((px, py), (py, px)))
    d = np.stack([fx, fy, z], -1)
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    occ = np.where(d @ sun > np.cos(np.deg2rad(75)), 1.0, rng.integers(0, 33, (P, R, R)) / 64).astype(F)
    rgb, one = np.zeros((P, R, R, 3), F), np.full(M, 0.5, F)
    at = sop.make_atlas(cuda(pp), R, dtype, with_depth=False)
    sop.atlas_pack(cuda(rgb), cuda(occ), None, at)
    out = sop.query_shade(*[cuda(v) for v in (x, n, n, np.full((M, 3), 0.5, F), one, one)], at, cuda(env), 1, S,
                          mode=sop.MODE_SHADOW).cpu().numpy()
    sel = rng.integers(0, M, 200)
    args = [x[sel], n[sel], n[sel], np.full((200, 3), 0.5, F), one[sel], one[sel], pp, rgb, occ, env, 1, S]
    want, _, _ = orc.query_shade(*args, mode=orc.MODE_SHADOW)
    sens = orc.query_shade_sensitivity(*args, mode=orc.MODE_SHADOW)
    assert 0 < want.max() < 1e-3
    assert np.all(np.abs(out[sel] - want) <= 1e-5 * np.maximum(np.abs(want), 1e-3 * np.abs(want).mean()) + sens)


@pytest.mark.parametrize("K,radius", [(5, 0.0), (9, 0.0), (17, 0.0), (6, 0.01)])
@pytest.mark.parametrize("M", [262_144, 311_296])
def test_shadow_of_nothing(sop, K, radius, M):
    """Probes that hide nothing, and points with no probe within the radius:
    the ratio is exactly 1, also where a warp's points share their sums."""
    rng = np.random.default_rng(K)
    P, R = 64, 8
    pp = np.concatenate([rng.uniform(-1, 1, (P, 2)), np.full((P, 1), 0.02)], axis=1).astype(F)
    x = np.zeros((M, 3), F)
    x[:, 0] = np.linspace(-1.2, 1.2, M)
    n = np.tile(np.array([0.0, 0.0, 1.0], F), (M, 1))
    at = sop.make_atlas(cuda(pp), R, with_depth=False)
    sop.atlas_pack(cuda(np.zeros((P, R, R, 3), F)), cuda(np.zeros((P, R, R), F)), None, at)
    env = np.exp(rng.normal(0, 1.5, (16, 32, 3))).astype(F)
    one = np.full(M, 0.5, F)
    out = sop.query_shade(*[cuda(v) for v in (x, n, n, np.full((M, 3), 0.5, F), one, one)], at, cuda(env), K, 64,
                          mode=sop.MODE_SHADOW, radius=radius)
    assert bool((out == 1).all())


@pytest.mark.parametrize("R,M,K,S,dtype", [
    (2, 33_000, 4, 32, 0), (2, 33_000, 4, 40, 0),            # float32, several lanes: S K = 150
    (2, 160_000, 4, 128, 0), (2, 160_000, 5, 104, 0),        # two lanes: S (K - 2) = 300
    (3, 160_000, 4, 400, 0), (3, 160_000, 6, 400, 0),
    (2, 33_000, 5, 99, 2), (2, 33_000, 5, 100, 1),           # 16 bits, eight lanes: S (K - 1) = 400
    (2, 80_000, 6, 135, 1), (2, 80_000, 6, 137, 2),          # fewer: S (K - 3) = 400 + texels / 2
    (3, 1000, 1, 32, 0), (3, 16_384, 1, 32, 0), (3, 16_384, 8, 32, 1),  # few points
])
def test_shade_dispatch(sop, orc, R, M, K, S, dtype):
    """SHADE on both sides of the lines between its kernels on small maps (in
    which a footprint of texels is most of the map): a sample against the oracle,
    with the bound of the query's other tests, on maps that are exact in 16 bits."""
    rng = np.random.default_rng(R * M + S)
    P = 40
    pp, x = rng.uniform(-1, 1, (P, 3)).astype(F), rng.uniform(-1, 1, (M, 3)).astype(F)
    n = rng.standard_normal((M, 3))
    wo = rng.standard_normal((M, 3))
    wo *= np.sign(np.sum(wo * n, axis=1, keepdims=True))
    n, wo = ((v / np.linalg.norm(v, axis=1, keepdims=True)).astype(F) for v in (n, wo))
    th, ph = (np.arange(16) + 0.5) / 16 * np.pi, (np.arange(32) + 0.5) / 16 * np.pi
    env = (1.0 + 0.5 * np.sin(th)[:, None, None] * np.cos(ph[None, :, None] + np.arange(3))).astype(F)
    rgb, occ = ((rng.integers(0, 65, s) / 64).astype(F) for s in ((P, R, R, 3), (P, R, R)))
    pts = (x, n, wo, rng.uniform(0, 1, (M, 3)).astype(F), rng.uniform(0.3, 1, M).astype(F), rng.uniform(0, 1, M).astype(F))
    at = sop.make_atlas(cuda(pp), R, dtype, with_depth=False)
    sop.atlas_pack(cuda(rgb), cuda(occ), None, at)
    out = sop.query_shade(*[cuda(v) for v in pts], at, cuda(env), K, S).cpu().numpy()
    sel = np.unique(np.concatenate([rng.integers(0, M, 100), np.arange(M - 40, M)]))
    args = [v[sel] for v in pts] + [pp, rgb, occ, env, K, S]
    want, _, _ = orc.query_shade(*args)
    sens = orc.query_shade_sensitivity(*args)
    assert np.all(np.abs(out[sel] - want) <= 1e-5 * np.maximum(np.abs(want), 1e-3 * np.abs(want).mean()) + sens)


@pytest.mark.parametrize("R,M,K,S", [
    (24, 16_384, 4, 64), (24, 4096, 4, 40), (24, 4096, 2, 20), (16, 16_384, 4, 36), (16, 16_384, 4, 37),
    (8, 16_384, 4, 20), (8, 16_385, 4, 38), (8, 16_385, 12, 9), (2, 16_385, 4, 13), (2, 16_385, 4, 14),
    (16, 16_385, 17, 29), (64, 300, 16, 24), (64, 300, 32, 12),
])
@pytest.mark.parametrize("dtype", [0, 1, 2])
def test_adjoint_dispatch(sop, orc, R, M, K, S, dtype):
    """The adjoint on both sides of the lines between its kernels, every type of
    atlas and number of probes in each: a sample's own gradients, and for few
    points the summed ones, against the oracle, on maps that are exact in 16
    bits, with the tolerances of the adjoint's other tests."""
    rng = np.random.default_rng(R * M + S)
    P = 40
    pp, x = rng.uniform(-1, 1, (P, 3)).astype(F), rng.uniform(-1, 1, (M, 3)).astype(F)
    n = rng.standard_normal((M, 3))
    wo = rng.standard_normal((M, 3))
    wo *= np.sign(np.sum(wo * n, axis=1, keepdims=True))
    n, wo = ((v / np.linalg.norm(v, axis=1, keepdims=True)).astype(F) for v in (n, wo))
    th, ph = (np.arange(16) + 0.5) / 16 * np.pi, (np.arange(32) + 0.5) / 16 * np.pi
    env = (1.0 + 0.5 * np.sin(th)[:, None, None] * np.cos(ph[None, :, None] + np.arange(3))).astype(F)
    rgb, occ = ((rng.integers(0, 65, s) / 64).astype(F) for s in ((P, R, R, 3), (P, R, R)))
    pts = (x, n, wo, rng.uniform(0, 1, (M, 3)).astype(F), rng.uniform(0.3, 1, M).astype(F), rng.uniform(0, 1, M).astype(F))
    go = rng.standard_normal((M, 3)).astype(F)
    at = sop.make_atlas(cuda(pp), R, dtype, with_depth=False)
    sop.atlas_pack(cuda(rgb), cuda(occ), None, at)
    g = sop.query_shade_backward(*[cuda(v) for v in pts], at, cuda(env), K, S, cuda(go))
    sel = np.arange(M) if M <= 300 else np.unique(np.concatenate([rng.integers(0, M, 100), np.arange(M - 40, M)]))
    w = orc.query_shade_grad(*[v[sel] for v in pts], pp, rgb, occ, env, K, S, go[sel])
    for key in ("albedo", "rough", "metal", "normal"):
        d = np.abs(g[key].cpu().numpy()[sel] - w[key])
        terms = w["abs_" + key][:, None] if key == "normal" else w["abs_" + key]
        assert np.all(d <= 1e-4 * np.abs(w[key]) + 2e-4 * terms + 1e-12), key
    if M <= 300:
        for got, ref in ((g["env"], w["env"]), (g["maps"][..., :3], w["maps_rgb"]), (g["maps"][..., 3], w["maps_occ"])):
            d = np.abs(got.cpu().numpy() - ref)
            assert np.all(d <= 1e-4 * np.abs(ref) + 2e-5 * np.abs(ref).max() + 1e-12)


@pytest.mark.parametrize("n,k,lattice", [
    (1500, 300, False), (2048, 400, False), (2049, 400, False), (2049, 2049, False),  # one CTA / the least that many share
    (466_944, 30, False), (466_945, 30, False),      # 6 / 8 points a thread on 152 SMs
    (778_241, 30, False), (933_889, 30, False), (1_089_537, 30, False),  # 12, 14, 16
    (4913, 600, True), (110_592, 300, True),         # a lattice: equal keys everywhere
])
def test_placement_splits(sop, orc, n, k, lattice):
    """Probe placement at the edges of its splits, and where nearly every choice
    is a tie: the indices equal the oracle's, captured in a graph too."""
    rng = np.random.default_rng(n)
    if lattice:
        m = round(n ** (1 / 3))
        pts = (np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) / 64).astype(F)
        pts = pts[rng.permutation(len(pts))]
    else:
        pts = rng.standard_normal((n, 3))
        pts = (pts / np.linalg.norm(pts, axis=1, keepdims=True)).astype(F)
    d = cuda(pts)
    want, _ = orc.fps(pts, k, start=n // 2)
    idx, pos = sop.place_probes(d, k, start=n // 2)
    assert np.array_equal(idx.cpu().numpy(), want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        idx, pos = sop.place_probes(d, k, start=n // 2)
    for _ in range(2):
        idx.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(idx.cpu().numpy(), want) and np.array_equal(pos.cpu().numpy(), pts[want])
    sop.device_status()


@pytest.mark.parametrize("n", [1, 2, 33, 1024, 1025, 4096, 4097, 9000])
def test_bins_of_small_sets(sop, orc, n):
    """Sets of one Gaussian to a few CTAs' worth, sized so that rays hit whatever
    their number: the traced maps against the oracle."""
    rng = np.random.default_rng(n)
    size = 0.25 * n ** (-1 / 3)
    s = size * np.exp(rng.uniform(-0.5, 0.5, (n, 3)))
    q = rng.standard_normal((n, 4))
    g = dict(mean=rng.uniform(-0.3, 0.3, (n, 3)), scale=s, quat=q / np.linalg.norm(q, axis=1, keepdims=True),
             opacity=rng.uniform(0.3, 0.9, n), rgb=rng.uniform(0, 1, (n, 3)))
    g = {k: v.astype(F) for k, v in g.items()}
    pp, R = np.array([[0.02, -0.05, 0.01], [0.9, 0.1, 0.2], [-0.2, -0.8, 0.5]], F), 8
    at = sop.make_atlas(cuda(pp), R)
    sop.bake({k: cuda(v) for k, v in g.items()}, at)
    sop.device_status()
    rgb, occ, dep = (t.cpu().numpy() for t in at.interior())
    o_rgb, o_occ, o_dep, fl, sens = orc.bake(g, pp, R, with_sens=True)
    decided = (fl & (orc.FLAG_ALPHA_MIN | orc.FLAG_TNEAR | orc.FLAG_TSTOP)) == 0
    assert decided.mean() > 0.7 and (decided & (o_occ > 0.01)).sum() >= 8
    assert_close(occ[decided], o_occ[decided], what="O", absolute=sens[..., 3][decided])
    ok = decided & ((fl & orc.FLAG_ORDER) == 0)
    assert_close(rgb[ok], o_rgb[ok], what="L_in", absolute=sens[..., :3][ok])


@pytest.mark.parametrize("n", [2000, 20_000])
def test_bake_replayed_from_a_graph(sop, n):
    """A bake with default scratch captured in a graph and replayed beside plain
    bakes of other Gaussians: the plain call's maps, bit for bit."""
    pp = cuda(np.random.default_rng(2).uniform(-1, 1, (64, 3)).astype(F))
    g, other = ({k: cuda(v) for k, v in _rods(n, 0.05, 0.01, False, seed).items()} for seed in (5, 6))
    want, spare, at = (sop.make_atlas(pp, 8) for _ in range(3))
    sop.bake(g, want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sop.bake(g, at)
    for _ in range(3):
        at.rgbo.zero_()
        sop.bake(other, spare)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(at.rgbo, want.rgbo) and torch.equal(at.depth, want.depth)
