"""Calls at the ends of their ranges: parameters, types and set sizes far from
the workloads the kernels were tuned on; against the oracle, through the C ABI."""
import numpy as np
import pytest
import torch

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
