"""Kernels at the sizes where their launch shape changes: the edges of tiles
and of dispatch rules, remainders, the smallest and largest of a range;
against the oracle, through the C ABI."""
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
