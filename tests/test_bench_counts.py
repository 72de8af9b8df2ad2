"""bench.py's counts, on the host: the step's launches against the recorded
list of its present form, and the bytes that its query roof rests on."""
import os
import re

import numpy as np
import torch

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_step_launches_match_the_recorded_list():
    text = open(os.path.join(ROOT, "profiles", "launches_step.md")).read()
    rows = re.findall(r"^\| `[^`]+` \| \([^)]*\) \| [\d.]+ \|", text, flags=re.M)
    total = int(re.search(r"^\| (\d+) launches \|", text, flags=re.M).group(1))
    assert len(rows) == total == bench.step_launches(True, 2)


def test_shared_footprints():
    rng = np.random.default_rng(0)
    M, K = 32 * 40 + 7, 4
    idx = rng.integers(0, 12, (M, K)).astype(np.int32)
    idx[64:96] = rng.integers(0, 1000, (32, K))  # more than 32 probes
    n = np.tile(np.array([[0, 0, 1]], np.float32), (M, 1))
    n[33, 0] = 1e-7  # a group of two normals
    want = 0
    for g in range(0, M, 32):
        i, m = idx[g:g + 32], n[g:g + 32]
        d = len(np.unique(i))
        want += d if (m.view(np.int32) == m[:1].view(np.int32)).all() and d <= 32 else i.size
    assert bench.shared_footprints(torch.from_numpy(idx), torch.from_numpy(n)) == want


def test_touched_texels():
    up = np.array([[0.0, 0.0, 1.0]])
    assert bench.touched_texels(up, np.array([[0.0, 0.0, 1.0]]), 8) == 4.0  # one footprint
    # a direction set all over the upper half of the map touches about half of it
    rng = np.random.default_rng(0)
    d = rng.standard_normal((20000, 3))
    d[:, 2] = np.abs(d[:, 2])
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    assert 0.45 * 18 * 18 < bench.touched_texels(up, d, 16) < 0.65 * 18 * 18
