"""Voxel means where eight lanes share a run: run lengths around the pixels they
take at a time, radiance inside and outside the exact integer range (and
ranges that only the lanes together leave), bit-equal to the oracle's grid."""
import numpy as np
import pytest
import torch

import oracle as O
from workloads import cornell_box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["narrow", "wide", "signs"])
def test_run_lengths(kind):
    import paper_2304_05669_gb300 as F
    rng = np.random.default_rng(7)
    lengths = [1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 100, 257, 1000]
    R = 16
    cell = np.repeat(np.arange(len(lengths)), lengths)
    cell = rng.permutation(cell)
    x = np.stack([(cell + 0.5) / R, np.full(len(cell), 0.5 / R), np.full(len(cell), 0.5 / R)], 1).astype(np.float32)
    L = rng.uniform(0.25, 2.0, (len(cell), 3)).astype(np.float32)
    if kind == "wide":
        L *= np.float32(2.0) ** rng.integers(-14, 15, (len(cell), 1)).astype(np.float32)
    if kind == "signs":
        L *= rng.choice([-1, 0, 1], (len(cell), 3)).astype(np.float32)
    m = cornell_box()
    sc = F.Scene.from_mesh(m)
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    got = sc.voxel_cache(cu(x), cu(L), R).cpu().numpy()
    want = O.OracleScene.from_mesh(m).voxel_pool(x, L, R).astype(np.float32)
    assert np.array_equal(got, want)
