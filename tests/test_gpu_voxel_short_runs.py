"""Voxel means where the runs are short on average: a lane a run, four long
ones among them at a time, and runs outside the exact integer range held back
until ten fill a warp; bit-equal to the oracle's grid."""
import numpy as np
import pytest
import torch

import oracle as O
from workloads import cornell_box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["narrow", "wide", "some wide", "signs"])
@pytest.mark.parametrize("runs,long_runs", [(1, 0), (31, 0), (33, 1), (60, 5), (700, 4), (700, 17)])
def test_short_runs(kind, runs, long_runs):
    import paper_2304_05669_gb300 as F
    rng = np.random.default_rng(runs + long_runs)
    lengths = rng.integers(1, 5, runs)
    lengths[rng.permutation(runs)[:long_runs]] = rng.choice([31, 32, 33, 65], long_runs)
    assert lengths.sum() < 8 * runs                       # under the limit of the other path
    R = 32
    cell = rng.permutation(np.repeat(rng.permutation(R * R)[:runs], lengths))
    x = np.stack([(cell % R + 0.5) / R, (cell // R + 0.5) / R, np.full(len(cell), 0.5 / R)], 1).astype(np.float32)
    L = rng.uniform(0.25, 2.0, (len(cell), 3)).astype(np.float32)
    if kind == "wide":
        L *= np.float32(2.0) ** rng.integers(-30, 31, (len(cell), 1)).astype(np.float32)
    if kind == "some wide":
        L[cell % 3 == 0] *= np.float32(2.0) ** rng.integers(-30, 31, (int((cell % 3 == 0).sum()), 1)).astype(np.float32)
    if kind == "signs":
        L *= rng.choice([-1, 0, 1], (len(cell), 3)).astype(np.float32)
    m = cornell_box()
    sc = F.Scene.from_mesh(m)
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    got = sc.voxel_cache(cu(x), cu(L), R).cpu().numpy()
    want = O.OracleScene.from_mesh(m).voxel_pool(x, L, R).astype(np.float32)
    assert np.array_equal(got, want)
