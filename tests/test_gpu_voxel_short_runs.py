"""Voxel means where neighbouring runs are short: a lane a run, four long ones
among them at a time, dense neighbourhoods of 128 runs beside such ones (and a
last one that is not full), and runs outside the exact integer range listed by
their block; bit-equal to the oracle's grid."""
import numpy as np
import pytest
import torch

import oracle as O
from workloads import cornell_box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["narrow", "wide", "some wide", "signs"])
@pytest.mark.parametrize("runs,long_runs,dense", [(1, 0, 0), (31, 0, 0), (129, 1, 0), (140, 2, 128), (700, 4, 0), (700, 7, 256),
                                                  (1000, 9, 900)])
def test_short_runs(kind, runs, long_runs, dense):
    import paper_2304_05669_gb300 as F
    rng = np.random.default_rng(runs + long_runs)
    R = 32
    lengths = rng.integers(1, 4, runs)
    lengths[rng.permutation(runs)[:long_runs]] = rng.choice([31, 32, 33, 65], long_runs)
    lengths[:dense] += rng.integers(0, 40, dense)         # runs follow one another in the order of their cells
    cells = np.sort(rng.permutation(R * R)[:runs])
    cell = rng.permutation(np.repeat(cells, lengths))
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
