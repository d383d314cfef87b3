"""Emitter classification on both sides of the 52 samples from which four lanes
hold a row, and warps most or all of whose rows lie outside the exact integer
range: bit-equal means."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [48, 52, 56, 128])
@pytest.mark.parametrize("wide", ["none", "most", "all"])
def test_means(n, wide):
    import paper_2304_05669_gb300 as F
    T = 77
    rng = np.random.default_rng(n)
    a = rng.uniform(0, 0.03, (T, n)).astype(np.float32)
    rows = {"none": np.zeros(T, bool), "most": rng.random(T) < 0.7, "all": np.ones(T, bool)}[wide]
    a[rows] *= np.float32(2.0) ** rng.integers(-40, 41, (int(rows.sum()), n)).astype(np.float32)
    flag, mean = (x.cpu().numpy() for x in F.emitter_classify(torch.from_numpy(a.reshape(-1)).cuda(), n, 0.01))
    o_flag, o_mean = O.emitter_classify(a.reshape(-1), n, 0.01)
    assert np.array_equal(mean, o_mean) and np.array_equal(flag, o_flag)
