"""Emitter classification where rows are held by four lanes (a multiple of 4
samples, at most 128, 16-byte aligned) and where they are not: bit-equal means
for sample counts around those limits, a number of rows that does not fill a
warp, rows of zeros, of both signs, outside the exact integer range, with
subnormals, infinities and NaNs; shifted arrays."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 4, 12, 100, 124, 127, 128, 132])
@pytest.mark.parametrize("T", [1, 31, 33, 1000])
@pytest.mark.parametrize("shift", [0, 1])
def test_means(n, T, shift):
    import paper_2304_05669_gb300 as F
    rng = np.random.default_rng(n * T)
    a = rng.uniform(0, 0.03, (T, n)).astype(np.float32)
    for k, row in enumerate(a):
        if k % 9 == 1:
            row[:] = 0.0
        if k % 9 == 2:
            row[::2] *= -1
        if k % 9 == 3:
            row[0] = 1e20
        if k % 9 == 4:
            row[-1] = 1e-41
        if k % 9 == 5:
            row[n // 2] = np.inf
        if k % 9 == 6:
            row[0] = np.nan
        if k % 9 == 7:
            row[:] = np.float32(-0.0)
    buf = torch.zeros(T * n + shift, device="cuda")
    buf[shift:] = torch.from_numpy(a.reshape(-1)).cuda()
    flag, mean = (x.cpu().numpy() for x in F.emitter_classify(buf[shift:], n, 0.01))
    with np.errstate(invalid="ignore", over="ignore"):
        o_flag, o_mean = O.emitter_classify(a.reshape(-1), n, 0.01)
    assert np.array_equal(mean, o_mean, equal_nan=True) and np.array_equal(flag, o_flag)
