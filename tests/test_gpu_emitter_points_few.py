"""Sample points with 4 and with 16 consecutive samples a thread (from 16 per
triangle): samples that cross triangles within a thread, and blocks of 512 and
2,048 points that end just before and after the last of 36 triangles."""
import ctypes

import numpy as np
import pytest
import torch

import oracle as O
from workloads import cornell_box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 14, 15, 16, 17, 31, 56, 57, 114])     # 36 n points: 512 < 540, 2,016 < 2,048 < 2,052
@pytest.mark.parametrize("offset", [0, 1])
def test_points(n, offset):
    import paper_2304_05669_gb300 as F
    from paper_2304_05669_gb300._native import check, lib
    m = cornell_box()
    sc = F.Scene.from_mesh(m)
    x = torch.full((3 * 36 * n + 8,), -7.0, device="cuda")
    check(lib().fipt_emitter_sample_points(sc.handle, 11, 2, n, ctypes.c_void_p(x.data_ptr() + 4 * offset),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    got = x.cpu().numpy()
    want = O.OracleScene.from_mesh(m).emitter_points(n, seed=11, request_id=2)
    assert (got[:offset] == -7).all() and (got[offset + 3 * 36 * n:] == -7).all()
    got = got[offset:offset + 3 * 36 * n].reshape(-1, 3).astype(np.float64)
    # square root, two differences, two products and a sum of three products in float32
    assert np.max(np.abs(got - want)) <= 8 * np.abs(m.V).max() * 2.0 ** -24
