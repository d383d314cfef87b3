"""Sample points of the emitter extraction where a thread's four consecutive
samples cross triangles, a block is not full, or x is not 16-byte aligned
(then it is written without the bulk copy)."""
import ctypes

import numpy as np
import pytest
import torch

import oracle as O
from workloads import cornell_box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 29, 57, 100])     # 36 n samples: 1024 lies between 28 and 29
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
