"""The last restructuring pass leaves the subtree sizes the depth-first
renumbering reads.  A second renumbering counts them anew and has to leave a
depth-first tree as it is, so wrong sizes would show as other child links."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [3, 4, 5, 8, 33, 1000, 20_000])
@pytest.mark.parametrize("passes", [1, 2, 3])
def test_renumbering_again_changes_nothing(T, passes):
    import paper_2304_05669_gb300 as F
    from paper_2304_05669_gb300._native import check, lib
    rng = np.random.default_rng(T)
    V = (rng.uniform(-1, 1, (T, 1, 3)) + rng.uniform(-0.05, 0.05, (T, 3, 3))).astype(np.float32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    zero = t(np.zeros((T, 3), np.float32))
    sc = F.Scene(t(V.reshape(-1, 3)), t(np.arange(3 * T, dtype=np.int32).reshape(T, 3)), zero, zero, optimize=passes)
    one = {k: v.cpu().numpy() for k, v in sc.export().items()}
    check(lib().fipt_scene_relayout(sc.handle, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    two = {k: v.cpu().numpy() for k, v in sc.export().items()}
    assert F.context().sync_status() == 0
    for k in one:
        assert np.array_equal(one[k], two[k]), k
    child = one["child"]
    assert np.array_equal(np.sort(child[child >= 0]), np.arange(1, T - 1))          # every node but the root once
    assert (child[:, 0][child[:, 0] >= 0] == np.nonzero(child[:, 0] >= 0)[0] + 1).all()   # a first child follows its parent
