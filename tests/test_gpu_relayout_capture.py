"""Restructuring passes that were only captured leave no subtree sizes: a
renumbering after them counts the sizes of the tree as it is, and captured
behind them it counts those that its graph will find."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _scene(F, T, **kw):
    rng = np.random.default_rng(T)
    V = (rng.uniform(-1, 1, (T, 1, 3)) + rng.uniform(-0.05, 0.05, (T, 3, 3))).astype(np.float32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    zero = t(np.zeros((T, 3), np.float32))
    return F.Scene(t(V.reshape(-1, 3)), t(np.arange(3 * T, dtype=np.int32).reshape(T, 3)), zero, zero, **kw)


@pytest.mark.parametrize("replayed", [False, True])
def test_captured_passes(replayed):
    import paper_2304_05669_gb300 as F
    from paper_2304_05669_gb300._native import check, lib
    T = 1000
    sc = _scene(F, T, optimize=0)
    torch.cuda.synchronize()
    handle = lambda: ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        check(lib().fipt_scene_optimize(sc.handle, 2, handle()))
        if replayed:
            check(lib().fipt_scene_relayout(sc.handle, handle()))
    if replayed:
        graph.replay()
    else:
        check(lib().fipt_scene_relayout(sc.handle, handle()))
    sc.optimized = 2                          # no radix-tree ranges to export
    got = {k: v.cpu().numpy() for k, v in sc.export().items()}
    if replayed:
        want = {k: v.cpu().numpy() for k, v in _scene(F, T, optimize=2).export().items()}
        for k in want:
            assert np.array_equal(got[k], want[k]), k
    child = got["child"]
    assert np.array_equal(np.sort(child[child >= 0]), np.arange(1, T - 1))          # every node but the root once
    assert (child[:, 0][child[:, 0] >= 0] == np.nonzero(child[:, 0] >= 0)[0] + 1).all()   # a first child follows its parent
    assert F.context().sync_status() == 0
