"""A box with no area to compare (flat, with an infinite corner: infinity times
zero) is never opened by the restructuring, so a node over such a box and a
triangle is a treelet of two leaves.  Its subtree size is needed all the same:
the renumbering has to leave a depth-first tree, and rays that meet only sound
triangles hit them."""
import ctypes

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


def _mesh(groups):
    """Per group, along z: two triangles in the plane y = 0, the first with an infinite corner, a sound third in the
    plane, and two at y = 1; corners 0.2 apart."""
    V = []
    for g in range(groups):
        for y, z in ((0, 0.0), (0, 0.1), (0, 1.0), (1, 4.0), (1, 4.1)):
            V.append([[0, y, 8 * g + z], [0.2, y, 8 * g + z], [0, y, 8 * g + z + 0.2]])
    V = np.array(V, np.float32)
    V[::5, 1, 0] = np.inf
    return V


@pytest.mark.parametrize("groups", [1, 3, 64])
@pytest.mark.parametrize("passes", [1, 2, 3])
def test_sizes_of_boxes_without_area(groups, passes):
    import paper_2304_05669_gb300 as F
    from paper_2304_05669_gb300._native import check, lib
    V = _mesh(groups)
    T = len(V)
    Fi = np.arange(3 * T, dtype=np.int32).reshape(T, 3)
    if groups == 1:            # the radix tree has the node this is about: ((0, 1), 2), over a box of NaN area
        ref = O.lbvh_reference(V.reshape(-1, 3), Fi)
        assert ref["order"].tolist() == [0, 1, 2, 3, 4]
        nodes = set(zip(ref["first"].tolist(), ref["last"].tolist()))
        assert {(0, 4), (0, 2), (0, 1), (3, 4)} == nodes
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    zero = t(np.zeros((T, 3), np.float32))
    sc = F.Scene(t(V.reshape(-1, 3)), t(Fi), zero, zero, optimize=passes)
    one = {k: v.cpu().numpy() for k, v in sc.export().items()}
    check(lib().fipt_scene_relayout(sc.handle, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    two = {k: v.cpu().numpy() for k, v in sc.export().items()}
    for k in one:
        assert np.array_equal(one[k], two[k]), k
    child = one["child"]
    assert np.array_equal(np.sort(child[child >= 0]), np.arange(1, T - 1))          # every node but the root once
    assert (child[:, 0][child[:, 0] >= 0] == np.nonzero(child[:, 0] >= 0)[0] + 1).all()   # a first child follows its parent
    sound = np.nonzero(np.isfinite(V).all((1, 2)))[0]
    # over a part of the triangle that its neighbour in the plane does not reach
    o = (V[sound, 0] + [0.02, 0.5, 0.02] + np.isin(sound % 5, (1, 4))[:, None] * [0, 0, 0.13]).astype(np.float32)
    d = np.tile(np.array([0, -1, 0], np.float32), (len(sound), 1))
    tri, dist, _ = (a.cpu().numpy() for a in sc.trace(t(o), t(d)))
    assert F.context().sync_status() == 0
    assert np.array_equal(tri, sound) and np.allclose(dist, 0.5, rtol=16 * 2.0 ** -24, atol=0)
