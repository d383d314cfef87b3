"""The walk's stack at its limit of 32 entries, acted on once per eight visits.
Triangles at c / 2^j along x, y and z in turn, whose Morton codes each split one
triangle off the rest, make a chain of T - 1 nodes; a ray out of the corner
that all boxes hold finds the rest nearer at every one of them, pushes T - 1
leaves and parks the last.  Up to 33 remain in reach of a check; from 34 on the
ray is cut short, says so, and ends."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


def _chain(T):
    V = np.zeros((T, 3, 3), np.float32)
    for i in range(T):
        j, a = divmod(i, 3)
        u, v = (k for k in range(3) if k != a)
        V[i, :, a] = (0.75, 0.7, 0.65)[a] * 0.5 ** j
        V[i, :, u] = -1, 1, 0
        V[i, :, v] = -1, -1, 1
    return V


@pytest.mark.parametrize("T", [9, 31, 32, 33, 34, 35, 36, 41, 43, 60])
def test_stack_limit(T):
    import paper_2304_05669_gb300 as F
    V = _chain(T)
    Fi = np.arange(3 * T, dtype=np.int32).reshape(T, 3)
    ref = O.lbvh_reference(V.reshape(-1, 3), Fi)
    assert (ref["first"] == 0).all() and np.array_equal(np.sort(ref["last"]), np.arange(1, T))    # the chain
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    zero = t(np.zeros((T, 3), np.float32))
    sc = F.Scene(t(V.reshape(-1, 3)), t(Fi), zero, zero, optimize=0)
    n = 97                                    # a ragged last warp
    rng = np.random.default_rng(T)
    d = (1 + rng.uniform(-0.02, 0.02, (n, 3))).astype(np.float32)
    o = np.zeros((n, 3), np.float32)
    for last in (T - 1, T - 2):               # the nearest plane, and the next without it
        skip = np.full(n, -1 if last == T - 1 else T - 1, np.int32)
        tri = sc.trace(t(o), t(d), t(skip))[0].cpu().numpy()
        if T - 1 > 33:
            with pytest.raises(F.FiptError, match="0x1$"):
                F.context().sync_status()
            continue
        assert F.context().sync_status() == 0
        assert (tri == last).all()
    low = F.Scene(t(V[:9].reshape(-1, 3)), t(Fi[:9]), zero[:9], zero[:9], optimize=0)     # the next call is sound again
    assert (low.trace(t(o), t(d))[0].cpu().numpy() == 8).all()
    assert F.context().sync_status() == 0
