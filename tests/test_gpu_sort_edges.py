"""The radix sort at the edges of its paths (one block up to 8,192 pairs, with
2, 4 or 8 keys per thread; tiles of 2,048 pairs of 12 bytes and 4,096 of 8
above that): the points' Morton order against the host's, and the tree build's
order of 63-bit codes against the oracle's, many equal codes among both."""
import ctypes

import numpy as np
import pytest
import torch

import oracle as O
from workloads import cornell_box

pytestmark = pytest.mark.gpu
SIZES = [1, 2, 33, 1023, 2047, 2048, 2049, 4095, 4096, 4097, 8191, 8192, 8193, 12_289, 70_001]


@pytest.mark.parametrize("n", SIZES)
def test_point_order(n):
    import paper_2304_05669_gb300 as F
    from paper_2304_05669_gb300._native import check, lib
    sc = F.Scene.from_mesh(cornell_box())
    box = sc.info()
    rng = np.random.default_rng(n)
    q = np.zeros((n, 10), np.float32)
    q[:, :3] = rng.uniform(-0.1, 1.1, (n, 3))
    q[: n // 2, :3] = np.round(q[: n // 2, :3], 1)
    want = np.empty(n, np.int32)
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    lo, hi = (np.array(box[k], np.float32) for k in ("lo", "hi"))
    check(lib().fipt_debug_host_query_order(p(q), n, p(lo), p(hi), p(want)))
    assert np.array_equal(F.query_order(sc, torch.from_numpy(q).cuda()).cpu().numpy(), want)


@pytest.mark.parametrize("T", SIZES)
def test_code_order(T):
    import paper_2304_05669_gb300 as F
    rng = np.random.default_rng(T)
    V = rng.uniform(-1, 1, (T, 3, 3)).astype(np.float32)
    V[T // 2:] = V[: T - T // 2]                    # every code twice
    Fi = np.arange(3 * T, dtype=np.int32).reshape(T, 3)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    zero = t(np.zeros((T, 3), np.float32))
    ex = F.Scene(t(V.reshape(-1, 3)), t(Fi), zero, zero, optimize=0).export()
    ref = O.lbvh_reference(V.reshape(-1, 3), Fi)
    assert np.array_equal(ex["morton"].cpu().numpy().view(np.uint64), ref["sorted_codes"])
    assert np.array_equal(ex["order"].cpu().numpy(), ref["order"])
