"""The warp walk's guards are acted on once per block of node visits, so its
stack takes a whole block of pushes between two checks: rays that push at
every visit of a caterpillar tree (triangles at x = 0.75 / 2^k, whose Morton
codes each split one triangle off the rest) through one and several blocks,
against the hits known by construction."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 2, 8, 9, 10, 17, 18, 20])
@pytest.mark.parametrize("optimize", [0, 2])
def test_pushes_at_every_visit(T, optimize):
    import paper_2304_05669_gb300 as F
    x = 0.75 * 0.5 ** np.arange(T)
    V = np.stack([np.array([[a, -1.0, -1.0], [a, 3.0, -1.0], [a, -1.0, 3.0]]) for a in x]).reshape(-1, 3)
    t = lambda a, d: torch.from_numpy(np.ascontiguousarray(a, d)).cuda()
    zero = np.zeros((T, 3))
    sc = F.Scene(t(V, np.float32), t(np.arange(3 * T).reshape(T, 3), np.int32), t(zero, np.float32),
                 t(zero, np.float32), optimize=optimize)
    n = 97                                    # a ragged last warp
    up = np.arange(n) % 2 == 0                # along +x: every box is entered nearest last
    o = np.where(up, -1.0, 2.0)[:, None] * [1.0, 0, 0] + np.random.default_rng(0).uniform(-0.4, 0.4, (n, 3)) * [0, 1, 1]
    d = np.where(up, 1.0, -1.0)[:, None] * [1.0, 0, 0]
    for skip_nearest in (False, True):
        near = np.where(up, T - 1, 0)
        skip = near if skip_nearest else np.full(n, -1)
        want = np.where(up, T - 2, 1) if skip_nearest else near
        miss = (want < 0) | (want >= T)
        tri, dist, _ = (a.cpu().numpy() for a in sc.trace(t(o, np.float32), t(d, np.float32), t(skip, np.int32)))
        assert F.context().sync_status() == 0
        assert np.array_equal(tri, np.where(miss, -1, want))
        # one subtraction, one division and the products of the edge functions in float32
        far = np.abs(x[np.where(miss, 0, want)] - o[:, 0])
        assert np.all(np.isinf(dist[miss])) and np.allclose(dist[~miss], far[~miss], rtol=16 * 2.0 ** -24, atol=0)
