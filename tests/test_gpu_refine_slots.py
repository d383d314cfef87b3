"""Slots hold up to 32 samples of a point side by side and the points in Morton
order: whatever the sample counts leave over, a refinement equals the one of
each of its points alone, bit for bit."""
import numpy as np
import pytest
import torch

from workloads import cornell_box, surface_queries

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spp", [(1, 1), (3, 5), (32, 32), (33, 31), (40, 64)])
@pytest.mark.parametrize("K", [1, 3])
def test_points_alone_and_together(spp, K):
    import paper_2304_05669_gb300 as F
    m = cornell_box()
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    sc = F.Scene.from_mesh(m)
    rng = np.random.default_rng(2)
    sc.set_materials(cu(rng.uniform(0, 1, (m.T, 3)).astype(np.float32)), cu(rng.uniform(0.05, 1, m.T).astype(np.float32)),
                     cu(rng.uniform(0, 1, m.T).astype(np.float32)))
    b = surface_queries(m, 77, seed=4)
    q = F.pack_queries(*(cu(b[k]) for k in ("x", "n", "wo", "tri")))
    sigma = [0.1, 0.4, 0.9][:K]
    whole = F.bake_refine(sc, q, sigma, *spp, max_depth=3, seed=9, per_sample=True)
    for lo, n in ((0, 1), (5, 33), (40, 37)):
        part = F.bake_refine(sc, q[lo:lo + n], sigma, *spp, max_depth=3, seed=9, point_base=lo, per_sample=True)
        for x, y in zip(part, whole):
            assert torch.equal(x, y[lo:lo + n]), (lo, n)
    assert F.context().sync_status() == 0
