"""Lanes that share a (point, lobe) pair add its samples as one lane would:
chunks of a bake, small enough that 2 to 32 lanes share a pair, equal the rows
of one large bake, where a lane has a pair to itself, bit for bit -- sample
counts that do not divide by the lanes, fewer samples than lanes, ragged
warps, misses lit by a sky and voxel lookups among them."""
import numpy as np
import pytest
import torch

from workloads import cornell_box, surface_queries

pytestmark = pytest.mark.gpu
SIGMA = [0.1, 0.6]


@pytest.mark.parametrize("spp", [(33, 17), (3, 64), (1, 1)])
@pytest.mark.parametrize("extras", [False, True])
def test_chunks_equal_the_whole(spp, extras):
    import paper_2304_05669_gb300 as F
    m = cornell_box()
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    sc = F.Scene.from_mesh(m)
    base = surface_queries(m, 4096, seed=3)
    q = F.pack_queries(*(cu(base[k]) for k in ("x", "n", "wo", "tri")))
    if extras:
        rng = np.random.default_rng(1)
        sc.set_environment(cu(rng.uniform(0, 2, (16, 32, 3)).astype(np.float32)))
        sc.set_voxel_cache(sc.voxel_cache(q, cu(rng.uniform(0, 1, (4096, 3)).astype(np.float32)), 16))
    N = 2_200_000                              # over 60 fills of 311,296 lanes by 3 lobes, a small tree counting thrice
    q = q.repeat(N // 4096 + 1, 1)[:N].contiguous()
    whole = F.bake(sc, q, SIGMA, *spp, seed=5)
    for lo, n in ((0, 1), (7, 33), (1000, 1021), (5000, 20_011), (50_000, 90_001), (200_003, 300_000), (600_001, 1_500_000)):
        part = F.bake(sc, q[lo:lo + n], SIGMA, *spp, seed=5, point_base=lo, order=n % 2 == 1)
        for a, b in zip(part, whole):
            assert torch.equal(a, b[lo:lo + n]), (lo, n)
    assert F.context().sync_status() == 0
