"""Per-triangle error sums at the edges of the tiles they are computed in (rows
of 32 sorted pixels, tiles of 256): segments that end, begin and pass over
them, one triangle over many tiles, pixels without a triangle, triangles
without a pixel."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [1, 31, 32, 33, 255, 256, 257, 511, 512, 513, 8191, 20_000])
@pytest.mark.parametrize("kind", ["one", "few", "runs", "each"])
def test_segments_at_tile_edges(P, kind):
    import paper_2304_05669_gb300 as F
    rng = np.random.default_rng(P)
    T = {"one": 1, "few": 3, "runs": 40, "each": P + 5}[kind]
    tri = {"one": np.zeros(P), "few": rng.integers(-1, 3, P), "runs": np.sort(rng.integers(0, 39, P)) ** 2 // 38,
           "each": rng.permutation(P)}[kind].astype(np.int32)
    Lr, Lgt = (rng.uniform(0, 4, (P, 3)).astype(np.float32) for _ in "01")
    cu = lambda a: torch.from_numpy(a).cuda()
    err, count = (a.cpu().numpy() for a in F.tri_error(cu(tri), cu(Lr), cu(Lgt), T))
    want, n = O.tri_error(tri, Lr, Lgt, T)
    assert np.array_equal(count, n)
    # non-negative terms: n additions on each side and three products and sums a term, each within 2^-53
    assert np.all(np.abs(err - want) <= (2 * n + 8) * 2.0 ** -53 * want)
