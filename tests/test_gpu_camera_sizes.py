"""Images too small to fill their tiles are looked through 32 pixels in order,
across rows and views: first hits of both layouts at sizes around the limit of
28 pixels per tile of 32, against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from parity import ETA_TRACE
from workloads import pinhole_views, procedural_room

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("views,W,H", [(1, 1, 1), (33, 1, 1), (37, 2, 1), (11, 3, 3), (9, 5, 5), (7, 17, 5), (5, 25, 25),
                                       (3, 65, 49), (40, 7, 4), (13, 8, 4), (2, 1, 33), (2, 61, 1), (3, 97, 31)])
def test_small_images(views, W, H):
    import paper_2304_05669_gb300 as F
    m = procedural_room(1)
    sc = F.Scene.from_mesh(m)
    S = O.OracleScene.from_mesh(m)
    cams = pinhole_views(m, views, seed=2)
    P = views * W * H
    out = torch.full((P + 2, 10), -7.0, device="cuda")
    valid = torch.full((P + 2,), -7, dtype=torch.int32, device="cuda")
    sc.camera_queries(torch.from_numpy(cams).cuda(), W, H, out=out, valid=valid)
    q, valid = out.cpu().numpy(), valid.cpu().numpy()
    assert (q[P:] == -7).all() and (valid[P:] == -7).all()
    q, valid = q[:P], valid[:P]
    ora = S.camera_queries(cams, W, H, np.arange(P), eta=ETA_TRACE)
    tri = q[:, 9].copy().view(np.int32)
    unique = (ora["n_cand"] <= 1) & ~ora["miss_possible"]
    assert np.array_equal(tri[unique], ora["tri"][unique])
    assert np.array_equal(valid[unique], (ora["tri"][unique] >= 0).astype(np.int32))
    u = unique & (tri >= 0)
    assert np.max(np.abs(q[u, 0:3] - ora["x"][u]), initial=0) < 2e-6 * S.L * 4       # as at the larger sizes
    assert np.max(np.abs(q[u, 3:6] - ora["n"][u]), initial=0) < 1e-5
    assert np.max(np.abs(q[u, 6:9] - ora["wo"][u]), initial=0) < 1e-5
    for r in np.nonzero(~unique)[0]:
        cands = set(ora["cand_id"][r, :max(ora["n_cand"][r], 0)].tolist()) | {int(ora["tri"][r])}
        if ora["miss_possible"][r]:
            cands.add(-1)
        assert int(tri[r]) in cands
