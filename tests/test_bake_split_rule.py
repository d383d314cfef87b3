"""The lanes that share a pair of a bake (the library's rule, run on the host):
never more than samples, never so many that a lane's next sample index leaves
the int it is counted in (it would turn negative and the lane never end), and
fewer the more pairs there are."""
import ctypes

import numpy as np
import pytest

INT_MAX = 2 ** 31 - 1


def _log_lanes(pairs, T, spp_d, spp_s, sms=152):
    from paper_2304_05669_gb300._native import check, lib
    g = ctypes.c_int32(-1)
    check(lib().fipt_debug_bake_split(pairs, T, spp_d, spp_s, sms, ctypes.byref(g)))
    return g.value


@pytest.mark.parametrize("T", [0, 36, 200_000])
@pytest.mark.parametrize("spp", [1, 2, 3, 16, 33, 1000, INT_MAX - 32, INT_MAX - 31, INT_MAX - 16, INT_MAX - 1, INT_MAX])
def test_lanes(T, spp):
    before = 5
    for pairs in np.unique(np.geomspace(1, 2 ** 36, 200).astype(np.int64)).tolist():
        for d, s in ((spp, spp), (spp, 64), (64, spp)):
            g = _log_lanes(pairs, T, d, s)
            assert 0 <= g <= 5 and 2 ** g <= min(d, s)
            # the last lane's last step: from a sample below the count, G further
            assert max(d, s) - 1 + 2 ** g <= INT_MAX
        assert _log_lanes(pairs, T, spp, spp) <= before
        before = _log_lanes(pairs, T, spp, spp)
    assert _log_lanes(1, T, 64, 64) == 5 and _log_lanes(2 ** 36, T, 64, 64) == 0
