"""The self-boundness check where the number of CTAs per group depends on how many groups
there are: many medium groups (one, two and four CTAs each), few (eight), big ones alone
(128) and side by side (64).  The decisions must be those of the other ways."""
import numpy as np
import pytest

import paper_2501_10622_gb300 as pkg
from tests.gpu_util import dev
from tests.test_gpu_unbind_teams import _groups

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [
    [2049] * 400,                                             # one CTA each
    [2049, 3000] * 60,                                        # two
    [2100] * 60,                                              # four
    [2049 + i for i in range(20)],                            # eight
    [40000, 20000, 9000, 5000] + [2100] * 350,                # one, two, four and eight, by size
    [300000],                                                 # 128
    [140000, 131072],                                         # 128, side by side
    [70000] * 5 + [3000] * 3,                                 # 64, more groups than teams
    [300000, 65537, 65536, 2048, 1, 0, 50],                   # every kind
], ids=["one", "two", "four", "eight", "by-size", "big-alone", "big-pair", "big-many", "every-kind"])
def test_shares_decide_alike(sizes):
    L = 100.0
    pos, vel, grp = (dev(x) for x in _groups(sizes, L, len(sizes)))
    ctx = pkg.Context(0, max_ng=64, max_np=sum(sizes), max_scales=1, unbind=True)
    results = []
    try:
        # by share; every medium group on the whole grid; big groups on eight CTAs
        for grid_min in (1 << 16, 2000, 1 << 20):
            ctx.debug_set(pkg._lib.DEBUG_UNBIND_GRID_MIN, grid_min)
            out = ctx.unbind(pos, vel, grp, L, mass_unit=1e10, n_groups=len(sizes))
            ctx.check()
            results.append([x.cpu().numpy() for x in out])
    finally:
        ctx.close()
    kept = results[0][1]
    big = np.array(sizes) > 1000
    assert (kept[big] > 0.6 * np.array(sizes)[big]).all() and (kept < np.array(sizes))[big].all()
    for other in results[1:]:
        for a, b in zip(results[0], other):
            np.testing.assert_array_equal(a, b)
