"""The deposit's counter copies on large grids, where their number falls from eight to
four (beyond 2^17 counters), two (2^18) and one (2^19), with 16 particles per counter:
bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2501_10622_gb300 as pkg
from tests.gpu_util import dev, random_box
from tests.test_gpu_deposit_copies import _counters

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ng,masses,copies", [(322, True, 4), (420, False, 2), (514, False, 1)])
def test_copies_on_large_grids(ng, masses, copies):
    assert 2 ** 20 // (2 * copies) < _counters(ng) and (copies == 1 or _counters(ng) <= 2 ** 20 // copies)
    n, L = 16 * _counters(ng), 0.7 * ng
    pos = random_box(n, L, ng)
    mass = (np.random.default_rng(ng).random(n) * 5).astype(np.float32) if masses else None
    kw = {"mass_unit": 1.0 / 512} if masses else {}
    ctx = pkg.Context(0, max_ng=ng, max_np=n, max_scales=1)
    try:
        g = ctx.deposit(dev(pos), L, ng, mass=dev(mass) if masses else None, **kw)
        ctx.check()
    finally:
        ctx.close()
    ref, _ = oracle.cic(pos, L, ng, mass=mass, **kw)
    np.testing.assert_array_equal(g.cpu().numpy(), ref)
