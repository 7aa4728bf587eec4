"""The deposit's counter copies at the sizes where their number and the launch that
adds them up change: one counter set below 16 particles per counter, 16 copies from
there on (one block up to 4096 counters, the general scan above), 8 copies beyond
2^16 counters.  The grid is a sum of integers: bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2501_10622_gb300 as pkg
from tests.gpu_util import dev, random_box

pytestmark = pytest.mark.gpu


def _counters(ng):
    return -(-ng // 32) * -(-ng // 8) * -(-ng // 8) * 8


@pytest.mark.parametrize("masses", [False, True])
@pytest.mark.parametrize("ng,less", [(8, 1), (8, 0), (64, 0), (96, 1), (96, 0), (100, 0), (256, 0), (258, 0)])
def test_copies_bit_exact(ng, less, masses):
    n = 16 * _counters(ng) - less
    L = 0.7 * ng
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
