"""Mass quanta, rint(mass / mass_unit) with halves to even, where the deposit's integer
shortcut and the exact quotient are closest: fractions about one half, quotients up to 2^31.
Each particle sits on a node of its own, so its cell holds its quantum in units of 2^30."""
import numpy as np
import pytest
import torch

import paper_2501_10622_gb300 as pkg
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu
NG = 16


@pytest.fixture(scope="module")
def ctx():
    c = pkg.Context(0, max_ng=NG, max_np=NG ** 3, max_scales=1)
    yield c
    c.close()


def _quanta(ctx, mass, unit):
    """The quanta the deposit forms."""
    n = len(mass)
    i = np.arange(n)
    pos = np.stack([i % NG, i // NG % NG, i // NG ** 2], 1).astype(np.float32)
    mtot = torch.zeros(1, dtype=torch.int64, device="cuda")
    grid = ctx.deposit(dev(pos), float(NG), NG, mass=dev(mass), mass_unit=unit, mtot=mtot)
    ctx.check()
    q = grid.cpu().numpy().reshape(-1)
    assert (q % 2 ** 30 == 0).all() and int(mtot) == int(q.sum()) >> 30
    return q[:n] >> 30


@pytest.mark.parametrize("unit,mass", [("0x1.ffffff39fe004p+0", 4294797824.0), ("0x1.fffffd69fe035p+0", 4294916608.0),
                                       ("0x1.fffffc6df6065p+0", 4294783744.0)])
def test_quanta_near_2_31(ctx, unit, mass):
    # the shortcut's error is largest here: its fraction reads 2^-9 from one half, on the wrong side
    unit, mass = float.fromhex(unit), np.array([mass], np.float32)
    assert _quanta(ctx, mass, unit)[0] == np.rint(mass.astype(np.float64) / unit)[0]


@pytest.mark.parametrize("unit", [1.0, 0.01, 1.0 / 3.0, 7.3e-5, 1.9999999, 1e10])
@pytest.mark.parametrize("top", [4.0, 2.0 ** 12, 2.0 ** 20])
def test_quanta_about_halves(ctx, unit, top):
    # fractions exactly and nearly one half, 0 to 8 steps of 2^-11 to either side, whole quotients, any quotient
    rng = np.random.default_rng(int(top))
    n = NG ** 3
    q = np.floor(rng.uniform(0.0, top, n))
    q += np.where(rng.random(n) < 0.7, 0.5 + rng.integers(-8, 9, n) * 2.0 ** -11 * (rng.random(n) < 0.5),
                  np.where(rng.random(n) < 0.5, rng.random(n), 0.0))
    mass = (q * unit).astype(np.float32)
    want = np.rint(mass.astype(np.float64) / unit)
    assert want.sum() < 2 ** 33
    np.testing.assert_array_equal(_quanta(ctx, mass, unit), want.astype(np.int64))


def test_quotients_that_round_to_a_half(ctx):
    # units such that the fp64 quotient is a half, or a few units of its last place beside one, while the mass is
    # not that many units exactly
    rng = np.random.default_rng(3)
    halves = 0
    for k in range(400):
        mass = np.float32(rng.uniform(0.5, 4.0) * 2.0 ** rng.integers(-3, 28))
        h = np.floor(rng.uniform(0.0, 2.0 ** rng.integers(0, 31))) + 0.5
        unit = float(mass) / h
        for _ in range(abs(k % 5 - 2)):
            unit = float(np.nextafter(unit, 0.0 if k % 5 < 2 else np.inf))
        q = float(mass) / unit
        halves += q == h
        assert _quanta(ctx, np.array([mass]), unit)[0] == np.rint(q), (float(mass), unit.hex())
    assert 50 < halves < 350  # both kinds occur
