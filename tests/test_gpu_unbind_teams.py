"""The self-boundness check's ways of sharing a group among CTAs: one CTA (up
to 2048 members, sorted in shared memory), a team of 8, a team of 64
(above 65,536), the whole grid.  Group sizes sit on the edges between them; the
decisions must not depend on the way, nor on members at equal radii."""
import numpy as np
import pytest
import torch

import oracle
import paper_2501_10622_gb300 as pkg
from paper_2501_10622_gb300 import synth
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def uctx():
    c = pkg.Context(0, max_ng=64, max_np=1 << 18, max_scales=1, unbind=True)
    yield c
    c.close()


def _groups(sizes, L, seed):
    """Gaussian groups about random centres, with a tenth of the members too fast to be bound."""
    rng = np.random.default_rng(seed)
    pos, vel, grp = [], [], []
    for g, n in enumerate(sizes):
        centre = rng.uniform(0.1 * L, 0.9 * L, 3)
        sigma = np.sqrt(synth.G_MPC_KMS_MSUN * n * 1e10 / 0.3 / 6.0)
        v = sigma * rng.normal(size=(n, 3))
        v[: n // 10] *= 4.0
        pos.append(centre + 0.3 * rng.normal(size=(n, 3)))
        vel.append(v + 100.0 * rng.normal(size=3))
        grp.append(np.full(n, g))
    perm = rng.permutation(sum(sizes))
    return (np.concatenate(pos)[perm].astype(np.float32), np.concatenate(vel)[perm].astype(np.float32),
            np.concatenate(grp)[perm].astype(np.int32))


def test_every_way_decides_alike(uctx):
    sizes = [2047, 2048, 2049, 4096, 4097, 20000, 65536, 65537]
    L = 100.0
    pos, vel, grp = (dev(x) for x in _groups(sizes, L, 7))
    results = []
    # the default, the teams of 8 for everything above one CTA's share, the whole grid from 2001 members on
    # (groups of a big team's size excepted)
    for grid_min in (1 << 16, 1 << 20, 2000):
        uctx.debug_set(pkg._lib.DEBUG_UNBIND_GRID_MIN, grid_min)
        try:
            out = uctx.unbind(pos, vel, grp, L, mass_unit=1e10, n_groups=len(sizes))
            uctx.check()
            results.append([x.cpu().numpy() for x in out])
        finally:
            uctx.debug_set(pkg._lib.DEBUG_UNBIND_GRID_MIN, 1 << 16)
    kept, rounds = results[0][1], results[0][2]
    assert (kept > 0).all() and (kept < np.array(sizes)).all() and (rounds > 1).all()
    for r in results[1:]:
        for a, b in zip(results[0], r):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("copies", [20, 200])
def test_members_at_equal_radii(uctx, copies):
    # `copies` members at one point: their radii, and so the sort keys' upper halves, are equal (20: a short
    # run; 200: the sort falls back to all eight digits)
    L = 100.0
    pos, vel, grp = _groups([3000, 5000], L, 11)
    for g in (0, 1):
        i = np.flatnonzero(grp == g)[:copies]
        pos[i] = pos[i[0]]
    ref = oracle.unbind(pos, vel, grp, L, G=synth.G_MPC_KMS_MSUN, mass=None, mass_unit=1e10, n_groups=2, max_iter=100)
    out, nk, it = uctx.unbind(dev(pos), dev(vel), dev(grp), L, mass_unit=1e10, n_groups=2)
    uctx.check()
    if ref[3] > 1e-9:  # no decision within fp64 rounding of its threshold
        np.testing.assert_array_equal(out.cpu().numpy(), ref[0])
        np.testing.assert_array_equal(nk.cpu().numpy(), ref[1])
        np.testing.assert_array_equal(it.cpu().numpy(), ref[2])
