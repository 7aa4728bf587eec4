"""Plans of the run-time FFT kernels, which a caller's plan takes unless it is the built-in
one: other tile widths, other orders of the radices, one to three stages, odd x lengths,
y/z boxes that overhang the end of the axis (270, 350, 360, 486).  Against the built-in
compile-time instances; a plan with their very radices and width runs them."""
import math

import pytest
import torch

import paper_2501_10622_gb300 as pkg

pytestmark = pytest.mark.gpu

# grid size, y/z width and radices, x width and radices
PLANS = [
    (8, 16, (8,), 16, (4,)), (10, 16, (10,), 4, (5,)), (32, 4, (32,), 4, (16,)), (32, 4, (8, 4), 2, (2, 8)),
    (54, 16, (9, 6), 16, (27,)), (64, 4, (4, 4, 4), 4, (2, 4, 4)), (96, 2, (16, 6), 4, (2, 24)),
    (96, 4, (4, 6, 4), 4, (3, 4, 4)), (98, 16, (14, 7), 4, (7, 7)), (162, 16, (18, 9), 4, (3, 27)),
    (200, 4, (5, 8, 5), 4, (4, 5, 5)), (250, 16, (25, 10), 16, (5, 25)), (256, 4, (8, 32), 4, (32, 4)),
    (270, 16, (18, 15), 4, (9, 15)), (350, 16, (14, 25), 4, (7, 25)), (360, 4, (6, 6, 10), 8, (20, 9)),
    (486, 16, (18, 27), 4, (9, 27)),
]


@pytest.fixture()
def case(request):
    ng = request.param[0]
    ctx = pkg.Context(0, max_ng=ng, max_np=1, max_scales=1)
    gen = torch.Generator(device="cuda").manual_seed(ng)
    grid = (torch.rand((ng, ng, ng), generator=gen, device="cuda") ** 4 * 2 ** 33).long()
    yield ctx, grid, request.param
    ctx.close()


@pytest.mark.parametrize("case", PLANS, indirect=True, ids=lambda p: f"{p[0]}-{'x'.join(map(str, p[2]))}")
def test_runtime_plans(case):
    ctx, grid, (ng, c_yz, r_yz, c_x, r_x) = case
    L, w = 0.78125 * ng, 2.0
    want = ctx.transform(grid, L, w)
    for plans in (((0, c_yz, r_yz),), ((1, c_x, r_x),), ((0, c_yz, r_yz), (1, c_x, r_x))):
        for which, c, r in plans:
            assert ctx.set_fft_plan(ng, which, c, r)
        got = ctx.transform(grid, L, w)
        ctx.check()
        # either transform: six passes, each within 2^-24 log2(ng) of its values' norm
        diff = float((got - want).double().norm() / want.double().norm())
        assert diff <= 2 * 6 * 2.0 ** -24 * math.log2(ng), diff
        for which in (0, 1):
            assert ctx.set_fft_plan(ng, which)
    assert torch.equal(ctx.transform(grid, L, w), want)


@pytest.mark.parametrize("case", [(64, 8, (8, 8), 8, (32,)), (250, 8, (10, 25), 8, (5, 25))], indirect=True,
                         ids=["64", "250"])
def test_the_builtin_plan_set_by_a_caller(case):
    ctx, grid, (ng, c_yz, r_yz, c_x, r_x) = case
    want = ctx.transform(grid, float(ng), 2.0)
    assert ctx.set_fft_plan(ng, 0, c_yz, r_yz) and ctx.set_fft_plan(ng, 1, c_x, r_x)
    assert torch.equal(ctx.transform(grid, float(ng), 2.0), want)
    ctx.check()
