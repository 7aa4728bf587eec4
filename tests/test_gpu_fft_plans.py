"""The built-in FFT plans (compile-time instances) against the run-time kernels
that callers' plans use, with the same radices: lengths of one, two and three
stages, with one and several butterflies per thread, odd x lengths, and y/z
boxes that overhang the end of the axis (270, 350: two boxes, the second one
partial)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _radices(n):
    """Largest smallest radix first, as the built-in rule picks them."""
    from paper_2501_10622_gb300 import autotune
    fs = autotune.factorisations(n)
    short = min(len(f) for f in fs)
    return max((f for f in fs if len(f) == short), key=lambda f: (min(f), tuple(-x for x in f)))


@pytest.mark.parametrize("ng", [10, 32, 54, 98, 162, 250, 270, 350, 486])
def test_builtin_plans_equal_runtime_plans(ng):
    import paper_2501_10622_gb300 as pkg
    ctx = pkg.Context(0, max_ng=ng, max_np=1, max_scales=1)
    try:
        gen = torch.Generator(device="cuda").manual_seed(ng)
        grid = (torch.rand((ng, ng, ng), generator=gen, device="cuda") ** 4 * 2 ** 33).long()
        L, w = 0.78125 * ng, 2.0
        built_in = ctx.transform(grid, L, w)
        tiles = (8, 4, 2)
        assert any(ctx.set_fft_plan(ng, 0, c, _radices(ng)) for c in tiles)
        assert any(ctx.set_fft_plan(ng, 1, c, _radices(ng // 2)) for c in tiles)
        run_time = ctx.transform(grid, L, w)
        ctx.check()
        # the same butterflies and twiddles: at most a last-bit difference per pass in the contraction of
        # products (6 passes of relative error 2^-24 each, of the field's maximum)
        diff = float((built_in - run_time).abs().max()) / float(built_in.abs().max())
        assert diff <= 6 * 2.0 ** -24 * 4, diff
    finally:
        ctx.close()
