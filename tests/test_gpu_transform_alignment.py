"""cwthf_transform on buffers that are aligned to their own elements only (a grid 8 bytes
off a 16-byte boundary, a field 4 bytes off an 8-byte one): the same bits as on aligned
ones, with a radix plan, a Bluestein plan and a caller's plan."""
import pytest
import torch

import paper_2501_10622_gb300 as pkg

pytestmark = pytest.mark.gpu


def _off(shape, dtype, off):
    """A tensor whose first element lies `off` elements into its allocation."""
    n = shape[0] * shape[1] * shape[2]
    t = torch.zeros(n + off, dtype=dtype, device="cuda")[off:].view(shape)
    assert t.data_ptr() % 16 == off * t.element_size() % 16
    return t


@pytest.mark.parametrize("ng,plan", [(8, None), (64, None), (62, None), (230, None), (96, (4, (8, 12), (6, 8)))])
def test_element_aligned_buffers(ng, plan):
    ctx = pkg.Context(0, max_ng=ng, max_np=1, max_scales=1)
    try:
        if plan:
            assert ctx.set_fft_plan(ng, 0, plan[0], plan[1]) and ctx.set_fft_plan(ng, 1, plan[0], plan[2])
        gen = torch.Generator(device="cuda").manual_seed(ng)
        grid = (torch.rand((ng, ng, ng), generator=gen, device="cuda") ** 4 * 2 ** 33).long()
        want = ctx.transform(grid, float(ng), 2.0)
        for goff in (0, 1):
            for coff in (0, 1, 2, 3):
                g = _off((ng, ng, ng), torch.int64, goff)
                g.copy_(grid)
                out = ctx.transform(g, float(ng), 2.0, cwt=_off((ng, ng, ng), torch.float32, coff))
                ctx.check()
                assert torch.equal(out, want), (goff, coff)
    finally:
        ctx.close()
