"""The stencil CWT at the edges of its radius classes (4, 8, 12 and 16 run
register windows with zero taps beyond R; 17 the general kernels), on grids
narrower than a warp's columns, ragged, and barely wider than the stencil,
against the fp64 sum of the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2501_10622_gb300 import synth
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ng,R", [(8, 1), (10, 4), (12, 5), (18, 8), (20, 9), (26, 12), (28, 13), (34, 16), (36, 17),
                                  (66, 8), (70, 16)])
def test_radius_classes(gctx, ng, R):
    L, w = 0.78125 * ng, 1.0
    pos = synth.clumped_box(ng ** 3, L, 3, seed=ng).numpy()
    grid, _ = oracle.cic(pos, L, ng)
    ref = oracle.cwt_stencil(grid, L, w, R)
    c = gctx.transform_stencil(dev(grid), L, w, R)
    gctx.check()
    got = c.cpu().numpy().astype(np.float64)
    # three passes of 2 R + 1 fp32 terms each: 3 (2 R + 2) roundings of the sum of the terms' magnitudes, which
    # for this kernel is at most about ten times the largest result
    assert np.max(np.abs(got - ref)) <= 30 * (2 * R + 2) * 2.0 ** -24 * np.max(np.abs(ref))


def test_an_unaligned_grid(gctx):
    ng, L, w, R = 22, 20.0, 1.3, 7
    grid, _ = oracle.cic(synth.clumped_box(9000, L, 3, seed=4).numpy(), L, ng)
    buf = torch.empty(ng ** 3 + 1, dtype=torch.int64, device="cuda")
    view = buf[1:].view(ng, ng, ng)  # 8-byte aligned only
    view.copy_(dev(grid))
    a = gctx.transform_stencil(view, L, w, R)
    b = gctx.transform_stencil(dev(grid), L, w, R)
    gctx.check()
    assert torch.equal(a, b)
