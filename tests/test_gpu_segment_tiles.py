"""Segmentation at the tile kernel's edges: tiles full of seeds (one per 2 x 2 x 2
block, more than its counters hold at a time), ragged tiles, grids smaller than a
tile, plateaus across the periodic boundary, and a field that is not 8-byte
aligned."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _check(gctx, field, cwt_min=0.0, cwt=None):
    ng = field.shape[0]
    ref = oracle.segment(field, cwt_min)
    cwt = torch.as_tensor(field).cuda() if cwt is None else cwt
    lab = gctx.segment(cwt, cwt_min)
    seeds, n_cells, n = gctx.segment_sizes(ng ** 3 // 8 + 8)
    gctx.check()
    lab = lab.cpu().numpy()
    np.testing.assert_array_equal(lab, np.asarray(ref).reshape(lab.shape))
    # every seed's cell count, recounted from the labels
    s, c = np.unique(lab[lab >= 0], return_counts=True)
    np.testing.assert_array_equal(seeds.cpu().numpy(), s)
    np.testing.assert_array_equal(n_cells.cpu().numpy(), c)
    assert n == len(s)


@pytest.mark.parametrize("ng", [8, 16, 34, 64, 66, 130])
def test_a_seed_in_every_block(gctx, ng):
    rng = np.random.default_rng(ng)
    field = rng.random((ng, ng, ng)).astype(np.float32) * 0.1
    field[::2, ::2, ::2] += 1.0
    _check(gctx, field)


@pytest.mark.parametrize("ng", [10, 18, 36, 70])
def test_plateaus_across_the_boundary(gctx, ng):
    rng = np.random.default_rng(ng + 1)
    field = rng.integers(-2, 3, (ng, ng, ng)).astype(np.float32)  # few values: ties everywhere
    _check(gctx, field)


@pytest.mark.parametrize("ng", [20, 68])
def test_unaligned_field(gctx, ng):
    rng = np.random.default_rng(ng + 2)
    field = rng.normal(size=(ng, ng, ng)).astype(np.float32)
    buf = torch.empty(ng ** 3 + 1, dtype=torch.float32, device="cuda")
    view = buf[1:].view(ng, ng, ng)  # 4-byte aligned only
    view.copy_(torch.as_tensor(field))
    _check(gctx, field, cwt=view)
