"""Masks of block grids with more than 32 spatial or 64 temporal coordinates: window, word and 32-byte piece edges, grids of one
axis only, empty rows and rows that attend everything, odd numbers of blocks, and more heads than one launch carries.
Mask, row offsets and column lists bit for bit against the oracle, and nothing written beyond them."""
import numpy as np
import pytest
import torch

from oracle import psa_oracle as O

pytestmark = pytest.mark.gpu
INF = O.INF_STRIDE
KINDS = [(2, 0, INF, 5, 1, INF), (1, -2, 3, 33, 0, INF), (1, 1, 2, 3, -1, 5), (1, 0, 1, 1, 0, 1), (1, 7, INF, 1, 40, INF), (70, 0, INF, 1, 0, 31)]


@pytest.mark.parametrize("grid", [(1, 1, 33), (1, 33, 1), (65, 1, 1), (66, 1, 2), (65, 3, 5), (129, 1, 1), (3, 6, 6), (2, 8, 8), (4, 5, 13), (2, 11, 29), (7, 32, 2)],
                         ids=lambda g: "x".join(map(str, g)))
@pytest.mark.parametrize("n_heads", [1, 6, 131])
def test_wide_mask_grids(grid, n_heads):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    params = [KINDS[h % len(KINDS)] for h in range(n_heads)]
    om, orp, oc = O.block_index_lists(params, *grid, (1, 1, 1))
    guard = 64
    bufs = [torch.full((a.size + guard,), 77, dtype=t, device="cuda") for a, t in ((om, torch.uint8), (orp, torch.int32), (oc, torch.int32))]
    out = (bufs[0][:om.size].view(om.shape), bufs[1][:orp.size], bufs[2][:oc.size])
    B.psa_mask_build(params, grid, (1, 1, 1), out=out)
    torch.cuda.synchronize()
    for got, buf, want in zip(out, bufs, (om, orp, oc)):
        assert np.array_equal(got.cpu().numpy().ravel(), want.ravel())
        assert (buf[want.size:] == 77).all()
