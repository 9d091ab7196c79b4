"""What psa_last_attn_launch reports of planned launches on ragged grids: `ticket_edge` only where 3D-padding leaves some block a
slab without any token, `ticket` where it clips blocks and no slab is empty, also where such a block needs fewer slabs once it is cut
to its tokens and where the grid has no ordinary block at all."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,tile,n_heads,mode", [
    ((3, 23, 22), (1, 30, 8), 60, "ticket"),        # one clipped block row of 23 lines: 16 + 7
    ((3, 13, 22), (1, 30, 8), 120, "ticket_edge"),  # 13 lines: the second slab is empty
    ((6, 30, 24), (1, 15, 16), 20, "ticket"),       # a column of 120 tokens, in both slabs of a block as in one
    ((4, 48, 20), (1, 16, 16), 20, "ticket"),       # a column of 4 of 16
    ((4, 40, 32), (1, 16, 16), 20, "ticket_edge"),  # the last row has one slab
    ((90, 5, 33), (1, 8, 16), 3, "ticket"),         # one slab a block, one clipped block row
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_empty_slabs_are_reported(grid, tile, n_heads, mode):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    n = [-(-x // b) for x, b in zip(grid, tile)]
    params = [(n[0], 0, 0, n[1] * n[2], 0, 0)] * n_heads
    q, k, v = (torch.zeros((n_heads, math.prod(grid), 128), dtype=torch.bfloat16, device="cuda") for _ in range(3))
    B.psa_attn_fwd(q, k, v, params, grid, tile, 0.1)
    assert B.psa_last_attn_launch()[1] == mode
    assert B.psa_last_device_status() == (0, 0)
