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


def _call(B, grid, tile, n_heads):
    n = [-(-x // b) for x, b in zip(grid, tile)]
    q, k, v = (torch.zeros((n_heads, math.prod(grid), 128), dtype=torch.bfloat16, device="cuda") for _ in range(3))
    return B.psa_attn_fwd(q, k, v, [(n[0], 0, 0, n[1] * n[2], 0, 0)] * n_heads, grid, tile, 0.1)


@pytest.mark.parametrize("grid,tile,n_heads,kind", [
    ((3, 14, 32), (1, 14, 16), 2, "whole"),
    ((3, 16, 20), (1, 14, 16), 1, "padded"),    # 12 items: 20 us padded, 29 cut
    ((3, 16, 20), (1, 14, 16), 60, "cut"),      # the same grid, 720 items
    ((4, 18, 20), (2, 8, 8), 60, "padded"),     # one slab a block
    ((3, 20, 1100), (1, 1, 256), 9, "padded"),  # slabs along w
    ((10, 46, 41), (3, 32, 4), 1, "cut"),       # one head of 88 blocks
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_grids_are_cut_where_it_pays(grid, tile, n_heads, kind):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    _call(B, grid, tile, n_heads)
    assert B.psa_last_attn_grid()[0] == kind
    assert B.psa_last_device_status() == (0, 0)


def test_chunks_of_a_host_call_are_cut_as_the_whole_call():
    """60 heads are cut and one is not: the host-tensor call, which computes a few heads at a time, gives the device call's bits."""
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    grid, tile, nh = (3, 16, 20), (1, 14, 16), 60
    L = math.prod(grid)
    params = [(2 + h % 2, 0, 0, 3 + h % 2, 0, 0) for h in range(nh)]
    gen = torch.Generator(device="cuda").manual_seed(L)
    dev = [torch.randn((nh, L, 128), device="cuda", generator=gen).bfloat16() for _ in range(3)]
    want, want_lse = B.psa_attn_fwd(*dev, params, grid, tile, 0.1)
    assert B.psa_last_attn_grid()[0] == "cut"
    B.psa_attn_fwd(*(x[:1] for x in dev), params[:1], grid, tile, 0.1)
    assert B.psa_last_attn_grid()[0] == "padded"
    host = [x.cpu().pin_memory() for x in dev]
    out, lse = torch.empty_like(host[0]).pin_memory(), torch.empty((nh, L)).pin_memory()
    staging = (*(torch.empty_like(x) for x in dev), torch.empty_like(dev[0]), torch.empty((nh, L), device="cuda"))
    B.psa_attn_fwd_host(*host, out, lse, staging, params, grid, tile, 0.1)
    assert B.psa_last_attn_grid()[0] == "cut" and B.psa_last_device_status() == (0, 0)
    assert torch.equal(out.view(torch.int16), want.cpu().view(torch.int16)) and torch.equal(lse.view(torch.int32), want_lse.cpu().view(torch.int32))


@pytest.mark.parametrize("grid,tile,n_heads,axes,classes", [
    ((3, 16, 20), (1, 14, 16), 60, 6, {0: (2, 224, 1), 2: (1, 128, 4), 4: (1, 128, 2), 6: (1, 128, 16)}),   # cut: 224, 32, 56 and 8 rows
    ((4, 20, 32), (1, 16, 16), 20, 2, {0: (2, 256, 1), 2: (1, 128, 1)}),                                    # padded: the second slab is empty
    ((4, 18, 20), (2, 8, 8), 60, 0, {0: (1, 128, 1)}),
], ids=["cut", "empty_slab", "padded"])
def test_classes_of_blocks(grid, tile, n_heads, axes, classes):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    if axes == 2:
        n = [-(-x // b) for x, b in zip(grid, tile)]
        q, k, v = (torch.zeros((n_heads, math.prod(grid), 128), dtype=torch.bfloat16, device="cuda") for _ in range(3))
        B.psa_attn_fwd(q, k, v, [(1, 0, 0, 1, 0, 0)] * n_heads, grid, tile, 0.1)
    else:
        _call(B, grid, tile, n_heads)
    assert B.psa_last_attn_classes() == (axes, [classes.get(c, (0, 0, 1)) for c in range(8)])
