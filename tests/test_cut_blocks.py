"""Blocks at the grid's edge that are cut to their tokens: lines narrower than the block's, slabs put together from boxes of
several latent frames, slabs that several blocks share (a whole number of them and a rest), zeros behind the last row (in the same
box and in one of their own), grids without any ordinary block, text keys, rows without any key.  In launches that plan
their items (many heads) and in those that do not.  Every row of the checked heads against the fp64 oracle at the tolerances of the
other parity tests; infinite values in tokens that a query does not attend must not reach it."""
import math

import numpy as np
import pytest
import torch

from oracle import psa_oracle as O
from paper_2609_37001_b200 import workloads as WL

pytestmark = pytest.mark.gpu
INF = O.INF_STRIDE
SCALE = 1.0 / math.sqrt(128.0)


def _binding():
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding
    return binding


@pytest.mark.parametrize("n_heads", [1, 40])
@pytest.mark.parametrize("grid,tile,n_text", [
    ((3, 30, 20), (1, 30, 8), 0),     # w: 4 of 8 columns, 120 rows and 8 of zeros behind the last line
    ((3, 33, 20), (1, 15, 16), 0),    # w: lines of 8 (an odd height has no 4), h: 3 lines; the corner: both
    ((4, 21, 16), (3, 8, 16), 0),     # t and h: 5 lines in three frames, two slabs of two boxes
    ((2, 18, 33), (1, 8, 16), 50),    # w: 1 of 16 columns, 8 rows, up to 16 blocks a slab; h: 2 lines
    ((5, 15, 28), (2, 8, 8), 0),      # all three axes
    ((3, 23, 22), (1, 30, 8), 30),    # no ordinary block: the pattern is 128 + 64
    ((3, 30, 9), (2, 32, 4), 0),      # the same with 128 + 112, a box of another frame in the first slab
    ((2, 19, 70), (6, 8, 8), 0),      # one row of blocks in time
    ((2, 13, 35), (1, 16, 16), 0),    # the pattern is 128 + 96
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_cut_blocks(grid, tile, n_text, n_heads):
    B = _binding()
    T, H, W = grid
    L = T * H * W
    Tp, Hp, Wp = O.block_grid(T, H, W, tile)
    kinds = [(Tp, 0, INF, Hp * Wp, 0, INF), (1, 0, INF, 1, 0, INF), (1, 1, INF, Hp * Wp, 0, INF), (Tp, 0, INF, 1, 1, INF), (2, 0, 2, 2, -1, 3)]
    params = [kinds[h % len(kinds)] for h in range(n_heads)]
    checked = range(n_heads) if n_heads < 6 else range(n_heads - 5, n_heads)
    bits = {n: WL.tensor_bits(0xC07 + L, n, n_heads, L + n_text) for n in ("q", "k", "v")}
    q, k, v = (torch.from_numpy(bits[n].view(np.int16)).cuda().view(torch.bfloat16) for n in ("q", "k", "v"))
    out = torch.full_like(q, float("nan"))
    lse = torch.full((n_heads, L + n_text), float("nan"), dtype=torch.float32, device="cuda")
    B.psa_attn_fwd_joint(q, k, v, params, grid, tile, SCALE, n_text, out=out, lse=lse)
    st, detail = B.psa_last_device_status()
    assert st == 0, (st, hex(detail))
    out_h = O.bf16_bits_to_f64(out.view(torch.int16).cpu().numpy().view(np.uint16))
    lse_h = lse.cpu().numpy().astype(np.float64)
    assert not np.isnan(out_h).any() and not np.isnan(lse_h).any()   # every row was written
    for hd in checked:
        qf, kf, vf = (O.bf16_bits_to_f64(bits[n][hd]) for n in ("q", "k", "v"))
        ro, rl = O.attention_with_text(qf, kf, vf, params[hd], T, H, W, tile, SCALE, n_text)
        empty = np.isneginf(rl)
        assert np.array_equal(np.isneginf(lse_h[hd]), empty)
        assert np.all(out_h[hd][empty] == 0)
        err = np.abs(out_h[hd] - ro)
        assert err.max() <= 2e-2 and err.mean() <= 2e-3, (hd, params[hd], err.max(), err.mean())
        assert empty.all() or np.abs(lse_h[hd][~empty] - rl[~empty]).max() <= 1e-3


@pytest.mark.parametrize("grid,tile", [((2, 30, 20), (1, 15, 16)), ((2, 16, 36), (1, 8, 16)), ((2, 60, 20), (1, 30, 8))],
                         ids=["1x15x16", "1x8x16", "1x30x8"])
def test_values_of_other_blocks_stay_out(grid, tile):
    """Each block attends itself only, and every other block's values are infinite: a row of zero probability that came from
    there would make the result NaN."""
    B = _binding()
    T, H, W = grid
    L = T * H * W
    params = [(1, 0, INF, 1, 0, INF)] * 40
    gen = torch.Generator(device="cuda").manual_seed(L)
    q, k, v = (torch.randn((40, L, 128), device="cuda", generator=gen).bfloat16() for _ in range(3))
    want, want_lse = B.psa_attn_fwd(q, k, v, params, grid, tile, SCALE)
    t, h, w = torch.meshgrid(*(torch.arange(n, device="cuda") for n in grid), indexing="ij")
    odd = (((t // tile[0]) + (h // tile[1]) + (w // tile[2])) % 2 == 1).reshape(-1)
    for other in (odd, ~odd):
        bad = v.clone()
        bad[:, other] = float("inf")
        out, lse = B.psa_attn_fwd(q, k, bad, params, grid, tile, SCALE)
        assert B.psa_last_device_status()[0] == 0
        assert torch.equal(out[:, ~other].view(torch.int16), want[:, ~other].view(torch.int16))
        assert torch.equal(lse.view(torch.int32), want_lse.view(torch.int32))
