"""Slabs that 3D-padding leaves without a token are neither loaded nor computed: blocks at the grid's edge with one or two
of their two or three slabs, stacked along t, h and w, as keys and as queries, with text keys, with rows that attend
edge blocks only and rows without any key, in the kernel that plans its items (many heads) and in those that do not.
Every row of the checked heads against the fp64 oracle at the tolerances of the other parity tests."""
import math

import numpy as np
import pytest
import torch

from oracle import psa_oracle as O
from paper_2609_37001_b200 import workloads as WL

pytestmark = pytest.mark.gpu
INF = O.INF_STRIDE
SCALE = 1.0 / math.sqrt(128.0)


@pytest.mark.parametrize("n_heads", [1, 60])
@pytest.mark.parametrize("grid,tile,n_text", [
    ((3, 32, 8), (2, 32, 4), 0),      # t: 1 of 2 slabs
    ((4, 16, 16), (3, 8, 16), 0),     # t: 1 of 3
    ((5, 8, 20), (3, 8, 16), 40),     # t: 2 of 3, padded along w, text
    ((2, 23, 32), (1, 16, 16), 0),    # h: 1 of 2
    ((3, 16, 8), (1, 30, 8), 0),      # h: a single block row with 1 of its 2 slabs (128 + 112)
    ((2, 20, 17), (1, 15, 16), 130),  # h: 1 of 2, padded along w, text
    ((2, 31, 16), (1, 23, 16), 0),    # h: 1 of 3 (128 + 128 + 112)
    ((2, 3, 300), (1, 1, 256), 0),    # w: 1 of 2
    ((3, 2, 700), (1, 1, 384), 20),   # w: 3 of 3 (316 tokens)
    ((3, 2, 590), (1, 1, 384), 0),    # w: 2 of 3
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_empty_slabs(grid, tile, n_text, n_heads):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    T, H, W = grid
    L = T * H * W
    Tp, Hp, Wp = O.block_grid(T, H, W, tile)
    kinds = [(Tp, 0, INF, Hp * Wp, 0, INF), (1, 0, INF, 1, 0, INF), (1, 1, INF, Hp * Wp, 0, INF), (Tp, 0, INF, 1, 1, INF), (2, 0, 2, 2, -1, 3)]
    params = [kinds[h % len(kinds)] for h in range(n_heads)]
    checked = range(n_heads) if n_heads < 6 else range(n_heads - 5, n_heads)
    bits = {n: WL.tensor_bits(0xE59 + L, n, n_heads, L + n_text) for n in ("q", "k", "v")}
    q, k, v = (torch.from_numpy(bits[n].view(np.int16)).cuda().view(torch.bfloat16) for n in ("q", "k", "v"))
    out = torch.full_like(q, float("nan"))
    lse = torch.full((n_heads, L + n_text), float("nan"), dtype=torch.float32, device="cuda")
    B.psa_attn_fwd_joint(q, k, v, params, grid, tile, SCALE, n_text, out=out, lse=lse)
    mode = B.psa_last_attn_launch()[1]
    assert mode in (("direct", "shared_direct") if n_heads == 1 else ("ticket" if grid[2] == 700 else "ticket_edge", "shared")), mode
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
