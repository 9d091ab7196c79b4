"""Blocks of one slab, enough of them that the launch plans its items: the kernel that starts an item while the one before is
still being written out.  Items of no key, of one, two and three key slabs and of all of them follow one another, with text
queries (pairs of slabs, and an odd one) between them, padding rows, and both memory layouts of the tensors.  Every row of
the checked heads against the fp64 oracle at the tolerances of the other parity tests."""
import math

import numpy as np
import pytest
import torch

from oracle import psa_oracle as O
from paper_2609_37001_b200 import workloads as WL

pytestmark = pytest.mark.gpu
INF = O.INF_STRIDE
SCALE = 1.0 / math.sqrt(128.0)


@pytest.mark.parametrize("grid,tile,n_text,n_heads", [
    ((4, 16, 32), (1, 8, 16), 0, 24),     # 16 blocks
    ((3, 15, 33), (1, 8, 16), 0, 30),     # 18 blocks, padded along h and w
    ((3, 16, 32), (1, 8, 16), 300, 100),  # 12 blocks, text: two full slabs and 44 tokens
    ((5, 7, 18), (2, 8, 8), 128, 150),    # 9 blocks, padded along t, h and w; one text slab
    ((2, 3, 300), (1, 1, 128), 0, 20),    # along w
    ((7, 16, 32), (1, 8, 16), 0, 15),     # 28 blocks
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
@pytest.mark.parametrize("token_layout", [False, True])
def test_short_items(grid, tile, n_text, n_heads, token_layout):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    T, H, W = grid
    L = T * H * W
    Tp, Hp, Wp = O.block_grid(T, H, W, tile)
    kinds = [(Tp, 0, INF, Hp * Wp, 0, INF), (1, 0, INF, 1, 0, INF), (1, 1, INF, 2, 0, INF), (1, 0, INF, 3, -1, INF), (2, 0, 2, 2, -1, 3)]
    params = [kinds[h % len(kinds)] for h in range(n_heads)]
    checked = range(n_heads - 5, n_heads)
    bits = {n: WL.tensor_bits(0x5407 + L, n, n_heads, L + n_text) for n in ("q", "k", "v")}

    def place(t):   # (heads, tokens, 128), contiguous or a view of (tokens, heads, 128)
        return t.transpose(0, 1).contiguous().transpose(0, 1) if token_layout else t

    q, k, v = (place(torch.from_numpy(bits[n].view(np.int16)).cuda().view(torch.bfloat16)) for n in ("q", "k", "v"))
    out = place(torch.full_like(q, float("nan")))
    lse = torch.full((n_heads, L + n_text), float("nan"), dtype=torch.float32, device="cuda")
    B.psa_attn_fwd_joint(q, k, v, params, grid, tile, SCALE, n_text, out=out, lse=lse)
    assert B.psa_last_attn_launch()[1] == "ticket_short"
    st, detail = B.psa_last_device_status()
    assert st == 0, (st, hex(detail))
    out_h = O.bf16_bits_to_f64(out.contiguous().view(torch.int16).cpu().numpy().view(np.uint16))
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
