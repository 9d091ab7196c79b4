"""A split-KV item (one query slab, the key slabs dealt to both tiles) followed in the same CTA by a two-slab item without
any key: the second softmax warpgroup has nothing to wait for between the two.  It used to take the accumulator barrier's
phase before last for the empty item's own, release the query buffer early and leave the CTA waiting until its time limit.
Blocks of three slabs give both kinds of item; many heads give every CTA several."""
import math

import numpy as np
import pytest
import torch

from oracle import psa_oracle as O
from paper_2609_37001_b200 import workloads as WL

pytestmark = pytest.mark.gpu
INF = O.INF_STRIDE
SCALE = 1.0 / math.sqrt(128.0)


@pytest.mark.parametrize("n_heads", [40, 100])
def test_split_item_then_item_without_keys(n_heads):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    grid, tile = (6, 16, 32), (3, 8, 16)
    T, H, W = grid
    L = T * H * W
    # rows with all keys, with one block, and without any key
    kinds = [(2, 0, INF, 4, 0, INF), (1, 1, INF, 4, 0, INF), (1, 5, INF, 1, 0, INF), (1, 0, INF, 1, 0, INF), (2, 0, INF, 1, 2, INF)]
    params = [kinds[h % len(kinds)] for h in range(n_heads)]
    bits = {n: WL.tensor_bits(0x5E4, n, n_heads, L) for n in ("q", "k", "v")}
    q, k, v = (torch.from_numpy(bits[n].view(np.int16)).cuda().view(torch.bfloat16) for n in ("q", "k", "v"))
    for _ in range(5):
        out, lse = B.psa_attn_fwd(q, k, v, params, grid, tile, SCALE)
        st, detail = B.psa_last_device_status()
        assert st == 0, (st, hex(detail))
    out_h = O.bf16_bits_to_f64(out.view(torch.int16).cpu().numpy().view(np.uint16))
    lse_h = lse.cpu().numpy().astype(np.float64)
    for hd in range(len(kinds)):
        qf, kf, vf = (O.bf16_bits_to_f64(bits[n][hd]) for n in ("q", "k", "v"))
        ro, rl = O.attention(qf, kf, vf, params[hd], T, H, W, tile, SCALE)
        empty = np.isneginf(rl)
        assert np.array_equal(np.isneginf(lse_h[hd]), empty)
        err = np.abs(out_h[hd] - ro)
        assert err.max() <= 2e-2 and err.mean() <= 2e-3, (hd, err.max(), err.mean())
