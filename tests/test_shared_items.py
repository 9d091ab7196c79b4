"""Work items shared by a cluster of CTAs (problems of few items: 2, 4 or 8 CTAs each take a share of the attended key
blocks and merge through distributed shared memory), every row against the fp64 oracle at the tolerances of the other
parity tests.  The sizes cover few items (2), every cluster size, items that all run at once and items that are planned, one-,
two- and three-slab blocks, short last slabs, ragged grids, slabs without a token, shares without a key block, rows without
any key, and text keys, which go with the last share.  That the items were shared, and among how many, is checked."""
import math

import numpy as np
import pytest
import torch

from oracle import psa_oracle as O
from paper_2609_37001_b200 import workloads as WL

pytestmark = pytest.mark.gpu
INF = O.INF_STRIDE
SCALE = 1.0 / math.sqrt(128.0)


@pytest.mark.parametrize("grid,tile,params,n_text,ctas", [
    ((2, 16, 16), (1, 16, 16), [(2, 0, INF, 1, 0, INF)], 0, (2,)),                               # 2 items
    ((10, 16, 16), (1, 16, 16), [(10, 0, INF, 1, 0, INF)], 0, (8,)),                             # 10 items, dense
    ((16, 16, 16), (2, 8, 16), [(8, 0, INF, 2, 0, INF)], 0, (4,)),                               # 16 items, dense
    ((8, 16, 16), (2, 8, 8), [(1, 0, 3, 2, 0, 3), (4, 0, INF, 4, 0, INF)], 0, (2, 4)),           # single-slab items
    ((5, 29, 47), (1, 15, 16), [(5, 0, INF, 6, 0, INF), (2, 0, 3, 2, 1, INF)], 0, (2,)),         # 128 + 112 tokens, ragged
    ((7, 24, 30), (1, 12, 16), [(3, 0, INF, 2, 0, INF)], 0, (2, 4)),                             # 128 + 64 tokens, ragged
    ((6, 15, 40), (3, 8, 16), [(2, 0, INF, 6, 0, INF)], 0, (4,)),                                # three slabs, ragged
    ((8, 16, 32), (1, 16, 16), [(5, 5, INF, 2, 0, INF), (8, 2, INF, 2, 0, INF)], 0, (2, 4)),     # rows of 0 to all keys
    ((4, 16, 32), (1, 16, 16), [(1, 5, INF, 1, 0, INF), (4, 0, INF, 2, 0, INF)], 77, (4,)),      # only text keys / all
    ((6, 16, 32), (1, 8, 16), [(6, 0, INF, 4, 0, INF)], 300, (4,)),                              # a single text slab left over
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) and len(v) == 3 else None)
def test_shared_items(grid, tile, params, n_text, ctas):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    T, H, W = grid
    L, nh = T * H * W, len(params)
    bits = {n: WL.tensor_bits(0x51A + L, n, nh, L + n_text, threads=1) for n in ("q", "k", "v")}
    q, k, v = (torch.from_numpy(bits[n].view(np.int16)).cuda().view(torch.bfloat16) for n in ("q", "k", "v"))
    out = torch.full_like(q, float("nan"))
    lse = torch.full((nh, L + n_text), float("nan"), dtype=torch.float32, device="cuda")
    B.psa_attn_fwd_joint(q, k, v, params, grid, tile, SCALE, n_text, out=out, lse=lse)
    # (how many clusters of 4 run at a time differs from GPU to GPU: the sizes that come with 28 to 32 items may, too)
    items, mode, got = B.psa_last_attn_launch()
    assert mode == "shared_direct" and got in ctas, (items, mode, got)
    st, detail = B.psa_last_device_status()
    assert st == 0, (st, hex(detail))
    out_h = O.bf16_bits_to_f64(out.view(torch.int16).cpu().numpy().view(np.uint16))
    lse_h = lse.cpu().numpy().astype(np.float64)
    for hd in range(nh):
        qf, kf, vf = (O.bf16_bits_to_f64(bits[n][hd]) for n in ("q", "k", "v"))
        ro, rl = O.attention_with_text(qf, kf, vf, params[hd], T, H, W, tile, SCALE, n_text)
        empty = np.isneginf(rl)
        assert np.array_equal(np.isneginf(lse_h[hd]), empty)
        assert np.all(out_h[hd][empty] == 0)
        err = np.abs(out_h[hd] - ro)
        assert err.max() <= 2e-2 and err.mean() <= 2e-3, (hd, err.max(), err.mean())
        assert np.abs(lse_h[hd][~empty] - rl[~empty]).max() <= 1e-3


@pytest.mark.parametrize("grid,tile,params,n_text,ctas", [
    ((15, 16, 80), (1, 16, 16), [(5, 0, INF, 5, 0, INF)] * 2, 0, (2, 4)),                         # 150 items, half the keys
    ((15, 24, 48), (1, 16, 16), [(15, 0, INF, 6, 0, INF)] * 2, 0, (2, 4)),                        # 180, every second an edge block
    ((45, 15, 30), (1, 8, 16), [(45, 0, INF, 4, 0, INF)], 0, (2, 4)),                             # 180 of one slab, dense
    ((15, 24, 80), (1, 16, 16), [(15, 0, INF, 10, 0, INF)], 0, (4, 8)),                           # 150, edge blocks, dense
    ((28, 29, 12), (1, 8, 16), [(1, 0, INF, 1, 0, INF)], 219, (2, 4, 8)),                         # 113, a long one of text queries
    ((20, 24, 30), (1, 16, 16), [(1, 0, INF, 1, 0, INF)], 219, (4, 8)),                           # 81, edge blocks, text
], ids=["half", "edge", "one_slab", "edge_dense", "text", "edge_text"])
def test_shared_items_in_several_rounds(grid, tile, params, n_text, ctas):
    """More shared items than clusters that run at a time, which are planned, heaviest first.  Every row was written; sampled
    rows, the first and the last video row and all text rows against the oracle."""
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    T, H, W = grid
    L, nh = T * H * W, len(params)
    bits = {n: WL.tensor_bits(0x51B, n, nh, L + n_text) for n in ("q", "k", "v")}
    q, k, v = (torch.from_numpy(bits[n].view(np.int16)).cuda().view(torch.bfloat16) for n in ("q", "k", "v"))
    out = torch.full_like(q, float("nan"))
    lse = torch.full((nh, L + n_text), float("nan"), dtype=torch.float32, device="cuda")
    B.psa_attn_fwd_joint(q, k, v, params, grid, tile, SCALE, n_text, out=out, lse=lse)
    items, mode, got = B.psa_last_attn_launch()
    assert mode == "shared" and got in ctas, (items, mode, got)
    assert B.psa_last_device_status()[0] == 0
    out_h = O.bf16_bits_to_f64(out.view(torch.int16).cpu().numpy().view(np.uint16))
    lse_h = lse.cpu().numpy().astype(np.float64)
    assert not np.isnan(out_h).any() and not np.isnan(lse_h).any()
    for hd in range(nh):
        rows = sorted(set(WL.sample_rows(7, hd, L, 64)) | set(range(L, L + n_text)) | {0, L - 1})
        qf, kf, vf = (O.bf16_bits_to_f64(bits[n][hd]) for n in ("q", "k", "v"))
        ro, rl = O.attention_rows_with_text(qf, kf, vf, rows, params[hd], T, H, W, tile, SCALE, n_text)
        err = np.abs(out_h[hd][rows] - ro)
        assert err.max() <= 2e-2 and err.mean() <= 2e-3, (hd, err.max(), err.mean())
        assert np.abs(lse_h[hd][rows] - rl).max() <= 1e-3


@pytest.mark.parametrize("tile", [(1, 16, 16), (1, 8, 16)], ids=["two_slabs", "one_slab"])
def test_rows_whose_sums_are_no_numbers(tile):
    """NaN and infinite inputs leave the same rows 0 with lse = -inf, and the same elements infinite or NaN, whether items
    are shared (2 heads) or whole (the same 2 heads repeated until there are many items)."""
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    grid, params = (8, 16, 16), [(8, 0, INF, 2, 0, INF), (2, 0, INF, 2, 0, INF)]
    L, many = 8 * 16 * 16, 40
    gen = torch.Generator(device="cuda").manual_seed(5)
    q, k, v = (torch.randn((2, L, 128), device="cuda", generator=gen).bfloat16() for _ in range(3))
    k[0, 700, 5] = float("inf")    # scores of +inf and -inf, by the sign of the query's channel
    k[1, 300, 9] = float("nan")    # every score of that key; only rows near it attend it
    q[1, 1500, 3] = float("nan")   # every score of that query
    v[1, 1900, 77] = float("inf")
    v[1, 1910, 78] = float("nan")
    o2, l2 = B.psa_attn_fwd(q, k, v, params, grid, tile, SCALE)
    assert B.psa_last_attn_launch()[1] == "shared_direct"
    o80, l80 = B.psa_attn_fwd(*(x.repeat(many, 1, 1) for x in (q, k, v)), params * many, grid, tile, SCALE)
    assert B.psa_last_attn_launch()[2] == 1
    assert B.psa_last_device_status()[0] == 0
    for o, l in ((o80[:2], l80[:2]), (o80[-2:], l80[-2:])):
        assert torch.equal(torch.isneginf(l2), torch.isneginf(l))
        empty = torch.isneginf(l2)
        assert 0.3 < empty[0].float().mean() < 0.7 and empty[1, 1500] and empty[1, 300] and not empty[1, -1]
        assert (o2[empty] == 0).all() and (o[empty] == 0).all()
        assert torch.equal(o2.isnan(), o.isnan()) and torch.equal(o2.isinf(), o.isinf()) and o2.isinf().any() and o2.isnan().any()
        ok = ~empty
        a, b = (x.float().nan_to_num(0.0, 0.0, 0.0)[ok] for x in (o2, o))
        assert (a - b).abs().max() <= 4e-2 and (l2[ok] - l[ok]).abs().max() <= 2e-3   # twice the bounds against the oracle
