"""Work items shared by a cluster of CTAs (problems of few items: 2, 4 or 8 CTAs each take a share of the attended key
blocks and merge through distributed shared memory), every row against the fp64 oracle at the tolerances of the other
parity tests.  The sizes cover the smallest (one item), every cluster size, one-, two- and three-slab blocks, short last
slabs, ragged grids, shares without a key block, rows without any key, and text keys, which go with the last share."""
import math

import numpy as np
import pytest
import torch

from oracle import psa_oracle as O
from paper_2609_37001_b200 import workloads as WL

pytestmark = pytest.mark.gpu
INF = O.INF_STRIDE
SCALE = 1.0 / math.sqrt(128.0)


@pytest.mark.parametrize("grid,tile,params,n_text", [
    ((2, 16, 16), (1, 16, 16), [(2, 0, INF, 1, 0, INF)], 0),                                     # 2 items
    ((16, 16, 16), (2, 8, 16), [(8, 0, INF, 2, 0, INF)], 0),                                     # 16 items, dense
    ((8, 16, 16), (2, 8, 8), [(1, 0, 3, 2, 0, 3), (4, 0, INF, 4, 0, INF)], 0),                   # single-slab items
    ((5, 29, 47), (1, 15, 16), [(5, 0, INF, 6, 0, INF), (2, 0, 3, 2, 1, INF)], 0),               # 128 + 112 tokens, ragged
    ((7, 24, 30), (1, 12, 16), [(3, 0, INF, 2, 0, INF)], 0),                                     # 128 + 64 tokens, ragged
    ((6, 15, 40), (3, 8, 16), [(2, 0, INF, 6, 0, INF)], 0),                                      # three slabs, ragged
    ((8, 16, 32), (1, 16, 16), [(5, 5, INF, 2, 0, INF), (8, 2, INF, 2, 0, INF)], 0),             # rows of 0 to all keys
    ((4, 16, 32), (1, 16, 16), [(1, 5, INF, 1, 0, INF), (4, 0, INF, 2, 0, INF)], 77),            # only text keys / all
    ((6, 16, 32), (1, 8, 16), [(6, 0, INF, 4, 0, INF)], 300),                                    # a single text slab left over
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else None)
def test_shared_items(grid, tile, params, n_text):
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


def test_shared_items_in_several_rounds():
    """More shared items than clusters that run at a time (they are planned, heaviest first): long text-query items make
    sharing pay.  Sampled video rows, and the text rows of the ragged last slab."""
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    grid, tile, n_text = (28, 29, 12), (1, 8, 16), 347
    T, H, W = grid
    L = T * H * W
    params = [(28, 0, INF, 3, 0, INF), (28, 0, INF, 2, 0, INF)]
    bits = {n: WL.tensor_bits(0x51B, n, 2, L + n_text) for n in ("q", "k", "v")}
    q, k, v = (torch.from_numpy(bits[n].view(np.int16)).cuda().view(torch.bfloat16) for n in ("q", "k", "v"))
    out = torch.full_like(q, float("nan"))
    lse = torch.full((2, L + n_text), float("nan"), dtype=torch.float32, device="cuda")
    B.psa_attn_fwd_joint(q, k, v, params, grid, tile, SCALE, n_text, out=out, lse=lse)
    assert B.psa_last_device_status()[0] == 0
    out_h = O.bf16_bits_to_f64(out.view(torch.int16).cpu().numpy().view(np.uint16))
    lse_h = lse.cpu().numpy().astype(np.float64)
    assert not np.isnan(out_h).any() and not np.isnan(lse_h).any()
    for hd in range(2):
        rows = sorted(set(WL.sample_rows(7, hd, L, 64)) | set(range(L + 250, L + n_text)) | {0, L - 1})
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
    o80, l80 = B.psa_attn_fwd(*(x.repeat(many, 1, 1) for x in (q, k, v)), params * many, grid, tile, SCALE)
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
