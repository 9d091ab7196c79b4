"""The largest spatial block grids (2,048 blocks, in one column or in one row) and padding on each axis: the load warp
turns block ids into coordinates without divisions and tabulates the key positions of a slab.  Sampled rows, the first
and the last rows included, against the fp64 oracle at the tolerances of the other parity tests."""
import math

import numpy as np
import pytest
import torch

from oracle import psa_oracle as O
from paper_2609_37001_b200 import workloads as WL

pytestmark = pytest.mark.gpu
INF = O.INF_STRIDE
SCALE = 1.0 / math.sqrt(128.0)


@pytest.mark.parametrize("grid,tile,params", [
    ((1, 2048, 100), (1, 1, 128), (1, 0, INF, 2, 1, 700)),     # W' = 1, padded along w
    ((1, 7, 32760), (1, 8, 16), (1, 0, INF, 3, -1, 500)),      # H' = 1, padded along h and w
    ((5, 26, 70), (4, 8, 8), (2, 0, INF, 9, 0, 4)),            # two slabs stacked along t, padded on all axes
    ((7, 13, 30), (6, 8, 8), (2, 0, INF, 3, 0, INF)),          # three slabs stacked along t
    ((3, 46, 33), (1, 15, 16), (3, 0, INF, 4, 0, 2)),          # short last slab, padded along h and w
    ((2, 5, 300), (1, 3, 64), (2, 0, INF, 4, 0, INF)),         # 128 + 64 keys
], ids=lambda v: "x".join(map(str, v)) if len(v) == 3 else None)
def test_block_coordinates_and_padding(grid, tile, params):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    T, H, W = grid
    L = T * H * W
    bits = {n: WL.tensor_bits(0x61D + L, n, 1, L, threads=1) for n in ("q", "k", "v")}
    q, k, v = (torch.from_numpy(bits[n].view(np.int16)).cuda().view(torch.bfloat16) for n in ("q", "k", "v"))
    out, lse = B.psa_attn_fwd(q, k, v, [params], grid, tile, SCALE)
    st, detail = B.psa_last_device_status()
    assert st == 0, (st, hex(detail))
    rows = sorted(set(WL.sample_rows(L, 0, L, 40)) | {0, 1, W - 1, L - W, L - 1})
    qf, kf, vf = (O.bf16_bits_to_f64(bits[n][0]) for n in ("q", "k", "v"))
    ro, rl = O.attention_rows(qf, kf, vf, rows, params, T, H, W, tile, SCALE)
    got = O.bf16_bits_to_f64(out.view(torch.int16).cpu().numpy().view(np.uint16))[0][rows]
    got_l = lse.cpu().numpy().astype(np.float64)[0][rows]
    empty = np.isneginf(rl)
    assert np.array_equal(np.isneginf(got_l), empty)
    err = np.abs(got - ro)
    assert err.max() <= 2e-2 and err.mean() <= 2e-3, (err.max(), err.mean())
    assert np.abs(got_l[~empty] - rl[~empty]).max() <= 1e-3
