"""Blocks at the grid's edge that are cut to their tokens: lines narrower than the block's, slabs put together from boxes of
several latent frames, slabs that several blocks share (a whole number of them and a rest), zeros behind the last row (in the same
box and in one of their own), grids without any ordinary block, patterns of every width, text keys, rows without any key; in launches
of every kind.  That a grid was cut, its pattern of key slabs and the kind of launch are checked.  Against the fp64 oracle at the
tolerances of the other parity tests; infinite values in tokens that a query does not attend must not reach it."""
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


def _kinds(n):
    """Masks that attend everything, the block itself, the next frame, the next block, every second frame (rows without any key)."""
    return [(n[0], 0, INF, n[1] * n[2], 0, INF), (1, 0, INF, 1, 0, INF), (1, 1, INF, n[1] * n[2], 0, INF), (n[0], 0, INF, 1, 1, INF), (2, 0, 2, 2, -1, 3)]


@pytest.mark.parametrize("mode,pattern,grid,tile,n_heads,n_text", [   # blocks to a slab of those that are cut most
    ("direct", (2, 112), (12, 17, 49), (1, 15, 16), 1, 0),            # 4 and 16
    ("direct", (1, 128), (23, 20, 2), (3, 8, 16), 3, 200),            # 2, 4, 5 and 8
    ("direct", (3, 96), (34, 7, 48), (3, 8, 16), 2, 0),               # slabs of two boxes
    ("direct", (2, 128), (7, 78, 9), (2, 32, 4), 3, 200),             # all eight classes
    ("shared_direct", (2, 96), (2, 43, 17), (1, 14, 16), 1, 0),       # 2, 8 and 16
    ("shared_direct", (2, 112), (59, 5, 17), (3, 8, 16), 1, 0),       # 5 and 8
    ("shared_direct", (2, 64), (10, 18, 6), (3, 8, 16), 3, 50),       # 2
    ("shared_direct", (3, 64), (5, 10, 24), (6, 8, 8), 1, 0),
    ("shared", (2, 96), (8, 30, 35), (1, 14, 16), 3, 0),              # 2, 4 and 16
    ("shared", (2, 64), (20, 12, 35), (1, 15, 16), 3, 50),            # 2
    ("shared", (3, 96), (24, 7, 64), (3, 8, 16), 3, 0),
    ("shared", (2, 128), (39, 25, 13), (2, 8, 16), 2, 200),           # 4 and 8
    ("ticket", (2, 64), (4, 12, 18), (1, 12, 16), 40, 0),             # 5
    ("ticket", (2, 112), (2, 48, 9), (1, 30, 8), 40, 200),            # 2 and 5
    ("ticket", (1, 96), (24, 3, 33), (2, 8, 16), 40, 0),              # 8
    ("ticket", (3, 64), (60, 23, 8), (3, 32, 4), 3, 50),
    ("ticket_edge", (2, 128), (2, 40, 8), (3, 32, 4), 40, 0),         # 2
    ("ticket_edge", (1, 96), (45, 8, 2), (6, 8, 8), 40, 200),         # 2
    ("ticket_edge", (3, 128), (8, 32, 9), (6, 8, 8), 40, 0),          # 2 and 8
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_modes_and_patterns(mode, pattern, grid, tile, n_heads, n_text):
    """Sampled rows, those of the last frame's, row's and column's blocks among them, and all text rows."""
    B = _binding()
    T, H, W = grid
    L = T * H * W
    kinds = _kinds(O.block_grid(T, H, W, tile))
    params = [kinds[h % 5 if n_heads > 5 else 0] for h in range(n_heads)]
    checked = range(n_heads) if n_heads < 6 else range(n_heads - 5, n_heads)
    bits = {n: WL.tensor_bits(0xC08 + L, n, n_heads, L + n_text) for n in ("q", "k", "v")}
    q, k, v = (torch.from_numpy(bits[n].view(np.int16)).cuda().view(torch.bfloat16) for n in ("q", "k", "v"))
    out = torch.full_like(q, float("nan"))
    lse = torch.full((n_heads, L + n_text), float("nan"), dtype=torch.float32, device="cuda")
    B.psa_attn_fwd_joint(q, k, v, params, grid, tile, SCALE, n_text, out=out, lse=lse)
    assert B.psa_last_attn_launch()[1] == mode and B.psa_last_attn_grid() == ("cut", *pattern)
    st, detail = B.psa_last_device_status()
    assert st == 0, (st, hex(detail))
    out_h = O.bf16_bits_to_f64(out.view(torch.int16).cpu().numpy().view(np.uint16))
    lse_h = lse.cpu().numpy().astype(np.float64)
    assert not np.isnan(out_h).any() and not np.isnan(lse_h).any()   # every row was written
    rng = np.random.default_rng(L)
    at = np.arange(L).reshape(grid)
    ends = [rng.choice(x.reshape(-1), 24) for x in (at[-(T % tile[0] or tile[0]):], at[:, -(H % tile[1] or tile[1]):], at[:, :, -(W % tile[2] or tile[2]):])]
    for hd in checked:
        rows = sorted(set(WL.sample_rows(7, hd, L, 48)) | set(range(L, L + n_text)) | {0, L - 1} | {int(r) for x in ends for r in x})
        qf, kf, vf = (O.bf16_bits_to_f64(bits[n][hd]) for n in ("q", "k", "v"))
        ro, rl = O.attention_rows_with_text(qf, kf, vf, rows, params[hd], T, H, W, tile, SCALE, n_text)
        empty = np.isneginf(rl)
        assert np.array_equal(np.isneginf(lse_h[hd][rows]), empty)
        assert np.all(out_h[hd][rows][empty] == 0)
        err = np.abs(out_h[hd][rows] - ro)
        assert err.max() <= 2e-2 and err.mean() <= 2e-3, (hd, params[hd], err.max(), err.mean())
        assert empty.all() or np.abs(lse_h[hd][rows][~empty] - rl[~empty]).max() <= 1e-3


@pytest.mark.parametrize("n_heads", [1, 40])
@pytest.mark.parametrize("grid,tile,n_text", [
    ((3, 30, 20), (1, 30, 8), 0),     # w: 4 of 8 columns
    ((3, 33, 20), (1, 15, 16), 0),    # w: an odd height, h: 3 lines
    ((4, 21, 16), (3, 8, 16), 0),     # t and h
    ((2, 18, 33), (1, 8, 16), 50),    # one slab a block; w: 1 of 16 columns, h: 2 lines
    ((5, 15, 28), (2, 8, 8), 0),      # one slab a block; all three axes
    ((3, 23, 22), (1, 30, 8), 30),    # no ordinary block
    ((3, 30, 9), (2, 32, 4), 0),      # the same
    ((2, 19, 70), (6, 8, 8), 0),      # one row of blocks in time
    ((2, 13, 35), (1, 16, 16), 0),    # the same in height
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_cut_blocks(grid, tile, n_text, n_heads):
    """Every row of small grids, most of which are padded with so little to compute."""
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


@pytest.mark.parametrize("spatial,grid,tile", [
    (False, (24, 33, 20), (1, 15, 16)),   # each block attends its place in every frame: lines of 4 of 16 columns, 3 lines
    (False, (24, 60, 20), (1, 30, 8)),
    (False, (35, 18, 20), (2, 8, 16)),    # all eight classes
    (False, (34, 18, 20), (3, 8, 16)),
    (False, (30, 45, 22), (2, 32, 4)),
    (True, (7, 45, 42), (3, 8, 16)),      # each block attends its frames
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_values_of_other_blocks_stay_out_of_cut_ones(spatial, grid, tile):
    """Every block of which the query's block attends none has infinite values: a row of zero probability that came from there would
    make the result NaN."""
    B = _binding()
    T, H, W = grid
    L = T * H * W
    n = O.block_grid(T, H, W, tile)
    params = [(1, 0, INF, n[1] * n[2], 0, INF) if spatial else (n[0], 0, INF, 1, 0, INF)] * 20
    gen = torch.Generator(device="cuda").manual_seed(L)
    q, k, v = (torch.randn((20, L, 128), device="cuda", generator=gen).bfloat16() for _ in range(3))
    want, want_lse = B.psa_attn_fwd(q, k, v, params, grid, tile, SCALE)
    assert B.psa_last_attn_grid()[0] == "cut"
    t, h, w = torch.meshgrid(*(torch.arange(x, device="cuda") for x in grid), indexing="ij")
    odd = ((t // tile[0] if spatial else h // tile[1] + w // tile[2]) % 2 == 1).reshape(-1)
    for other in (odd, ~odd):
        bad = v.clone()
        bad[:, other] = float("inf")
        out, lse = B.psa_attn_fwd(q, k, bad, params, grid, tile, SCALE)
        assert B.psa_last_device_status()[0] == 0
        assert torch.equal(out[:, ~other].view(torch.int16), want[:, ~other].view(torch.int16))
        assert torch.equal(lse.view(torch.int32), want_lse.view(torch.int32))


def test_more_spatial_blocks_than_a_cut_grid_has():
    """1,056 blocks a frame, ragged in height and width: padded; in width only: cut."""
    B = _binding()
    for grid, kind in (((1, 525, 503), "padded"), ((1, 528, 504), "cut")):
        T, H, W = grid
        L, tile = T * H * W, (1, 16, 16)
        params = [(1, 0, INF, 2, 0, 7)]
        gen = torch.Generator(device="cuda").manual_seed(L)
        q, k, v = (torch.randn((1, L, 128), device="cuda", generator=gen).bfloat16() for _ in range(3))
        out, lse = B.psa_attn_fwd(q, k, v, params, grid, tile, SCALE)
        assert B.psa_last_attn_grid()[0] == kind and B.psa_last_device_status()[0] == 0
        rows = sorted(set(WL.sample_rows(7, 0, L, 12)) | {0, W - 1, L - W, L - 1})
        qf, kf, vf = (x[0].double().cpu().numpy() for x in (q, k, v))
        ro, rl = O.attention_rows(qf, kf, vf, rows, params[0], T, H, W, tile, SCALE)
        err = np.abs(out[0, rows].double().cpu().numpy() - ro)
        assert err.max() <= 2e-2 and err.mean() <= 2e-3, (err.max(), err.mean())
        assert np.abs(lse[0, rows].double().cpu().numpy() - rl).max() <= 1e-3


@pytest.mark.parametrize("grid,tile", [((2, 30, 20), (1, 15, 16)), ((2, 16, 36), (1, 8, 16)), ((2, 60, 20), (1, 30, 8))],
                         ids=["1x15x16", "1x8x16", "1x30x8"])
def test_values_of_other_blocks_stay_out(grid, tile):
    """Each block attends itself only (too little for a cut), and every other block's values are infinite: a row of zero
    probability that came from there would make the result NaN."""
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
