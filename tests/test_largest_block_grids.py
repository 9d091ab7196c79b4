"""The largest block grids that the planning kernel takes: T'S' + T' + S' words of shared memory of 58,112."""
import ctypes
import math

import pytest
import torch

SCALE = 1.0 / math.sqrt(128.0)
PARAMS = [(2, 0, 0, 1, 0, 0)]   # a block attends itself and its neighbours in time


def test_grids_beyond_the_planning_kernel_are_refused():
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    prob = B.make_problem(1, (1, 8, 16), SCALE, 128, 128)
    refused = {}
    for tp, sp in ((28, 2048), (33, 1760), (32, 1761), (29, 1937)):
        assert tp * sp + tp + sp > 58112
        # pointers that are refused after the grid: q and out alias
        refused[tp, sp] = B.lib().psa_attn_fwd(16, 32, 48, 16, 80, B._params_array(PARAMS), ctypes.byref(prob), tp, 8 * sp, 1, None)
    assert set(refused.values()) == {B.PSA_ERR_UNSUPPORTED}, refused
    for tp, sp in ((27, 2048), (32, 1760)):
        assert tp * sp + tp + sp <= 58112
        rc = B.lib().psa_attn_fwd(16, 32, 48, 16, 80, B._params_array(PARAMS), ctypes.byref(prob), tp, 8 * sp, 1, None)
        assert rc == B.PSA_ERR_INVALID_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("T,Sp,bh", [(27, 2048, 8), (32, 1760, 8), (27, 2048, 16), (32, 1760, 16)])
def test_largest_grids(T, Sp, bh):
    """Blocks of 8 or 16 rows of a grid one column wide, the last block of each frame one row high (with 16 rows, two slabs,
    it is an edge block).  Every row against plain torch in 32 bits, at the tolerances of the other parity tests."""
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    H = (Sp - 1) * bh + 1
    L = T * H
    gen = torch.Generator(device="cuda").manual_seed(L)
    q, k, v = (torch.randn((1, L, 128), device="cuda", generator=gen).bfloat16() for _ in range(3))
    out, lse = B.psa_attn_fwd(q, k, v, PARAMS, (T, H, 1), (1, bh, 16), SCALE)
    assert B.psa_last_device_status() == (0, 0)

    def blocks(x):   # (T, blocks, rows, 128), frames and rows beyond the grid zero
        x = x[0].float().reshape(T, H, 128)
        return torch.nn.functional.pad(x, (0, 0, 0, Sp * bh - H)).reshape(T, Sp, bh, 128)

    real = torch.zeros((T, Sp * bh), dtype=torch.bool, device="cuda")
    real[:, :H] = True
    real = real.reshape(T, Sp, bh)
    qb, kb, vb = blocks(q), blocks(k), blocks(v)
    for t in range(T):
        near = [u for u in (t - 1, t, t + 1) if 0 <= u < T]
        keys, vals = torch.cat([kb[u] for u in near], 1), torch.cat([vb[u] for u in near], 1)
        s = torch.einsum("bqd,bkd->bqk", qb[t].double(), keys.double()) * SCALE
        s.masked_fill_(~torch.cat([real[u] for u in near], 1)[:, None, :], float("-inf"))
        ro = torch.einsum("bqk,bkd->bqd", s.softmax(-1), vals.double())[real[t]]
        rl = s.logsumexp(-1)[real[t]]
        err = (out[0, t * H:(t + 1) * H].double() - ro).abs()
        assert err.max() <= 2e-2 and err.mean() <= 2e-3, (t, err.max().item())
        assert (lse[0, t * H:(t + 1) * H].double() - rl).abs().max() <= 1e-3
