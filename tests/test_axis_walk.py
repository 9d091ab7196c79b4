"""psa_mask_sizes (host code: the incremental walk over an axis' coordinate differences) against the oracle's axis
masks: short and long axes, strides of 1, short, longer than the axis and infinite, offsets inside and far outside."""
import random

import pytest

from oracle import psa_oracle as O


@pytest.mark.parametrize("seed", range(4))
def test_pair_counts_match_the_axis_masks(seed):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    rng = random.Random(seed)
    for _ in range(150):
        T, H, W = rng.choice([1, 2, 21, 64, 65, 130]), rng.randint(1, 12), rng.randint(1, 12)
        p = (rng.randint(1, T + 3), rng.choice([0, 1, -2, T, -T, 5 * T, -(1 << 29)]), rng.choice([0, 1, 2, 3, T, T + 1, 1 << 20]),
             rng.randint(1, H * W + 3), rng.choice([0, -1, 3, H * W, -3 * H * W]), rng.choice([0, 1, 5, 6, H * W + 7]))
        nb, nnz = B.psa_mask_sizes([p], (T, H, W), (1, 1, 1))
        want = int(O.axis_mask(T, *p[:3]).sum()) * int(O.axis_mask(H * W, *p[3:]).sum())
        assert (nb, nnz) == (T * H * W, want), (p, T, H, W)


def test_parameters_given_as_lists_or_floats():
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    grid, tile = (21, 45, 80), (1, 15, 16)
    want = B.psa_mask_sizes([(4, 2, 0, 5, 1, 3)], grid, tile)
    assert B.psa_mask_sizes([[4, 2, 0, 5, 1, 3]], grid, tile) == want
    assert B.psa_mask_sizes([(4.0, 2.0, 0.0, 5.0, 1.0, 3.0)], grid, tile) == want


def test_parameters_are_looked_up_by_value():
    """Rows that hash by identity and change between calls, and rows of other lengths than six."""
    import numpy as np
    import torch
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    grid, tile = (21, 45, 80), (1, 15, 16)
    want = {w: B.psa_mask_sizes([(w, 2, 0, 5, 1, 3)], grid, tile) for w in (4, 21)}
    assert want[4] != want[21]

    class Row:
        def __init__(self, values):
            self.values = values

        def __iter__(self):
            return iter(self.values)

    row = torch.tensor([4, 2, 0, 5, 1, 3], dtype=torch.int32)
    cells = tuple(torch.tensor(x) for x in (4, 2, 0, 5, 1, 3))
    obj, arr = Row([4, 2, 0, 5, 1, 3]), np.array([4, 2, 0, 5, 1, 3], dtype=np.int64)
    given = ([row], (row,), [cells], [obj], [arr], torch.stack([row]))
    assert [B.psa_mask_sizes(g, grid, tile) for g in given] == [want[4]] * 6
    row[0], obj.values[0], arr[0] = 21, 21, 21
    cells[0].fill_(21)
    given = ([row], (row,), [cells], [obj], [arr], torch.stack([row]))
    assert [B.psa_mask_sizes(g, grid, tile) for g in given] == [want[21]] * 6
    # a row of five leaves the spatial stride 0 (infinite), whatever row stands beside it; one of seven is an error
    five, six = (4, 2, 0, 5, 1), (3, 4, 2, 5, 1, 3)
    assert B.psa_mask_sizes([five, six], grid, tile) == B.psa_mask_sizes([five + (0,), six], grid, tile)
    for rows in ([five, six + (3,)], [six + (3,), five], [six + (3,)]):
        with pytest.raises(TypeError):
            B.psa_mask_sizes(rows, grid, tile)


@pytest.mark.parametrize("n", [32, 33, 36, 60, 63, 64, 65])
def test_pair_counts_of_axes_around_the_bit_set_widths(n):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    for w in (1, 2, n - 1, n, 2 * n, 200):
        for o in (0, 1, -1, n - 1, 1 - n, n, -n, 128 - n, 129 - n):
            for s in (0, 1, 2, 3, n, 63, 64, 65, 127, 128):
                got = B.psa_mask_sizes([(w, o, s, 1, 0, 0)], (n, 1, 1), (1, 1, 1))
                assert got == (n, int(O.axis_mask(n, w, o, s).sum())), (n, w, o, s)
