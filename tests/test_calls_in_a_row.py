"""Calls enqueued one behind the other without a synchronisation, in every order of the ways a launch may hand out its work
items, on whole, padded and cut grids, and through both scratch areas: a call's kernels start while the ones before are still running, so each must wait for
what it reads and overwrites.  Every result bit for bit that of the call alone; the inputs of a group of calls are
overwritten right in front of it, and again behind it."""
import math
import random

import pytest
import torch

pytestmark = pytest.mark.gpu
SCALE = 1.0 / math.sqrt(128.0)
KINDS = {   # mode (and grid): grid, tile, heads, text tokens
    "shared_direct": ((8, 16, 16), (2, 8, 8), 2, 0),
    "direct": ((7, 16, 32), (1, 8, 16), 4, 0),
    "ticket": ((4, 16, 32), (1, 16, 16), 40, 0),
    "ticket_short": ((4, 16, 32), (1, 8, 16), 24, 0),
    "ticket_edge": ((2, 23, 32), (1, 16, 16), 90, 0),
    "shared": ((20, 24, 32), (1, 16, 16), 1, 219),
    "shared whole": ((20, 32, 32), (1, 16, 16), 1, 219),
    "shared_direct padded": ((6, 15, 23), (2, 8, 8), 3, 0),
    "direct padded": ((2, 24, 27), (2, 8, 8), 11, 0),
    "ticket padded": ((5, 11, 60), (1, 15, 16), 17, 0),
    "ticket_short padded": ((3, 15, 33), (1, 8, 16), 30, 0),
    "shared_direct cut": ((5, 10, 45), (3, 32, 4), 2, 0),
    "direct cut": ((11, 9, 16), (2, 32, 4), 6, 0),
    "ticket cut": ((6, 16, 20), (3, 32, 4), 20, 0),
    "ticket_edge cut": ((9, 11, 60), (2, 32, 4), 2, 0),
    "shared cut": ((20, 12, 35), (1, 15, 16), 3, 50),
}
GRIDS = {"shared_direct": "whole", "direct": "whole", "ticket": "whole", "ticket_short": "whole", "ticket_edge": "padded", "shared": "padded"}


class Problem:
    def __init__(self, B, mode, noalloc):
        self.B, self.noalloc, self.mode = B, noalloc, mode
        self.grid, self.tile, heads, self.n_text = KINDS[mode]
        self.params = [((2, 0, 0, 3, 0, 0), (1, 0, 0, 1, 0, 0), (1, 1, 0, 2, 0, 0))[h % 3] for h in range(heads)]
        L = self.grid[0] * self.grid[1] * self.grid[2] + self.n_text
        gen = torch.Generator(device="cuda").manual_seed(L + heads)
        self.variants = [[torch.randn((heads, L, 128), device="cuda", generator=gen).bfloat16() for _ in range(3)] for _ in range(2)]
        self.qkv = [torch.empty_like(x) for x in self.variants[0]]
        self.want = []
        for v in range(2):
            self.fill(v)
            torch.cuda.synchronize()
            got = self.call(*self.outputs())
            assert B.psa_last_attn_launch()[1] == mode.split()[0]
            assert B.psa_last_attn_grid()[0] == (GRIDS[mode] if mode in GRIDS else mode.split()[1])
            torch.cuda.synchronize()
            self.want.append([x.clone() for x in got])

    def outputs(self):
        out = torch.full_like(self.qkv[0], float("nan"))
        return out, torch.full(out.shape[:2], float("nan"), dtype=torch.float32, device="cuda")

    def fill(self, variant):
        for x, y in zip(self.qkv, self.variants[variant]):
            x.copy_(y)

    def call(self, out, lse):
        if self.noalloc:
            self.B.psa_attn_fwd_noalloc(*self.qkv, out, lse, self.params, self.grid, self.tile, SCALE, check=False)
        elif self.n_text:
            self.B.psa_attn_fwd_joint(*self.qkv, self.params, self.grid, self.tile, SCALE, self.n_text, out=out, lse=lse)
        else:
            self.B.psa_attn_fwd(*self.qkv, self.params, self.grid, self.tile, SCALE, out=out, lse=lse)
        return out, lse


@pytest.mark.parametrize("captured", [False, True], ids=["enqueued", "captured"])
def test_every_order_of_launch_modes(captured):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    problems = [Problem(B, mode, noalloc) for mode in KINDS for noalloc in ((False, True) if KINDS[mode][3] == 0 else (False,))]
    # every problem directly behind every other and behind itself, in pairs and in longer groups; one variant of a problem's
    # inputs within a group
    rng = random.Random(7)
    orders = [[a, b] for a in problems for b in problems] + [rng.sample(problems, 4) for _ in range(20)]
    rng.shuffle(orders)
    groups = []
    for order in orders:
        variant = {id(p): rng.randrange(2) for p in order}
        groups.append([(p, variant[id(p)], *p.outputs()) for p in order])

    def enqueue():
        for group in groups:
            for p, v, _, _ in group:
                p.fill(v)
            for p, _, out, lse in group:
                p.call(out, lse)
            for p, v, _, _ in group:
                p.fill(1 - v)

    torch.cuda.synchronize()
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            enqueue()
        for _ in range(3):
            graph.replay()
    else:
        enqueue()
    assert B.psa_last_device_status() == (0, 0)
    for group in groups:
        for p, v, out, lse in group:
            assert torch.equal(out.view(torch.int16), p.want[v][0].view(torch.int16)), p.mode
            assert torch.equal(lse.view(torch.int32), p.want[v][1].view(torch.int32)), p.mode
