"""A call behind a kernel that lets the call's kernels start early and then runs for longer than the time limit of the
waits inside them: the limits may only start when that kernel has finished.  Calls that share items without and with
planning, that run every item at once and that draw planned items; each result bit for bit that of the call alone."""
import ctypes
import math
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SCALE = 1.0 / math.sqrt(128.0)
LIMIT_MS = 2000   # of a wait inside the attention kernel


@pytest.fixture(scope="module")
def early_trigger(tmp_path_factory):
    from paper_2609_37001_b200 import build
    lib = str(tmp_path_factory.mktemp("early") / "libearly.so")
    subprocess.run([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-Xcompiler", "-fPIC", "-shared",
                    "-o", lib, os.path.join(ROOT, "tests", "c_abi", "early_trigger.cu")], check=True, capture_output=True)
    f = ctypes.CDLL(lib).early_trigger
    f.argtypes = [ctypes.c_int, ctypes.c_void_p]
    return f


@pytest.mark.parametrize("grid,tile,n_heads,n_text", [
    ((8, 16, 16), (2, 8, 8), 2, 0),       # shared items, all at once
    ((20, 24, 32), (1, 16, 16), 1, 219),  # shared items, planned
    ((7, 16, 32), (1, 8, 16), 4, 0),      # 112 items
    ((21, 30, 24), (1, 15, 16), 12, 0),   # planned items
], ids=["shared_direct", "shared", "direct", "ticket"])
def test_time_limits_start_when_the_predecessor_has_finished(early_trigger, request, grid, tile, n_heads, n_text):
    from paper_2609_37001_b200 import build
    build.build()
    from paper_2609_37001_b200 import binding as B
    L = grid[0] * grid[1] * grid[2] + n_text
    params = [(3, 0, 0, 2, 0, 0) if n_text == 0 else (1, 0, 0, 1, 0, 0)] * n_heads
    gen = torch.Generator(device="cuda").manual_seed(L)
    q, k, v = (torch.randn((n_heads, L, 128), device="cuda", generator=gen).bfloat16() for _ in range(3))
    want = B.psa_attn_fwd_joint(q, k, v, params, grid, tile, SCALE, n_text)
    assert B.psa_last_attn_launch()[1] == request.node.callspec.id
    assert B.psa_last_device_status() == (0, 0)
    t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    out, lse = (torch.empty_like(x) for x in want)
    stream = torch.cuda.current_stream()
    t0.record()
    assert early_trigger(LIMIT_MS + 300, stream.cuda_stream) == 0
    B.psa_attn_fwd_joint(q, k, v, params, grid, tile, SCALE, n_text, out=out, lse=lse)
    t1.record()
    assert B.psa_last_device_status() == (0, 0)
    assert t0.elapsed_time(t1) > LIMIT_MS
    assert torch.equal(out.view(torch.int16), want[0].view(torch.int16)) and torch.equal(lse.view(torch.int32), want[1].view(torch.int32))
