"""Performance cases of the library: the calls a video-DiT program makes, from the smallest to the largest.

A case names one entry point of paper_2609_37001_b200.binding ("call") and its problem: token grid, mask block
("tile"), heads, per-head stripe masks (those of a committed workload, or drawn from the ranges the paper searches),
memory layout of the activations and the call's own options.

    listed()   the fixed cases        draw(rng)   one more of the same ranges
    prepare()  inputs on the device   run()       one pass through the public entry point
    work()     bytes and operations a pass cannot do without
    tolerance()  how far another correct implementation may be
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2609_37001_b200 import binding as psa
from paper_2609_37001_b200 import workloads

HEAD_DIM = 128
SCALE = 1.0 / math.sqrt(HEAD_DIM)
INF = 0   # an infinite stride

# Mask blocks the attention kernel takes, by slabs per block: 128 tokens, two slabs (192 to 256 tokens), three.
TILES = {1: [(1, 8, 16), (2, 8, 8), (1, 32, 4)],
         2: [(1, 16, 16), (1, 15, 16), (1, 30, 8), (2, 32, 4), (2, 8, 16), (1, 14, 16), (1, 12, 16)],
         3: [(3, 8, 16), (6, 8, 8), (3, 32, 4)]}


def _case(name, call, grid, tile, heads, **more):
    T, H, W = grid
    bt, bh, bw = tile
    case = {"call": call, "T": T, "H": H, "W": W, "bt": bt, "bh": bh, "bw": bw, "heads": heads}
    if name:
        case["name"] = name
    case.update(more)
    return case


def _listed(name, call, workload_name, heads=None, **more):
    w = workloads.workload(workload_name)
    return _case(name, call, w["grid"], w["tile"], heads or w["n_heads"], workload=workload_name, **more)


def listed():
    return [
        # One attention call on a few latent frames (128-token blocks): launches and host work are all there is.
        _listed("tiny_call", "attn", "tiny"),
        # The same size with 256-token blocks through the entry point that allocates nothing (plugins, serving loops).
        _listed("tiny_noalloc", "noalloc", "tiny_b256"),
        # One layer of the 1.3B model at 480p, [heads, tokens, 128] activations.
        _listed("wan13b_480p", "attn", "wan13b_480p_b1x30x8"),
        # The conditional / unconditional pair of classifier-free guidance in the layout the projections leave:
        # [batch, tokens, heads, 128], so heads are interleaved and the samples are not evenly spaced heads.
        _listed("wan13b_480p_cfg", "batched", "wan13b_480p", batch=2, layout="token"),
        # One layer of the 14B model at 720p: the headline workload.
        _listed("wan14b_720p", "attn", "wan14b_720p"),
        # The same layer with the paper's 384-token block (H is padded from 45 to 48).
        _listed("wan14b_720p_b3x8x16", "attn", "wan14b_720p_b3x8x16"),
        # The five heads that one of eight ranks holds of that layer when heads are sharded.
        _listed("wan14b_720p_5heads", "noalloc", "wan14b_720p", heads=5),
        # A grid that no block tiles: ragged in height and width.
        _listed("ragged_75", "attn", "ragged_75", layout="token"),
        # A multimodal layer at 768p: 115,200 video tokens and the prompt's 256 text tokens.  The largest case.
        _listed("hunyuan_768p_text", "joint", "hunyuan_768p", text=256),
        # The block mask and index lists of one 720p layer, as a caller of other kernels asks for them.
        _listed("mask_build_720p", "mask", "wan14b_720p"),
        # Mask search: every candidate mask of one head against full attention.
        _case("search_480p", "search", (21, 30, 52), (1, 30, 8), 32, masks=7),
        # One 480p layer whose activations live in (pinned) host memory: copies in, kernel, copies out.
        _listed("host_480p", "host", "wan13b_480p"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# Bounds on a drawn case: attended pairs (well below the largest listed case, as some blocks run slower), bytes of a mask build.
_MAX_PAIRS = 4.0e10
_MAX_MASK_BYTES = 2.0e8


def draw(rng):
    while True:
        call = rng.choice(["attn", "attn", "attn", "noalloc", "batched", "joint", "mask", "search", "host"])
        tile = rng.choice(TILES[rng.choice([1, 2, 2, 2, 3])])
        # a grid from a few frames of a thumbnail to 33 latent frames of 768p, ragged as often as not
        grid = [_log_int(rng, 2, 33), _log_int(rng, 12, 48), _log_int(rng, 12, 80)]
        if rng.random() < 0.4:
            grid = [-(-x // b) * b for x, b in zip(grid, tile)]
        grid = tuple(grid)
        heads = _log_int(rng, 1, 40)
        more = {"masks": rng.randrange(1 << 20)}
        lo = rng.choice([0.0, 0.25, 0.5, 0.6, 0.75, 0.85])
        more["lo"], more["hi"] = lo, min(0.95, lo + 0.25)
        if call in ("attn", "noalloc", "joint"):
            more["layout"] = rng.choice(["head", "token"])
        if call == "batched":
            more["batch"], more["layout"] = rng.choice([2, 2, 3]), rng.choice(["head", "token"])
        if call == "joint":
            more["text"] = _log_int(rng, 16, 512)
        if call == "search":
            heads = _log_int(rng, 4, 128)
            more["lo"], more["hi"] = 0.0, 0.95
        if call == "mask" and rng.random() < 0.4:
            tile = rng.choice([(1, 8, 8), (1, 4, 16), (2, 4, 8)])   # finer than the attention kernel's blocks
        case = _case(None, call, grid, tile, heads, **more)
        nb = _blocks(case)[2]
        tokens = grid[0] * grid[1] * grid[2]
        if call == "mask":
            if heads * nb * nb > _MAX_MASK_BYTES or heads < 6 or nb < 16:
                continue
        elif call == "noalloc" and heads * nb * (2 if tile in TILES[3] else 1) > 16384:
            continue
        elif call == "host" and heads * tokens > 600_000:
            continue
        elif (call == "search" and heads * tokens > 4_000_000) or _pairs(case) > _MAX_PAIRS:
            continue
        return case


# ---------------------------------------------------------------------------------------------- masks of a case
def _blocks(case):
    tp, hp, wp = (-(-case[x] // case[b]) for x, b in (("T", "bt"), ("H", "bh"), ("W", "bw")))
    return tp, hp * wp, tp * hp * wp


@functools.lru_cache(maxsize=None)
def _axis(n, w, o, s):
    """The axis mask of the stripe rule: n x n truth values, query by key."""
    d = np.abs(np.arange(n)[None, :] - np.arange(n)[:, None] - o)
    return ((d % s if s else d) <= w - 1)


def _masks(case):
    """The six stripe parameters of every head (of every candidate for a search)."""
    if "workload" in case:
        return [tuple(p) for p in workloads.workload(case["workload"])["head_params"][:case["heads"]]]
    tp, sp, _ = _blocks(case)
    wp = -(-case["W"] // case["bw"])
    lo, hi = case.get("lo", 0.0), case.get("hi", 0.95)
    rng = random.Random(case["masks"])
    got = []
    for h in range(case["heads"]):
        kind, best = ("temporal", "spatial", "joint")[h % 3], None
        for _ in range(60):   # the draw of wanted sparsity, or the nearest one on grids that have none
            t = (rng.randint(1, tp), rng.choice([0, 1, -1, 2, -2]), rng.choice([1, 2, 3, INF]))
            s = (rng.randint(1, wp), rng.choice([0, 1, -1]), rng.choice([1, 3, 5, 6, INF]))
            if kind == "temporal":
                s = (sp, 0, INF)
            elif kind == "spatial":
                t = (tp, 0, INF)
            mt, ms = _axis(tp, *t), _axis(sp, *s)
            if not (mt.any(1).all() and ms.any(1).all()):
                continue   # a query block without any key
            sparsity = 1.0 - mt.mean() * ms.mean()
            miss = max(lo - sparsity, sparsity - hi, 0.0)
            if best is None or miss < best[0]:
                best = (miss, t + s)
            if miss == 0.0:
                break
        got.append(best[1] if best else (tp, 0, INF, sp, 0, INF))
    return got


def _sizes(extent, block):
    n = -(-extent // block)
    return np.minimum(block, extent - block * np.arange(n)).astype(np.float64)


def _pairs(case):
    """Attended (query, key) pairs of real tokens in one pass."""
    tp, sp, _ = _blocks(case)
    nt = _sizes(case["T"], case["bt"])
    ns = np.outer(_sizes(case["H"], case["bh"]), _sizes(case["W"], case["bw"])).reshape(-1)
    tokens = float(case["T"] * case["H"] * case["W"])
    total = 0.0
    for p in _masks(case):
        total += float(nt @ _axis(tp, *p[:3]) @ nt) * float(ns @ _axis(sp, *p[3:]) @ ns)
    if case["call"] == "search":
        total += tokens * tokens   # full attention, which the candidates are held against
    text = case.get("text", 0)
    total += case["heads"] * (2.0 * tokens * text + float(text) * text)
    return total * case.get("batch", 1)


# ---------------------------------------------------------------------------------------------- inputs and passes
def _activations(case, seed, count):
    """`count` bf16 tensors [(batch,) heads, tokens, 128], standard normal, in the case's memory layout."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    heads = 1 if case["call"] == "search" else case["heads"]
    tokens = case["T"] * case["H"] * case["W"] + case.get("text", 0)
    got = []
    for _ in range(count):
        shape = [case.get("batch", 1), heads, tokens, HEAD_DIM]
        if case.get("layout", "head") == "token":
            shape[1], shape[2] = shape[2], shape[1]
        x = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
        for part in x:
            part.normal_(generator=gen)
        if case.get("layout", "head") == "token":
            x = x.transpose(1, 2)
        got.append(x if "batch" in case else x[0])
    return got


def prepare(case, seed):
    state = {"call": case["call"], "grid": (case["T"], case["H"], case["W"]), "tile": (case["bt"], case["bh"], case["bw"]),
             "masks": _masks(case), "text": case.get("text", 0)}
    call = case["call"]
    if call == "mask":
        # other heads' masks with another seed: the same ones in another order, so that a pass costs the same
        random.Random(seed).shuffle(state["masks"])
        nb, nnz = psa.psa_mask_sizes(state["masks"], state["grid"], state["tile"])
        state["out"] = (torch.empty((case["heads"], nb, nb), dtype=torch.uint8, device="cuda"),
                        torch.empty(case["heads"] * nb + 1, dtype=torch.int32, device="cuda"),
                        torch.empty(max(nnz, 1), dtype=torch.int32, device="cuda"))
        return state
    state["qkv"] = _activations(case, seed, 3)
    if call == "search":
        state["qkv"] = [x[0] for x in state["qkv"]]
        n = psa.psa_search_scratch_bytes(case["heads"], state["grid"])
        state["scratch"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    if call == "noalloc":
        q = state["qkv"][0]
        state["out"] = torch.empty_strided(q.shape, q.stride(), dtype=q.dtype, device="cuda")
        state["lse"] = torch.empty(q.shape[:2], dtype=torch.float32, device="cuda")
    if call == "host":
        dev = state["qkv"]
        state["qkv"] = [torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x) for x in dev]
        state["out"] = torch.empty(dev[0].shape, dtype=torch.bfloat16, pin_memory=True)
        state["lse"] = torch.empty(dev[0].shape[:2], dtype=torch.float32, pin_memory=True)
        state["staging"] = dev + [torch.empty_like(dev[0]), torch.empty(dev[0].shape[:2], dtype=torch.float32, device="cuda")]
    return state


def run(state):
    call, masks, grid, tile = state["call"], state["masks"], state["grid"], state["tile"]
    if call == "mask":
        return psa.psa_mask_build(masks, grid, tile, out=state["out"])
    q, k, v = state["qkv"]
    if call == "attn":
        return psa.psa_attn_fwd(q, k, v, masks, grid, tile, SCALE)
    if call == "batched":
        return psa.psa_attn_fwd_batched(q, k, v, masks, grid, tile, SCALE)
    if call == "joint":
        return psa.psa_attn_fwd_joint(q, k, v, masks, grid, tile, SCALE, state["text"])
    if call == "noalloc":
        psa.psa_attn_fwd_noalloc(q, k, v, state["out"], state["lse"], masks, grid, tile, SCALE, check=False)
    elif call == "host":
        psa.psa_attn_fwd_host(q, k, v, state["out"], state["lse"], state["staging"], masks, grid, tile, SCALE)
    elif call == "search":
        return psa.psa_search_losses(q, k, v, masks, grid, tile, SCALE, scratch=state["scratch"])
    return state["out"], state["lse"]


# ---------------------------------------------------------------------------------------------- work and tolerance
def work(case):
    heads, (tp, sp, nb) = case["heads"], _blocks(case)
    if case["call"] == "mask":
        nnz = sum(int(_axis(tp, *p[:3]).sum()) * int(_axis(sp, *p[3:]).sum()) for p in _masks(case))
        return {"bytes": heads * nb * nb + 4 * (heads * nb + 1) + 4 * nnz, "flops": 0}
    tokens = case["T"] * case["H"] * case["W"] + case.get("text", 0)
    rows = (1 if case["call"] == "search" else heads) * tokens * case.get("batch", 1)
    # q, k, v read once; out and lse written once (a search returns one number per candidate)
    moved = rows * 3 * HEAD_DIM * 2 + (4 * heads if case["call"] == "search" else rows * (HEAD_DIM * 2 + 4))
    return {"bytes": moved, "flops": 4 * HEAD_DIM * _pairs(case)}


def tolerance(case):
    if case["call"] == "mask":
        return "exact"
    if case["call"] == "search":
        # losses of sampled rows against 64-bit arithmetic: rel 2.5e-5, max 9e-5; smaller grids average over fewer rows
        return {"rel": 2e-4, "max": 2e-3}
    # against 64-bit arithmetic on the bf16 inputs: rel 2.3e-3 (the rounding of the output alone is 1.7e-3), max 1.4e-2
    return {"rel": 1e-2, "max": 6e-2}
