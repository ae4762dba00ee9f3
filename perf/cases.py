"""The requests whose speed this repository watches, and how one pass of each is made.

A case is one attention request of a video-diffusion transformer as a user's program sends it: a logical block mask
over (heads, query blocks, key blocks), the tensors Q, K, V and the entry point that is called.

Fields of a case
    path     "request"  a new mask on every call: ``bsa.request`` (mask analysis, plan, attention), plan given back
             "plan"     one mask for many calls: a kept ``Plan`` and its ``forward``
             "cache"    a mask that repeats from step to step and is not tracked by the caller: ``PlanCache.request``
             "host"     mask and tensors in (pinned) host memory: ``bsa.request_host``
    heads, N, N_kv, d, B_Q, B_KV, dtype, layout, packed    as the arguments of those calls (N_kv = N: self-attention)
    pattern  "window"   3-D neighbourhood of a latent cut into grid tiles of one block each, plus random blocks
             "mixed"    neighbourhood, then column stripes, then random blocks up to each row's budget
             "runs"     a few contiguous runs of key blocks per row, different from row to row
             "random"   independent random blocks and the diagonal
    density  share of active blocks; with ``skewed`` one head in eight is up to ten times heavier than the others
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_25869_b200 import bsa

# the block geometries of the repository's configurations, sweep and tests
_GEOMETRIES = [(16, 16), (16, 64), (32, 16), (32, 32), (64, 32), (64, 64), (64, 64), (64, 128), (128, 64), (128, 128),
               (128, 128), (256, 256)]
_MAX_DRAWN_FLOPS = 2.5e12   # a drawn case stays below a quarter of the largest listed one
_MAX_DRAWN_BLOCKS = 1.0e8   # mask elements


def _case(name, path, heads, N, d, B, density, pattern, N_kv=0, dtype="bf16", layout="hnd", packed=False, skewed=False,
          grid="", window="", extra=0.0):
    c = {"path": path, "heads": heads, "N": N, "N_kv": N_kv or N, "d": d, "B_Q": B[0], "B_KV": B[1], "density": density,
         "pattern": pattern, "dtype": dtype, "layout": layout, "packed": packed, "skewed": skewed, "grid": grid,
         "window": window, "extra": extra}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: two heads of a short clip; launches and the host's share are everything
        _case("tiny_request", "request", 2, 2048, 64, (64, 64), 0.25, "random"),
        # attention of video tokens to another, shorter and ragged token sequence, half tensors as a fused projection
        # leaves them ([tokens, heads, d]); several such calls per layer
        _case("cross_ragged", "plan", 16, 3600, 64, (64, 32), 0.2, "mixed", N_kv=1111, dtype="fp16", layout="nhd"),
        # one layer of a short clip with a mask of its own: the ordinary cold request
        _case("mid_request", "request", 8, 16384, 128, (128, 128), 0.15, "window", grid="8x4x4", window="1,1,1", extra=0.02),
        # the same layer in the next denoising steps, the mask unchanged: the warm request
        _case("mid_repeated", "cache", 8, 16384, 128, (128, 128), 0.15, "window", grid="8x4x4", window="1,1,1", extra=0.02),
        # the same layer for a caller whose tensors live in host memory (offloaded activations)
        _case("mid_host", "host", 8, 16384, 128, (128, 128), 0.15, "window", grid="8x4x4", window="1,1,1", extra=0.02),
        # fine row blocks that each keep their own runs of keys
        _case("fine_rows_runs", "request", 16, 32768, 64, (16, 64), 0.15, "runs"),
        # coarse blocks and a small head dimension, one mask for all steps
        _case("coarse_plan", "plan", 16, 32768, 64, (256, 256), 0.2, "random"),
        # 75600 tokens (not a multiple of any block), heads of very different weight, a new mask per request: the
        # block sizes that mask predictors emit, from fine to coarse
        _case("long_32x32_packed", "request", 24, 75600, 128, (32, 32), 0.1, "mixed", packed=True, skewed=True),
        _case("long_64x64", "request", 24, 75600, 128, (64, 64), 0.1, "mixed", skewed=True),
        _case("long_64x128_nhd", "plan", 12, 75600, 128, (64, 128), 0.1, "mixed", layout="nhd", skewed=True),
        _case("long_128x64_fp16", "request", 12, 75600, 128, (128, 64), 0.3, "mixed", dtype="fp16", skewed=True),
        # the largest: one layer of a 720p clip, 115200 tokens
        _case("huge_request", "request", 24, 115200, 128, (128, 128), 0.08, "window", grid="15x6x10", window="1,1,2",
              extra=0.03),
    ]


def draw(rng):
    while True:
        B = rng.choice(_GEOMETRIES)
        d = rng.choice([64, 64, 64, 64, 128, 128, 128, 128, 128, 256])
        N = int(round(2.0 ** rng.uniform(10.0, math.log2(115200))))
        if rng.random() < 0.5:
            N -= N % B[0] - B[0]  # half of the drawn requests are whole blocks, the others ragged
        N_kv = N if rng.random() < 0.8 else max(64, int(N * rng.uniform(0.2, 1.5)))
        heads = int(round(2.0 ** rng.uniform(0.0, math.log2(24))))
        density = 2.0 ** rng.uniform(math.log2(0.03), math.log2(0.5))
        pattern = rng.choice(["mixed", "mixed", "runs", "random"])
        c = _case("", rng.choice(["request", "request", "plan", "cache"]), heads, N, d, B, density, pattern, N_kv=N_kv,
                  dtype="fp16" if rng.random() < 0.25 else "bf16", layout="nhd" if rng.random() < 0.3 else "hnd",
                  packed=rng.random() < 0.25, skewed=heads >= 4 and rng.random() < 0.4)
        nq, nk = _blocks(c)
        if work(c)["flops"] <= _MAX_DRAWN_FLOPS and heads * nq * nk <= _MAX_DRAWN_BLOCKS:
            return c


# ------------------------------------------------------------------ masks
def _blocks(c):
    return -(-c["N"] // c["B_Q"]), -(-c["N_kv"] // c["B_KV"])


def _row_budgets(c):
    """Active blocks of every row, [heads, nQb]: a function of the case alone (which columns they are is the seed's)."""
    nq, nk = _blocks(c)
    H, rho = c["heads"], c["density"]
    r = np.random.RandomState(20240607)
    rho_h = np.full(H, rho)
    if c["skewed"]:
        w = np.ones(H)
        w[r.permutation(H)[: -(-H // 8)]] = 10.0
        rho_h = np.minimum(rho * w / w.mean(), 0.95)
        light = w == 1.0
        rho_h[light] += (rho * H - rho_h.sum()) / light.sum()
    jitter = np.exp(0.4 * r.randn(H, nq) - 0.08)
    return np.clip(np.rint(np.minimum(rho_h[:, None] * jitter, 1.0) * nk), 1, nk).astype(np.int64)


def _tile_coords(centres, n_tokens):
    """3-D tile coordinate of each token in ``centres``: tiles of 120 tokens, about five frames of square grids."""
    tiles = -(-n_tokens // 120)
    side = max(1, int(round(math.sqrt(tiles / 5.0))))
    t = centres // 120
    return torch.stack([t // (side * side), (t // side) % side, t % side], dim=1)


def _window(c):
    grid = [int(x) for x in c["grid"].split("x")]
    win = torch.tensor([int(x) for x in c["window"].split(",")], device="cuda")
    b = torch.arange(math.prod(grid), device="cuda")
    xyz = torch.stack([b // (grid[1] * grid[2]), (b // grid[2]) % grid[1], b % grid[2]], dim=1)
    return ((xyz[:, None] - xyz[None]).abs() <= win).all(dim=2)


def _window_blocks(c):
    n = 1
    for g, w in zip(c["grid"].split("x"), c["window"].split(",")):
        n *= sum(min(int(g), i + int(w) + 1) - max(0, i - int(w)) for i in range(int(g)))
    return n


def _make_mask(c, gen):
    nq, nk = _blocks(c)
    H = c["heads"]
    M = torch.empty((H, nq, nk), dtype=torch.uint8, device="cuda")
    if c["pattern"] == "window":
        W = _window(c)
        for h in range(H):
            M[h] = W | (torch.rand((nq, nk), device="cuda", generator=gen) < c["extra"])
        return M
    budget = torch.from_numpy(_row_budgets(c)).cuda()
    near = None
    if c["pattern"] == "mixed":
        cq = torch.clamp(torch.arange(nq, device="cuda") * c["B_Q"] + c["B_Q"] // 2, max=c["N"] - 1)
        ck = torch.clamp(torch.arange(nk, device="cuda") * c["B_KV"] + c["B_KV"] // 2, max=c["N_kv"] - 1)
        ck = ck * c["N"] // c["N_kv"]  # the key sequence spans the same clip
        dist = (_tile_coords(cq, c["N"])[:, None] - _tile_coords(ck, c["N"])[None]).abs().amax(dim=2)
        near = torch.clamp(dist, max=2).float()
        near[near == 2] = 3.0
    for h in range(H):
        key = torch.rand((nq, nk), device="cuda", generator=gen)
        if c["pattern"] == "mixed":
            rank = near.clone()
            rank[:, h % 8::8].clamp_(max=2.0)
            key += rank
        elif c["pattern"] == "runs":
            ctl = torch.rand((nq, 1, max(4, min(24, nk))), device="cuda", generator=gen)
            wave = torch.nn.functional.interpolate(ctl, size=nk, mode="linear", align_corners=True)[:, 0]
            key = wave + 1e-5 * key
        else:
            diag = torch.arange(nq, device="cuda") * nk // nq
            key[torch.arange(nq, device="cuda"), diag] = -1.0
        kth = key.sort(dim=1).values.gather(1, budget[h][:, None] - 1)
        M[h] = key <= kth
    return M


# ------------------------------------------------------------------ one case
def _inputs(case, seed):
    """The block mask (one byte per block) and Q, K, V of one seed."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    mask = _make_mask(case, gen)
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float16
    H, d = case["heads"], case["d"]

    def tokens(n):
        shape = (H, n, d) if case["layout"] == "hnd" else (n, H, d)
        return torch.randn(shape, device="cuda", generator=gen, dtype=torch.float32).to(dt)

    return mask, tokens(case["N"]), tokens(case["N_kv"]), tokens(case["N_kv"])


def prepare(case, seed):
    mask, q, k, v = _inputs(case, seed)
    H, d = case["heads"], case["d"]
    kw = {"N_kv": case["N_kv"], "dtype": case["dtype"], "layout": case["layout"]}
    st = {"path": case["path"], "args": (case["B_Q"], case["B_KV"], case["N"], H, d), "kw": kw}
    stride = 0
    if case["packed"]:
        mask, stride = bsa.pack_mask(mask)
    if case["path"] == "host":
        st["mask"] = mask.cpu().pin_memory()
        st["qkv"] = tuple(t.cpu().pin_memory() for t in (q, k, v))
        st["O"] = torch.empty_like(st["qkv"][0]).pin_memory()
        st["LSE"] = torch.empty((H, case["N"]), dtype=torch.float32).pin_memory()
        return st
    st["qkv"] = (q, k, v)
    if case["path"] == "plan":
        if stride:
            st["plan"] = bsa.plan_create_packed(mask, stride, *st["args"], **kw)
        else:
            st["plan"] = bsa.plan_create(mask, *st["args"], **kw)
        st["mask"] = mask
        return st
    st["mask"], st["row_stride"] = mask, stride
    if case["path"] == "cache":
        st["cache"] = bsa.PlanCache(16)
    return st


def run(state):
    q, k, v = state["qkv"]
    path = state["path"]
    if path == "plan":
        return state["plan"].forward(q, k, v)
    if path == "host":
        bsa.request_host(state["mask"], *state["args"], q, k, v, state["O"], state["LSE"], **state["kw"])
        return state["O"], state["LSE"]
    if path == "cache":
        O = torch.empty_like(q)
        LSE = torch.empty((state["args"][3], state["args"][2]), dtype=torch.float32, device="cuda")
        plan, _ = state["cache"].request(state["mask"], *state["args"], q, k, v, O, LSE, row_stride=state["row_stride"],
                                         **state["kw"])
    else:
        plan, O, LSE = bsa.request(state["mask"], *state["args"], q, k, v, row_stride=state["row_stride"], **state["kw"])
    plan.destroy()
    return O, LSE


def work(case):
    """Active token pairs times 4 d flops; Q, K, V and the mask read once, O and LSE written once."""
    nq, nk = _blocks(case)
    H, N, N_kv, d = case["heads"], case["N"], case["N_kv"], case["d"]
    if case["pattern"] == "window":
        w = _window_blocks(case)
        active = H * (w + (nq * nk - w) * case["extra"])
    else:
        active = float(_row_budgets(case).sum())
    pairs = active * (N / nq) * (N_kv / nk)
    mask_bytes = H * nq * (((nk + 31) // 32) * 4 if case["packed"] else nk)
    return {"bytes": 2 * H * d * (2 * N + 2 * N_kv) + 4 * H * N + mask_bytes, "flops": 4.0 * d * pairs}


def tolerance(case):
    # P and O are rounded to the element type once each, sums are fp32; measured against the same rows in 64-bit
    # arithmetic (2.3e-3 in bf16, 2.9e-4 in fp16 on every case), times four
    return {"rel": 1e-2} if case["dtype"] == "bf16" else {"rel": 1.2e-3}


def exact(case, seed):
    """O and LSE by dense masked softmax in 64 bits, a strip of query rows at a time."""
    mask, q, k, v = _inputs(case, seed)
    if case["layout"] == "nhd":
        q, k, v = (t.transpose(0, 1) for t in (q, k, v))
    H, N, N_kv, d = case["heads"], case["N"], case["N_kv"], case["d"]
    O = torch.empty((H, N, d), dtype=torch.float64, device="cuda")
    LSE = torch.empty((H, N), dtype=torch.float64, device="cuda")
    key_block = torch.arange(N_kv, device="cuda") // case["B_KV"]
    strip = max(case["B_Q"], (1 << 28) // N_kv // case["B_Q"] * case["B_Q"])  # 2 GB of scores
    for h in range(H):
        kt, vh = k[h].double().t() / math.sqrt(d), v[h].double()
        for r in range(0, N, strip):
            e = min(N, r + strip)
            off = mask[h, r // case["B_Q"]:-(-e // case["B_Q"])] == 0
            S = q[h, r:e].double() @ kt
            S.masked_fill_(off[:, key_block].repeat_interleave(case["B_Q"], dim=0)[:e - r], -math.inf)
            LSE[h, r:e] = torch.logsumexp(S, dim=1)
            O[h, r:e] = S.sub_(LSE[h, r:e, None]).exp_() @ vh
    return (O if case["layout"] == "hnd" else O.transpose(0, 1).contiguous()), LSE
