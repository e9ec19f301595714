"""The calls that users of this library make, as cases that can be timed and compared.

A case is one layer's worth of work through the public entry points of ``paper_2604_16429_b200.binding``:

* ``infer``           selection, then the forward of the one-softmax form
* ``train``           the same, then its backward
* ``branches_infer``  selection, then the forward of the three-branch form
* ``branches_train``  the same, then its backward

with, where ``rope`` is set, the rotary embedding of Q and K in front (and, after a backward, its transpose on the
gradients).  ``kept``: the program allocated outputs and workspaces once, as an inference loop does; otherwise the
binding allocates them on every call, as in the README's example and under an autograd function.
"""
from __future__ import annotations

import math

import torch

from paper_2604_16429_b200 import binding as mb
from paper_2604_16429_b200 import flops, synth

D = 64  # head dimension of the library


def _case(name, path, B, H, nlat, nlon, bh, bw, topk, **over):
    c = dict(name=name, path=path, B=B, H=H, Hkv=H, nlat=nlat, nlon=nlon, bh=bh, bw=bw, topk=topk, rlat=1, rlon=1,
             groups=False, f16=False, scale=0.0, rope=False, kept=False, smooth=True)
    c.update(over)
    return c


def _sequence(name, path, B, H, Hkv, tokens, topk, **over):
    """The layout of a token sequence: blocks of 128 contiguous tokens, local attention inside groups of 1024."""
    return _case(name, path, B, H, tokens // 16, 16, 8, 16, topk, Hkv=Hkv, rlat=8, rlon=1, groups=True, **over)


def listed():
    return [
        # a toy grid (32 x 64, i.i.d. inputs): the smallest call, where launches and host time count
        _case("tiny_infer", "infer", 1, 4, 32, 64, 8, 8, 4, kept=True, smooth=False),
        # one layer of one member on the 1.5-degree grid: a deterministic forecast step
        _case("infer_1p5deg", "infer", 1, 8, 120, 240, 8, 8, 8, kept=True),
        # the same for a 24-member ensemble: the batched inference of a probabilistic forecast
        _case("ensemble_1p5deg", "infer", 24, 8, 120, 240, 8, 8, 8, kept=True),
        # one layer on the 0.25-degree grid with 16 x 16 blocks: the largest problem
        _case("infer_0p25deg", "infer", 1, 8, 720, 1440, 16, 16, 16, kept=True),
        # a training step's layer on the 1.5-degree grid
        _case("train_1p5deg", "train", 4, 16, 120, 240, 8, 8, 8),
        # a regional grid with odd numbers of blocks both ways and a caller's softmax scale
        _case("train_ragged", "train", 2, 3, 88, 152, 8, 8, 5, scale=0.1),
        # a wide neighbourhood on 16 x 8 blocks, odd numbers of blocks, grouped-query heads
        _case("infer_wide_ragged", "infer", 3, 6, 176, 216, 16, 8, 7, Hkv=2, rlat=2, rlon=2),
        # three-branch form on the 1.5-degree grid, training
        _case("branches_train_1p5deg", "branches_train", 1, 8, 120, 240, 8, 8, 8),
        # 49152-token sequence with grouped-query heads in binary16 and the rotary embedding: a layer of the
        # finest stage of the U-shaped model, inference of two members
        _sequence("branches_infer_49152", "branches_infer", 2, 12, 3, 49152, 24, f16=True, rope=True, kept=True),
        # the same stage in training
        _sequence("branches_train_49152", "branches_train", 1, 12, 3, 49152, 24, f16=True, rope=True),
        # the middle stage, one-softmax form, training
        _sequence("train_12288", "train", 2, 16, 4, 12288, 12, rope=True),
        # the coarsest stage in training: short sequence, many heads
        _sequence("branches_train_3072", "branches_train", 1, 20, 5, 3072, 4, f16=True, rope=True),
    ]


def draw(rng):
    """One more case of the ranges above: any path, grid layout, block shape, neighbourhood, head grouping and type;
    8 thousand to 4 million (token, head) pairs per call, 1 million in the three-branch form, half a million where a
    backward follows."""
    path = rng.choice(["infer", "infer", "train", "branches_infer", "branches_train"])
    most = 4.0e6 if path == "infer" else 1.0e6 if path == "branches_infer" else 5.0e5
    pairs = math.exp(rng.uniform(math.log(8.0e3), math.log(most)))
    H = rng.choice([1, 2, 3, 4, 5, 6, 8, 12, 16, 20])
    B = rng.choice([1, 1, 1, 2, 3, 4])
    tokens = max(1024.0, pairs / (B * H))
    Hkv = rng.choice([h for h in range(1, H + 1) if H % h == 0 and H // h <= 4])
    common = dict(f16=rng.random() < 0.4, scale=rng.choice([0.0, 0.0, 0.1]), rope=rng.random() < 0.5,
                  kept=rng.random() < 0.5)
    if rng.random() < 0.35:  # token sequence; the last local group may be ragged
        blocks = max(9, round(tokens / 128))
        return {k: v for k, v in _sequence("", path, B, H, Hkv, 128 * blocks, rng.randint(2, 24), **common).items()
                if k != "name"}
    bh, bw = rng.choice([(8, 8), (8, 8), (8, 8), (16, 16), (8, 16), (16, 8)])
    blocks = max(12.0, tokens / (bh * bw))
    nbh = max(3, round(math.sqrt(blocks) * rng.uniform(0.5, 1.0)))
    nbw = max(4, round(blocks / nbh))
    rlat, rlon = rng.choice([(1, 1), (1, 1), (1, 1), (2, 1), (2, 2)])
    c = _case("", path, B, H, nbh * bh, nbw * bw, bh, bw, rng.randint(2, 16), Hkv=Hkv, rlat=rlat, rlon=rlon, **common)
    del c["name"]
    return c


def _workload(c):
    return synth.Workload("case", 0, c["B"], c["H"], c["nlat"], c["nlon"], c["bh"], c["bw"], c["topk"], "smooth", rlat=c["rlat"],
                          rlon=c["rlon"], local_groups=c["groups"], Hkv=c["Hkv"], f16=c["f16"])


def _fields(gen, c, heads):
    """[B, heads, N, 64]: smooth fields (eight waves per head and channel, the same for all members) plus a tenth of
    N(0, 1) per element, or N(0, 1) alone."""
    B, nlat, nlon = c["B"], c["nlat"], c["nlon"]
    dt = torch.float16 if c["f16"] else torch.bfloat16
    out = torch.empty((B, heads, nlat * nlon, D), dtype=dt, device="cuda")
    rand = lambda *s: torch.rand(s, generator=gen, device="cuda")  # noqa: E731
    normal = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    lon, lat = torch.arange(nlon, device="cuda") / nlon, torch.arange(nlat, device="cuda") / nlat
    for h in range(heads):
        if c["smooth"]:
            kx, ky = (rand(D, 8) * 7).floor(), (rand(D, 8) * 7).floor()
            s_lon = torch.sin(2 * math.pi * (kx[..., None] * lon + rand(D, 8)[..., None]))
            c_lat = (normal(D, 8) / math.sqrt(8))[..., None] * torch.cos(
                math.pi * (ky[..., None] * lat + 2 * rand(D, 8)[..., None]))
            base = torch.einsum("cwl,cwo->loc", c_lat, s_lon).reshape(nlat * nlon, D)
        for b in range(B):
            e = normal(nlat * nlon, D)
            out[b, h] = (base + 0.1 * e if c["smooth"] else e).to(dt)
    return out


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    w = _workload(c)
    p = mb.Params.from_workload(w, scale=c["scale"])
    s = {"p": p, "path": c["path"], "rope": c["rope"]}
    s["q"], s["k"], s["v"] = _fields(gen, c, c["H"]), _fields(gen, c, c["Hkv"]), _fields(gen, c, c["Hkv"])
    training, branches = c["path"].endswith("train"), c["path"].startswith("branches")
    if training:
        s["d_o"] = torch.randn(s["q"].shape, generator=gen, device="cuda").to(s["q"].dtype)
    if branches:  # gates are sigmoids of a learned projection
        s["gates"] = torch.sigmoid(torch.randn((p.B, p.H, p.N, 3), generator=gen, device="cuda"))
    if c["rope"]:  # longitude and latitude of every token
        u = torch.rand((p.N, 2), generator=gen, device="cuda")
        s["pos"] = torch.stack([2 * math.pi * u[:, 0], torch.asin(2 * u[:, 1] - 1)], dim=1).contiguous()
        s["neg_pos"] = -s["pos"]
    s["buf"] = {k: {} for k in ("rope", "select", "fwd", "bwd", "rope_t")}
    if c["kept"]:
        b = s["buf"]
        row = lambda: torch.empty((p.B, p.H, p.N), dtype=torch.float32, device="cuda")  # noqa: E731
        if c["rope"]:
            b["rope"] = dict(q_out=torch.empty_like(s["q"]), k_out=torch.empty_like(s["k"]))
        b["select"] = dict(block_idx=torch.empty((p.B, p.H, p.m, p.topk), dtype=torch.int32, device="cuda"),
                           ws=mb.alloc_workspace(p, mb.OP_SELECT))
        b["fwd"] = dict(o=torch.empty_like(s["q"]),
                        ws=mb.alloc_workspace(p, mb.OP_FWD_BRANCHES if branches else mb.OP_FWD))
        b["fwd"].update(dict(lse_fg=row(), lse_l=row()) if branches else dict(lse=row()))
        if training:
            b["bwd"] = dict(dq=torch.empty_like(s["q"]), dk=torch.empty_like(s["k"]), dv=torch.empty_like(s["v"]),
                            ws=mb.alloc_workspace(p, mb.OP_BWD_BRANCHES if branches else mb.OP_BWD))
            if branches:
                b["bwd"]["dgates"] = torch.empty_like(s["gates"])
            if c["rope"]:
                b["rope_t"] = dict(q_out=torch.empty_like(s["q"]), k_out=torch.empty_like(s["k"]))
    return s


def run(state):
    s, b, p = state, state["buf"], state["p"]
    q, k, v = s["q"], s["k"], s["v"]
    out = {}
    if s["rope"]:
        q, k = mb.mosaic_bsa_rope(p, q, k, s["pos"], **b["rope"])
        out["q_rot"], out["k_rot"] = q, k
    idx = out["block_idx"] = mb.mosaic_bsa_select(p, q, k, **b["select"])
    if s["path"].startswith("branches"):
        out["o"], out["lse_fg"], out["lse_l"] = mb.mosaic_bsa_fwd_branches(p, q, k, v, idx, s["gates"], **b["fwd"])
        if s["path"] == "branches_train":
            dq, dk, out["dv"], out["dgates"] = mb.mosaic_bsa_bwd_branches(p, q, k, v, idx, s["gates"], s["d_o"], **b["bwd"])
    else:
        o, lse = out["o"], out["lse"] = mb.mosaic_bsa_fwd(p, q, k, v, idx, **b["fwd"])
        if s["path"] == "train":
            dq, dk, out["dv"] = mb.mosaic_bsa_bwd(p, q, k, v, o, lse, s["d_o"], idx, **b["bwd"])
    if s["path"].endswith("train"):
        if s["rope"]:  # the transpose of a rotation turns the other way
            dq, dk = mb.mosaic_bsa_rope(p, dq, dk, s["neg_pos"], **b["rope_t"])
        out["dq"], out["dk"] = dq, dk
    return out


def work(case):
    """Tensors that come in or go out, once each, and the products of the attended (query block, key block) pairs
    (two in the forward, five in the backward; the same for the block level of the three-branch form)."""
    c, w = case, _workload(case)
    training, branches = c["path"].endswith("train"), c["path"].startswith("branches")
    rows = w.U * w.N
    q, kv = 2 * rows * D, 2 * w.B * w.kv_heads * w.N * D  # bytes of Q, and of K or V
    nbytes = q + 2 * kv + q + 4 * rows + 4 * w.U * w.m * w.topk  # Q, K, V in; O, log-sum-exp, ids out
    if c["rope"]:
        nbytes += q + kv + 8 * w.N  # rotated Q and K out, positions in
    if branches:
        nbytes += 12 * rows + 4 * rows  # gates in, the second log-sum-exp out
    if training:
        nbytes += q + q + 2 * kv + (12 * rows if branches else 0)  # dO in; dQ, dK, dV, gate gradients out
    fwd = flops.fwd_flops(w) + (4.0 * w.m * w.m * D * w.U if branches else 0.0)
    select = 2.0 * w.m * w.m * D * w.U
    return {"bytes": float(nbytes), "flops": fwd * (3.5 if training else 1.0) + select}


def tolerance(case):
    """Against dense masked attention in fp64 (small grids of every path) the outputs were off by at most 3.3e-3 in the
    2-norm and 2.7e-2 in the largest element with bf16 tensors, 4.2e-4 and 3.3e-3 with binary16: the rounding of the
    16-bit operands and results.  The ids of the selection are exact."""
    return {"rel": 1.6e-3, "max": 1.3e-2} if case["f16"] else {"rel": 1.2e-2, "max": 0.1}
