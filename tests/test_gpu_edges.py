"""GPU parity at the edges of the kernels' tiles and of their launch rules, against the oracle, through the C ABI: the
sizes on both sides of every line at which a kernel changes its width, its split or its work queue.  Tolerances are those
of the full tests: ids and rotated values exact (one 16-bit step at rounding ties), outputs and gradients the bounds of
the shared helpers."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2604_16429_b200 import binding as mb
from paper_2604_16429_b200 import synth
from tests import gpu_util as G
from tests import test_gpu_rope as R
from tests import test_gpu_three_branch as T

pytestmark = pytest.mark.gpu


def _name(w):
    return f"m{w.m}_k{w.topk}_U{w.U}" if hasattr(w, "m") else str(w)


# Ranking: 16 query blocks per CTA, 32 from 296 CTAs of 32 on (148 units of 33 blocks), 64 keys per chunk; room for 96
# survivors per row, 192 beyond top-k 16.  Pooling: 2, 4 or 8 channels per lane from 75000 / 16 and 75000 / 8 pooled
# blocks on (Q and K together).
RANK = [synth.small_case(8 * a, 8 * b, 8, 8, k, H=h, seed=300 + i) for i, (a, b, k, h) in enumerate([
    (3, 5, 16, 1), (4, 4, 4, 2), (17, 1, 17, 1), (3, 21, 16, 1), (8, 8, 17, 1), (5, 13, 32, 2), (3, 43, 31, 1),
    (3, 11, 16, 147), (3, 11, 16, 148), (3, 11, 17, 148), (3, 11, 32, 71), (1, 11, 8, 213), (1, 11, 8, 214), (1, 11, 8, 426),
    (1, 11, 8, 427)])] + [synth.small_case(24, 176, 8, 16, 5, H=h, seed=320 + h) for h in (1, 100, 148)]


@pytest.mark.parametrize("w", RANK, ids=_name)
def test_ranking_and_pooling_at_tile_and_rule_edges(w):
    x = synth.make_inputs(w)
    got = G.gpu_select(w, G.device_inputs(x)).cpu().numpy()
    want = G.oracle_select_all(w, x)
    assert np.array_equal(got, want), f"{(got != want).sum()} of {want.size} ids differ"


@pytest.mark.parametrize("offset", [1.0, 16.0, 64.0])
def test_ranking_of_vectors_with_a_large_common_part(offset):
    """A constant on every channel of Q and K: all scores of a row are alike in their leading bits, down to below the width
    of the screening's bounds, so that from few to all rows keep more candidates than there is room for and score every key."""
    w = synth.small_case(3072, 16, 8, 16, 24, H=2, kind="smooth", seed=335)
    x = synth.make_inputs(w)
    for n in ("q", "k"):
        x[n] = synth.to_bf16_bits(synth.bf16_bits_to_f32(x[n]) + np.float32(offset))
    got = G.gpu_select(w, G.device_inputs(x)).cpu().numpy()
    want = G.oracle_select_all(w, x)
    assert np.array_equal(got, want), f"{(got != want).sum()} of {want.size} ids differ"


# Work queue of the row-stationary kernels on 148 SMs: the items left over after full waves are cut into four parts up to
# 37 of them, into two up to 74.  One item per unit here (2 x 2 blocks, and three blocks in a row, whose fourth part is empty).
QUEUE = [(16, 16, h) for h in (1, 37, 38, 74, 75, 148, 149, 593, 630)] + [(8, 24, h) for h in (1, 38, 75, 594, 631)]


@pytest.mark.parametrize("nlat,nlon,heads", QUEUE)
def test_left_over_items_in_parts(nlat, nlon, heads):
    w = synth.small_case(nlat, nlon, 8, 8, 2, H=heads, seed=340 + heads, rlat=0, rlon=0, backward=True)
    x = synth.make_inputs(w)
    dx = G.device_inputs(x)
    idx = G.gpu_select(w, dx)
    o, lse = G.gpu_fwd(w, dx, idx)
    grads = G.gpu_bwd(w, dx, o, lse, idx)
    gates = np.random.default_rng(heads).standard_normal((1, heads, w.N, 3))
    three = T._run(w, x, idx, gates)
    assert all(bool(torch.isfinite(t.float()).all()) for t in (o, lse, *grads)) and np.isfinite(three[0]).all()
    idx_h = idx.cpu().numpy()
    units = range(heads) if heads <= 12 else [0, 1, heads // 2, *range(heads - 4, heads)]
    for h in units:
        G.compare_fwd_unit(w, x, 0, h, idx_h[0, h], o, lse)
        ref = oracle.bwd(G.geom_of(w), x["q"][0, h], x["k"][0, h], x["v"][0, h], x["do"][0, h], idx_h[0, h])
        for name, got, want in zip(("dQ", "dK", "dV"), grads, ref):
            G.assert_bwd_close(f"{name} unit {h}", got[0, h], want)
    _compare3_units(w, x, idx_h, gates, three, units, T._compare)


def _compare3_units(w, x, idx_h, gates, got, units, compare):
    """A three-branch comparison of some units only (one key/value head per query head)."""
    one = dataclasses.replace(w, H=1, Hkv=0)
    for h in units:
        s = slice(h, h + 1)
        compare(one, {k: v[:, s] for k, v in x.items()}, idx_h[:, s], gates[:, s], [t[:, s] for t in got])


@pytest.mark.parametrize("nlat,nlon,heads,topk", [(16, 16, 37, 0), (16, 16, 74, 0), (16, 16, 80, 0), (16, 16, 444, 0), (8, 24, 38, 3),
                                                  (16, 16, 37, 4), (64, 64, 5, 4)])
def test_lists_that_a_tile_does_not_attend(nlat, nlon, heads, topk):
    """Without selected blocks every list of the selection branch is empty, and a part of an item leaves one tile empty in
    both of its lists: the roles of a tile that has nothing to do stay in step, pass after pass.  No block is selected here
    (top-k 0, or rows of -1); on the largest grid every fourth row selects one."""
    w = synth.small_case(nlat, nlon, 8, 8, topk, H=heads, seed=350 + heads, rlat=0, rlon=0, backward=True)
    x = synth.make_inputs(w)
    idx_h = np.full((1, heads, w.m, topk), -1, np.int32)
    if w.m > 4:
        idx_h[:, :, ::4, 1] = (np.arange(0, w.m, 4) + 5) % w.m
    idx = torch.from_numpy(idx_h).cuda()
    gates = np.random.default_rng(heads).standard_normal((1, heads, w.N, 3))
    first = T._run(w, x, idx, gates), T._run_bwd3(w, x, idx, gates)
    units = sorted({0, heads // 2, heads - 1})
    _compare3_units(w, x, idx_h, gates, first[0], units, T._compare)
    _compare3_units(w, x, idx_h, gates, first[1], units, T._compare_bwd3)
    for _ in range(20):
        for run, want in zip((T._run, T._run_bwd3), first):
            assert all(np.array_equal(a, b) for a, b in zip(run(w, x, idx, gates), want))


# A unit's bits depend on its own inputs only: not on its place in the batch, nor on how many units there are, by which the
# work queue cuts items into parts (every number on 148 SMs: 8 units of 113 items leave 16, cut into four; one unit is not cut;
# 2 leave 78, not cut, 3 leave 43, cut into two; 7 items are cut into four, 70 into two, 77 not).  The block level sums
# 450, 21, 24, 15 and 8 blocks in four, one, one, one and one parts.
ALONE = [(synth.small_case(120, 240, 8, 8, 8, kind="smooth", seed=501, backward=True), (1, 3, 8)),
         (synth.small_case(24, 56, 8, 8, 5, seed=502, backward=True), (1, 7, 10, 11)),                 # ragged groups
         (synth.small_case(192, 16, 8, 16, 4, seed=503, rlat=8, rlon=1, local_groups=True, backward=True), (1, 6, 8, 13)),
         (synth.small_case(24, 80, 8, 16, 3, seed=504, backward=True), (1, 6, 12)),
         (synth.small_case(32, 64, 16, 16, 3, seed=505, backward=True), (1, 8, 10))]


@pytest.mark.parametrize("w,counts", ALONE, ids=_name)
def test_a_units_bits_do_not_depend_on_the_other_units(w, counts):
    gen = torch.Generator("cuda").manual_seed(w.cfg)
    one = G.device_inputs(synth.make_inputs(w))
    gates = torch.randn((1, 1, w.N, 3), device="cuda", generator=gen)
    want = None
    for n in counts:
        wn = dataclasses.replace(w, H=n)
        dx = {k: torch.cat([v] + [torch.randn(v.shape, device="cuda", generator=gen).to(v.dtype)] * (n - 2) + [v] * (n > 1), dim=1)
              for k, v in one.items()}
        idx = G.gpu_select(wn, dx)
        o, lse = G.gpu_fwd(wn, dx, idx)
        p, gt = mb.Params.from_workload(wn), gates.expand(1, n, w.N, 3).contiguous()
        three = mb.mosaic_bsa_fwd_branches(p, dx["q"], dx["k"], dx["v"], idx, gt)
        three += mb.mosaic_bsa_bwd_branches(p, dx["q"], dx["k"], dx["v"], idx, gt, dx["do"])
        got = [idx, o, lse, *G.gpu_bwd(wn, dx, o, lse, idx), *three]
        want = [t[:, 0].clone() for t in got] if want is None else want
        for i, (t, ref) in enumerate(zip(got, want)):
            assert torch.equal(t[:, 0], ref) and torch.equal(t[:, -1], ref), (n, i)


# Block level of the three-branch form: 64 x 64 tiles, a tile's streams over a cluster of 1, 2 or 4 CTAs (at most one per
# chunk; on the key side the chunks of all query heads of a group count).
COMPRESS = [synth.small_case(8 * m, 8, 8, 8, 2, H=h, Hkv=kv, seed=360 + i, backward=True) for i, (m, h, kv) in enumerate([
    (63, 1, 0), (64, 1, 0), (65, 1, 0), (129, 1, 0), (193, 1, 0), (449, 1, 0), (65, 4, 1), (65, 6, 2)])]


@pytest.mark.parametrize("w", COMPRESS, ids=_name)
def test_block_level_tiles_and_cluster_sizes(w):
    x = synth.make_inputs(w)
    idx = G.gpu_select(w, G.device_inputs(x))
    gates = np.random.default_rng(w.cfg).standard_normal((w.B, w.H, w.N, 3))
    if not w.Hkv:
        T._compare(w, x, idx.cpu().numpy(), gates, T._run(w, x, idx, gates))
    T._compare_bwd3(w, x, idx.cpu().numpy(), gates, T._run_bwd3(w, x, idx, gates))


@pytest.mark.parametrize("heads", [16, 40, 148])
def test_block_level_many_units(heads):
    """Gated pooling with 2, 4 and 8 channels per lane (4 * heads * 65 pooled blocks), and with 148 units a block level of
    many CTAs per SM."""
    w = synth.small_case(40, 104, 8, 8, 3, H=heads, seed=380 + heads, backward=True)
    x = synth.make_inputs(w)
    idx = G.gpu_select(w, G.device_inputs(x))
    gates = np.random.default_rng(w.cfg).standard_normal((w.B, w.H, w.N, 3))
    got = T._run_bwd3(w, x, idx, gates)
    assert all(np.isfinite(t).all() for t in got)
    _compare3_units(w, x, idx.cpu().numpy(), gates, got, (0, heads - 1), T._compare_bwd3)


@pytest.mark.parametrize("topk", [1, 3, 7, 17, 32])
def test_transposed_lists_for_any_topk(topk):
    """A warp of the transposed-pattern kernel takes 32 / topk rows at a time; rows of repeated, local and absent ids."""
    w = synth.small_case(40, 56, 8, 8, topk, H=1, seed=400 + topk, backward=True)
    x = synth.make_inputs(w)
    dx = G.device_inputs(x)
    idx = G.gpu_select(w, dx)
    idx[0, 0, 9, :] = -1
    clean = idx.clone()
    if topk > 2:                                            # the oracle gets the rows without the ids that are to be skipped
        idx[0, 0, 12, 1] = idx[0, 0, 12, 0]                 # a repeat
        idx[0, 0, 13, 2] = 13                               # the block itself, local already
        clean[0, 0, 12, 1] = clean[0, 0, 13, 2] = -1
    idx_h = clean.cpu().numpy()
    p = mb.Params.from_workload(w)
    ws = mb.alloc_workspace(p, mb.OP_FWD)
    o, lse = mb.mosaic_bsa_fwd(p, dx["q"], dx["k"], dx["v"], idx, ws=ws)
    ws = mb.alloc_workspace(p, mb.OP_BWD)
    grads = mb.mosaic_bsa_bwd(p, dx["q"], dx["k"], dx["v"], o, lse, dx["do"], idx, ws=ws)
    ref = oracle.bwd(G.geom_of(w), x["q"][0, 0], x["k"][0, 0], x["v"][0, 0], x["do"][0, 0], idx_h[0, 0])
    for name, got, want in zip(("dQ", "dK", "dV"), grads, ref):
        G.assert_bwd_close(name, got[0, 0], want)


@pytest.mark.parametrize("bh,bw,nlat,nlon", [(8, 8, 64, 64), (8, 16, 64, 128)])
def test_a_tile_that_skips_most_of_its_items_list(bh, bw, nlat, nlon):
    """The two tiles of an item walk their own entries of a merged list of 64, and rows without entries stand beside full ones.
    (The planner pairs the blocks that have most in common, so the two tiles take turns; with one unit every item is cut into
    parts.  Lists whose tiles wait for one another over the whole key ring: test_lists_of_very_different_lengths.)"""
    w = synth.small_case(nlat, nlon, bh, bw, 30, H=1, seed=420 + bw, rlat=0, rlon=0, backward=True)
    x = synth.make_inputs(w)
    dx = G.device_inputs(x)
    nbw = nlon // bw
    idx_h = np.full((1, 1, w.m, 30), -1, np.int32)
    for y in range(0, nlat // bh, 2):
        for c in range(0, nbw, 2):
            far = [j for j in range(w.m) if j not in (y * nbw + c, y * nbw + c + 1, (y + 1) * nbw + c, (y + 1) * nbw + c + 1)]
            idx_h[0, 0, y * nbw + c] = far[:30]
            idx_h[0, 0, y * nbw + c + 1] = far[30:60]
            idx_h[0, 0, (y + 1) * nbw + c, :2] = [far[0], far[59]]
            idx_h[0, 0, (y + 1) * nbw + c + 1, :1] = [far[59]]
    idx_h[0, 0, -1, :] = -1
    idx = torch.from_numpy(idx_h).cuda()
    o, lse = G.gpu_fwd(w, dx, idx)
    G.compare_fwd_unit(w, x, 0, 0, idx_h[0, 0], o, lse)
    grads = G.gpu_bwd(w, dx, o, lse, idx)
    ref = oracle.bwd(G.geom_of(w), x["q"][0, 0], x["k"][0, 0], x["v"][0, 0], x["do"][0, 0], idx_h[0, 0])
    for name, got, want in zip(("dQ", "dK", "dV"), grads, ref):
        G.assert_bwd_close(name, got[0, 0], want)
    gates = np.random.default_rng(w.cfg).standard_normal((1, 1, w.N, 3))
    T._compare(w, x, idx_h, gates, T._run(w, x, idx, gates))
    T._compare_bwd3(w, x, idx_h, gates, T._run_bwd3(w, x, idx, gates))


@pytest.mark.parametrize("bh,bw,nlat,nlon,heads,f16", [(8, 8, 64, 64, 5, False), (8, 16, 64, 128, 3, False), (16, 8, 128, 64, 3, True)])
def test_lists_of_very_different_lengths(bh, bw, nlat, nlon, heads, f16):
    """The key ring goes round several times between two entries of a tile: in every other 2 x 2 group the upper two blocks
    (128-token blocks: the left one of a pair) select 56 blocks of which the lower two (the right one) select none, the first
    or the last; four common blocks make sure that the two long lists share a tile.  The other groups' rows have 0, 1 or 30
    entries at random.  80 and 96 items, which the work queue does not cut."""
    w = synth.small_case(nlat, nlon, bh, bw, 30, H=heads, seed=430 + bw + bh, rlat=0, rlon=0, backward=True, f16=f16)
    x = synth.make_inputs(w)
    dx = G.device_inputs(x, f16=f16)
    nbh, nbw = nlat // bh, nlon // bw
    rng = np.random.default_rng(w.cfg)
    idx_h = np.full((1, heads, w.m, 30), -1, np.int32)
    for n, (h, y, c) in enumerate((h, y, c) for h in range(heads) for y in range(0, nbh, 2) for c in range(0, nbw, 2)):
        own = [y * nbw + c, y * nbw + c + 1, (y + 1) * nbw + c, (y + 1) * nbw + c + 1]
        far = [int(j) for j in rng.permutation([j for j in range(w.m) if j not in own])]
        if n % 2:
            rows = [list(rng.permutation(far)[:k]) for k in rng.choice([0, 1, 30], size=4)]
        else:
            long = [far[:30], far[26:56]]
            short = [[far[0]] if n & 2 else [], [far[55]] if n & 4 else []]
            rows = long + short if bh * bw == 64 else [long[0], short[0], long[1], short[1]]
        for j, r in zip(own, rows):
            idx_h[0, h, j, :len(r)] = r
    idx = torch.from_numpy(idx_h).cuda()
    o, lse = G.gpu_fwd(w, dx, idx)
    grads = G.gpu_bwd(w, dx, o, lse, idx)
    for h in range(heads):
        G.compare_fwd_unit(w, x, 0, h, idx_h[0, h], o, lse)
        ref = oracle.bwd(G.geom_of(w), x["q"][0, h], x["k"][0, h], x["v"][0, h], x["do"][0, h], idx_h[0, h])
        for name, got, want in zip(("dQ", "dK", "dV"), grads, ref):
            G.assert_bwd_close(f"{name} unit {h}", got[0, h], want)
    if not f16:
        gates = rng.standard_normal((1, heads, w.N, 3))
        _compare3_units(w, x, idx_h, gates, T._run(w, x, idx, gates), range(heads), T._compare)
        _compare3_units(w, x, idx_h, gates, T._run_bwd3(w, x, idx, gates), range(heads), T._compare_bwd3)


@pytest.mark.parametrize("f16", [False, True])
@pytest.mark.parametrize("heads,kv", [(1, 1), (6, 1), (7, 1), (6, 6), (24, 1), (15, 15)])
def test_rope_unit_shares_and_non_finite_values(heads, kv, f16):
    """Short sequences split the units over blocks from eight units on (shares that end inside Q's or K's units, or run
    over their border); infinities and NaNs take the plain conversion, subnormals and zeros the exact scaled one."""
    w = synth.small_case(24, 40, 8, 8, 2, H=heads, Hkv=kv, seed=440 + heads, f16=f16)
    x = synth.make_inputs(w)
    inf = 0x7C00 if f16 else 0x7F80
    for a in (x["q"], x["k"]):
        a[0, :, 5, :8] = [inf, inf | 0x8000, inf | 1, 0, 0x8000, 1, 0x8001, inf - 1]
    pos = R._positions(w, np.random.default_rng(w.cfg))
    p = mb.Params.from_workload(w)
    dx = G.device_inputs(x, f16=f16)
    out = mb.mosaic_bsa_rope(p, dx["q"], dx["k"], torch.from_numpy(pos).cuda())
    g = G.geom_of(w)
    total = same = 0
    for got, src in zip(out, (x["q"], x["k"])):
        bits = got.view(torch.int16).cpu().numpy().view(np.uint16)
        for h in range(src.shape[1]):
            _, want = oracle.rope(g, src[0, h], pos.astype(np.float64))
            nan = (want & 0x7FFF) > inf
            assert np.array_equal(nan, (bits[0, h] & 0x7FFF) > inf)
            dist = np.abs(R._ordered(bits[0, h]) - R._ordered(want))[~nan]
            assert dist.max() <= 1
            total += dist.size
            same += int((dist == 0).sum())
    assert same >= 0.9999 * total


@pytest.mark.parametrize("nlat,nlon,heads", [(16, 24, 2), (64, 128, 4), (120, 160, 6)])
def test_passes_back_to_back_on_the_same_buffers(nlat, nlon, heads):
    """Launches overlap the kernel ahead of them: passes over two inputs in turn, with one workspace and one set of outputs
    and no synchronisation between them, give the bits of passes that ran alone."""
    w = synth.small_case(nlat, nlon, 8, 8, 3, H=heads, seed=460 + heads, backward=True)
    p = mb.Params.from_workload(w)
    xs = [G.device_inputs(synth.make_inputs(dataclasses.replace(w, cfg=w.cfg + 7 * i))) for i in range(2)]
    gates = torch.randn((1, heads, w.N, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(heads))
    ws = torch.empty(max(mb.workspace_bytes(p, op) for op in range(5)), dtype=torch.uint8, device="cuda")
    idx = torch.empty((1, heads, w.m, 3), dtype=torch.int32, device="cuda")
    o, lse = torch.empty_like(xs[0]["q"]), torch.empty((1, heads, w.N), device="cuda")
    grads, three, dg = [[torch.empty_like(o) for _ in range(3)] for _ in range(2)] + [torch.empty_like(gates)]
    pos = torch.rand((w.N, 2), device="cuda", generator=torch.Generator("cuda").manual_seed(heads + 1))
    qr, kr, o3, lse3 = torch.empty_like(o), torch.empty_like(o), torch.empty_like(o), [torch.empty_like(lse) for _ in range(2)]

    def run(x):
        mb.mosaic_bsa_rope(p, x["q"], x["k"], pos, q_out=qr, k_out=kr)
        mb.mosaic_bsa_select(p, qr, kr, block_idx=idx, ws=ws)
        mb.mosaic_bsa_fwd_branches(p, qr, kr, x["v"], idx, gates, o=o3, lse_fg=lse3[0], lse_l=lse3[1], ws=ws)
        mb.mosaic_bsa_fwd(p, x["q"], x["k"], x["v"], idx, o=o, lse=lse, ws=ws)
        mb.mosaic_bsa_bwd(p, x["q"], x["k"], x["v"], o, lse, x["do"], idx, dq=grads[0], dk=grads[1], dv=grads[2], ws=ws)
        mb.mosaic_bsa_bwd_branches(p, x["q"], x["k"], x["v"], idx, gates, x["do"], dq=three[0], dk=three[1], dv=three[2],
                                   dgates=dg, ws=ws)
        return [t.clone() for t in (qr, kr, idx, o3, *lse3, o, lse, *grads, *three, dg)]

    alone = []
    for x in xs:
        torch.cuda.synchronize()
        alone.append(run(x))
    torch.cuda.synchronize()
    for i, got in enumerate([run(xs[i % 2]) for i in range(6)]):
        for a, b in zip(got, alone[i % 2]):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), i
