"""GPU parity of the warp-matrix kernel that AMSKV_PATH_AUTO uses for calls of few items or few queries: edges of its
16-query blocks and 64-key chunks, key sets longer than its ring of stages, several cache ranges, fused appends of
several copies, the never-stored last scale, and the densities from its third product."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2511_16047_b200 import binding as B

from gpu_common import Cache, check_close, make_qkv, oracle_outputs, run_pass, to_items

pytestmark = pytest.mark.gpu

# sides -> T = 4, 9, 16, 25, 36, 49, 64, 81: one to six query blocks, full and partial; the key counts of the layers below run
# from 13 to 285, across the chunk edges, with and without a refilled stage
SIDES = (2, 3, 4, 5, 6, 7, 8, 9)
POLICIES = [(1, 1, False), (2, 3, False), (0, 9, True)]


def _run(D, rows, heads, fused, budgets=None, flags=0, peaked=False, packed=False, density=False):
    qkv = make_qkv(rows, heads, SIDES, D, seed=91, peaked=peaked)
    if packed:
        qkv = [tuple(x.transpose(1, 2).contiguous().transpose(1, 2) for x in t) for t in qkv]
    Ks, Vs = [to_items(k) for _, k, _ in qkv], [to_items(v) for _, _, v in qkv]
    scale = 1.0 / math.sqrt(D)
    with Cache(len(POLICIES), heads, D, rows, SIDES, POLICIES, flags=flags, token_budgets=budgets) as c:
        for k, (q, kk, v) in enumerate(qkv):
            for layer in range(len(POLICIES)):
                out = torch.full_like(q, float("nan"))
                n0 = B.amskv_launch_count()
                if fused:
                    B.amskv_append_attend(c.h, layer, k, kk, v, q, out)
                    assert B.amskv_launch_count() - n0 == 1      # whatever the number of copies of the append
                else:
                    B.amskv_append(c.h, layer, k, kk, v)
                runs = B.amskv_attended_tokens(c.h, layer, k)
                if density:
                    den = torch.full((heads, len(runs)), float("nan"), dtype=torch.float64, device="cuda")
                    B.amskv_attend_density(c.h, layer, k, q, out, den, den.numel())
                elif not fused:
                    B.amskv_attend(c.h, layer, k, q, out)
                torch.cuda.synchronize()
                tokens = [(s, t) for s, first, count in runs for t in range(first, first + count)]
                check_close(out, oracle.attend_tokens(to_items(q), Ks, Vs, tokens, scale),
                            "layer %d scale %d" % (layer, k), max_abs=4e-2 if peaked else 1e-2)
                if density:
                    want = oracle.attention_density(to_items(q), Ks, runs, scale, heads)
                    assert np.allclose(den.cpu().numpy(), want, rtol=2e-4, atol=1e-7), (layer, k)
        assert B.amskv_status(c.h) == 0


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("fused", [False, True], ids=["separate", "fused"])
@pytest.mark.parametrize("rows,heads", [(1, 1), (3, 5)])
def test_blocks_chunks_and_ranges(D, fused, rows, heads):
    _run(D, rows, heads, fused, peaked=True, packed=(rows == 3))


@pytest.mark.parametrize("D", [64, 128])
def test_appends_of_several_copies_are_one_launch(D):
    """Token budgets whose ring wraps inside a scale, a scale cut by its own roll, one larger than the budget."""
    _run(D, 2, 3, True, budgets=[(70, 5), (40, 0), (130, 20)])


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("path", [B.PATH_AUTO, B.PATH_TENSOR_PAIR], ids=["auto", "pair"])
def test_tokens_with_two_places(D, path):
    """Scales that are attended from a slot of their own and also leave tokens in the ring or its pinned head: those tokens are
    written twice by one append, and later scales read them from the ring."""
    budgets = [(58, 12), (40, 30), (70, 60), (100, 95), (45, 20), (30, 7)]
    rows, heads, scale = 2, 3, 1.0 / math.sqrt(D)
    qkv = make_qkv(rows, heads, SIDES, D, seed=106, peaked=True)
    Ks, Vs = [to_items(k) for _, k, _ in qkv], [to_items(v) for _, _, v in qkv]
    twice, read_later = [set() for _ in budgets], [False] * len(budgets)
    with Cache(len(budgets), heads, D, rows, SIDES, [(1, 1, False)] * len(budgets), token_budgets=budgets) as c:
        c.arena.fill_(0x3f)                                    # a place that is not written holds 0.75
        torch.cuda.synchronize()
        c.arena[:4].zero_()                                    # (the status word)
        B.amskv_set_attend_path(c.h, path)
        for k, (q, kk, v) in enumerate(qkv):
            for layer in range(len(budgets)):
                out = torch.full_like(q, float("nan"))
                B.amskv_append_attend(c.h, layer, k, kk, v, q, out)
                runs = B.amskv_attended_tokens(c.h, layer, k)
                copies = sorted((src, src + n) for src, _, n in B.amskv_append_copies(c.h, layer, k))
                if any(b[0] < a[1] for a, b in zip(copies, copies[1:])):
                    twice[layer].add(k)
                read_later[layer] |= any(s in twice[layer] and s != k for s, _, _ in runs)
                tokens = [(s, t) for s, first, count in runs for t in range(first, first + count)]
                check_close(out, oracle.attend_tokens(to_items(q), Ks, Vs, tokens, scale), "layer %d scale %d" % (layer, k), max_abs=4e-2)
        assert B.amskv_status(c.h) == 0
    assert all(read_later)


@pytest.mark.parametrize("D", [64, 128])
def test_never_stored_last_scale(D):
    _run(D, 2, 3, True, flags=B.FLAG_TRANSIENT_LAST_SCALE)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("budgets", [None, [(70, 5), (40, 0), (130, 20)]], ids=["scales", "tokens"])
def test_densities(D, budgets):
    _run(D, 2, 3, False, budgets=budgets, density=True, peaked=True)


def test_item_counts_on_both_sides_of_the_line():
    """The same scale served by this kernel and, with more items, by the paired one."""
    sides, D, heads = (4, 5, 6), 64, 30
    for rows in (2, 13, 17, 60):
        qkv = make_qkv(rows, heads, sides, D, seed=92)
        with Cache(1, heads, D, rows, sides, [(1, 2, False)]) as c:
            for k, (q, kk, v) in enumerate(qkv):
                out = torch.full_like(q, float("nan"))
                B.amskv_append_attend(c.h, 0, k, kk, v, q, out)
                pick = [0, rows * heads // 2, rows * heads - 1]
                got = out.reshape(rows * heads, -1, D)[pick].cpu().double().numpy()
                items = [x.reshape(rows * heads, -1, D)[pick].cpu().double().numpy() for t in qkv[: k + 1] for x in t]
                keep = oracle.keep_set(k, 1, 2, False)
                want = oracle.attend_selected(items[3 * k], items[1::3], items[2::3], keep, 0.125)
                check_close(torch.from_numpy(got), want, "rows %d scale %d" % (rows, k))
            assert B.amskv_status(c.h) == 0


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("path", [B.PATH_AUTO, B.PATH_TENSOR_PAIR], ids=["auto", "pair"])
@pytest.mark.parametrize("fused", [False, True], ids=["separate", "fused"])
def test_one_query_tile_per_sm(D, path, fused):
    """The paired kernel with a query tile per CTA (auto, as many tiles as SMs, 148, at the most): one to three tiles per item with
    full and ragged last ones, up to nine key tiles, fused writes from the CTA of an item's first tile; and the launches
    with one tile too many for it, which take pairs again."""
    sides = (4, 8, 11, 13, 17)                                 # T = 16, 64, 121, 169 (two tiles), 289 (three)
    pols = [(1, 2, False), (0, 9, True)]
    for rows, heads in ((1, 3), (7, 7), (1, 74), (3, 25)):     # 49 x 3 = 147, 74 x 2 = 148, 75 x 2 = 150 tiles
        qkv = make_qkv(rows, heads, sides, D, seed=93, peaked=(rows == 7))
        with Cache(len(pols), heads, D, rows, sides, pols) as c:
            outs = run_pass(c, qkv, path, fused=fused)
            for layer, pol in enumerate(pols):
                items = sorted({0, rows * heads // 2, rows * heads - 1})
                want = oracle_outputs(qkv, pol, 1.0 / math.sqrt(D), items=items)
                for k in range(len(sides)):
                    got = outs[layer][k].reshape(rows * heads, -1, D)[items].cpu().double()
                    check_close(got, want[k], "%d items layer %d scale %d" % (rows * heads, layer, k), max_abs=4e-2 if rows == 7 else 1e-2)


@pytest.mark.parametrize("D", [64, 128])
def test_paired_kernel_writes_an_append_in_pieces(D):
    """Token budgets under the paired kernel: rings that wrap inside a key tile, a head and a ring filled by the same scale,
    scales cut by their own roll, pieces that end inside the last tile.  One launch each; every output of every later scale
    depends on what was written."""
    sides = (2, 8, 8, 9, 11, 8, 13, 12)
    budgets = [(133, 5), (128, 64), (200, 70), (150, 0), (64, 64)]
    pols = [(1, 1, False)] * len(budgets)
    rows, heads = 2, 3
    qkv = make_qkv(rows, heads, sides, D, seed=94)
    Ks, Vs = [to_items(k) for _, k, _ in qkv], [to_items(v) for _, _, v in qkv]
    copies = set()
    with Cache(len(pols), heads, D, rows, sides, pols, token_budgets=budgets) as c:
        B.amskv_set_attend_path(c.h, B.PATH_TENSOR_PAIR)
        for k, (q, kk, v) in enumerate(qkv):
            for layer in range(len(pols)):
                out = torch.full_like(q, float("nan"))
                n0 = B.amskv_launch_count()
                B.amskv_append_attend(c.h, layer, k, kk, v, q, out)
                assert B.amskv_launch_count() - n0 == 1
                copies.add(len(B.amskv_append_copies(c.h, layer, k)))
                tokens = [(s, t) for s, first, count in B.amskv_attended_tokens(c.h, layer, k) for t in range(first, first + count)]
                check_close(out, oracle.attend_tokens(to_items(q), Ks, Vs, tokens, 1.0 / math.sqrt(D)), "layer %d scale %d" % (layer, k))
        assert B.amskv_status(c.h) == 0
    assert copies == {1, 2, 3}


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("rows,heads,path", [(10, 30, B.PATH_TENSOR_PAIR), (10, 30, B.PATH_AUTO), (5, 40, B.PATH_AUTO), (2, 37, B.PATH_AUTO)],
                         ids=["300-pair", "300-auto", "200-auto", "74-auto"])
def test_appends_in_pieces_of_launches_that_fill_the_chip(D, rows, heads, path):
    """The same in the forms of larger launches: 64 channels, two CTAs per SM with pairs of both kinds (150 to 300 units), one CTA per SM
    with two streams of their own tiles (T = 81 and 121 of 200 items) and with one (T = 169 of 74 items, the budget of 200); 128
    channels with one and with two streams."""
    sides = (2, 8, 8, 9, 11, 8, 13, 12)
    budgets = [(133, 5), (128, 64), (200, 70), (150, 0), (64, 64)]
    pols = [(1, 1, False)] * len(budgets)
    n = rows * heads
    pick = [0, 1, n // 2, n - 1]
    qkv = make_qkv(rows, heads, sides, D, seed=104, peaked=True)

    def items(x):
        return x.reshape(n, -1, D)[pick].cpu().double().numpy()

    Ks, Vs = [items(k) for _, k, _ in qkv], [items(v) for _, _, v in qkv]
    copies = set()
    with Cache(len(pols), heads, D, rows, sides, pols, token_budgets=budgets) as c:
        B.amskv_set_attend_path(c.h, path)
        for k, (q, kk, v) in enumerate(qkv):
            for layer in range(len(pols)):
                out = torch.full_like(q, float("nan"))
                n0 = B.amskv_launch_count()
                B.amskv_append_attend(c.h, layer, k, kk, v, q, out)
                assert path == B.PATH_AUTO or B.amskv_launch_count() - n0 == 1
                copies.add(len(B.amskv_append_copies(c.h, layer, k)))
                tokens = [(s, t) for s, first, count in B.amskv_attended_tokens(c.h, layer, k) for t in range(first, first + count)]
                check_close(torch.from_numpy(items(out)), oracle.attend_tokens(items(q), Ks, Vs, tokens, 1.0 / math.sqrt(D)),
                            "layer %d scale %d" % (layer, k), max_abs=4e-2)
        assert B.amskv_status(c.h) == 0
    assert copies == {1, 2, 3}


@pytest.mark.parametrize("fused", [False, True], ids=["separate", "fused"])
@pytest.mark.parametrize("rows,heads,sides", [
    (5, 31, (3, 28)),          # 155 items, seven query tiles: 543 units, 99 left over after three rounds of 148: not split
    (2, 16, (16, 17, 25)),     # 32 items, five query tiles at the end, pairs of both kinds: 80 units: not split
    (1, 150, (5, 27)),         # 150 items, six query tiles (the last ragged): 450 units, six left over
    (8, 11, (12, 25)),         # 88 items, five query tiles: 220 units, of both kinds, 72 left over, 28 of two tiles of an item
    (2, 35, (12, 25)),         # 70 items: 175 units, 27 left over, all of two items' last tiles
])
def test_last_round_shared_by_two_ctas(rows, heads, sides, fused):
    """128 channels, launches whose last round of units is split over clusters of two CTAs: odd and even numbers of key tiles,
    a ragged last query tile, streams with tiles of their own, fused writes from both halves, moving references."""
    D = 128
    pols = [(0, 9, True)]
    qkv = make_qkv(rows, heads, sides, D, seed=95, peaked=True)
    n = rows * heads
    items = sorted({0, 1, n // 2, n - 28, n - 13, n - 2, n - 1})
    with Cache(1, heads, D, rows, sides, pols) as c:
        outs = run_pass(c, qkv, B.PATH_AUTO, fused=fused)
        want = oracle_outputs(qkv, pols[0], 1.0 / math.sqrt(D), items=items)
        for k in range(len(sides)):
            got = outs[0][k].reshape(n, -1, D)[items].cpu().double()
            check_close(got, want[k], "scale %d" % k, max_abs=4e-2)
        again = run_pass(c, qkv, B.PATH_AUTO, fused=fused)
        assert all(torch.equal(x, y) for x, y in zip(outs[0], again[0]))


@pytest.mark.parametrize("rows", [16, 17])
def test_densities_of_one_query_block_with_two_and_with_four_warps(rows):
    """One query block per CTA: two warps with more than four items per SM (148 x 4 = 592), four up to there."""
    sides, heads, D = (1, 3, 4, 4, 4, 4), 37, 64               # 592 and 629 items; one and two key chunks
    qkv = make_qkv(rows, heads, sides, D, seed=98)
    Ks, Vs = [to_items(k) for _, k, _ in qkv], [to_items(v) for _, _, v in qkv]
    with Cache(1, heads, D, rows, sides, [(0, 9, True)]) as c:
        for k, (q, kk, v) in enumerate(qkv):
            B.amskv_append(c.h, 0, k, kk, v)
            runs = B.amskv_attended_tokens(c.h, 0, k)
            out = torch.full_like(q, float("nan"))
            den = torch.full((heads, len(runs)), float("nan"), dtype=torch.float64, device="cuda")
            B.amskv_attend_density(c.h, 0, k, q, out, den, den.numel())
            torch.cuda.synchronize()
            tokens = [(s, t) for s, first, count in runs for t in range(first, first + count)]
            check_close(out, oracle.attend_tokens(to_items(q), Ks, Vs, tokens, 0.125), "scale %d" % k)
            want = oracle.attention_density(to_items(q), Ks, runs, 0.125, heads)
            assert np.allclose(den.cpu().numpy(), want, rtol=2e-4, atol=1e-7), k
        assert B.amskv_status(c.h) == 0


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("side,items", [(6, (148, 150, 296, 300)), (9, (148, 150)), (10, (72, 76)), (11, (42, 46))])
def test_more_ctas_than_are_resident_at_once(D, side, items):
    """T = 36, 81, 100 and 121 at the item counts where the kernel changes: the second wave of its CTAs, and 7 units per SM."""
    sides = (5, side)
    for n in items:
        rows, heads = n // 4 if n % 4 == 0 else n // 2, 4 if n % 4 == 0 else 2
        qkv = make_qkv(rows, heads, sides, D, seed=103)
        pick = [0, n // 2, n - 1]
        for fused in (False, True):
            with Cache(1, heads, D, rows, sides, [(1, 2, False)]) as c:
                outs = run_pass(c, qkv, fused=fused)
                want = oracle_outputs(qkv, (1, 2, False), 1.0 / math.sqrt(D), items=pick)
                for k in range(2):
                    got = outs[0][k].reshape(n, -1, D)[pick].cpu().double()
                    check_close(got, want[k], "%d items scale %d" % (n, k))


@pytest.mark.parametrize("D,sides,rows_of", [(64, (1, 3, 4, 6, 8, 11, 17), (1, 13, 40, 80)), (128, (1, 3, 4, 6, 8, 11, 17), (1, 13, 40, 80)),
                                             (128, (12, 25), (1, 22))])
@pytest.mark.parametrize("path", ["SIMT", "TENSOR", "SMALL", "TENSOR_PAIR", "AUTO"])
def test_an_item_does_not_depend_on_the_values_of_others_nor_beyond_rounding_on_their_number(D, sides, rows_of, path):
    """The items of one image alone and as the last of many, in all forms that the number of items chooses (with 88 items and 128
    channels, a shared last round): bit-equal under every path but AUTO, whose kernels are each within 2.5e-3 of exact sums."""
    heads = 4
    most = make_qkv(rows_of[-1], heads, sides, D, seed=105, peaked=True)
    outs = {}
    for rows in rows_of:
        qkv = [tuple(torch.cat([x[1:rows], x[:1]]) for x in t) for t in most]      # the image is the last of many
        with Cache(1, heads, D, rows, sides, [(2, 2, False)]) as c:
            outs[rows] = [o.double() for o in run_pass(c, qkv, getattr(B, "PATH_" + path), fused=path not in ("SIMT", "TENSOR"))[0]]
            again = run_pass(c, [(t[0], t[1], torch.cat([-t[2][:-1], t[2][-1:]])) for t in qkv], getattr(B, "PATH_" + path),
                             fused=path not in ("SIMT", "TENSOR"))[0]
            assert all(torch.equal(x[-1:], y[-1:].double()) for x, y in zip(outs[rows], again))
    for rows in rows_of[1:]:
        for x, y in zip(outs[1], outs[rows]):
            y = y[-1:]
            if path == "AUTO":
                assert (x - y).norm() <= 5e-3 * x.norm()
            else:
                assert torch.equal(x, y)


@pytest.mark.parametrize("D,side,items", [(64, 8, (184, 186)), (64, 9, (148, 150)), (128, 6, (98, 100)), (128, 8, (98, 100))])
def test_lines_between_the_kernels_of_fused_and_separate_appends(D, side, items):
    """T = 64 of 185 items, T = 81 with and without an SM for every query tile, T = 36 and 64 of 128 channels at two thirds of the SMs:
    the outputs of fused and of separate appends, whatever kernel serves them, against the oracle."""
    sides = (5, side)
    for n in items:
        rows, heads = n // 2, 2
        qkv = make_qkv(rows, heads, sides, D, seed=108)
        pick = [0, n // 2, n - 1]
        want = oracle_outputs(qkv, (1, 2, False), 1.0 / math.sqrt(D), items=pick)
        for fused in (False, True):
            with Cache(1, heads, D, rows, sides, [(1, 2, False)]) as c:
                outs = run_pass(c, qkv, fused=fused)
                for k in range(2):
                    got = outs[0][k].reshape(n, -1, D)[pick].cpu().double()
                    check_close(got, want[k], "%d items scale %d" % (n, k))


@pytest.mark.parametrize("D,side,share", [(64, 8, 240 / 148), (64, 9, 100 / 148), (64, 10, 60 / 148), (128, 6, 60 / 148), (128, 8, 60 / 148)])
def test_fused_and_separate_appends_choose_the_same_kernel(D, side, share):
    """T = 64, 81, 100 and, 128 channels, 36 and 64, at item counts (per SM) that the lines of the warp-matrix kernel leave to it whether
    or not the append is fused: its packed key sequence is then the same, so the outputs are, bit for bit.  (The paired kernel's,
    asked for by its path, are not.)"""
    items = int(torch.cuda.get_device_properties(0).multi_processor_count * share)
    qkv = make_qkv(items, 1, (5, side), D, seed=108, peaked=True)
    outs = []
    with Cache(1, 1, D, items, (5, side), [(1, 2, False)]) as c:
        for path, fused in ((B.PATH_AUTO, False), (B.PATH_AUTO, True), (B.PATH_TENSOR_PAIR, True)):
            outs.append(run_pass(c, qkv, path, fused=fused)[0][1])
    assert torch.equal(outs[0], outs[1])
    assert not torch.equal(outs[1], outs[2])
