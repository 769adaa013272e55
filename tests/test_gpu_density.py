"""GPU parity: amskv_attention_density through the C ABI against the oracle."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2511_16047_b200 import binding as B
from paper_2511_16047_b200 import synth

from gpu_common import Cache, check_close, make_qkv, to_items

pytestmark = pytest.mark.gpu


def _density(cache, layer, k, q, heads):
    runs = B.amskv_attended_tokens(cache.h, layer, k)
    out = torch.full((heads, len(runs)), float("nan"), dtype=torch.float64, device="cuda")
    B.amskv_attention_density(cache.h, layer, k, q, out, out.numel())
    torch.cuda.synchronize()
    return runs, out.cpu().numpy()


@pytest.mark.parametrize("D", [64, 128])
def test_matches_oracle_for_whole_scales_and_token_budgets(D):
    sides, rows, heads = (1, 2, 3, 4, 5, 6, 8), 3, 5
    qkv = make_qkv(rows, heads, sides, D, seed=61, peaked=(D == 64))
    pols = [(2, 2, False), (2, 2, True), (1, 3, False), (2, 2, False), (2, 2, False)]
    budgets = [(0, 0), (0, 0), (0, 0), (40, 5), (13, 3)]
    scale = 1.0 / math.sqrt(D)
    Ks = [to_items(k) for _, k, _ in qkv]
    with Cache(len(pols), heads, D, rows, sides, pols, token_budgets=budgets) as c:
        for k, (q, kk, v) in enumerate(qkv):
            for layer in range(len(pols)):
                B.amskv_append(c.h, layer, k, kk, v)
                runs, got = _density(c, layer, k, q, heads)
                want = oracle.attention_density(to_items(q), Ks, runs, scale, heads)
                assert np.allclose(got, want, rtol=2e-4, atol=1e-7), (layer, k, np.abs(got - want).max())
                counts = np.array([n for _, _, n in runs], dtype=np.float64)
                assert np.allclose(got @ counts, sides[k] ** 2, rtol=1e-5)
        assert B.amskv_status(c.h) == 0


def test_order_and_argument_errors():
    sides, rows, heads, D = (2, 3), 1, 2, 64
    qkv = make_qkv(rows, heads, sides, D, seed=62)
    with Cache(1, heads, D, rows, sides, [(2, 2, False)]) as c:
        q, k, v = qkv[0]
        out = torch.zeros(heads * 2, dtype=torch.float64, device="cuda")
        f = B.lib.amskv_attention_density
        assert f(c.h, 0, 0, q.data_ptr(), None, out.data_ptr(), out.numel(), None) == B.ERR_ORDER
        B.amskv_append(c.h, 0, 0, k, v)
        assert f(c.h, 0, 0, q.data_ptr(), None, out.data_ptr(), 1, None) == B.ERR_NOMEM
        assert f(c.h, 0, 0, q.data_ptr(), None, None, out.numel(), None) == B.ERR_INVALID
        assert f(c.h, 0, 0, q.data_ptr(), None, out.data_ptr(), out.numel(), None) == B.OK
    with Cache(1, heads, D, rows, sides, [(2, 2, False)], flags=B.FLAG_TRANSIENT_LAST_SCALE) as c:
        for kk, (q, k, v) in enumerate(qkv):
            o = torch.empty_like(q)
            B.amskv_append_attend(c.h, 0, kk, k, v, q, o)
        out = torch.zeros(heads * 2, dtype=torch.float64, device="cuda")
        assert B.lib.amskv_attention_density(c.h, 0, 1, q.data_ptr(), None, out.data_ptr(), out.numel(), None) == B.ERR_UNSUPPORTED
        torch.cuda.synchronize()


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("peaked", [False, True], ids=["flat", "peaked"])
def test_density_as_a_by_product_of_the_attention_launch(D, peaked):
    """amskv_attend_density: the output and the density are the oracle's -- whole scales and token budgets, more units than CTAs, query tiles with idle warps, rows whose reference maximum moves (peaked)."""
    from gpu_common import check_close, oracle_outputs
    sides, rows, heads = (1, 2, 3, 5, 6, 8, 13), 6, 40
    qkv = make_qkv(rows, heads, sides, D, seed=63, peaked=peaked)
    pols = [(2, 2, False), (2, 2, True), (1, 3, False), (2, 2, False)]
    budgets = [(0, 0), (0, 0), (0, 0), (120, 5)]
    scale = 1.0 / math.sqrt(D)
    Ks = [to_items(k) for _, k, _ in qkv]
    Vs = [to_items(v) for _, _, v in qkv]
    with Cache(len(pols), heads, D, rows, sides, pols, token_budgets=budgets) as c:
        for k, (q, kk, v) in enumerate(qkv):
            for layer in range(len(pols)):
                B.amskv_append(c.h, layer, k, kk, v)
                runs = B.amskv_attended_tokens(c.h, layer, k)
                den = torch.full((heads, len(runs)), float("nan"), dtype=torch.float64, device="cuda")
                out = torch.full_like(q, float("nan"))
                B.amskv_attend_density(c.h, layer, k, q, out, den, den.numel())
                torch.cuda.synchronize()
                tokens = [(s, t) for s, first, count in runs for t in range(first, first + count)]
                want_out = oracle.attend_tokens(to_items(q), Ks, Vs, tokens, scale)
                check_close(out, want_out, "output, layer %d scale %d" % (layer, k), max_abs=4e-2 if peaked else 1e-2)
                want = oracle.attention_density(to_items(q), Ks, runs, scale, heads)
                got = den.cpu().numpy()
                assert np.allclose(got, want, rtol=2e-4, atol=1e-7), (layer, k, np.abs(got / want - 1).max())
                counts = np.array([n for _, _, n in runs], dtype=np.float64)
                assert np.allclose(got @ counts, sides[k] ** 2, rtol=1e-4)
        assert B.amskv_status(c.h) == 0


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("rows,budgets", [(1, None), (3, None), (2, [(70, 5), (40, 0), (130, 20)])], ids=["r1", "r3", "tokens"])
def test_key_tiles_of_several_runs(D, rows, budgets):
    """The paired kernel packs what whole 64-token tiles leave of each run into tiles of four 16-token boxes: runs of 1, 16,
    49 (four boxes, one key in the last), 64 (none left), 81 and 121 tokens, and the pieces of rings cut anywhere."""
    sides, heads, scale = (1, 4, 7, 8, 9, 11), 3, 1.0 / math.sqrt(D)
    pols = [(1, 1, False), (2, 3, False), (0, 9, True)]
    qkv = make_qkv(rows, heads, sides, D, seed=95, peaked=True)
    Ks, Vs = [to_items(k) for _, k, _ in qkv], [to_items(v) for _, _, v in qkv]
    with Cache(len(pols), heads, D, rows, sides, pols, token_budgets=budgets) as c:
        B.amskv_set_attend_path(c.h, B.PATH_TENSOR_PAIR)
        for k, (q, kk, v) in enumerate(qkv):
            for layer in range(len(pols)):
                B.amskv_append(c.h, layer, k, kk, v)
                runs = B.amskv_attended_tokens(c.h, layer, k)
                out = torch.full_like(q, float("nan"))
                den = torch.full((heads, len(runs)), float("nan"), dtype=torch.float64, device="cuda")
                n0 = B.amskv_launch_count()
                B.amskv_attend_density(c.h, layer, k, q, out, den, den.numel())
                assert B.amskv_launch_count() - n0 == 2      # the result zeroed, one attention launch
                torch.cuda.synchronize()
                tokens = [(s, t) for s, first, count in runs for t in range(first, first + count)]
                check_close(out, oracle.attend_tokens(to_items(q), Ks, Vs, tokens, scale), "layer %d scale %d" % (layer, k), max_abs=4e-2)
                want = oracle.attention_density(to_items(q), Ks, runs, scale, heads)
                assert np.allclose(den.cpu().numpy(), want, rtol=2e-4, atol=1e-7), (layer, k)
        assert B.amskv_status(c.h) == 0


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("path", [B.PATH_AUTO, B.PATH_TENSOR_PAIR], ids=["auto", "pair"])
@pytest.mark.parametrize("peaked", [False, True], ids=["flat", "peaked"])
def test_masses_are_those_of_fp32_probabilities(D, path, peaked):
    """Masses are sums of fp32 probabilities in every kernel, of runs of one key as of long ones: relative to the oracle an
    exponential is off by 2^-22 (its instruction) and by the rounding of its argument, which is at most 2^-24 of a logit's size
    (in units of log 2: under 2 for the flat inputs, under 48 for the peaked ones) times a few roundings; sums of up to 274
    terms in fp32 add less.  Twice that: 1e-6 and 1e-5.  (Probabilities rounded to 16 bits are off by 2e-3, the polynomial that the
    attention outputs take every sixth pair from by up to 8e-4, and two bf16 terms by 8e-6 of one probability.)"""
    sides, rows, heads, scale = (1, 2, 3, 4, 5, 7, 10, 13), 1, 3, 1.0 / math.sqrt(D)
    pols = [(2, 2, False), (0, 9, True)]
    qkv = make_qkv(rows, heads, sides, D, seed=99, peaked=peaked)
    Ks = [to_items(k) for _, k, _ in qkv]
    worst = 0.0
    with Cache(len(pols), heads, D, rows, sides, pols) as c:
        B.amskv_set_attend_path(c.h, path)
        for k, (q, kk, v) in enumerate(qkv):
            for layer in range(len(pols)):
                B.amskv_append(c.h, layer, k, kk, v)
                runs = B.amskv_attended_tokens(c.h, layer, k)
                out = torch.full_like(q, float("nan"))
                den = torch.full((heads, len(runs)), float("nan"), dtype=torch.float64, device="cuda")
                B.amskv_attend_density(c.h, layer, k, q, out, den, den.numel())
                torch.cuda.synchronize()
                want = oracle.attention_density(to_items(q), Ks, runs, scale, heads)
                worst = max(worst, np.abs(den.cpu().numpy() / want - 1).max())
    assert worst <= (1e-5 if peaked else 1e-6), worst


@pytest.mark.parametrize("side", [4, 10])
def test_a_result_in_pageable_host_memory_is_refused(side):
    """As a fill of it is; nothing is launched and the cache stays usable."""
    qkv = make_qkv(1, 2, (side,), 64, seed=100)
    q, kk, v = qkv[0]
    with Cache(1, 2, 64, 1, (side,), [(1, 1, True)]) as c:
        B.amskv_append(c.h, 0, 0, kk, v)
        out = torch.empty_like(q)
        runs = B.amskv_attended_tokens(c.h, 0, 0)
        host = np.full(2, np.nan)
        n0 = B.amskv_launch_count()
        assert B.lib.amskv_attend_density(c.h, 0, 0, q.data_ptr(), out.data_ptr(), None, None, host.ctypes.data_as(B.ctypes.c_void_p),
                                          2, None) == B.ERR_CUDA
        assert B.amskv_launch_count() == n0
        den = torch.full((2, 1), float("nan"), dtype=torch.float64, device="cuda")
        B.amskv_attend_density(c.h, 0, 0, q, out, den, 2)
        torch.cuda.synchronize()
        want = oracle.attention_density(to_items(q), [to_items(kk)], runs, 0.125, 2)
        assert np.allclose(den.cpu().numpy(), want, rtol=1e-5)
        assert B.amskv_status(c.h) == 0


@pytest.mark.parametrize("D", [64, 128])
def test_a_single_token_with_several_keys_keeps_fp32_probabilities(D):
    """The output of the call with densities is amskv_attend's bit for bit: the CUDA-core kernel's, which rounds no probability."""
    sides, rows, heads = (3, 1, 5, 1, 1), 2, 3
    qkv = make_qkv(rows, heads, sides, D, seed=101, peaked=True)
    with Cache(1, heads, D, rows, sides, [(0, 9, True)]) as c:
        for k, (q, kk, v) in enumerate(qkv):
            B.amskv_append(c.h, 0, k, kk, v)
            runs = B.amskv_attended_tokens(c.h, 0, k)
            den = torch.zeros((heads, len(runs)), dtype=torch.float64, device="cuda")
            out, want = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
            B.amskv_attend_density(c.h, 0, k, q, out, den, den.numel())
            B.amskv_attend(c.h, 0, k, q, want)
            torch.cuda.synchronize()
            if sides[k] == 1:
                assert torch.equal(out, want)
        assert B.amskv_status(c.h) == 0


@pytest.mark.parametrize("D,sides,items", [(64, (1, 2), (1480, 1488)), (128, (1, 2), (296, 304, 740, 744)), (128, (2, 3, 4), (740, 744))])
def test_one_query_block_on_both_sides_of_the_lines(D, sides, items):
    """Single tokens, four and more queries at the item counts where the kernel changes (10, 2 and 5 per SM of 148): the
    densities of an item do not depend on it."""
    for n in items:
        heads, scale = 8, 1.0 / math.sqrt(D)
        rows = n // heads
        qkv = make_qkv(rows, heads, sides, D, seed=102)
        with Cache(1, heads, D, rows, sides, [(0, 9, True)]) as c:
            for k, (q, kk, v) in enumerate(qkv):
                B.amskv_append(c.h, 0, k, kk, v)
                runs = B.amskv_attended_tokens(c.h, 0, k)
                out = torch.full_like(q, float("nan"))
                den = torch.full((heads, len(runs)), float("nan"), dtype=torch.float64, device="cuda")
                B.amskv_attend_density(c.h, 0, k, q, out, den, den.numel())
                torch.cuda.synchronize()
                Ks, Vs = [to_items(t[1]) for t in qkv[:k + 1]], [to_items(t[2]) for t in qkv[:k + 1]]
                check_close(out, oracle.attend_tokens(to_items(q), Ks, Vs, [(s, t) for s, f, m in runs for t in range(f, f + m)], scale),
                            "%d items, scale %d" % (n, k))
                assert np.allclose(den.cpu().numpy(), oracle.attention_density(to_items(q), Ks, runs, scale, heads), rtol=1e-6), (n, k)
            assert B.amskv_status(c.h) == 0
