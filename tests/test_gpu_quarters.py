"""Decode rows whose heads' softmax is shared out over the warps by keys, 32 of a tile each: contexts on both sides of those edges,
one tile, two and several, group sizes up to the limit and beyond it, parts of rows, references that grow in one warp alone, many items
on an SM and items of other kinds between them, values and scores that are not finite."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2608_26523_b200 import workloads as W
from parity import ABS_TOL, LSE_TOL, compare, oracle_rows, packed_index, run_gpu

pytestmark = pytest.mark.gpu


def filled(ctx, heads):
    """The contexts with as many rows of one key behind them as make a batch whose keys are shared out: three items to an SM."""
    return ctx + [1] * max(0, -(-3 * torch.cuda.get_device_properties(0).multi_processor_count // heads[1]) - len(ctx))


@pytest.mark.parametrize("heads", [(1, 1), (8, 1), (16, 1), (17, 1), (24, 3), (64, 4)])
@pytest.mark.parametrize("splits", [0, 1, 2])
def test_contexts_around_the_edges_of_quarters(heads, splits):
    ctx = filled([1, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 160, 255, 256, 257, 289, 383, 385, 513, 700], heads)
    prob = W.make_problem(8950 + heads[0], [c - 1 for c in ctx], [1] * len(ctx), heads[0], heads[1], 128, 128, block_size=16, std=1.0)
    out, lse, _ = run_gpu(prob.to("cuda"), splits)
    print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), heads[0]), "quarters"))


def test_a_reference_that_grows_late_in_one_quarter():
    """References that rise by far, so that each outweighs all before it: the weights at the join.  (What was summed before they grow
    does not show in this result: test_what_was_summed_before_a_reference_grows.)"""
    ctx = filled([640], (8, 1))
    prob = W.make_problem(8990, [c - 1 for c in ctx], [1] * len(ctx), 8, 1, 128, 128, block_size=64, std=0.1)
    for i, pos in enumerate((5, 200, 330, 470, 601, 639)):
        prob.k_cache[int(prob.block_table[0, pos // 64]), pos % 64, 0] = prob.q[0, 0] * (40.0 * (i + 1))
    out, lse, _ = run_gpu(prob.to("cuda"), 1)
    print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), 8), "late"))


def _edge_problem(ctx, hq, hkv):
    return W.make_problem(9010 + hq, [c - 1 for c in ctx], [1] * len(ctx), hq, hkv, 128, 128, block_size=16, std=1.0)


def _slot(prob, r, pos):
    return int(prob.block_table[r, pos // prob.block_size]), pos % prob.block_size


@pytest.mark.parametrize("heads", [(8, 1), (16, 1), (12, 4)])
def test_infinite_values(heads):
    """Values of visible keys may be infinite: the feature is infinite with their sign then (NaN where both signs meet), and the
    other features are what they are.  (A key's value must meet the weights of its own key alone: 0 * inf would be NaN.)"""
    ctx = [1, 40, 128, 129, 300, 513, 700]
    prob = _edge_problem(filled(ctx, heads), *heads)
    for r, c in enumerate(ctx):
        for pos, feature, v in ((0, 3, "inf"), (c // 2, 64, "-inf"), (c - 1, 127, "inf"), (c // 3, 10, "inf"), (c - 1 - c // 5, 10, "-inf")):
            prob.v_cache[_slot(prob, r, pos) + (slice(None), feature)] = float(v)
    out, lse, _ = run_gpu(prob.to("cuda"), 1)
    rows = oracle.all_rows(prob.chunk_len.numpy(), heads[0])
    rows = rows[rows[:, 0] < len(ctx)]
    ref_o, ref_l = oracle_rows(prob, rows)
    ti, hi = packed_index(prob, rows)
    got_o, got_l = out.double().cpu().numpy()[ti, hi], lse.double().cpu().numpy()[ti, hi]
    assert not np.isfinite(ref_o[:, [3, 64, 127, 10]]).any() and np.isinf(ref_o[:, [3, 64, 127]]).sum() > 2 * rows.shape[0]
    fin = np.isfinite(ref_o)
    np.testing.assert_array_equal(got_o[~fin], ref_o[~fin])
    assert np.abs(got_o[fin] - ref_o[fin]).max() <= ABS_TOL      # (values of N(0, 1): averages stay below 4)
    assert (np.abs(got_l - ref_l) / np.maximum(1.0, np.abs(ref_l))).max() <= LSE_TOL


@pytest.mark.parametrize("ctx", [20, 100, 128, 250, 600])
def test_scores_that_are_no_numbers(ctx):
    """A row with a key of NaN has no result, wherever the key is and however many of its neighbours are NaN too; nor has a row
    whose scores are all -inf.  Rows beside them keep theirs."""
    nan, ninf = float("nan"), float("-inf")
    spans = [(0, ctx), (0, 1), (ctx - 1, ctx), (0, min(32, ctx)), (ctx // 2, ctx), (ctx // 128 * 128, ctx // 128 * 128 + min(ctx % 128, 32))]
    prob = _edge_problem(filled([ctx] * (len(spans) + 2), (8, 1)), 8, 1)
    bad = [r for r, (a, b) in enumerate(spans) if b > a]
    for r in bad:
        for pos in range(*spans[r]):
            prob.k_cache[_slot(prob, r, pos)] = nan
    no_scores = len(spans)
    prob.q[no_scores, :, 5] = 1.0
    for pos in range(ctx):
        prob.k_cache[_slot(prob, no_scores, pos) + (0, 5)] = ninf
    out, lse, _ = run_gpu(prob.to("cuda"), 1)
    out, lse = out.cpu(), lse.cpu()
    assert out[bad].isnan().all() and lse[bad].isnan().all()
    assert out[no_scores].isnan().all() and (lse[no_scores] == ninf).all()
    rows = oracle.all_rows(prob.chunk_len.numpy(), 8)
    rest = [r for r in range(prob.num_reqs) if r not in bad and r != no_scores]
    print(compare(out, lse, prob, rows[np.isin(rows[:, 0], rest)], "rows beside them"))


@pytest.mark.parametrize("heads,rows", [((64, 8), 200), ((8, 1), 450), ((8, 1), 290), ((16, 1), 450), ((32, 32), 40)])
def test_many_items_of_a_cta(heads, rows):
    """Several items to an SM one after the other, of one tile, two, three and several, odd and even numbers, in the order of their
    lengths and the ends of long and of one-tile items next to each other: every element."""
    rng = np.random.default_rng(rows + heads[0])
    ctx = rng.choice([1, 7, 31, 32, 33, 64, 100, 127, 128, 129, 200, 256, 257, 300, 384, 385, 400, 530], size=rows)
    # (std 0.5: a result of few keys is off by half an ulp of its own and 2^-9 of the largest value, whose weight is rounded: below 2 that
    # is 3.9e-3 + 4.5e-3 at most, under the tolerance of 1e-2; values of N(0, 1) reach 4.5, and 1.05e-2)
    prob = W.make_problem(9040 + heads[0], [int(c) - 1 for c in ctx], [1] * rows, heads[0], heads[1], 128, 128, block_size=16, std=0.5)
    out, lse, _ = run_gpu(prob.to("cuda"), 1)
    print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), heads[0]), "many items"))


@pytest.mark.parametrize("heads", [(64, 8), (16, 1), (32, 32)])
def test_items_of_every_kind_on_a_cta(heads):
    """More requests than tokens: rows of one token between units of a few tokens and of several hundred, which share barriers, the
    stage and the exchange area with them."""
    rng = np.random.default_rng(heads[0])
    chunk = [0] * 900 + [1] * 150 + [2, 3, 5, 8, 16] * 4 + [300, 130]
    if heads[0] == heads[1]:
        chunk = [0] * 700 + [1] * 40 + [2, 100, 128, 300]
    assert sum(chunk) <= len(chunk)
    order = rng.permutation(len(chunk))
    chunk = [chunk[i] for i in order]
    prefix = [int(rng.choice([0, 1, 30, 100, 127, 128, 250, 400])) if c else 0 for c in chunk]
    # (std 0.5: see above)
    prob = W.make_problem(9060 + heads[0], prefix, chunk, heads[0], heads[1], 128, 128, block_size=16, std=0.5)
    out, lse, _ = run_gpu(prob.to("cuda"), 1)
    print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), heads[0]), "mixed kinds"))


def growing_problem(levels):
    """Scores by design: head h sees every key at log2 weight 0 but for one key of the last tiles, in the tile parity and quarter
    of h, which is `levels[h]` above.  The earlier keys of each quarter and parity, as many as 2^9 together, have values of their
    own about 1, so that what a warp held before its reference grew is a tenth of the result."""
    n_heads, tiles = len(levels), 32
    ctx = filled([tiles * 128], (n_heads, 1))
    prob = W.make_problem(9080, [c - 1 for c in ctx], [1] * len(ctx), n_heads, 1, 128, 128, block_size=128, std=0.1)
    gen = torch.Generator().manual_seed(9081)
    base = torch.randn((2, 4, 128), generator=gen)
    pos = torch.arange(tiles * 128)
    part = base[pos // 128 % 2, pos // 32 % 4]
    k = torch.zeros((tiles * 128, 128))
    v = part + 0.1 * torch.randn((tiles * 128, 128), generator=gen)
    prob.q[0] = 0
    for h, level in enumerate(levels):
        prob.q[0, h, h] = 8.0
        late = (tiles - 2 + (h >> 2 & 1)) * 128 + (h & 3) * 32 + 5 + h
        k[late, h] = level * math.log(2.0) / (8.0 * prob.scale)
    table = prob.block_table[0].long()
    prob.k_cache[table, :, 0] = k.view(tiles, 128, 128).to(torch.bfloat16)
    prob.v_cache[table, :, 0] = v.view(tiles, 128, 128).to(torch.bfloat16)
    return prob


def test_what_was_summed_before_a_reference_grows():
    """Rescales of a warp's O and sum that the result shows: in every quarter of both tile parities, by different factors."""
    prob = growing_problem([8.5, 9.0, 9.5, 10.0, 8.6, 9.2, 9.8, 10.4, 9.4, 8.8, 10.2, 9.6, 9.1, 9.9, 8.7, 9.3])
    out, lse, _ = run_gpu(prob.to("cuda"), 1)
    print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), 16), "rescaled"))
