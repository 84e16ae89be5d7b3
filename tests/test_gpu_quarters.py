"""Decode rows whose heads' softmax is shared out over the warps by keys, 32 of a tile each: contexts on both sides of those edges,
one tile, two and several, group sizes up to the limit and beyond it, parts of rows, references that grow in one warp alone, values and scores that are not finite."""
import numpy as np
import pytest

import oracle
from paper_2608_26523_b200 import workloads as W
from parity import ABS_TOL, LSE_TOL, compare, oracle_rows, packed_index, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [(1, 1), (8, 1), (16, 1), (17, 1), (24, 3), (64, 4)])
@pytest.mark.parametrize("splits", [0, 1, 2])
def test_contexts_around_the_edges_of_quarters(heads, splits):
    ctx = [1, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 160, 255, 256, 257, 289, 383, 385, 513, 700]
    prob = W.make_problem(8950 + heads[0], [c - 1 for c in ctx], [1] * len(ctx), heads[0], heads[1], 128, 128, block_size=16, std=1.0)
    out, lse, _ = run_gpu(prob.to("cuda"), splits)
    print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), heads[0]), "quarters"))


def test_a_reference_that_grows_late_in_one_quarter():
    """Rescales of O in one warp while the others' references stand: keys whose scores rise by far, in different quarters and tiles."""
    prob = W.make_problem(8990, [639], [1], 8, 1, 128, 128, block_size=64, std=0.1)
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
    prob = _edge_problem(ctx, *heads)
    for r, c in enumerate(ctx):
        for pos, feature, v in ((0, 3, "inf"), (c // 2, 64, "-inf"), (c - 1, 127, "inf"), (c // 3, 10, "inf"), (c - 1 - c // 5, 10, "-inf")):
            prob.v_cache[_slot(prob, r, pos) + (slice(None), feature)] = float(v)
    out, lse, _ = run_gpu(prob.to("cuda"), 1)
    rows = oracle.all_rows(prob.chunk_len.numpy(), heads[0])
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
    prob = _edge_problem([ctx] * (len(spans) + 2), 8, 1)
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
    rest = [r for r in range(len(spans) + 2) if r not in bad and r != no_scores]
    print(compare(out, lse, prob, rows[np.isin(rows[:, 0], rest)], "rows beside them"))
