"""Decode rows whose heads' softmax is shared out over the warps by keys, 32 of a tile each: contexts on both sides of those edges,
one tile, two and several, group sizes up to the limit and beyond it, parts of rows, and references that grow in one warp alone."""
import pytest

import oracle
from paper_2608_26523_b200 import workloads as W
from parity import compare, run_gpu

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
