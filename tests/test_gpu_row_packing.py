"""Tiles whose rows are (token, q-head) pairs: every way a kv-head's group fills a tile (whole, in part, with rows left over, one
head at a time), chunk lengths on both sides of a tile's and a unit's tokens, decode rows among them, every element."""
import pytest

import oracle
from paper_2608_26523_b200 import workloads as W
from parity import compare, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group", [1, 2, 3, 5, 6, 7, 11, 16, 42, 48, 64, 128, 130])
def test_groups_and_chunk_lengths_around_a_tile(group):
    per = max((d for d in range(1, min(group, 128) + 1) if group % d == 0 and d * (128 // d) >= 125), default=1)
    tok = 128 // per                                     # tokens of a tile; a unit has twice as many
    chunk = sorted({1, tok - 1, tok, tok + 1, 2 * tok - 1, 2 * tok, 2 * tok + 1, 4 * tok + 3} - {0})
    prefix = [(37 * i) % 300 for i in range(len(chunk))]
    prob = W.make_problem(9500 + group, prefix, chunk, 2 * group if group < 64 else group, 2 if group < 64 else 1, 128, 128,
                          block_size=32, std=0.8)
    for splits in (0, 3):
        out, lse, _ = run_gpu(prob.to("cuda"), splits)
        print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), prob.num_q_heads), "group %d S=%d" % (group, splits)))


def test_units_of_very_different_length_in_one_launch():
    """The item order goes by smaller blocks of units here than when all are about equally long."""
    prob = W.make_problem(9600, [0, 3000, 700, 0], [900, 64, 1, 300], 8, 4, 128, 128, block_size=64, std=0.8)
    out, lse, _ = run_gpu(prob.to("cuda"), 1)
    print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), 8), "ragged units"))


@pytest.mark.parametrize("group,chunk", [(3, 256), (3, 512), (5, 256), (6, 768), (7, 512), (3, 341)])
def test_one_chunk_in_parts_of_its_groups(group, chunk):
    prob = W.make_problem(9650 + group, [500], [chunk], 2 * group, 2, 128, 128, block_size=64, std=0.8)
    for splits in (0, 2):
        out, lse, _ = run_gpu(prob.to("cuda"), splits)
        print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), 2 * group), "group %d, %d tokens, S=%d" % (group, chunk, splits)))
