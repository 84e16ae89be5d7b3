"""Launches of few work items, whose KV tiles the work decomposition shares out evenly over the SMs: one long context among
short ones, equal ones, a single token, a short chunk deep in a prompt, prefill and decode together, both head-dim families, every
element; and the same launches uncut."""
import pytest
import torch

import oracle
from paper_2608_26523_b200 import api, workloads as W
from parity import compare, run_gpu

pytestmark = pytest.mark.gpu

CASES = [
    # prefix, chunk, (hq, hkv), MLA hq, page
    ([6000, 3, 100, 129, 700], [1] * 5, (16, 2), 128, 16),          # ragged decode rows
    ([1023] * 12, [1] * 12, (8, 8), 128, 64),                       # equal ones
    ([9000], [1], (4, 1), 64, 128),                                 # one token: all SMs on it
    ([8000], [60], (4, 1), 4, 64),                                  # a short chunk deep in a prompt
    ([0], [700], (4, 1), 2, 32),                                    # a first chunk: cuts end at a row's own position
    ([5000, 2000, 1, 900], [1, 70, 200, 1], (8, 2), 16, 64),        # decode rows and chunks in one launch
    ([127, 128, 255, 0], [1, 1, 2, 1], (2, 1), 3, 16),              # hardly any keys
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("mla", [False, True])
def test_balanced_cut_matches_the_oracle(case, mla):
    prefix, chunk, heads, mla_hq, page = CASES[case]
    if mla:
        prob = W.make_problem(9700 + case, prefix, chunk, mla_hq, 1, 576, 512, block_size=page, std=0.5, scale=1.0 / 192 ** 0.5,
                              v_aliases_k=True)
    else:
        prob = W.make_problem(9800 + case, prefix, chunk, heads[0], heads[1], 128, 128, block_size=page, std=0.8)
    rows = oracle.all_rows(prob.chunk_len.numpy(), prob.num_q_heads)
    gpu = prob.to("cuda")
    out, lse, runner = run_gpu(gpu, 0)
    print(compare(out, lse, prob, rows, "cut %d" % case))
    first = out.clone()
    for _ in range(3):                       # (which unit of equal cost comes first is left open; the cuts are not)
        assert torch.equal(runner.run()[0], first)
    out, lse, _ = run_gpu(gpu, 1)
    print(compare(out, lse, prob, rows, "uncut %d" % case))


def test_more_requests_than_the_decomposition_keeps_in_shared_memory():
    R = 1100
    prob = W.make_problem(9900, [(7 * r) % 90 for r in range(R)], [1 + (r % 3) for r in range(R)], 2, 1, 128, 128, block_size=16, std=0.8)
    out, lse, _ = run_gpu(prob.to("cuda"), 0)
    print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), 2), "many requests"))


@pytest.mark.parametrize("chunk", [640, 577, 650])   # whole units, one row more than nine of them, ten of them and a bit
def test_slivers_of_long_shares(chunk):
    """Shares of 33 KV tiles: parts from the fewest tiles worth a start on are cut off."""
    prob = W.make_problem(9950 + chunk, [60000], [chunk], 4, 1, 128, 128, block_size=64, std=0.8)
    rows = oracle.all_rows(prob.chunk_len.numpy(), 4)[::13]
    out, lse, _ = run_gpu(prob.to("cuda"), 0)
    print(compare(out, lse, prob, rows, "slivers %d" % chunk))


def test_forced_splits_of_more_units_than_threads():
    """Uniform splits, placed in rounds: requests of one to four splits, 1100 units."""
    R = 1100
    prob = W.make_problem(9990, [(7 * r) % 500 for r in range(R)], [1 + (r % 3) for r in range(R)], 2, 1, 128, 128, block_size=16, std=0.8)
    out, lse, _ = run_gpu(prob.to("cuda"), 4)
    print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), 2), "many requests, four splits"))
