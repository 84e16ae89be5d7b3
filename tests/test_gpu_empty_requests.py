"""Batches of more requests than tokens (a server's fixed slots, most of them empty), whose requests with tokens have one, a few
or many of them: every element, over the groups of q-heads that fill a tile in different ways, uncut and cut, and as key ranges
that are merged afterwards."""
import pytest
import torch

import oracle
from paper_2608_26523_b200 import api, workloads as W
from parity import compare, run_gpu

pytestmark = pytest.mark.gpu

CHUNKS = [[2, 0], [5, 1, 1, 0, 0, 0, 0, 0], [0] * 99 + [100] + [0] * 156, [1, 0, 3, 0, 0, 1, 0, 0, 20, 0, 1, 0] + [0] * 30]


def _problem(chunk, group, hkv=2):
    prefix = [300 + 61 * (i % 7) if c else 5 for i, c in enumerate(chunk)]
    return W.make_problem(9700 + group + len(chunk), prefix, chunk, hkv * group, hkv, 128, 128, block_size=16, std=0.8)


@pytest.mark.parametrize("chunk", CHUNKS, ids=lambda c: "%dof%d" % (sum(c), len(c)))
@pytest.mark.parametrize("group", [1, 3, 8, 16])
def test_more_requests_than_tokens(chunk, group):
    assert sum(chunk) <= len(chunk)
    prob = _problem(chunk, group)
    gpu = prob.to("cuda")
    rows = oracle.all_rows(prob.chunk_len.numpy(), prob.num_q_heads)
    for splits in (0, 1, 3):
        out, lse, _ = run_gpu(gpu, splits)
        print(compare(out, lse, prob, rows, "S=%d" % splits))


@pytest.mark.parametrize("chunk", CHUNKS, ids=lambda c: "%dof%d" % (sum(c), len(c)))
@pytest.mark.parametrize("group", [1, 8])
def test_key_ranges_of_more_requests_than_tokens(chunk, group):
    prob = _problem(chunk, group)
    gpu = prob.to("cuda")
    runner = api.ChunkAttn(gpu, num_kv_splits=1)
    bounds = [(0, 256), (256, 1 << 30)]
    o = torch.full((len(bounds), prob.total_q, prob.num_q_heads, 128), float("nan"), device="cuda")
    l = torch.full((len(bounds), prob.total_q, prob.num_q_heads), float("nan"), device="cuda")
    for s, (b, e) in enumerate(bounds):
        api.vpp_chunk_attn_partial_fwd(runner.args, b, e, o[s], l[s])
        torch.cuda.synchronize()
        assert int(runner.status.item()) == 0
    api.vpp_lse_merge(o, l, runner.out, runner.lse)
    torch.cuda.synchronize()
    print(compare(runner.out, runner.lse, prob, oracle.all_rows(prob.chunk_len.numpy(), prob.num_q_heads), "key ranges"))
