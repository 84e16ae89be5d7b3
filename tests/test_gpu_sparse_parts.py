"""Sparse launches of few tokens: their lists are cut into parts whose results are merged.  Token counts on both sides of where
the number of parts changes, short lists, parts of which no entry takes part, a workspace that has room for an uncut launch
only, and many tokens after one another on the same pairs."""
import numpy as np
import pytest
import torch

from paper_2608_26523_b200 import api, workloads as W
from test_gpu_sparse import _check, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tokens", [1, 9, 10, 18, 37, 38])      # 74 pairs: 8 / 8 / 7 / 4 / 2 / 1 parts
@pytest.mark.parametrize("topk", [130, 257, 1100])              # 2, 3 and 9 KV tiles: parts of at least two tiles
def test_cut_lists_match_the_oracle(tokens, topk):
    prefix = [1200 + 3 * r for r in range(tokens)]
    p = _problem(5800 + tokens, prefix, [1] * tokens, 128 if topk != 257 else 72)
    idx = W.make_sparse_indices(70 + topk, prefix, [1] * tokens, topk)
    idx[0, 256:] = -1                       # every later part of the first list is empty
    idx[tokens // 2, :256] = 5000           # the future: the first part takes no part
    if tokens > 2:
        idx[2] = -1                         # nothing listed at all
    print(_check(p, idx, label="cut lists"))


def test_a_workspace_without_room_for_partials_runs_uncut():
    p = _problem(5900, [900, 40], [3, 4], 128).to("cuda")
    idx = torch.from_numpy(W.make_sparse_indices(71, [900, 40], [3, 4], 700)).cuda()
    a, b = api.SparseAttn(p, idx), api.SparseAttn(p, idx)
    assert api.vpp_sparse_attn_workspace_size(7) > 256 + 8 * 7
    b.args.workspace_bytes = 256 + 8 * 7
    oa, la = a.run()
    ob, lb = b.run()
    torch.cuda.synchronize()
    assert int(a.status.item()) == 0 and int(b.status.item()) == 0
    # the same sums in another order, rounded to bf16 once: half an ulp of results below 4 either way
    assert (oa.float() - ob.float()).abs().max().item() <= 1e-2
    assert (la - lb).abs().max().item() <= 1e-5 * max(1.0, lb.abs().max().item())


def test_repeated_launches_of_many_tokens_give_the_same_bits():
    """Hundreds of tokens in turn on every pair, lists of many tiles: the query tile of a token may be replaced only when the
    scores of the token before are done, whatever warp runs ahead."""
    p = _problem(6000, [3000], [700], 128).to("cuda")
    idx = torch.from_numpy(W.make_sparse_indices_strata(72, [3000], [700], 1024, kind="clustered").numpy()).cuda()
    r = api.SparseAttn(p, idx)
    first = r.run()[0].clone()
    for _ in range(4):
        assert torch.equal(r.run()[0], first)
    assert int(r.status.item()) == 0
