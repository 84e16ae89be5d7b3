"""Append rows wider than a warp's piece (256 vectors of 16 bytes), narrower ones and the sizes around it, bit for bit; a page
out of range is reported wherever its row stands."""
import pytest
import torch

from paper_2608_26523_b200 import api, workloads as W
from test_gpu_kv_append import run_case

pytestmark = pytest.mark.gpu


# 16-byte vectors per row: 32 hkv (K and V of 128), 72 for an absorbed-MLA row
@pytest.mark.parametrize("hkv,dqk,dv,alias", [(1, 128, 128, False), (7, 128, 128, False), (8, 128, 128, False), (9, 128, 128, False),
                                              (32, 128, 128, False), (1, 576, 512, True)])
@pytest.mark.parametrize("chunk", [[1], [1, 0, 9], [300]])
def test_rows_of_every_width(hkv, dqk, dv, alias, chunk):
    run_case(3300 + hkv, [5 + 17 * i for i in range(len(chunk))], chunk, hkv, dqk, dv, 16, alias)


@pytest.mark.parametrize("reqs,chunk", [(1, 700), (300, 1), (20, 40)])
def test_a_page_out_of_range_is_reported_wherever_it_stands(reqs, chunk):
    prob = W.make_problem(3400, [3] * reqs, [chunk] * reqs, 2, 1, 128, 128, block_size=16, device="cuda", unused_fill=None)
    new = torch.zeros((reqs * chunk, 1, 128), dtype=torch.bfloat16, device="cuda")
    status = torch.full((1,), 9, dtype=torch.int32, device="cuda")
    last = (3 + chunk - 1) // 16
    for r, b, want in [(0, 0, 2), (reqs - 1, last, 2), (reqs // 2, last // 2, 2), (0, 0, 0)]:
        bt = prob.block_table.clone()
        if want:
            bt[r, b] = prob.k_cache.shape[0]
        api.vpp_kv_append(new, new, prob.k_cache, prob.v_cache, bt, prob.prefix_len, prob.chunk_len, 16, prob.max_seq_len, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == want, (r, b)
