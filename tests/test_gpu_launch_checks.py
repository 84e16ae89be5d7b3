"""The work decomposition checks the block table with several blocks while it cuts the work: one entry out of range, wherever
it stands, stops the launch before it writes anything, and the next launch is unaffected."""
import pytest
import torch

from paper_2608_26523_b200 import api, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reqs,seq,page", [(1, 40, 16), (3, 9000, 16), (300, 200, 16), (40, 6000, 64)])
@pytest.mark.parametrize("chunk", [1, 33])
def test_a_bad_block_table_entry_is_found_wherever_it_stands(reqs, seq, page, chunk):
    prob = W.make_problem(11, [seq - chunk - (r % 7) for r in range(reqs)], [chunk] * reqs, 4, 1, 128, 128, block_size=page,
                          device="cuda", unused_fill=None)
    runner = api.ChunkAttn(prob)
    good = prob.block_table.clone()
    ref = runner.run()[0].clone()
    need = [(int(p) + chunk + page - 1) // page for p in prob.prefix_len.tolist()]
    places = {(0, 0), (0, need[0] - 1), (reqs - 1, need[-1] - 1), (reqs // 2, need[reqs // 2] // 2)}
    for r, b in sorted(places):
        for bad in (-1, prob.k_cache.shape[0]):
            prob.block_table.copy_(good)
            prob.block_table[r, b] = bad
            runner.out.fill_(3.0)
            runner.run()
            torch.cuda.synchronize()
            assert int(runner.status.item()) == 2, (r, b, bad)      # VPP_DEV_BAD_BLOCK
            assert (runner.out == 3.0).all()
    prob.block_table.copy_(good)
    for r in range(reqs):                                           # entries no request needs may hold anything
        prob.block_table[r, need[r]:] = -7
    out, _ = runner.run()
    torch.cuda.synchronize()
    assert int(runner.status.item()) == 0 and torch.equal(out, ref)
