"""The status word of an append: every page that a row needs is looked at, whatever the batch looks like, and what that costs does
not depend on how the rows are shared out among the requests."""
import pytest
import torch

from paper_2608_26523_b200 import api, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("page,prefix,chunk", [
    (16, [0, 5, 30, 7, 16, 15], [0, 300, 1, 0, 33, 2]), (16, [3], [500]), (1, [0, 4, 9], [70, 0, 31]),
    (64, [63] * 300, [2] * 300), (16, [15, 14] * 700, [1, 3] * 700), (128, [100, 0], [4000, 17])])
def test_every_page_is_looked_at(page, prefix, chunk):
    prob = W.make_problem(3500, prefix, chunk, 1, 1, 128, 128, block_size=page, device="cuda", unused_fill=None)
    new = torch.zeros((sum(chunk), 1, 128), dtype=torch.bfloat16, device="cuda")
    status = torch.full((1,), 9, dtype=torch.int32, device="cuda")
    good = prob.block_table.clone()
    need = torch.zeros_like(good, dtype=torch.bool)
    for r, (a, n) in enumerate(zip(prefix, chunk)):
        if n:
            need[r, a // page:(a + n - 1) // page + 1] = True
    good[~need] = -5                                   # entries that no row needs may hold anything

    def run(bt):
        api.vpp_kv_append(new, new, prob.k_cache, prob.v_cache, bt, prob.prefix_len, prob.chunk_len, page, prob.max_seq_len, status=status)
        return int(status.item())

    assert run(good) == 0
    places = need.nonzero().tolist()
    for r, b in places[::max(1, len(places) // 400)] + places[-1:]:
        bt = good.clone()
        bt[r, b] = prob.k_cache.shape[0] if (r + b) % 2 else -1
        assert run(bt) == 2, (r, b)


@pytest.mark.parametrize("reqs", [8, 64, 256, 1024])
def test_the_look_at_the_pages_hides_behind_the_copy(reqs):
    """One chunk of 8192 rows in pages of 16 among single rows (a mixed batch): the call with a status word takes at most half as
    long again as the call without (a thread per request walking its pages took three times as long)."""
    prob = W.make_problem(3600, [100] * reqs, [8192] + [1] * (reqs - 1), 8, 8, 128, 128, block_size=16, device="cuda", unused_fill=None)
    new = torch.zeros((prob.total_q, 8, 128), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def graph(st):
        def call():
            api.vpp_kv_append(new, new, prob.k_cache, prob.v_cache, prob.block_table, prob.prefix_len, prob.chunk_len, 16, prob.max_seq_len,
                              status=st)
        call()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(20):
                call()
        return g

    def us(g):
        best = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.replay()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3 / 20)
        return best

    with_status, without = us(graph(status)), us(graph(None))
    print("%d requests: %.1f us with a status word, %.1f without" % (reqs, with_status, without))
    assert with_status <= 1.5 * without
