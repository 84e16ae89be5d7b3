"""When the library cuts a launch of few work items into parts (host arithmetic; 148 SMs assumed on a box without a GPU): only
where the share saved outweighs the merge and the partial results.  The workspace says what was chosen: without parts it holds no
partial results."""
import ctypes

import pytest
import torch

from paper_2608_26523_b200 import api


def _workspace(total_q, num_reqs, hq, hkv, seq, splits, mla=False):
    a = api.ChunkAttnArgs()
    fake = ctypes.c_void_p(1 << 20)
    a.q = a.k_cache = a.v_cache = a.block_table = a.prefix_len = a.chunk_len = a.out = fake
    a.num_reqs, a.total_q, a.max_seq_len = num_reqs, total_q, seq
    a.max_blocks_per_req, a.block_size, a.num_blocks = (seq + 63) // 64, 64, 1 << 16
    a.num_q_heads, a.num_kv_heads = hq, hkv
    a.head_dim_qk, a.head_dim_v = (576, 512) if mla else (128, 128)
    a.softmax_scale, a.num_kv_splits = 0.1, splits
    return api.vpp_chunk_attn_workspace_size(a)


# measured on both sides of the line: cutting loses where False stands, wins where True does
@pytest.mark.parametrize("total_q,num_reqs,hq,hkv,seq,mla,cut", [
    (256, 1, 4, 1, 512, False, False), (256, 1, 4, 1, 1024, False, True),           # a short chunk of a few heads
    (200, 1, 64, 8, 1536, False, False), (200, 1, 64, 8, 6144, False, True),        # many heads: more partial results
    (1, 1, 64, 8, 1024, False, False), (1, 1, 64, 8, 2048, False, True),            # a decode row
    (200, 1, 16, 1, 2048, True, False), (200, 1, 16, 1, 8192, True, True),          # MLA chunk
    (4, 4, 128, 1, 1024, True, False), (4, 4, 128, 1, 2048, True, True),            # MLA decode rows
    (110, 110, 128, 1, 8192, True, False),                                          # more items than pairs of SMs
])
def test_cutting_is_chosen_where_it_pays(total_q, num_reqs, hq, hkv, seq, mla, cut):
    if torch.cuda.is_available() and torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the expectations are for 148 SMs")
    auto, uncut = (_workspace(total_q, num_reqs, hq, hkv, seq, s, mla) for s in (0, 1))
    assert (auto > uncut) == cut


@pytest.mark.parametrize("total_q,hq,hkv,seq,cut", [
    (1280, 32, 32, 32768, True), (1280, 32, 16, 32768, True),     # 160 items either way: twelve would run a second wave alone
    (4096, 32, 32, 4096, False), (4096, 32, 16, 4096, False),     # items of all lengths: longest first fills the last wave
    (8192, 16, 2, 73728, True), (8192, 64, 4, 73728, False)])     # 3.5 and 14 waves of equally long items
def test_equal_splits_go_by_the_items_that_run(total_q, hq, hkv, seq, cut):
    if torch.cuda.is_available() and torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the expectations are for 148 SMs")
    auto, uncut = (_workspace(total_q, 1, hq, hkv, seq, s) for s in (0, 1))
    assert (auto > uncut) == cut


@pytest.mark.parametrize("rows,heads", [(5, (32, 32)), (20, (24, 8)), (8, (40, 40))])
def test_decode_rows_of_odd_groups_are_cut_like_those_of_even_ones(rows, heads):
    hq, hkv = heads
    one = lambda q: _workspace(rows, rows, q, hkv, 16384, 0) - _workspace(rows, rows, q, hkv, 16384, 1)
    assert one(2 * hkv) / (2 * hkv) == pytest.approx(one(hq) / hq, rel=0.02)
