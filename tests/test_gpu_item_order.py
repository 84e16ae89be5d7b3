"""The order in which a launch of few work items hands them out, read from the work list that it leaves in its workspace: the parts
of a balanced cut are of very different lengths, so they go longest first over all heads, and the time that the SMs then need is
close to an equal share; in a batch, chunks whose items are longer than the decode rows' go before these."""
import heapq
import struct

import pytest
import torch

from paper_2608_26523_b200 import api, workloads as W

pytestmark = pytest.mark.gpu

LEAD = 2                                                 # what starting and ending an item costs, in KV tiles


def _launch(prefix, chunk, hq, hkv, splits=0):
    """(header, units) of a launch: WorkHeader and WorkUnit of csrc/common.cuh."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the sizes are for 148 SMs")
    prob = W.make_problem(9200, prefix, chunk, hq, hkv, 128, 128, block_size=128, device="cuda", unused_fill=None, tail_fill=None)
    runner = api.ChunkAttn(prob, num_kv_splits=splits)
    runner.run()
    torch.cuda.synchronize()
    assert int(runner.status.item()) == 0
    raw = runner.workspace.cpu().numpy().tobytes()
    head = dict(zip(("units", "short", "block", "error", "counter", "checkers", "lead"), struct.unpack_from("<7i", raw, 0)))
    keys = ("req", "row0", "rows", "pos0", "begin", "end", "split", "kv_len")
    units = [dict(zip(keys, struct.unpack_from("<8i", raw, 256 + 32 * i))) for i in range(head["units"])]
    for u in units:
        u["rows"] &= 0xffff
        u["tiles"] = u["end"] - u["begin"]
    assert head["error"] == 0 and head["block"] >= 1
    return head, units


def _items(units, block, unit_items, per_kv_head):
    """KV tiles of the items of units of two tiles, in the order they are handed out."""
    order = []
    for b0 in range(0, len(units), block):
        for _ in range(unit_items // per_kv_head):
            order += [u["tiles"] for u in units[b0:b0 + block] for _ in range(per_kv_head)]
    return order


# head counts, q-heads per item (the largest divisor of the group that fills a tile), tokens, keys
@pytest.mark.parametrize("hq,hkv,per_item,chunk,seq", [
    (64, 8, 8, 256, 8192), (64, 8, 8, 256, 16384), (32, 16, 2, 512, 8192), (24, 8, 3, 504, 16384), (40, 40, 1, 512, 4096),
    (16, 2, 8, 1024, 32768), (8, 1, 8, 2048, 16369), (96, 8, 4, 200, 16384)])
def test_parts_of_a_balanced_cut_go_longest_first(hq, hkv, per_item, chunk, seq):
    head, units = _launch([seq - chunk], [chunk], hq, hkv)
    assert head["short"] == 0 and api.vpp_last_launch_count() == 3
    order = _items(units, head["block"], hq // per_item, hq // per_item // hkv)
    busy = [0] * 148
    for n in order:                                      # whoever is free first takes the next item
        heapq.heapreplace(busy, busy[0] + n + LEAD)
    share = (sum(order) + LEAD * len(order)) / 148
    print("longest %d tiles, share %.1f, items %d" % (max(busy), share, len(order)))
    assert max(busy) <= 1.3 * share                       # (40 heads in three ranges: 120 of the 148 SMs, 1.24)


@pytest.mark.parametrize("chunk,rows,hq,hkv,first", [(64, 30, 64, 8, True), (300, 8, 16, 16, True), (64, 8, 64, 8, False), (1000, 300, 64, 8, False)])
def test_chunks_of_longer_items_go_before_decode_rows(chunk, rows, hq, hkv, first):
    """... in batches of fewer than four items to an SM; there as many units are put in front as take longer than every row."""
    prefix = [8000] + [4000 + 13 * (i % 30) for i in range(rows)] if hq == 64 else [6000] + [2000] * rows
    if not first and rows == 8:
        prefix = [2000] + [9000] * rows
    head, units = _launch(prefix, [chunk] + [1] * rows, hq, hkv, splits=1)
    normal, short = units[:head["units"] - head["short"]], units[head["units"] - head["short"]:]
    us = lambda u: (u["tiles"] + 2) * 1.75 if u in normal else (u["tiles"] + 3) * 0.85
    longest = max(us(u) for u in short)
    longer = [u for u in normal if us(u) > 1.05 * longest]                  # (bins of lengths: 1 / 128 of the longest)
    assert all(us(u) > 0.95 * longest for u in normal[:head["lead"]])
    assert head["lead"] >= len(longer) > 0 if first else head["lead"] == 0, (head, len(longer))


@pytest.mark.parametrize("hq,hkv,chunk,seq", [(64, 8, 400, 65536), (32, 8, 300, 131072), (32, 16, 512, 32768)])
def test_units_whose_keys_exceed_l2_are_cut_at_the_same_places(hq, hkv, chunk, seq):
    """Equal splits of all units: units that run together go over the same keys."""
    head, units = _launch([seq - chunk], [chunk], hq, hkv)
    assert api.vpp_last_launch_count() == 3
    for s in range(max(u["split"] for u in units) + 1):
        part = [u for u in units if u["split"] == s]
        assert max(u["begin"] for u in part) - min(u["begin"] for u in part) <= chunk // 128 + 1


@pytest.mark.parametrize("hq,hkv,chunk,rows", [(24, 8, 512, 256), (24, 8, 504, 84), (15, 5, 256, 256), (48, 8, 768, 128), (64, 8, 268, 32)])
def test_tiles_of_a_chunk_whose_tail_would_go_over_all_keys_again(hq, hkv, chunk, rows):
    """A part of the group of q-heads that divides the chunk better is taken where the largest leaves a few tokens over."""
    _, units = _launch([4096 - chunk], [chunk], hq, hkv, splits=1)
    assert max(u["rows"] for u in units) == rows
