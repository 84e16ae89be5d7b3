"""The order in which a cut launch hands out its work items, read from the work list that the launch leaves in its workspace: the
parts of a balanced cut are of very different lengths, so they go longest first over all heads, and the time that the SMs then
need is close to an equal share."""
import heapq
import struct

import pytest
import torch

from paper_2608_26523_b200 import api, workloads as W

pytestmark = pytest.mark.gpu


def _items(ws, unit_items, per_kv_head):
    """KV tiles of the items of units of two tiles, in the order they are handed out (WorkHeader and WorkUnit of csrc/common.cuh)."""
    raw = ws.cpu().numpy().tobytes()
    num_units, num_short, block, error = struct.unpack_from("<4i", raw, 0)
    assert error == 0 and num_short == 0 and block >= 1
    units = [struct.unpack_from("<8i", raw, 256 + 32 * i) for i in range(num_units)]
    order = []
    for b0 in range(0, num_units, block):
        block_units = units[b0:b0 + block]
        for _ in range(unit_items // per_kv_head):
            order += [u[5] - u[4] for u in block_units for _ in range(per_kv_head)]
    return order


# head counts, q-heads per item (the largest divisor of the group that fills a tile), tokens, keys
@pytest.mark.parametrize("hq,hkv,per_item,chunk,seq", [
    (64, 8, 8, 256, 32768), (64, 8, 8, 256, 8192), (64, 4, 16, 256, 32768), (24, 8, 3, 504, 32768), (40, 40, 1, 512, 16384),
    (16, 2, 8, 1024, 32768), (8, 1, 8, 2048, 16369), (96, 8, 4, 200, 32768)])
def test_parts_of_a_balanced_cut_go_longest_first(hq, hkv, per_item, chunk, seq):
    slots = torch.cuda.get_device_properties(0).multi_processor_count
    if slots != 148:
        pytest.skip("the sizes are for 148 SMs")
    prob = W.make_problem(9200, [seq - chunk], [chunk], hq, hkv, 128, 128, block_size=128, device="cuda", unused_fill=None, tail_fill=None)
    runner = api.ChunkAttn(prob)
    runner.run()
    torch.cuda.synchronize()
    assert api.vpp_last_launch_count() == 3 and int(runner.status.item()) == 0
    order = _items(runner.workspace, hq // per_item, hq // per_item // hkv)
    assert len(order) > slots
    lead = 2                                             # what starting and ending an item costs, in KV tiles
    busy = [0] * slots
    for n in order:                                      # whoever is free first takes the next item
        heapq.heapreplace(busy, busy[0] + n + lead)
    share = (sum(order) + lead * len(order)) / slots
    print("longest %d tiles, share %.1f, items %d" % (max(busy), share, len(order)))
    assert max(busy) <= 1.3 * share                      # (40 heads in three ranges: 120 of the 148 SMs, 1.24)
