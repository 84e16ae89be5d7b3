"""The allocation-free entry point with the library's own cut finer than its scratch array holds: the launch is cut into as many
parts as fit -- three kernels, the merge among them -- and not left whole.  (One whose cut fits is cut too.)"""
import pytest
import torch

import oracle
from paper_2608_26523_b200 import api, workloads as W
from parity import compare, sample_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prefix,chunk,hq,hkv,mla", [
    ([14321], [2048], 8, 1, False), ([32512], [256], 64, 8, False), ([31744], [1024], 16, 2, False), ([16128] * 4, [256] * 4, 8, 1, False),
    ([4200 + 700 * i for i in range(17)], [1] * 17, 128, 1, True)])
def test_a_cut_that_does_not_fit_is_made_coarser(prefix, chunk, hq, hkv, mla):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the sizes are for 148 SMs")
    prob = W.make_problem(9100 + hq, prefix, chunk, hq, hkv, 576 if mla else 128, 512 if mla else 128, block_size=64, std=0.5,
                          scale=1.0 / 192 ** 0.5 if mla else None, v_aliases_k=mla)
    runner = api.ChunkAttn(prob.to("cuda"))
    assert api.vpp_chunk_attn_workspace_size(runner.args) > api.vpp_static_scratch_bytes() or hq == 64
    runner.args.workspace, runner.args.workspace_bytes = None, 0
    runner.out.fill_(float("nan"))
    api.vpp_chunk_attn_fwd_static(runner.args)
    torch.cuda.synchronize()
    assert int(runner.status.item()) == 0 and torch.isfinite(runner.out).all()
    assert api.vpp_last_launch_count() == 3
    print(compare(runner.out, runner.lse, prob, sample_rows(prob, 64), "static, cut to fit"))
