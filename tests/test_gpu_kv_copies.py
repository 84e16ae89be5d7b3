"""K/V copies of the d = 128 kernel: pages of every size (one copy each), contiguous caches whose length is no multiple of eight
(the last tile comes in copies of eight keys of a map with the exact extent), strides with hardly a common divisor, and pages so
far apart that (page, head) does not fit one coordinate (every tile in copies of eight keys)."""
import pytest
import torch

import oracle
from paper_2608_26523_b200 import workloads as W
from parity import compare, run_gpu

pytestmark = pytest.mark.gpu


def check(prob, gpu, label, splits=0):
    out, lse, _ = run_gpu(gpu, splits)
    print(compare(out, lse, prob, oracle.all_rows(prob.chunk_len.numpy(), prob.num_q_heads), label))


@pytest.mark.parametrize("seq", [1, 5, 8, 9, 127, 130, 255, 256, 257, 391])
@pytest.mark.parametrize("chunk", [1, 70])
def test_contiguous_lengths(seq, chunk):
    c = min(seq, chunk)
    prob = W.make_problem(9950 + seq, [seq - c, 0], [c, min(3, seq)], 4, 2, 128, 128, block_size=None, std=0.8, seq_lens=[seq, seq])
    check(prob, prob.to("cuda"), "contiguous %d" % seq)


@pytest.mark.parametrize("page", [16, 32, 64, 128, 256])
@pytest.mark.parametrize("chunk", [[1] * 9, [150]])
def test_pages(page, chunk):
    prob = W.make_problem(9960 + page, [300 + 31 * i for i in range(len(chunk))], chunk, 8, 4, 128, 128, block_size=page, std=0.8)
    check(prob, prob.to("cuda"), "pages of %d" % page)


@pytest.mark.parametrize("page", [16, 128])
def test_strides_with_hardly_a_common_divisor(page):
    prob = W.make_problem(9970, [200, 0], [90, 33], 6, 3, 128, 128, block_size=page, std=0.8)
    gpu = prob.to("cuda")
    for name in ("k_cache", "v_cache"):
        x = getattr(gpu, name)
        nb, bs, h, d = x.shape
        store = torch.full((nb * (bs * h * 136 + 8) + 8,), float("nan"), dtype=x.dtype, device="cuda")
        view = store.as_strided(x.shape, (bs * h * 136 + 8, h * 136, 136, 1))
        view.copy_(x)
        setattr(gpu, name, view)
    check(prob, gpu, "odd strides")


def test_pages_tens_of_gigabytes_apart():
    prob = W.make_problem(9980, [40], [60], 4, 2, 128, 128, block_size=64, std=0.8, pool_factor=1.0)
    gpu = prob.to("cuda")
    nb, bs, h, d = gpu.k_cache.shape
    far = 18 * (1 << 30) + 8                        # elements between pages: 36 GB, and hardly a divisor in common with a head
    if torch.cuda.mem_get_info()[0] < far * 2 * (nb - 1) + (1 << 30):
        pytest.skip("needs a cache of %d GB" % (far * 2 * (nb - 1) >> 30))
    store = torch.empty((nb - 1) * far + bs * h * d, dtype=torch.bfloat16, device="cuda")
    view = store.as_strided(gpu.k_cache.shape, (far, h * d, d, 1))
    view.copy_(gpu.k_cache)
    gpu.k_cache = view
    check(prob, gpu, "pages far apart")
