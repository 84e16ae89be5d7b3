"""The work this library is used for, as measurable cases: one attention layer's step over a paged KV cache.

A serving engine calls the library once per layer and step: `vpp_kv_append` writes the step's new keys and values into the
cache, then the attention entry point runs over everything cached.  The listed cases are that step for the shapes of
workloads.py, bench.py and the tests: chunks of a prompt (first, later, head-sharded), a mixed batch, decode batches,
the absorbed-MLA forms of the same, index-selected attention, and the cache write by itself.  `draw` gives more cases of the
same ranges.  A case holds sizes only; ragged lengths follow from its `lens` number, values from the seed.
"""
import math

import numpy as np
import torch

from paper_2608_26523_b200 import api
from paper_2608_26523_b200 import workloads as W

GQA = dict(dqk=128, dv=128)
MLA = dict(dqk=576, dv=512)


def listed():
    return [
        # the smallest call: a 512-token chunk of a short prompt on a small head shard, contiguous cache (cfg 1)
        dict(GQA, name="chunk_small", kind="chunk", hq=4, hkv=1, page=0, chunk=512, prefix=1536),
        # one rank's heads of a GQA 64/8 model sharded eight ways, an ordinary chunk at an unaligned place of a prompt
        dict(GQA, name="chunk_shard", kind="chunk", hq=8, hkv=1, page=64, chunk=2048, prefix=14321),
        # the first chunk of a prompt (nothing cached before it), MHA
        dict(GQA, name="chunk_first", kind="chunk", hq=32, hkv=32, page=128, chunk=4096, prefix=0),
        # a full-size chunk deep in a long prompt, GQA 64/4 (cfg 2): the headline shape
        dict(GQA, name="chunk_long", kind="chunk", hq=64, hkv=4, page=128, chunk=8192, prefix=65536),
        # continuous batching: 32 requests' ragged chunks of together 8192 tokens with 16 decode rows among them (cfg 5)
        dict(GQA, name="mixed", kind="mixed", hq=64, hkv=8, page=128, reqs=32, rows=16, budget=8192, longest=65536, lens=5),
        # a small decode batch, where latency counts: 8 rows
        dict(GQA, name="decode_few", kind="decode", hq=64, hkv=8, page=16, rows=8, longest=8192, lens=6),
        # a large decode batch: 256 rows, ragged contexts
        dict(GQA, name="decode_many", kind="decode", hq=64, hkv=8, page=16, rows=256, longest=8192, lens=7),
        # absorbed MLA: a chunk deep in a prompt (cfg 3)
        dict(MLA, name="mla_chunk", kind="chunk", hq=128, hkv=1, page=64, chunk=2048, prefix=32768),
        # absorbed MLA: a decode batch
        dict(MLA, name="mla_decode", kind="decode", hq=128, hkv=1, page=64, rows=32, longest=16384, lens=9),
        # index-selected MLA attention: a chunk of 2048 tokens, 2048 listed keys each
        dict(MLA, name="sparse_chunk", kind="sparse", hq=128, hkv=1, page=64, reqs=1, chunk=2048, prefix=65536, topk=2048),
        # the same for a decode batch: one token of each of 16 requests
        dict(MLA, name="sparse_decode", kind="sparse", hq=128, hkv=1, page=64, reqs=16, chunk=1, prefix=32768, topk=2048),
        # the cache write of a 16384-token chunk by itself (cfg 4)
        dict(GQA, name="append", kind="append", hq=64, hkv=8, page=128, chunk=16384, prefix=65536),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng):
    kind = rng.choice(["chunk", "chunk", "mixed", "decode", "decode", "mla_chunk", "mla_decode", "sparse", "sparse", "append"])
    page = rng.choice([16, 32, 64, 128])
    hq, hkv = rng.choice([(64, 4), (64, 8), (32, 8), (32, 32), (16, 2), (8, 1), (4, 1), (15, 5)])
    if kind == "chunk":
        return dict(GQA, kind="chunk", hq=hq, hkv=hkv, page=rng.choice([0, page, page]), chunk=_log(rng, 200, 8192),
                    prefix=rng.choice([0, _log(rng, 100, 65536), _log(rng, 100, 65536)]))
    if kind == "mixed":
        reqs = _log(rng, 4, 48)
        return dict(GQA, kind="mixed", hq=hq, hkv=hkv, page=page, reqs=reqs, rows=rng.choice([0, _log(rng, 1, 64)]),
                    budget=max(8 * reqs, _log(rng, 1000, 8192)), longest=_log(rng, 2000, 65536), lens=rng.randrange(1 << 20))
    if kind == "decode":
        return dict(GQA, kind="decode", hq=hq, hkv=hkv, page=page, rows=_log(rng, 1, 256), longest=_log(rng, 1000, 32768),
                    lens=rng.randrange(1 << 20))
    if kind == "mla_chunk":
        return dict(MLA, kind="chunk", hq=rng.choice([128, 64, 16]), hkv=1, page=page, chunk=_log(rng, 200, 2048),
                    prefix=rng.choice([0, _log(rng, 100, 32768)]))
    if kind == "mla_decode":
        return dict(MLA, kind="decode", hq=rng.choice([128, 64, 16]), hkv=1, page=page, rows=_log(rng, 1, 128),
                    longest=_log(rng, 1000, 32768), lens=rng.randrange(1 << 20))
    if kind == "sparse":
        one = rng.random() < 0.5
        return dict(MLA, kind="sparse", hq=rng.choice([128, 64]), hkv=1, page=page, reqs=_log(rng, 1, 64) if one else rng.choice([1, 2]),
                    chunk=1 if one else _log(rng, 64, 2048), prefix=_log(rng, 4000, 65536), topk=rng.choice([1024, 2048]))
    return dict(GQA, kind="append", hq=hq, hkv=hkv, page=page, chunk=_log(rng, 64, 16384), prefix=_log(rng, 100, 65536))


def draw(rng):
    """One more case of these ranges that costs no more than the largest listed one."""
    def cost(case):
        w = work(case)
        return max(w["bytes"], w["flops"] / 200)      # (about the ratio of the card's matrix rate to its memory rate)
    most = max(cost(c) for c in listed())
    while True:
        case = _draw(rng)
        if cost(case) <= most:
            return case


def lengths(case):
    """(prefix, chunk) lengths of the case's requests."""
    kind = case["kind"]
    if kind in ("chunk", "append"):
        return [case["prefix"]], [case["chunk"]]
    if kind == "sparse":
        return [case["prefix"] + 37 * r for r in range(case["reqs"])], [case["chunk"]] * case["reqs"]
    rng = np.random.default_rng(case["lens"])
    if kind == "decode":
        # contexts from a sixteenth of the longest to the longest, one of them the longest
        p = np.exp(rng.uniform(math.log(case["longest"] / 16), math.log(case["longest"]), size=case["rows"])).astype(int)
        p[0] = case["longest"]
        return [int(x) - 1 for x in p], [1] * case["rows"]
    n = case["reqs"]
    share = rng.dirichlet(np.full(n, 2.0))
    c = 1 + np.floor(share * (case["budget"] - n)).astype(int)
    c[0] += case["budget"] - int(c.sum())
    total = np.exp(rng.uniform(math.log(case["longest"] / 64), math.log(case["longest"]), size=n)).astype(int)
    p = np.array([int(rng.integers(0, max(1, t - k) + 1)) for t, k in zip(total, c)])
    d = np.exp(rng.uniform(math.log(case["longest"] / 16), math.log(case["longest"]), size=case["rows"])).astype(int)
    order = rng.permutation(n + case["rows"])
    pre, chk = np.concatenate([p, d]), np.concatenate([c, np.ones(case["rows"], int)])
    return [int(pre[i]) for i in order], [int(chk[i]) for i in order]


def selected_keys(pos, topk, gen, group=64):
    """Key positions for tokens at positions `pos`: the topk / 4 most recent ones and one draw from each of equal strata of
    the earlier ones, shared by a group of consecutive tokens (as a trained indexer's lists mostly are); -1 where a token has
    fewer than topk positions to list; shuffled."""
    dev, n = pos.device, pos.numel()
    window = topk // 4
    far = topk - window
    first = pos[torch.arange(n, device=dev) // group * group]
    same = (pos - first >= 0) & (pos - first < group)
    first = torch.where(same, first, pos)
    u = torch.rand((n, far), generator=gen, device=dev)
    u = torch.where(same[:, None], u[torch.arange(n, device=dev) // group * group], u)
    width = (first + 1 - window).clamp(min=0).double()[:, None] / far
    k = torch.arange(far, device=dev, dtype=torch.float64)[None]
    lo, hi = (k * width).floor(), ((k + 1) * width).floor()
    idx = torch.cat([pos[:, None] - torch.arange(window, device=dev)[None], (lo + (u * (hi - lo)).floor()).long()], dim=1)
    short = (width[:, 0] < 1)
    every = torch.arange(topk, device=dev)[None].expand(n, topk)
    idx = torch.where(short[:, None], torch.where(every <= pos[:, None], every, -1), idx)
    order = torch.argsort(torch.rand((n, topk), generator=gen, device=dev), dim=1)
    return idx.gather(1, order).to(torch.int32).contiguous()


def prepare(case, seed):
    p, c = lengths(case)
    mla = case["dqk"] == 576
    prob = W.make_problem(seed, p, c, case["hq"], case["hkv"], case["dqk"], case["dv"], block_size=case["page"] or None,
                          std=0.5 if mla else 1.0, scale=1.0 / math.sqrt(192.0) if mla else None, v_aliases_k=mla,
                          unused_fill=None, tail_fill=None, device="cuda", name=case["kind"])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) + 1)
    tokens = sum(c)

    def fresh(d):
        return (torch.randn((tokens, case["hkv"], d), generator=gen, device="cuda") * (0.5 if mla else 1.0)).to(torch.bfloat16)

    state = dict(prob=prob, k_new=fresh(case["dqk"]), v_new=None if mla else fresh(case["dv"]),
                 status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if case["kind"] == "sparse":
        pos = torch.cat([torch.arange(a, a + n, device="cuda") for a, n in zip(p, c)])
        state["attn"] = api.SparseAttn(prob, selected_keys(pos, case["topk"], gen))
    elif case["kind"] != "append":
        state["attn"] = api.ChunkAttn(prob)
    return state


def run(state):
    """One layer's step: the new rows join the cache, then the attention over all of it.  The cache is an output too."""
    p = state["prob"]
    api.vpp_kv_append(state["k_new"], state["v_new"], p.k_cache, p.v_cache if state["v_new"] is not None else None, p.block_table,
                      p.prefix_len, p.chunk_len, p.block_size, p.max_seq_len, status=state["status"])
    caches = [p.k_cache] if state["v_new"] is None else [p.k_cache, p.v_cache]
    if "attn" not in state:
        return caches
    out, lse = state["attn"].run()
    return [out, lse] + caches


def work(case):
    """New rows read and written once; queries and the keys and values that are attended to read once, results written once;
    2 (dqk + dv) operations for each visible (query, key) pair and q-head."""
    p, c = lengths(case)
    dqk, dv, hq, hkv = case["dqk"], case["dv"], case["hq"], case["hkv"]
    tokens = sum(c)
    row = hkv * (dqk if dqk == 576 else dqk + dv) * 2          # the cached bytes of a token
    moved, flops = 2 * tokens * row, 0
    if case["kind"] != "append":
        moved += tokens * hq * (2 * dqk + 2 * dv + 4)
        if case["kind"] == "sparse":
            keys = [min(case["topk"], x + i + 1) for x, n in zip(p, c) for i in range(n)]
            # every listed row is read at least once; consecutive tokens share most of their lists, so at most what is cached
            moved += sum(min(x + n, case["topk"] * n) for x, n in zip(p, c)) * row + 4 * tokens * case["topk"]
            pairs = sum(keys)
        else:
            moved += sum(x + n for x, n in zip(p, c)) * row
            pairs = sum(n * x + n * (n + 1) // 2 for x, n in zip(p, c))
        flops = 2 * hq * (dqk + dv) * pairs
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    """Measured: the same step with its keys split in three differs by rel 1.5e-3 to 2.9e-3, max 0.8e-2 to 1.4e-2 (weights and
    results rounded to bf16 in another order), the path against 64 bits by rel 2.3e-3; four times that.  A copy is exact."""
    if case["kind"] == "append":
        return "exact"
    return {"rel": 1.2e-2, "max": 5.6e-2}
