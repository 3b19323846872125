"""The half-SM attention kernel (batches of few requests): against the CPU oracle's attention at the geometries and edges
of the other kernels' test, at the widths of its row tiles and its key parts, and on a batch in which one request's
context is another request's chunk."""
import pytest
import torch

from workloads import gen
from workloads.configs import TINY, Workload

import test_gpu_attention as base
from harness import cpu_model, to_cuda

pytestmark = pytest.mark.gpu

CASES = base.CASES + [
    (128, 8, 2, [63, 64, 65], [1, 4, 5]),        # one, two and three 64-key blocks; 1 and 2 row tiles
    (64, 8, 2, [4000], [9]),                     # 63 blocks over the most parts of one unit, 36 rows
    (128, 8, 8, [900, 31, 2047], [1, 16, 2]),    # G = 1
    (128, 8, 2, [6000], [12]),                   # parts of several blocks
]


@pytest.mark.parametrize("hd,Hq,Hkv,ctx,chunk", CASES)
def test_thin_attention_matches_oracle(hd, Hq, Hkv, ctx, chunk):
    import paper_2511_07423_b200 as syn
    syn.debug_set_attention(3)
    try:
        base._run(hd, Hq, Hkv, ctx, chunk)
    finally:
        syn.debug_set_attention(0)


@pytest.mark.parametrize("hd", [128, 64])
def test_scores_that_keep_growing(hd):
    base.test_scores_that_keep_growing_along_the_keys(hd, 8, 2, 3)


def test_a_context_written_by_another_request_of_the_batch():
    """Two requests over one page table, the second one's context ending with the first one's chunk (a long run of
    uncached tokens in one step): its keys must not be read before they are written.  The first request writes whole pages
    of the second one's first stage of 64 keys, which without a look at the other requests' chunks would be read early."""
    import paper_2511_07423_b200 as syn
    shape, seed = TINY, 31
    glob, layers = cpu_model(shape, seed)
    model = syn.Model(shape, *to_cuda(glob, layers))
    toks = gen.gen_context_tokens(Workload("w", shape, seed, 1, None, None, 0.5), 0, 90)
    table = torch.tensor([[5, 1, 7, 2, 0, 4]], dtype=torch.int32)
    two = dict(chunk_tokens=toks[48:90], chunk_offsets=[0, 32, 42], page_tables=table.repeat(2, 1), ctx_lens=[48, 80])
    syn.debug_set_attention(3)
    try:
        safe = {int(r[3]): int(r[9]) for r in syn.plan_work_host(shape, 8, **two)["items"]}
        assert safe == {0: 48, 1: 48}
        kv = syn.KVCache(model, 8)
        for at, n in ((0, 32), (32, 16)):
            kv.verify_batch(toks[at:at + n], [0, n], table, [at], [n])
        # the pieces one after the other ...
        kv.verify_batch(toks[48:80], [0, 32], table, [48], [32])
        _, _, want = kv.verify_batch(toks[80:90], [0, 10], table, [80], [10], want_logits=True)
        # ... and as two requests of one batch, over slots that hold something else before
        for _ in range(3):
            kv.verify_batch(toks[:32].flip(0), [0, 32], table, [48], [32])
            kv.verify_batch(toks[:10].flip(0), [0, 10], table, [80], [10])
            _, _, got = kv.verify_batch(*two.values(), [32, 10], want_logits=True)
            assert torch.equal(got[32:], want)
    finally:
        syn.debug_set_attention(0)


@pytest.mark.parametrize("hd,Hq,Hkv,ctx,chunk", [
    (128, 8, 4, [2500], [16]),          # 32 parts and fewer of 32 rows
    (64, 32, 8, [3000], [16]),          # 64 rows
    (128, 16, 8, [1400, 700], [9, 5]),  # fewer than 17 parts
])
def test_parts_are_merged_in_their_order(hd, Hq, Hkv, ctx, chunk):
    """Keys of zero make every weight 1 and every sum of a part a whole number, so the merge alone decides the last bits: the
    weight of a part is divided by the row's sum, then the parts are added in order with fused multiply-adds."""
    import numpy as np
    import paper_2511_07423_b200 as syn
    from workloads.configs import ModelShape
    shape, seed = ModelShape("merge", 1, 256, Hq, Hkv, hd, 256, 512), 5
    batch = base._batch(ctx, chunk, seed=seed)
    model = syn.Model(shape, *to_cuda(*cpu_model(shape, seed)))
    kv = syn.KVCache(model, batch.n_pages)
    g = torch.Generator().manual_seed(seed)
    values = []
    for r in range(batch.n_req):
        n = ctx[r] + chunk[r]
        v = torch.randint(-27, 28, (n, Hkv, hd), generator=g) + torch.where(torch.arange(n) < n // 2, 100, -100).view(n, 1, 1)
        kv.import_kv(0, batch.page_tables[r], 0, torch.zeros(n, Hkv, hd, dtype=torch.bfloat16, device="cuda"), v.to(torch.bfloat16).cuda())
        values.append(v.numpy().astype(np.float64).cumsum(0))
    T = batch.n_tokens
    q = torch.randn(T, shape.q_dim, generator=g).to(torch.float16)
    args = (torch.zeros(T, dtype=torch.int32), batch.chunk_offsets, batch.page_tables, batch.ctx_lens)
    syn.debug_set_attention(3)
    try:
        out = syn.Plan(kv, *args).attention(0, q.cuda())
        work = syn.plan_work_host(shape, batch.n_pages, *args, n_sm=torch.cuda.get_device_properties(0).multi_processor_count)
    finally:
        syn.debug_set_attention(0)
    torch.cuda.synchronize()
    assert model.status() == 0 and work["attention"] == 3
    groups = {}
    for q_tok, nj, kvh, req, k0, k1, pos0, part, grp, _ in work["items"].tolist():
        if part >= 0:
            groups.setdefault(grp, []).append((part, q_tok, nj, kvh, req, k0, k1, pos0))
    assert max(map(len, groups.values())) > 2
    got = out.cpu().view(T, Hkv, Hq // Hkv, hd)
    for items in groups.values():
        for j in range(items[0][2]):
            _, q_tok, _, kvh, req, _, _, pos0 = items[0]
            seen = [(k0, min(k1, pos0 + j + 1)) for _, _, _, _, _, k0, k1, _ in sorted(items)]
            inv = np.float32(1) / np.float32(pos0 + j + 1)
            acc = np.zeros(hd, dtype=np.float32)
            for k0, k1 in seen:
                if k1 > k0:   # (in 64 bits the product is exact, so this rounds once, like a fused multiply-add)
                    s = values[req][k1 - 1, kvh] - (values[req][k0 - 1, kvh] if k0 else 0)
                    acc = (s * np.float64(inv) + acc).astype(np.float32)
            want = torch.from_numpy(acc).to(torch.float16).expand(Hq // Hkv, hd)
            assert torch.equal(got[q_tok + j, kvh], want), (req, kvh, j)
