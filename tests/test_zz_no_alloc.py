"""syn_op_attention_static, the attention entry point for callers that cannot allocate device
memory while they run (inside a stream capture, or in a server whose memory was handed out up
front), against the ordinary syn_op_attention on the same plan.  Collected last on purpose."""
import numpy as np
import pytest
import torch

from workloads import gen, rng
from workloads.configs import ModelShape, Workload

from harness import cpu_model, to_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd", [128, 64])
def test_static_scratch_attention_equals_the_allocating_one_twice_in_a_row(hd, attention_kind):
    import paper_2511_07423_b200 as syn
    shape = ModelShape("att-static", 1, 256, 8, 2, hd, 256, 512)
    seed = 21
    # long contexts, so that key ranges are split over work items and the partial-result array is used
    wl = Workload("t", None, seed, 4, ("list", (1500, 40, 2300, 900)), ("list", (16, 3, 9, 1)), 0.5)
    batch = gen.gen_batch(wl)
    glob, layers = cpu_model(shape, seed)
    gg, gl = to_cuda(glob, layers)
    model = syn.Model(shape, gg, gl)
    kv = syn.KVCache(model, batch.n_pages)
    T = batch.n_tokens
    for r in range(batch.n_req):
        tot = int(batch.ctx_lens[r] + batch.chunk_lens[r])
        k, v = gen.gen_kv(shape, seed, 0, r, 0, tot, device="cuda")
        kv.import_kv(0, batch.page_tables[r], 0, k, v)
    plan = syn.Plan(kv, torch.zeros(T, dtype=torch.int32), batch.chunk_offsets, batch.page_tables, batch.ctx_lens)
    assert plan.stats().attn_split_items > 0
    out_static = torch.empty(T, shape.q_dim, dtype=torch.float16, device="cuda")
    for call in range(2):   # the second call finds the first call's partials in the shared array
        q = rng.normal_f32(rng.stream_key(seed, 77 + call), 0, T * shape.q_dim, 1.5, device="cuda") \
            .view(T, shape.q_dim).to(torch.float16)
        ref = plan.attention(0, q)
        torch.cuda.synchronize()
        out_static.fill_(float("nan"))
        torch.cuda.synchronize()
        free_before, _ = torch.cuda.mem_get_info()
        plan.attention_static(0, q, out=out_static)
        torch.cuda.synchronize()
        free_after, _ = torch.cuda.mem_get_info()
        # what the entry point is for: the device's free memory is the same before and after the call
        # (from the second call on: the first one on a device looks the array's address up)
        if call > 0:
            assert free_after == free_before
        assert model.status() == 0
        a, b = out_static.float().cpu().numpy(), ref.float().cpu().numpy()
        assert np.isfinite(a).all()
        assert np.abs(a - b).max() <= 0.02 * np.abs(b).max()   # the tolerance of the attention parity test


@pytest.mark.parametrize("kind,n_req,ctx,Hq,Hkv,chunk,n_parts", [
    (0, 7, 2000, 21, 21, 1, 294),     # 147 equal (request, kv head) units, two parts each
    (1, 19, 2000, 32, 8, 5, 282),     # 152 units laid end to end over 148 CTAs
    (3, 19, 2000, 32, 8, 5, 418),     # ... over 296
    (2, 19, 3000, 32, 8, 32, 274),    # partials of 128 rows
])
def test_static_scratch_attention_takes_what_its_array_holds(kind, n_req, ctx, Hq, Hkv, chunk, n_parts):
    """Plans of more partials than one a CTA.  (None exceeds the array: a host test in test_attention_cuts.py.)"""
    import paper_2511_07423_b200 as syn
    shape = ModelShape("att-static", 1, 256, Hq, Hkv, 128, 256, 512)
    seed = 22
    wl = Workload("t", None, seed, n_req, ("const", ctx), ("const", chunk), 0.5)
    batch = gen.gen_batch(wl)
    glob, layers = cpu_model(shape, seed)
    gg, gl = to_cuda(glob, layers)
    model = syn.Model(shape, gg, gl)
    kv = syn.KVCache(model, batch.n_pages)
    for r in range(batch.n_req):
        k, v = gen.gen_kv(shape, seed, 0, r, 0, int(batch.ctx_lens[r] + batch.chunk_lens[r]), device="cuda")
        kv.import_kv(0, batch.page_tables[r], 0, k, v)
    T = batch.n_tokens
    syn.debug_set_attention(kind)
    try:
        plan = syn.Plan(kv, torch.zeros(T, dtype=torch.int32), batch.chunk_offsets, batch.page_tables, batch.ctx_lens)
    finally:
        syn.debug_set_attention(0)
    assert (plan.stats().attn_split_items, plan.stats().attn_rows) == (n_parts, 128 if kind == 2 else 64)
    q = rng.normal_f32(rng.stream_key(seed, 78), 0, T * shape.q_dim, 1.5, device="cuda").view(T, shape.q_dim).to(torch.float16)
    ref = plan.attention(0, q)
    out = torch.full_like(ref, float("nan"))
    plan.attention_static(0, q, out=out)
    torch.cuda.synchronize()
    assert model.status() == 0
    assert torch.equal(out, ref)   # the same kernel, list and order of sums; only the scratch is another
