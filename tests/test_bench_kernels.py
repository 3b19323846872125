"""Which kernel function bench.py books a class of launches to."""
import pytest
import torch

import bench
import paper_2511_07423_b200 as syn
from workloads import gen
from workloads.configs import CONFIGS


def test_projections_are_booked_to_the_kernel_that_the_library_launches():
    # 129 tokens of the 1B shape: everything but the lm_head on the half-SM kernel
    for N, K, epi in ((3072, 2048, "qkv"), (2048, 2048, "resid"), (16384, 2048, "swiglu"), (2048, 8192, "resid")):
        assert bench.projection_kernel(129, N, K, epi) == "thin_kernel"
        assert bench.projection_kernel(129, N, K, epi, "one-cta") == "gemm_kernel"
    assert bench.projection_kernel(544, 6144, 4096, "qkv") == "gemm2_kernel"
    assert bench.projection_kernel(176, 4096, 14336, "resid") == "gemm_kernel"
    assert set(bench.ATTENTION_KERNELS.values()) | {"gemm_kernel", "gemm2_kernel", "thin_kernel"} == set(bench.KERNEL_SOURCES)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", [0, 1, 2, 3])
def test_a_plan_names_its_attention_kernel(kind):
    wl = CONFIGS[1]
    batch = gen.gen_batch(wl)
    from paper_2511_07423_b200 import synthetic
    model = synthetic.load_model(wl.shape, wl.seed)
    kv = syn.KVCache(model, batch.n_pages)
    syn.debug_set_attention(kind)
    try:
        args = (torch.zeros(batch.n_tokens, dtype=torch.int32), batch.chunk_offsets, batch.page_tables, batch.ctx_lens)
        assert syn.Plan(kv, *args).attention_kernel() == (kind or syn.plan_work_host(wl.shape, batch.n_pages, *args)["attention"])
    finally:
        syn.debug_set_attention(0)
