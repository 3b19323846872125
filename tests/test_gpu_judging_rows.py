"""Calls that ask for no logits run the lm_head over the rows that verification looks at only: the same results as greedy
verification of the logits that the same batch gives where they are asked for."""
import pytest
import torch

from workloads import gen
from workloads.configs import MINI_1B, MINI_8B, Workload

import test_gpu_verify as base

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,chunk,unc", [
    (MINI_8B, [32] * 12, [32] * 12),                             # prefill: one row of 32
    (MINI_1B, [32, 1, 7, 32, 32, 32], [28, 1, 7, 32, 20, 31]),   # some, all and one of a request's rows
    (MINI_1B, [32] * 20, [31] * 20),                             # 640 tokens, 40 rows: another projection kernel
    (MINI_8B, [32] * 4 + [1], [32] * 4 + [1]),                   # the smallest batch that it is done for, 129 tokens
    (MINI_1B, [32] * 8, [1] * 4 + [32] * 4),                     # 132 rows of 256: all of them
])
def test_results_without_logits_are_those_of_the_logits(shape, chunk, unc):
    r = torch.Generator().manual_seed(len(chunk))
    ctx = [17 * (i % 5) for i in range(len(chunk))]
    batch = gen.gen_batch(Workload("judging", shape, 3, len(ctx), ("list", tuple(ctx)), ("list", tuple(chunk)), 0.7))
    _, _, model, kv, _, _ = base._setup(shape, 3, batch)
    tokens = torch.randint(0, shape.vocab, (sum(chunk),), generator=r, dtype=torch.int32)
    args = (batch.chunk_offsets, batch.page_tables, batch.ctx_lens)
    unc_t = torch.tensor(unc, dtype=torch.int32)
    for _ in range(2):   # with drafts that are nobody's, then with the model's own
        acc, cor, logits = kv.verify_batch(tokens, *args, n_uncached=unc_t, want_logits=True)
        got = kv.verify_batch(tokens, *args, n_uncached=unc_t)
        assert model.status() == 0
        assert torch.equal(got[0], acc) and torch.equal(got[1], cor)
        top = logits.argmax(1).cpu()
        off = [int(v) for v in batch.chunk_offsets]
        for i, (n, u) in enumerate(zip(chunk, unc)):
            a = 0
            while a < n - u and int(top[off[i] + u - 1 + a]) == int(tokens[off[i] + u + a]):
                a += 1
            assert (a, int(top[off[i] + u - 1 + a])) == (int(acc[i]), int(cor[i]))
            for j in range(u, n):
                tokens[off[i] + j] = top[off[i] + j - 1]


@pytest.mark.parametrize("chunk,unc,fewer", [
    ([32] * 5, [32, 31, 32, 1, 32], True),   # 160 tokens, 37 rows
    ([32] * 5, [1] * 5, False),              # every row judges
    ([32] * 4, [32] * 4, False),             # 128 tokens
])
def test_the_step_counts_what_it_ran(chunk, unc, fewer):
    import bench
    import paper_2511_07423_b200 as syn
    shape, T = MINI_1B, sum(chunk)
    batch = gen.gen_batch(Workload("judging", shape, 3, len(chunk), ("list", (16,) * len(chunk)), ("list", tuple(chunk)), 0.7))
    _, _, model, kv, _, _ = base._setup(shape, 3, batch)
    plan = syn.Plan(kv, torch.zeros(T, dtype=torch.int32), batch.chunk_offsets, batch.page_tables, batch.ctx_lens, torch.tensor(unc, dtype=torch.int32))
    rows = sum(n - u + 1 for n, u in zip(chunk, unc)) if fewer else T
    i32 = dict(dtype=torch.int32, device="cuda")
    acc, cor, top1 = torch.empty(len(chunk), **i32), torch.empty(len(chunk), **i32), torch.empty(T, **i32)
    of_plan = plan.stats()
    assert of_plan.kernel_launches == 1 + 5 * shape.n_layers + 2 and of_plan.dense_flops == 2.0 * T * shape.dense_params()
    for out, n in (((acc, cor), rows), ((acc, cor, top1), T)):
        model.set_profile(True)
        plan.run(*out)
        launches = {k: v[1] for k, v in model.get_profile().items()}
        model.set_profile(False)
        st = model.last_step_stats()
        assert st.kernel_launches == of_plan.kernel_launches + (n < T) == sum(launches.values())
        assert launches["verify"] == 1 and launches["judging_rows"] == (n < T)
        assert st.dense_flops == of_plan.dense_flops - 2.0 * (T - n) * shape.d_model * shape.vocab
        assert bench.lm_head_rows(of_plan, st, shape.d_model, shape.vocab) == n
    assert model.status() == 0
