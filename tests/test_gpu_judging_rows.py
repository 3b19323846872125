"""Calls that ask for no logits run the lm_head over the rows that verification looks at only: the same results as greedy
verification of the logits that the same batch gives where they are asked for.  The small models are compared token for token,
on seeds whose closest pair of logits is decided alike (0.001 apart, below what fp32 sums could move it in the worst case); the
full widths allow for ties at rounding level."""
import dataclasses

import pytest
import torch

from workloads import gen
from workloads.configs import MINI_1B, MINI_8B, SHAPE_1B, Workload

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


@pytest.mark.parametrize("n_req,unc", [(5, 28), (20, 31)])
def test_full_width_tokens_differ_at_rounding_level_ties_only(n_req, unc):
    """The widths of the 1B shape: the lm_head over 25 of 160 and 40 of 640 rows against the logits of the same batch.  A row's
    sums may be taken in another order, so a token whose logit is within the bound of fp32 sums of the largest is as good."""
    import paper_2511_07423_b200 as syn
    from paper_2511_07423_b200 import synthetic
    shape = dataclasses.replace(SHAPE_1B, n_layers=2)
    chunk = [32] * n_req
    batch = gen.gen_batch(Workload("judging", shape, 3, n_req, ("list", (24,) * n_req), ("list", tuple(chunk)), 0.7))
    model = synthetic.load_model(shape, 3)
    kv = syn.KVCache(model, batch.n_pages)
    synthetic.fill_cache(kv, shape, 3, batch)
    # |error| of a sum of d exact products in any order <= d 2^-24 sum |x w| <= d 2^-24 |x| |w|, |x| = sqrt(d) after the norm; two
    # sums of each of two logits
    glob = gen.gen_globals(shape, 3, device="cuda")
    d = shape.d_model
    x_norm = d ** 0.5 * float(glob["final_norm"].float().abs().max())
    bound = 4 * d * 2.0 ** -24 * x_norm * float(glob["lm_head"].float().norm(dim=1).max())
    tokens = torch.randint(0, shape.vocab, (sum(chunk),), generator=torch.Generator().manual_seed(n_req), dtype=torch.int32)
    args, unc_t = (batch.chunk_offsets, batch.page_tables, batch.ctx_lens), torch.full((n_req,), unc, dtype=torch.int32)
    accepted = 0
    for _ in range(4):   # with drafts that are nobody's, then with more and more of the model's own
        _, _, logits = kv.verify_batch(tokens, *args, n_uncached=unc_t, want_logits=True)
        acc, cor = kv.verify_batch(tokens, *args, n_uncached=unc_t)[:2]
        assert model.status() == 0
        for i, n in enumerate(chunk):
            b, rows = 32 * i, logits[32 * i + unc - 1:32 * i + n]
            near = [set(torch.nonzero(r >= r.max() - bound).flatten().tolist()) for r in rows]
            a = int(acc[i])
            accepted += a
            assert all(int(tokens[b + unc + j]) in near[j] for j in range(a)) and int(cor[i]) in near[a]
            if a < n - unc:   # the draft that was turned down is not the only token that the row allows
                assert near[a] != {int(tokens[b + unc + a])}
                tokens[b + unc + a] = int(cor[i])
    assert accepted >= n_req
