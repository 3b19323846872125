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
