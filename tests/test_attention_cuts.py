"""Work lists of batches with about one (request, kv head) unit to a CTA: units laid end to end over the CTAs and cut where
one is full.  On the CPU the cover of every unit; on the device the attention of such lists against the oracle."""
import random

import numpy as np
import pytest
import torch

import paper_2511_07423_b200 as syn
from workloads.configs import ModelShape

import test_gpu_attention as base


def _lengths(n, seed, hi):
    r = random.Random(seed)
    return [r.choice([0, 1, 63, 64, 65, r.randint(2, hi)]) for _ in range(n)], [r.randint(1, 8) for _ in range(n)]


@pytest.mark.parametrize("export", [syn.plan_work_host, syn.plan_host], ids=["step", "one_cta_per_sm"])
@pytest.mark.parametrize("kind", [0, 1, 2, 3])
@pytest.mark.parametrize("n_req,heads,hd,hi", [(10, 8, 128, 900), (17, 8, 128, 4000), (19, 8, 128, 4000), (36, 8, 64, 2000), (7, 21, 128, 2000), (1, 1, 64, 20)])
def test_cut_units_are_covered_exactly_once(kind, n_req, heads, hd, hi, export):
    ctx, chunk = _lengths(n_req, n_req, hi)
    off = np.concatenate([[0], np.cumsum(chunk)]).tolist()
    pages = [(a + b + 15) // 16 for a, b in zip(ctx, chunk)]
    table = torch.zeros(n_req, max(pages), dtype=torch.int32)
    for i, first in enumerate(np.cumsum([0] + pages[:-1])):
        table[i, :pages[i]] = torch.arange(first, first + pages[i], dtype=torch.int32)
    syn.debug_set_attention(kind)
    try:
        p = export(ModelShape("cut", 1, 256, 4 * heads, heads, hd, 256, 512), sum(pages),
                   torch.zeros(off[-1], dtype=torch.int32), off, table, ctx)
    finally:
        syn.debug_set_attention(0)
    cb, n_cta = p["cta_begin"].numpy(), p["n_cta"]
    items = p["items"].numpy()
    assert cb[0] == 0 and cb[n_cta] == len(items) and (np.diff(cb[:n_cta + 1]) >= 1).all()
    assert n_cta <= (296 if p.get("attention") == 3 else 148)   # the half-SM kernel runs two CTAs to an SM
    assert p.get("attention", kind) == (kind or p.get("attention", 0))
    units = {}
    for q, nj, h, req, kb, ke, _, part, group in items[:, :9]:
        assert kb % 64 == 0 and kb < ke and off[req] <= q and q + nj <= off[req + 1]
        units.setdefault((req, q, nj, h), []).append((kb, ke, part, group))
    assert len(units) == sum(-(-n // (16 if p["stats"].attn_rows == 64 else 32)) for n in chunk) * heads
    for (req, q, nj, h), v in units.items():
        v.sort()
        assert v[0][0] == 0 and v[-1][1] == ctx[req] + q - off[req] + nj
        assert (len(v) == 1) == (v[0][2] < 0)
        for a, b in zip(v, v[1:]):
            assert b[0] == a[1] and b[2] == a[2] + 1 and b[3] == a[3]   # one group, its partials side by side
    parts = sorted(x[7] for x in items if x[7] >= 0)
    assert parts == list(range(len(parts)))


@pytest.mark.parametrize("kind", [0, 1, 2, 3])
@pytest.mark.parametrize("heads,hd", [(8, 128), (8, 64)])
def test_few_long_requests_among_many_short_ones_are_not_cut_small(kind, heads, hd):
    """More than two units to a CTA: a long one is cut into parts of about a CTA's fair share, no smaller, so there are no more
    parts than CTAs."""
    ctx, chunk = [5953] * 3 + [100] * 80, [32] * 3 + [4] * 80
    off = np.concatenate([[0], np.cumsum(chunk)]).tolist()
    pages = [(a + b + 15) // 16 for a, b in zip(ctx, chunk)]
    table = torch.zeros(len(ctx), max(pages), dtype=torch.int32)
    for i, first in enumerate(np.cumsum([0] + pages[:-1])):
        table[i, :pages[i]] = torch.arange(first, first + pages[i], dtype=torch.int32)
    syn.debug_set_attention(kind)
    try:
        p = syn.plan_work_host(ModelShape("cut", 1, 256, 4 * heads, heads, hd, 256, 512), sum(pages),
                               torch.zeros(off[-1], dtype=torch.int32), off, table, ctx)
    finally:
        syn.debug_set_attention(0)
    cb, items = p["cta_begin"].numpy(), p["items"].numpy()
    keys = [int((items[a:b, 5] - items[a:b, 4]).sum()) for a, b in zip(cb, cb[1:])]
    assert 0 < p["stats"].attn_split_items <= p["n_cta"], p["stats"].attn_split_items
    assert max(keys) <= 1.5 * sum(keys) / len(keys)


@pytest.mark.parametrize("n_req", range(15, 21))
def test_a_little_less_than_one_or_one_unit_to_an_sm_is_shared_out_over_all_ctas(n_req):
    """120 to 160 units of unequal lengths on the 296 CTAs of the half-SM kernel."""
    syn.debug_set_attention(3)
    try:
        for seed in range(8):
            r = random.Random(seed)
            ctx = [r.randint(256, 2048) for _ in range(n_req)]
            pages = [(n + 20) // 16 for n in ctx]
            table = torch.zeros(n_req, max(pages), dtype=torch.int32)
            for i, first in enumerate(np.cumsum([0] + pages[:-1])):
                table[i, :pages[i]] = torch.arange(first, first + pages[i], dtype=torch.int32)
            p = syn.plan_work_host(ModelShape("cut", 1, 256, 32, 8, 128, 256, 512), sum(pages),
                                   torch.zeros(5 * n_req, dtype=torch.int32), list(range(0, 5 * n_req + 1, 5)), table, ctx)
            cb, items = p["cta_begin"].numpy(), p["items"].numpy()
            keys = [int((items[a:b, 5] - items[a:b, 4]).sum()) for a, b in zip(cb, cb[1:])]
            assert len(keys) > 256 and max(keys) <= 1.95 * sum(keys) / 296, (seed, len(keys), max(keys))
    finally:
        syn.debug_set_attention(0)


@pytest.mark.parametrize("kind", [0, 1, 2, 3])
@pytest.mark.parametrize("heads,hd,group", [(8, 128, 4), (8, 64, 4), (21, 128, 1), (2, 64, 5)])
def test_no_plan_has_more_partials_than_the_static_array_holds(kind, heads, hd, group):
    """syn_op_attention_static: 592 partials of 64 rows, 296 of 128.  Lists end to end have two a CTA at most, equal parts no
    more than CTAs, and where a CTA has several units fewer than one a CTA and one more for each unit that is cut."""
    r = random.Random(heads * hd + kind)
    syn.debug_set_attention(kind)
    try:
        for _ in range(60):
            n_long, n_short = r.randint(1, max(1, 320 // heads)), r.choice([0, r.randint(0, 620 // heads)])
            hi = r.randint(300, 6000)
            ctx = [hi + r.randint(0, hi // r.choice([1, 4, 1000])) for _ in range(n_long)] + [r.randint(1, 60) for _ in range(n_short)]
            chunk = [r.choice([1, 5, 32])] * n_long + [r.choice([1, 4])] * n_short
            off = np.concatenate([[0], np.cumsum(chunk)]).tolist()
            pages = [(a + b + 15) // 16 for a, b in zip(ctx, chunk)]
            table = torch.zeros(len(ctx), max(pages), dtype=torch.int32)
            for i, first in enumerate(np.cumsum([0] + pages[:-1])):
                table[i, :pages[i]] = torch.arange(first, first + pages[i], dtype=torch.int32)
            s = syn.plan_work_host(ModelShape("cut", 1, 256, group * heads, heads, hd, 256, 512), sum(pages),
                                   torch.zeros(off[-1], dtype=torch.int32), off, table, ctx)["stats"]
            assert s.attn_split_items * s.attn_rows <= 592 * 64, (ctx, chunk)
    finally:
        syn.debug_set_attention(0)


def test_keys_that_may_be_read_before_the_chunks_are_written():
    """Up to the first page of a request that any request of the batch writes, over shared pages too; nothing in the lists of the
    kernels that wait for the projection first."""
    table = torch.tensor([[5, 1, 7, 2, 0, 4, 9], [5, 1, 7, 2, 0, 4, 8], [3, 6, 10, -1, -1, -1, -1], [5, 1, 7, 2, 11, -1, -1],
                          [12, -1, -1, -1, -1, -1, -1]], dtype=torch.int32)
    # request 0 writes 48..79 (pages 2 and 0), request 1 reads up to 95 through the same pages and writes page 8, request 2
    # ends on a page boundary, request 3 shares pages 5, 1, 7 and writes 64.. in a page of its own, request 4 has three keys
    ctx, chunk = [48, 96, 32, 64, 3], [32, 4, 16, 2, 1]
    off = [0] + np.cumsum(chunk).tolist()
    for kind, want in ((3, {0: 48, 1: 48, 2: 32, 3: 48, 4: 0}), (1, dict.fromkeys(range(5), 0)), (2, dict.fromkeys(range(5), 0))):
        syn.debug_set_attention(kind)
        try:
            p = syn.plan_work_host(ModelShape("safe", 1, 256, 8, 2, 64, 256, 512), 13, torch.zeros(off[-1], dtype=torch.int32), off, table, ctx)
        finally:
            syn.debug_set_attention(0)
        assert p["attention"] == kind
        assert {(int(r[3]), int(r[9])) for r in p["items"]} == set(want.items())


@pytest.mark.gpu
@pytest.mark.parametrize("kind", [0, 1, 2, 3])
@pytest.mark.parametrize("hd,Hkv,n_req", [(128, 8, 20), (64, 8, 20), (128, 8, 36)])
def test_cut_units_match_the_oracle(hd, Hkv, n_req, kind):
    ctx, chunk = _lengths(n_req, 5, 900)
    syn.debug_set_attention(kind)
    try:
        base._run(hd, 4 * Hkv, Hkv, ctx, chunk)
    finally:
        syn.debug_set_attention(0)
