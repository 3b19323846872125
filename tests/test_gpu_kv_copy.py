"""syn_kv_import / syn_kv_export: what goes in at any split of a range of positions comes out of any other split."""
import pytest
import torch

from workloads.configs import ModelShape

from harness import cpu_model, to_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd,Hkv,n,cuts", [
    (64, 2, 37, (1, 17)),               # a few rows of three pages
    (128, 1, 300, (16, 16, 255)),       # page boundaries, an empty piece left out
    (64, 2, 192 * 16 + 5, (7,)),        # one page more than the small launch carries
    (64, 2, 960 * 16 + 40, (3, 4000)),  # more pages than one launch carries
])
@pytest.mark.parametrize("offset", [0, 1], ids=["aligned", "odd_address"])
def test_pieces_in_whole_out(hd, Hkv, n, cuts, offset):
    import paper_2511_07423_b200 as syn
    shape = ModelShape("kv", 2, 128, 2 * Hkv, Hkv, hd, 128, 256)
    model = syn.Model(shape, *to_cuda(*cpu_model(shape, 3)))
    n_pages = (n + 15) // 16 + 3
    kv = syn.KVCache(model, n_pages)
    gen = torch.Generator().manual_seed(n)
    table = torch.randperm(n_pages, generator=gen).to(torch.int32)
    # eighths of integers: exact in bf16 and in half precision (a normal deviate below 2^-17 would not be)
    flat = (torch.randint(-128, 129, (2 * n * Hkv * hd + offset,), generator=gen) / 8).to(torch.bfloat16).cuda()[offset:]
    k, v = flat.view(2, n, Hkv, hd)
    edges = sorted({0, *cuts, n})
    for a, b in zip(edges, edges[1:]):
        kv.import_kv(1, table, a, k[a:b], v[a:b])
    out = kv.export_kv(1, table, 0, n)
    assert torch.equal(out[0], k) and torch.equal(out[1], v)
    a = n // 3
    out = kv.export_kv(1, table, a, n - a)
    assert torch.equal(out[0], k[a:]) and torch.equal(out[1], v[a:])
    assert not kv.export_kv(0, table, 0, n)[0].any()          # the other layer is untouched
