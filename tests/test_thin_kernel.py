"""The thin projection kernel of the batches of few tokens: its launch shape on the CPU, and its product against the
CPU oracle's linear map at the edges of its tiles, of its K parts and of its operand ring."""
import numpy as np
import pytest
import torch

import paper_2511_07423_b200 as syn
from workloads import rng
from workloads.configs import TINY

SHAPES = [(3072, 2048), (2048, 2048), (16384, 2048), (2048, 8192), (32000, 2048), (6144, 4096), (4096, 4096), (28672, 4096),
          (4096, 14336), (128256, 4096), (7168, 5120), (55296, 5120), (5120, 27648), (512, 256), (128, 64), (1408, 688)]


def test_launch_shapes():
    for T in list(range(1, 260)) + [300, 512, 513, 640, 769, 897, 1024]:
        for N, K in SHAPES:
            p = syn.thin_plan_host(T, N, K)
            S, nkb, U = p["splits"], p["num_kb"], p["TN"] // 16 * 4
            assert p["n_tiles"] == -(-N // 128) and nkb == -(-K // 64)
            assert 16 <= p["TN"] <= 128 and p["TN"] % 16 == 0 and (p["n_tt"] - 1) * p["TN"] < T <= p["n_tt"] * p["TN"]
            assert 1 <= S <= min(8, nkb) and 2 <= p["n_stages"] <= 6
            assert p["ring_left"] >= 0                                           # received units and scratch fit in the ring
            bounds = [s * nkb // S for s in range(S + 1)]
            assert all(a < b for a, b in zip(bounds, bounds[1:]))                 # every part of K has a k-block
            for n_units in {U, 4}:                                                # a last token tile may have fewer chunks
                first = [r * n_units // S for r in range(S + 1)]
                for u in range(n_units):
                    o = ((u + 1) * S - 1) // n_units
                    assert first[o] <= u < first[o + 1]
                assert max(b - a for a, b in zip(first, first[1:])) <= -(-U // S)


def test_which_projections_take_it():
    def takes(T, N, K, epi):
        return bool(syn.thin_plan_host(T, N, K, epi)["takes_it"])
    # one token tile: all projections of a layer; the lm_head of a large vocabulary only at very few tokens
    for N, K, epi in ((6144, 4096, "qkv"), (4096, 4096, "resid"), (28672, 4096, "swiglu"), (4096, 14336, "resid"), (32000, 2048, "lmhead")):
        assert takes(128, N, K, epi)
    assert takes(64, 128256, 4096, "lmhead") and not takes(65, 128256, 4096, "lmhead")
    # several: only where a CTA has little to do
    assert takes(256, 3072, 2048, "qkv") and takes(256, 2048, 8192, "resid") and takes(256, 4096, 4096, "resid")
    assert not takes(129, 6144, 4096, "qkv") and not takes(176, 4096, 14336, "resid") and not takes(320, 16384, 2048, "swiglu")
    assert not takes(513, 2048, 2048, "resid")


@pytest.mark.gpu
@pytest.mark.parametrize("T,N,K", [
    (1, 128, 64),         # one token, one k-block
    (16, 128, 688),       # K tail
    (17, 300, 2048),      # two chunks, ragged features, K shared by eight
    (40, 4096, 4096),     # three chunks, K shared by four
    (128, 2048, 2048),    # eight chunks, three stages
    (112, 5120, 1024),    # seven chunks, K shared by three
    (129, 3072, 2048),    # two token tiles of 80 and 49
    (200, 28672, 512),    # whole K per CTA, 448 CTAs
    (256, 6144, 4096),    # two full token tiles
    (97, 640, 14336),     # a long K, seven chunks
])
def test_product_matches_oracle(T, N, K):
    from oracle import Oracle
    key = rng.stream_key(T + N + K, 99)
    x = rng.normal_f32(key, 0, T * K, 1.0).view(T, K).to(torch.float16)
    w = rng.normal_f32(key, T * K, N * K, 0.05).view(N, K).to(torch.bfloat16)
    y = syn.syn_op_linear(x.cuda(), w.cuda(), schedule_as="thin")
    assert torch.equal(y, syn.syn_op_linear(x.cuda(), w.cuda(), schedule_as="thin"))   # fixed summation order
    ref = Oracle(TINY).linear(x.double().numpy(), w)
    scale = np.abs(ref).max()
    err = np.abs(y.cpu().double().numpy() - ref).max()
    assert err <= 2e-5 * scale * max(1.0, (K / 256) ** 0.5), (err, scale)   # fp32 sums, as for the other kernels


def test_two_ctas_to_an_sm():
    """Several token tiles, 56 to 70 items and a K of 64 k-blocks and more: parts in clusters of four, 16 k-blocks or more each.
    Clusters of four beyond 70 do not all run at a time."""
    for T, N, K, splits in ((600, 1408, 4096, 2), (160, 3584, 4096, 4), (272, 2944, 4096, 4), (160, 4480, 4096, 4), (160, 4608, 4096, 2),   # 55, 56, 69, 70, 72
                            (400, 2304, 8192, 2), (256, 4736, 8192, 2), (320, 3200, 4096, 1), (160, 3584, 4032, 2),   # 72, 74, 75; 63 k-blocks
                            (448, 2048, 8192, 4), (512, 2048, 8192, 4), (160, 4096, 4096, 4), (256, 4096, 4096, 4),
                            (320, 2048, 8192, 3), (448, 2048, 2048, 2), (128, 4096, 4096, 4), (160, 6144, 4096, 1), (1024, 3072, 2048, 1)):
        p = syn.thin_plan_host(T, N, K)
        assert p["splits"] == splits, (T, N, K, p)
    assert syn.thin_plan_host(1024, 3072, 2048, "qkv")["takes_it"] and not syn.thin_plan_host(1025, 3072, 2048, "qkv")["takes_it"]
    assert not syn.thin_plan_host(576, 6144, 4096, "qkv")["takes_it"]


@pytest.mark.gpu
@pytest.mark.parametrize("T,N,K", [
    (385, 2048, 4096),    # four token tiles of 112, 49 tokens in the last; 64 items in clusters of four
    (449, 2048, 8192),    # four token tiles of 128, 65 tokens in the last
    (160, 4096, 4160),    # two token tiles of 80, 65 k-blocks in parts of 16 and 17
    (1024, 384, 2048),    # eight token tiles
    (897, 384, 2048),     # the last of eight token tiles has one token: four units for six parts of K, two of which finish nothing
])
def test_products_of_several_token_tiles_match_the_oracle(T, N, K):
    test_product_matches_oracle(T, N, K)
