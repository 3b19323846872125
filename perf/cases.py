"""The measured work of this framework: verification batches, sampled verification, a serving loop and
K/V transfers, through the public entry points, from one device's four drafts on a small model to 256
devices on the 8B shape.

A case is a dict of plain values:
  entry     "batch"    KVCache.verify_batch: host metadata in, results and logits out (blocking)
            "resident" Plan.run: the same step with the batch description kept on the device
            "sampled"  verify_batch_sampled: sampling-based verification (top-k / top-p)
            "serve"    Scheduler: prompts arrive, are prefilled in 32-token chunks, then rounds of verification
            "move"     KVCache.import_kv and export_kv of one request's prefix, every layer
  model     shape of workloads.configs; layers: how many of its layers (fewer than the shape has where three
            copies of weights and cache would not fit one GPU)
  requests  devices in the batch; ctx_lo..ctx_hi cached tokens of each (log-uniform when the range spans more
            than a factor of ten); chunk_lo..chunk_hi tokens a device offloads, of which at most `drafts` at the end are
            drafts and the others accepted tokens that the cache does not hold yet; short: share of the devices
            that send a single token
Lengths follow from the case, contents from the seed.

The weights are random but the model is not: row next[v] of the lm_head leans towards the embedding of v, and
the projections that write the residual stream are scaled down with the depth, so that the model predicts
next[v] after v with the kind of margin a trained model has (ten and more standard deviations of the logits against
the 4.5 that the best of 128 000 random ones reach).  A device's drafts follow that chain with probability
P_MATCH, as the configurations have it, so accept lengths are spread over their range and do not hang on ties.
"""
from __future__ import annotations

import dataclasses
import math
import random

import numpy as np
import torch

import paper_2511_07423_b200 as syn
from workloads.configs import SHAPE_1B, SHAPE_32B, SHAPE_8B, TINY

SHAPES = {"tiny": TINY, "1b": SHAPE_1B, "8b": SHAPE_8B, "32b": SHAPE_32B}
P_MATCH = 0.65
EMBED_STD = 2.0
PAGE = 16
SERVE_ROUNDS = 2
SLM_K, TOP_K, TOP_P, TEMPERATURE = 20, 50, 0.95, 1.5


def _case(name, entry, model, layers, requests, ctx, chunk, drafts=31, short=0.0):
    c = dict(entry=entry, model=model, layers=layers, requests=requests, ctx_lo=ctx[0], ctx_hi=ctx[1], chunk_lo=chunk[0],
             chunk_hi=chunk[1], drafts=drafts, short=short)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a handful of devices on a draft-sized model: launches and latency only
        _case("tiny-4", "batch", "tiny", 2, 4, (48, 128), (4, 4)),
        # one device waits for its verdict on four drafts: the latency a user feels when the cloud is idle
        _case("1b-one-device", "batch", "1b", 16, 1, (777, 777), (5, 5)),
        # the ordinary batch of the 1B shape: ragged chunks of 1 to 8 tokens
        _case("1b-32", "batch", "1b", 16, 32, (256, 2048), (1, 8)),
        # a lightly loaded 8B cloud: eight devices, four drafts each
        _case("8b-8", "batch", "8b", 32, 8, (512, 4096), (5, 5)),
        # sampling-based verification at moderate load
        _case("8b-24-sampled", "sampled", "8b", 32, 24, (512, 4096), (2, 9)),
        # the benchmark's workload: 64 devices, chunks of 1 to 16, batch description resident on the device
        _case("8b-64-resident", "resident", "8b", 32, 64, (512, 4096), (1, 16)),
        # many devices with contexts from short to very long, most of them sending one token
        _case("8b-256-mixed", "batch", "8b", 16, 256, (128, 8192), (2, 16), short=0.6),
        # chunked partial prefill: 28 tokens to cache and four drafts in every chunk
        _case("8b-64-chunk32", "batch", "8b", 32, 64, (512, 4096), (32, 32), drafts=4),
        # the 32B width, five query heads to a kv head, long contexts
        _case("32b-128", "batch", "32b", 8, 128, (1024, 6000), (1, 16)),
        # a serving loop from prompt to verdict: prefill iterations of up to 768 tokens, then verification rounds
        _case("1b-serve-24", "serve", "1b", 16, 24, (40, 200), (3, 8)),
        # a prefix that another server computed is placed in the cache, and one is handed on
        _case("8b-move", "move", "8b", 32, 1, (2600, 2600), (1, 1)),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    entry = rng.choice(("batch", "batch", "batch", "resident", "resident", "sampled", "serve", "move"))
    model = rng.choice(("tiny", "1b", "1b", "8b", "8b", "32b"))
    if entry == "move":
        n = _log(rng, 17, 4096)
        model = rng.choice(("1b", "8b"))
        return _case(None, entry, model, 16 if model == "1b" else 32, 1, (n, n), (1, 1))
    layers = {"tiny": 2, "1b": 16, "8b": rng.choice((12, 20)), "32b": rng.choice((4, 8))}[model]
    if entry == "serve":
        model, layers = rng.choice((("tiny", 2), ("1b", 16)))
        lo = _log(rng, 8, 100)
        hi = lo + _log(rng, 8, 120)
        if model == "tiny":
            return _case(None, entry, model, layers, _log(rng, 1, 8), (lo, hi), (2, rng.randint(3, 6)))
        return _case(None, entry, model, layers, _log(rng, 1, 48), (lo, hi), (2, rng.randint(3, 9)))
    lo = _log(rng, 16, 1024)
    hi = _log(rng, lo, 8192 if model != "tiny" else 1024)
    requests = _log(rng, 1, {"tiny": 8, "1b": 192, "8b": 192, "32b": 96}[model])
    shape = rng.choice(("drafts", "drafts", "ragged", "mixed", "prefill"))
    short = 0.0
    drafts = 31
    if shape == "drafts":
        n = rng.randint(2, 8)
        chunk = (n, n)
    elif shape == "ragged":
        chunk = (1, rng.randint(3, 16))
    elif shape == "mixed":
        chunk, short = (2, rng.randint(3, 16)), 0.6
    else:
        n = rng.randint(17, 32)
        chunk, drafts, requests = (n, n), rng.randint(1, 5), min(requests, 48)
    if entry == "sampled":
        requests = min(requests, 64)
    return _case(None, entry, model, layers, requests, (lo, hi), chunk, drafts, short)


# ------------------------------------------------------------------------------------------ what a case is made of

def _shape(case):
    return dataclasses.replace(SHAPES[case["model"]], n_layers=case["layers"])


def _lengths(case):
    """Context, chunk and accepted-token lengths of every request."""
    rng = random.Random("/".join("%s=%s" % (k, case[k]) for k in sorted(case) if k != "name"))
    lo, hi = case["ctx_lo"], case["ctx_hi"]
    ctx = [_log(rng, lo, hi) if hi > 10 * lo else rng.randint(lo, hi) for _ in range(case["requests"])]
    chunk = [1 if rng.random() < case["short"] else rng.randint(case["chunk_lo"], case["chunk_hi"]) for _ in ctx]
    return ctx, chunk, [max(1, n - case["drafts"]) for n in chunk]


def _next_token(shape, gen):
    return torch.randperm(shape.vocab, generator=gen, device="cuda")


def _weights(shape, gen):
    d, std = shape.d_model, shape.weight_std
    out_std = std / math.sqrt(2 * shape.n_layers)   # the projections that write the residual stream

    def normal(rows, cols, s):
        return torch.empty(rows, cols, dtype=torch.bfloat16, device="cuda").normal_(0.0, s, generator=gen)

    def gain():
        return torch.empty(d, dtype=torch.float32, device="cuda").normal_(1.0, shape.gain_std, generator=gen).to(torch.bfloat16)

    nxt = _next_token(shape, gen)
    embed = normal(shape.vocab, d, EMBED_STD)
    lean = min(0.9, 18.0 / math.sqrt(d))
    head = normal(shape.vocab, d, math.sqrt(1.0 - lean * lean))
    head[nxt] += (lean / EMBED_STD) * embed
    head /= math.sqrt(d)
    glob = {"embed": embed, "lm_head": head, "final_norm": gain()}
    layers = [{"wq": normal(shape.q_dim, d, std), "wk": normal(shape.kv_dim, d, std), "wv": normal(shape.kv_dim, d, std),
               "wo": normal(d, shape.q_dim, out_std), "wg": normal(shape.d_ffn, d, std), "wu": normal(shape.d_ffn, d, std),
               "wd": normal(d, shape.d_ffn, out_std), "norm1": gain(), "norm2": gain()} for _ in range(shape.n_layers)]
    return glob, layers, nxt


def _fill_cache(kv, shape, gen):
    """K and V of every slot of the pool, at the scale a projection of a normalised vector has."""
    s = shape.weight_std * math.sqrt(shape.d_model)
    pages = torch.arange(kv.n_pages, dtype=torch.int32)
    for layer in range(shape.n_layers):
        k, v = (torch.empty(kv.n_pages * PAGE, shape.n_kv_heads, shape.head_dim, dtype=torch.bfloat16, device="cuda")
                .normal_(0.0, s, generator=gen) for _ in range(2))
        kv.import_kv(layer, pages, 0, k, v)


def _chain(nxt, start, n, right):
    """n tokens from `start` on: the model's own continuation where `right`, otherwise the given stray token."""
    out = [start]
    for j in range(1, n):
        out.append(int(nxt[out[-1]]) if right[j] < 0 else int(right[j]))
    return out


def _strays(np_rng, vocab, n, first):
    """-1 where a token follows the chain; a random token with probability 1 - P_MATCH from index `first` on."""
    miss = np_rng.random(n) >= P_MATCH
    miss[:first] = False
    return np.where(miss, np_rng.integers(0, vocab, n), -1)


def prepare(case, seed):
    shape = _shape(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    np_rng = np.random.default_rng(seed)
    ctx, chunk, uncached = _lengths(case)
    if case["entry"] == "move":
        return _prepare_move(shape, gen, np_rng, ctx[0])
    glob, layers, nxt = _weights(shape, gen)
    model = syn.Model(shape, glob, layers)
    del glob, layers
    torch.cuda.empty_cache()   # the library holds its own copy
    nxt = nxt.cpu().numpy()
    state = {"case": case, "model": model}
    if case["entry"] == "serve":
        extra = SERVE_ROUNDS * (case["chunk_hi"] + 1)
        state["kv"] = syn.KVCache(model, sum(-(-(c + extra) // PAGE) + 1 for c in ctx))
        state["sched"] = syn.Scheduler(state["kv"])
        state["prompts"] = [torch.tensor(_chain(nxt, int(np_rng.integers(shape.vocab)), n, np.full(n, -1)), dtype=torch.int32) for n in ctx]
        state["chunk"], state["next"] = chunk, nxt.tolist()
        state["strays"] = [[_strays(np_rng, shape.vocab, n, 1).tolist() for _ in range(SERVE_ROUNDS)] for n in chunk]
        return state
    pages = [-(-(c + n) // PAGE) for c, n in zip(ctx, chunk)]
    perm = np_rng.permutation(sum(pages)).astype(np.int32)   # logical neighbours lie anywhere in the pool
    table = np.full((len(ctx), max(pages)), -1, dtype=np.int32)
    at = 0
    for i, n in enumerate(pages):
        table[i, :n] = perm[at:at + n]
        at += n
    kv = syn.KVCache(model, sum(pages))
    _fill_cache(kv, shape, gen)
    toks = []
    for n, u in zip(chunk, uncached):
        toks += _chain(nxt, int(np_rng.integers(shape.vocab)), n, _strays(np_rng, shape.vocab, n, u))
    T = len(toks)
    state.update(kv=kv, tokens=torch.tensor(toks, dtype=torch.int32), tables=torch.from_numpy(table),
                 offsets=torch.tensor([0] + np.cumsum(chunk).tolist(), dtype=torch.int32),
                 ctx=torch.tensor(ctx, dtype=torch.int32), uncached=torch.tensor(uncached, dtype=torch.int32))
    if case["entry"] == "resident":
        dev = dict(dtype=torch.int32, device="cuda")
        state["plan"] = syn.Plan(kv, state["tokens"], state["offsets"], state["tables"], state["ctx"], state["uncached"])
        state["out"] = (torch.empty(len(ctx), **dev), torch.empty(len(ctx), **dev), torch.empty(T, **dev),
                        torch.empty(T, shape.vocab, dtype=torch.float32, device="cuda"))
    elif case["entry"] == "sampled":
        # what a device transmits: its draft with 0.7, the rest of its distribution spread over other tokens
        ids = np_rng.integers(0, shape.vocab, (T, SLM_K)).astype(np.int32)
        ids[:, 0] = toks
        probs = np.full((T, SLM_K), 0.3 / (SLM_K - 1), dtype=np.float32)
        probs[:, 0] = 0.7
        state["sampling"] = (syn.Sampling(TOP_K, TOP_P, TEMPERATURE, SLM_K), torch.from_numpy(ids), torch.from_numpy(probs),
                             torch.from_numpy(np_rng.random(T, dtype=np.float32)), torch.from_numpy(np_rng.random(len(ctx), dtype=np.float32)))
    return state


def _prepare_move(shape, gen, np_rng, n):
    # a cache belongs to a model: the same K/V geometry over a narrow MLP and vocabulary
    narrow = dataclasses.replace(shape, d_ffn=256, vocab=256)
    glob, layers, _ = _weights(narrow, gen)
    model = syn.Model(narrow, glob, layers)
    pages = -(-n // PAGE)
    kv = syn.KVCache(model, 2 * pages)
    s = shape.weight_std * math.sqrt(shape.d_model)
    kvs = torch.empty(shape.n_layers, 2, n, shape.n_kv_heads, shape.head_dim, dtype=torch.bfloat16, device="cuda").normal_(0.0, s, generator=gen)
    return {"case": {"entry": "move"}, "model": model, "kv": kv, "k_v": kvs,
            "table": torch.from_numpy(np_rng.permutation(2 * pages)[:pages].astype(np.int32))}


# ------------------------------------------------------------------------------------------ one pass

def run(state):
    entry = state["case"]["entry"]
    if entry == "batch":
        return state["kv"].verify_batch(state["tokens"], state["offsets"], state["tables"], state["ctx"], state["uncached"], want_logits=True)
    if entry == "resident":
        state["plan"].run(*state["out"])
        return state["out"]
    if entry == "sampled":
        return syn.verify_batch_sampled(state["kv"], state["tokens"], state["offsets"], state["tables"], state["ctx"], state["uncached"],
                                        *state["sampling"], want_logits=True)
    if entry == "serve":
        return _serve(state)
    kv, table, k_v = state["kv"], state["table"], state["k_v"]
    n = k_v.shape[2]
    for layer in range(k_v.shape[0]):
        kv.import_kv(layer, table, 0, k_v[layer, 0], k_v[layer, 1])
    return [kv.export_kv(layer, table, 0, n) for layer in range(k_v.shape[0])]


def _serve(state):
    """Every prompt arrives, is prefilled, offloads SERVE_ROUNDS chunks and leaves."""
    sched, nxt = state["sched"], state["next"]
    rounds = [0] * len(state["prompts"])
    log = []
    for r, prompt in enumerate(state["prompts"]):
        sched.add_request(r, prompt)
    while True:
        kind, results = sched.step()
        if kind == "idle":
            return torch.tensor(log, dtype=torch.int32)
        for x in results:
            r = x["req_id"]
            log.append((r, x["kind"], x["n_tokens"], x["accept_len"], x["correction_token"], x["ctx_len"]))
            if not x["prompt_done"]:
                continue
            if rounds[r] == SERVE_ROUNDS:
                sched.finish(r)
                continue
            chunk = _chain(nxt, x["correction_token"], state["chunk"][r], state["strays"][r][rounds[r]])
            sched.add_verify(r, chunk, 1)
            rounds[r] += 1


# ------------------------------------------------------------------------------------------ work and tolerance

def _step_work(shape, T, keys_read, keys_seen, logit_rows):
    """One step: projections, the lm_head and the cached K and V read once, new K and V and the logits written once."""
    kv_token = shape.kv_bytes_per_token()
    by = 2.0 * shape.dense_params() + keys_read * kv_token + T * kv_token + 4.0 * logit_rows * shape.vocab + 2.0 * T * shape.d_model
    fl = 2.0 * T * shape.dense_params() + 4.0 * shape.q_dim * shape.n_layers * keys_seen
    return by, fl


def work(case):
    shape = _shape(case)
    ctx, chunk, _ = _lengths(case)
    if case["entry"] == "move":   # placed and handed on: each a read and a write
        return {"bytes": 4.0 * ctx[0] * shape.kv_bytes_per_token(), "flops": 0.0}
    if case["entry"] == "serve":
        by = fl = 0.0
        steps = [[(at, min(32, n - at)) for n in ctx if at < n] for at in range(0, max(ctx), 32)]
        steps += [[(c + 1 + r * (n + 1) // 2, n) for c, n in zip(ctx, chunk)] for r in range(SERVE_ROUNDS)]
        for s in steps:
            b, f = _step_work(shape, sum(n for _, n in s), sum(c + n for c, n in s), sum(n * c + n * (n + 1) / 2 for c, n in s), 0)
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    T = sum(chunk)
    by, fl = _step_work(shape, T, sum(c + n for c, n in zip(ctx, chunk)), sum(n * c + n * (n + 1) / 2 for c, n in zip(ctx, chunk)), T)
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """Half-precision operands, fp32 sums.  The logits of one batch under the other schedules of the projections and
    of the attention (the same operands, sums in another order) are off by at most 0.00063 in the 2-norm and by 0.0037
    of their root mean square, about the same at 32 layers of the 8B width as at 8 of the 32B width; four times that is
    stated.  The tokens have margins far wider than that, and a K/V copy is exact."""
    if case["entry"] in ("move", "serve"):
        return "exact"
    return {"rel": 0.0025, "max": 0.015, "differ": 0.0}
