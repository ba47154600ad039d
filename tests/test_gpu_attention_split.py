"""Attention with a sequence's pages split over several CTAs (csrc/attn.cu): page counts on both sides of every split, uneven
runs, one and several row tiles, chain and tree masks, grouped heads, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from helpers import dev_i32, ensure_built, weights_to
from oracle import forward as O
from paper_2408_05676_b200 import synth
from test_gpu_forward import TOL, _fill_both, _step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    ensure_built()
    from paper_2408_05676_b200 import binding
    return binding


# caches of 16 pages or more are split: runs of twelve pages (192 tokens), dealt to up to eight CTAs in turn
@pytest.mark.parametrize("over,ctx,precise", [
    (dict(), [230], 0), (dict(), [231], 1), (dict(), [247], 1), (dict(), [248, 3], 1), (dict(), [300], 0), (dict(), [640, 77], 1), (dict(), [1000], 0),
    (dict(max_draft=16), [700], 1), (dict(max_draft=40), [300, 9, 500], 1), (dict(n_kv_heads=2, max_draft=3), [410, 0, 170], 1),
    (dict(d_model=512, head_dim=128, d_ffn=512), [333], 0),
])
def test_split_pages_match_the_oracle(L, over, ctx, precise):
    cfg = synth.model_cfg("tiny", **dict(over, precise=precise))
    Wc = synth.make_weights(cfg, seed=0, gain_jitter=0.1)
    B, K = len(ctx), cfg["max_draft"]
    pages = max(32, (max(ctx) + K + 16) // 16 + 1)
    m = L.model_create(cfg, weights_to(Wc, "cuda"), max_batch=B)
    kv = L.kv_create(m, B, B * pages)
    L.kv_set_page_table(kv, np.random.default_rng(1).permutation(B * pages).astype(np.int32))
    okv = O.KVCache(cfg, B, pages * 16)
    _fill_both(L, cfg, kv, okv, range(B), ctx, seed=7)
    rows = [synth.make_prompt(K + 1 - b % 2, cfg["vocab"], 30 + b) for b in range(B)]
    err, logits = _step(L, m, kv, cfg, Wc, okv, list(range(B)), rows)
    print("max-abs logit error %.2e" % err)
    assert err <= (TOL / 10 if precise else TOL)
    # a chain given as a tree uses the row masks instead of the causal limit
    tokens, parents = np.full((B, K + 1), -1, np.int32), np.full((B, K + 1), -1, np.int32)
    for b, r in enumerate(rows):
        tokens[b, :len(r)] = r
        parents[b, 1:len(r)] = np.arange(len(r) - 1)
    n_rows = [len(r) for r in rows]
    tree = L.verify_step_tree(m, kv, dev_i32(range(B)), dev_i32(tokens), dev_i32(parents), dev_i32(n_rows))
    L.check(m)
    for b in range(B):
        assert (tree[b, :n_rows[b]] - logits[b, :n_rows[b]]).abs().max().item() <= (TOL / 100 if precise else TOL / 2)


# Splits in six, four, three and two (64, 96, 144 and 192 pairs of sequence and head), none with the deep ring (240) and with the
# short one (448); one run against two (192 and 193 keys) and uneven deals of runs to CTAs, in a cache larger than the texts
@pytest.mark.parametrize("B,K,precise", [(16, 8, 0), (24, 8, 0), (24, 8, 1), (36, 3, 1), (48, 2, 1), (12, 20, 1), (60, 2, 0), (112, 1, 1)])
def test_fewer_splits(L, B, K, precise):
    cfg = synth.model_cfg("tiny", max_draft=K, precise=precise)
    Wc = synth.make_weights(cfg, seed=0, gain_jitter=0.1)
    pages = 64
    m = L.model_create(cfg, weights_to(Wc, "cuda"), max_batch=B)
    kv = L.kv_create(m, B, B * pages)
    okv = O.KVCache(cfg, B, pages * 16)
    ctx = ([192 - K - 1, 192 - K, 191, 192, 383 - K, 384 - K, 500, 640, 650, 0, 1000] * 11)[:B]
    _fill_both(L, cfg, kv, okv, range(B), ctx, seed=7)
    rows = [synth.make_prompt(K + 1, cfg["vocab"], 30 + b) for b in range(B)]
    err, _ = _step(L, m, kv, cfg, Wc, okv, list(range(B)), rows)
    print("max-abs logit error %.2e" % err)
    assert err <= (TOL / 10 if precise else TOL)


# What is summed in which order follows from the page numbers alone: the same bits in a cache of any capacity, and for a row
# among drafts and alone, also where the drafts reach into another page or run
@pytest.mark.parametrize("B,K,ctx", [(1, 8, 189), (2, 8, 505), (1, 20, 380), (24, 8, 380), (48, 4, 190), (60, 4, 126)])
def test_same_bits_in_any_capacity_and_alone(L, B, K, ctx):
    cfg = synth.model_cfg("tiny", max_draft=K)
    m = L.model_create(cfg, weights_to(synth.make_weights(cfg, seed=0, gain_jitter=0.1), "cuda"), max_batch=B)
    text, ids = synth.make_prompt(K + 1, cfg["vocab"], 30), dev_i32(range(B))
    first = None
    for pages in (34, 100, 256):
        kv = L.kv_create(m, B, B * pages)
        for l in range(cfg["n_layers"]):
            k, v = synth.make_kv_layer(ctx, cfg["n_kv_heads"] * cfg["head_dim"], 7, l, device="cuda")
            for b in range(B):
                L.kv_import(kv, b, l, 0, k, v)
        L.kv_set_len(kv, list(range(B)), [ctx] * B)
        full = L.verify_step(m, kv, ids, dev_i32(np.tile(text, (B, 1))), dev_i32([K + 1] * B))
        first = full if first is None else first
        assert torch.equal(first, full), "%d pages" % pages
        rows = np.full((B, K + 1), -1, np.int32)
        for i in range(K + 1):
            rows[:, 0] = text[i]
            L.kv_set_len(kv, list(range(B)), [ctx + i] * B)
            alone = L.verify_step(m, kv, ids, dev_i32(rows), dev_i32([1] * B))
            assert torch.equal(alone[:, 0], full[:, i]), "row %d, %d pages" % (i, pages)
    L.check(m)
