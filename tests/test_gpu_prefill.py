"""Prompt processing (csrc/attn_prefill.cu, prefill passes): what a generation leaves in the cache for its prompts, against the
fp64 oracle.  Prompt lengths on both sides of a chunk, of a page and of the four chunks that share a CTA; prompts of one token, whose
neighbours share a CTA with theirs; grouped heads, both head sizes, the precise mode, several passes."""
import numpy as np
import pytest

from helpers import ensure_built, weights_to
from oracle import forward as O
from oracle import generate as G
from paper_2408_05676_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    ensure_built()
    from paper_2408_05676_b200 import binding
    return binding


@pytest.mark.parametrize("over,lens", [
    (dict(), [1, 2, 17, 33, 34, 1, 65, 66, 97, 128, 129, 130, 161]),
    (dict(n_kv_heads=2), [130, 5, 257, 48]),
    (dict(d_model=512, head_dim=128, d_ffn=512), [40, 1, 290, 33, 32]),
    (dict(precise=1), [70, 1, 150]),
    (dict(n_layers=2), [260] * 11 + [7]),          # 2855 tokens: more than one pass
])
def test_cache_of_the_prompts(L, over, lens):
    cfg = synth.model_cfg("tiny", **dict(dict(n_layers=3), **over))
    Wc = synth.make_weights(cfg, seed=0, gain_jitter=0.1)
    B, pages = len(lens), (max(lens) + 1 + cfg["max_draft"] + 15) // 16
    m = L.model_create(cfg, weights_to(Wc, "cuda"), max_batch=B)
    kv = L.kv_create(m, B, B * pages)
    L.kv_set_page_table(kv, np.random.default_rng(1).permutation(B * pages).astype(np.int32))
    prompts = [synth.make_prompt(n, cfg["vocab"], 40 + b) for b, n in enumerate(lens)]
    L.generate(m, kv, None, prompts, [0] * B, L.make_params(K=cfg["max_draft"], max_new=1))
    L.check(m)
    okv = O.KVCache(cfg, B, max(lens))
    for b in range(B):
        G.prefill(Wc, cfg, okv, b, prompts[b])
    for b in range(B):
        n = lens[b] - 1
        for l in range(cfg["n_layers"] if n else 0):
            for got, want in zip(L.kv_export(kv, b, l, 0, n), (okv.k[l, b, :n], okv.v[l, b, :n])):
                d = (got.cpu().float() - want.reshape(n, -1).float()).abs()
                # Products of bf16-rounded operands, rounded to bf16: two steps of the format at the largest magnitude (which
                # are 2^-8 of the next power of two each), and half a step of its least spacing on average.
                top = max(1.0, float(want.float().abs().max()))
                step = 2.0 ** (np.ceil(np.log2(top)) - 8)
                assert d.max() <= 2 * step and d.mean() <= 2.0 ** -9 * top, (b, l, float(d.max()), float(d.mean()))


# A layer of 16 M weights, whose passes take up to 2304 rows: prompts that end just below, at and just above a full pass, in it and in its last
# chunk; a single long prompt over two passes; both modes
@pytest.mark.parametrize("precise", [0, 1])
@pytest.mark.parametrize("lens", [[449] * 4 + [500], [449] * 4 + [513], [449] * 4 + [513, 2], [2400]])
def test_cache_of_the_largest_passes(L, precise, lens):
    cfg = dict(synth.model_cfg("tiny", n_layers=2, d_model=2048, n_heads=16, n_kv_heads=16, head_dim=128, d_ffn=1024, vocab=512), precise=precise)
    assert cfg["d_model"] * (4 * 2048 + 3 * cfg["d_ffn"]) >= 16 << 20
    Wc = synth.make_weights(cfg, seed=0, gain_jitter=0.1)
    B, n = len(lens), max(lens) - 1
    pages = (max(lens) + 1 + cfg["max_draft"] + 15) // 16
    m = L.model_create(cfg, weights_to(Wc, "cuda"), max_batch=B)
    kv = L.kv_create(m, B, B * pages)
    L.kv_set_page_table(kv, np.random.default_rng(1).permutation(B * pages).astype(np.int32))
    prompts = [synth.make_prompt(n, cfg["vocab"], 40 + b) for b, n in enumerate(lens)]
    L.generate(m, kv, None, prompts, [0] * B, L.make_params(K=cfg["max_draft"], max_new=1))
    L.check(m)
    # the shortest prompt and the longest against the oracle; the others, whose chunks lie elsewhere in the passes, against a cache
    # that holds each of them alone
    okv = O.KVCache(cfg, B, max(lens))
    one = L.kv_create(m, 1, pages)
    for b in range(B):
        n = lens[b] - 1
        if b in (0, B - 1) and n < 1000:
            G.prefill(Wc, cfg, okv, b, prompts[b])
        L.kv_reset(one)
        L.generate(m, one, None, [prompts[b]], [0], L.make_params(K=cfg["max_draft"], max_new=1))
        for l in range(cfg["n_layers"]):
            got = L.kv_export(kv, b, l, 0, n)
            twice = not (b in (0, B - 1) and n < 1000)        # (both are within the bound of what is exact)
            for x, y, want in zip(got, L.kv_export(one, 0, l, 0, n), (okv.k[l, b, :n], okv.v[l, b, :n])):
                if twice:
                    want = y.cpu()
                d = (x.cpu().float() - want.reshape(n, -1).float()).abs()
                top = max(1.0, float(want.float().abs().max()))           # (the bound: see above)
                assert d.max() <= (2 + 2 * twice) * 2.0 ** (np.ceil(np.log2(top)) - 8) and d.mean() <= 2.0 ** -9 * top * (1 + twice), (b, l, float(d.max()), float(d.mean()))
