"""The generation loop's step bookkeeping where it can go wrong: more sequences than the step kernel has warps, drafts
longer than a warp, an EOS token in the middle of a long accepted draft, texts of one token, and the steps that are queued
before the earlier ones have reported.  Verification is strict, so whatever was drafted the texts must be those of plain
greedy decoding (Section 2.1), which runs the same rows one at a time; with an EOS token they end at its first occurrence."""
import numpy as np
import pytest

from helpers import ensure_built, weights_to
from paper_2408_05676_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    ensure_built()
    from paper_2408_05676_b200 import binding
    return binding


@pytest.mark.parametrize("B,K,max_new,fused", [(1, 1, 1, 0), (1, 40, 90, 0), (33, 8, 50, 1), (40, 40, 100, 0), (70, 3, 17, 0)])
def test_texts_equal_greedy(L, B, K, max_new, fused):
    cfg = dict(synth.model_cfg("tiny"), max_draft=K)
    m = L.model_create(cfg, weights_to(synth.make_weights(cfg, seed=0), "cuda"), max_batch=B)
    kv = L.kv_create(m, B, B * 16)
    prompts = [synth.make_prompt(20 + b, cfg["vocab"], 300 + b) for b in range(B)]
    gid = list(range(B))
    greedy = L.generate(m, kv, None, prompts, gid, L.make_params(K=K, max_new=max_new))
    assert greedy["verify_calls"] == max_new and greedy["emitted"] == greedy["steps"] == B * max_new
    # every group holds its sequence's text to come, cut into pieces by wrong tokens: long drafts and rejected ones
    docs = [[[int(prompts[b][-1])] + [t if j % 37 else (t + 1) % cfg["vocab"] for j, t in enumerate(greedy["out"][b], 1)]] for b in range(B)]
    pool, offs = synth.pool_from_documents(docs)
    h = L.pool_build(pool, offs, 1, 3)
    prm = dict(K=K, n_min=1, n_max=3, max_occ=64, max_new=max_new, fused_accept=fused)
    spec = L.generate(m, kv, h, prompts, gid, L.make_params(**prm))
    assert spec["out"] == greedy["out"] and spec["emitted"] == B * max_new
    assert K * max_new == 1 or spec["steps"] < greedy["steps"]
    assert (L.kv_get_len(kv, gid) == np.asarray([len(p) for p in prompts]) - 1 + max_new).all()
    # an EOS token from the middle of a text ends every text at its first occurrence
    eos = greedy["out"][0][max_new // 2]
    cut = [o[:o.index(eos) + 1] if eos in o else o for o in greedy["out"]]
    for pool_or_none in (h, None):
        r = L.generate(m, kv, pool_or_none, prompts, gid, L.make_params(eos_id=eos, **prm))
        assert r["out"] == cut and r["emitted"] == sum(map(len, cut))
        assert (L.kv_get_len(kv, gid) == np.asarray([len(p) - 1 + len(c) for p, c in zip(prompts, cut)])).all()
        assert all(r[k] >= 0 for k in ("ms_draft", "ms_verify", "ms_accept")) and r["ms_verify"] > 0
