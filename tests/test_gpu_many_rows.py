"""Steps of many token rows (csrc/gemm_pair.cu): the contraction that pairs two SMs on a tile, at the edges of its token
tiles and with the left-over tiles cut along K between two, a few and many contributors, against the fp64 oracle."""
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


# rows of a step = B x (K + 1); the pair form starts above 160 rows (64 in the precise mode)
@pytest.mark.parametrize("B,K,precise", [(18, 8, 0), (8, 8, 1), (16, 15, 0), (17, 15, 1), (33, 15, 0), (5, 12, 1)])
def test_layers_at_the_tile_edges(L, B, K, precise):
    cfg = synth.model_cfg("tiny", max_draft=K, precise=precise)
    Wc = synth.make_weights(cfg, seed=0, gain_jitter=0.1)
    m = L.model_create(cfg, weights_to(Wc, "cuda"), max_batch=B)
    kv = L.kv_create(m, B, B * 6)
    okv = O.KVCache(cfg, B, 6 * 16)
    rng = np.random.default_rng(B)
    ctx = [int(x) for x in rng.integers(0, 70, B)]
    _fill_both(L, cfg, kv, okv, range(B), ctx, seed=7)
    rows = [synth.make_prompt(K + 1 if b % 3 else int(rng.integers(1, K + 2)), cfg["vocab"], 50 + b) for b in range(B)]
    err, _ = _step(L, m, kv, cfg, Wc, okv, list(range(B)), rows)
    assert err <= (TOL / 10 if precise else TOL)


# No layers: the LM head alone, whose [vocab, d_model] shape sets how its 256-row tiles fall on the 74 SM pairs.
# Cut: 2 weight tiles x 3 token tiles (twelve contributors each), 12 x 2 (three), with operands as pairs 2 x 4 (nine) and 12 x 3
# (two).  Whole: 20 x 3, 30 x 2, 60 x 1 (more than half of the pairs), 125 x 2 (three waves and part of a fourth), 74 x 3.
@pytest.mark.parametrize("tiles,d,precise", [(2, 8192, 0), (20, 8192, 0), (30, 8192, 0), (60, 8192, 1), (125, 2048, 1), (74, 512, 0),
                                             (12, 8192, 0), (2, 8192, 1), (12, 8192, 1)])
def test_left_over_tiles_cut_along_k(L, tiles, d, precise):
    B, K = 20, 8                                     # 180 rows
    V = tiles * 256 - 8                              # the last weight tile overhangs
    cfg = synth.model_cfg("tiny", n_layers=0, d_model=d, vocab=V, max_draft=K, precise=precise)
    Wc = synth.make_weights(cfg, seed=1, gain_jitter=0.1)
    m = L.model_create(cfg, weights_to(Wc, "cuda"), max_batch=B)
    kv = L.kv_create(m, B, B * 2)
    okv = O.KVCache(cfg, B, 32)
    rows = [synth.make_prompt(K + 1, V, 70 + b) for b in range(B)]
    err, first = _step(L, m, kv, cfg, Wc, okv, list(range(B)), rows)
    # A logit is a sum of d products.  Rounding: the activation is off by at most 2^-9 of itself (as a hi + lo pair 2^-17),
    # signs independent, so the error has at most that share of the logits' deviation; six of these over millions of logits.
    # Accumulation: d / 16 MMA steps (twice that for pairs), each of which may cut the fp32 sum below its last bit, 2^-23.
    steps = d / 16 * (2 if precise else 1)
    bound = 6 * 2.0 ** (-17 if precise else -9) * float(first.std()) + steps * 2.0 ** -23 * float(first.abs().max())
    print("max-abs logit error %.2e, bound %.2e" % (err, bound))
    assert err <= bound
    for _ in range(3):                               # the partial sums are added in a fixed order
        again = L.verify_step(m, kv, dev_i32(range(B)), dev_i32(np.stack(rows)), dev_i32([K + 1] * B))
        assert torch.equal(first, again)
    L.check(m)


# A contributor that finds its peers late leaves its slice of the rows to the last one: with no time to wait nearly every slice
# is handed over.  LM heads whose tiles have twelve, three, four and (behind a full wave) two contributors; a layer whose gate/up
# and down projections are cut.
@pytest.mark.parametrize("over", [dict(n_layers=0, d_model=8192, vocab=2 * 256 - 8), dict(n_layers=0, d_model=8192, vocab=12 * 256),
                                  dict(n_layers=0, d_model=8192, vocab=30 * 256, precise=1), dict(n_layers=0, d_model=8192, vocab=60 * 256, precise=1),
                                  dict(shape="7b", n_layers=1, vocab=4096)])
def test_slices_handed_to_the_last_contributor(L, over):
    B, K = 30, 8                                     # 270 rows
    over = dict(over)
    cfg = synth.model_cfg(over.pop("shape", "tiny"), max_draft=K, **over)
    m = L.model_create(cfg, synth.make_weights(cfg, seed=1, device="cuda", gain_jitter=0.1), max_batch=B)
    kv = L.kv_create(m, B, B * 2)
    ids, n_rows = dev_i32(range(B)), dev_i32([K + 1] * B)
    tokens = dev_i32(np.stack([synth.make_prompt(K + 1, cfg["vocab"], 70 + b) for b in range(B)]))
    want = L.verify_step(m, kv, ids, tokens, n_rows)
    for cycles in (0, 0, 300, 1500, 200000):
        assert L.selftest_peers(m, cycles) == 0
        for _ in range(4):
            assert torch.equal(want, L.verify_step(m, kv, ids, tokens, n_rows))
    assert L.selftest_peers(m) == 0
    L.check(m)
