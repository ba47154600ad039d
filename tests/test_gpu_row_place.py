"""A row's result does not depend on its place in the step (csrc/gemm_pair.cu, csrc/attn.cu): the same text in every sequence
of a step, all K + 1 rows at once and one row after the other, gives the same bits.  Strict decoding equals plain greedy decoding
by this, also where two logits nearly tie."""
import numpy as np
import pytest
import torch

from helpers import dev_i32, ensure_built
from paper_2408_05676_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    ensure_built()
    from paper_2408_05676_b200 import binding
    return binding


# Steps whose left-over tiles are cut along K.  13B: 731 rows (down, LM head), 714 (every matrix but O), 1088 (gate/up, LM
# head), 1056 with pairs of operands (down); 7B with pairs: 396 rows (down).  Last: 144 rows, the form of gemm.cu
@pytest.mark.parametrize("shape,B,K,precise", [("13b", 43, 16, 0), ("13b", 42, 16, 0), ("13b", 64, 16, 0), ("13b", 66, 15, 1), ("7b", 44, 8, 1), ("7b", 16, 8, 0)])
def test_same_bits_at_every_place_and_alone(L, shape, B, K, precise):
    cfg = synth.model_cfg(shape, n_layers=1, max_draft=K, precise=precise)
    W = synth.make_weights(cfg, seed=0, device="cuda", gain_jitter=0.1)
    m = L.model_create(cfg, W, max_batch=B)
    ctx = 130
    kv = L.kv_create(m, B, B * ((ctx + K + 16) // 16))
    k, v = synth.make_kv_layer(ctx, cfg["n_kv_heads"] * cfg["head_dim"], 7, 0, device="cuda")
    for b in range(B):
        L.kv_import(kv, b, 0, 0, k, v)
    ids, text = dev_i32(range(B)), synth.make_prompt(K + 1, cfg["vocab"], 50)
    L.kv_set_len(kv, list(range(B)), [ctx] * B)
    full = L.verify_step(m, kv, ids, dev_i32(np.tile(text, (B, 1))), dev_i32([K + 1] * B))
    for b in range(1, B):
        assert torch.equal(full[0], full[b]), "sequence %d of %d" % (b, B)
    rows = np.full((B, K + 1), -1, np.int32)
    for i in range(K + 1):
        rows[:, 0] = text[i]
        L.kv_set_len(kv, list(range(B)), [ctx + i] * B)
        alone = L.verify_step(m, kv, ids, dev_i32(rows), dev_i32([1] * B))
        assert torch.equal(alone[:, 0], full[:, i]), "row %d" % i
    L.check(m)
