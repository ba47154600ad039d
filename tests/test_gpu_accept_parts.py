"""Acceptance with a row's CTAs (csrc/accept.cu): few rows are cut into two or four parts, many rows are read whole, and more
rows of a sequence than the last CTA has threads are judged in turn; against the oracle's rule, the fp64 decision included."""
import numpy as np
import pytest
import torch

from helpers import dev_i32, ensure_built
from oracle import accept as A

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    ensure_built()
    from paper_2408_05676_b200 import binding
    return binding


# parts of at least 4096 values while there are at most 1184 launched and 592 active ones (800 of rows longer than 24576)
@pytest.mark.parametrize("B,R,V", [
    (1, 2, 8195), (1, 3, 12287), (2, 5, 32003), (13, 9, 33001), (66, 9, 32002), (65, 9, 8200), (65, 9, 12001), (1, 256, 40), (1, 257, 31), (2, 300, 17), (1, 513, 9),
])
def test_parts_and_many_rows(L, B, R, V):
    rng = np.random.default_rng(B * 1000 + R)
    logits = (rng.standard_normal((B, R, V)) * 3).astype(np.float32)
    logits[:, ::3] = np.round(logits[:, ::3])             # ties across the parts
    top = logits.argmax(axis=2)
    tokens = rng.integers(0, V, (B, R)).astype(np.int32)
    tokens[:, 1:] = top[:, :-1]                           # all of it passes ...
    for b in range(B):
        if R > 2 and b % 2:
            tokens[b, 1 + int(rng.integers(0, R - 1))] = int(rng.integers(0, V))     # ... or all but one
    n_rows = rng.integers(1, R + 1, B).astype(np.int32)
    n_rows[0] = R
    q = A.prob_of(logits[0, 0], int(tokens[0, 1]))
    for mode, k, p in [(A.STRICT, 1, 0.0), (A.RELAXED, 2, 0.0), (A.RELAXED, 2, q * (1 + 1e-5)), (A.TOPP, 1, q * (1 - 1e-5))]:
        prm = L.make_params(K=R - 1, mode=mode, topk=k, p=p)
        got = L.accept_commit(None, None, torch.as_tensor(logits, device="cuda"), dev_i32(tokens), dev_i32(n_rows), prm)
        want = A.accept_batch(logits, tokens, n_rows, mode, k, float(np.float32(p)))
        for g, w in zip(got, want):
            assert (g.cpu().numpy() == w).all(), (mode, k, p)


# the allocation-free call keeps whole rows and parts in one array of fixed size: parts, then whole rows, then parts again
def test_parts_in_the_fixed_array(L):
    for B, R, V in [(2, 5, 32003), (66, 9, 8200), (130, 9, 8200), (1, 2, 16384)]:
        rng = np.random.default_rng(B)
        logits = torch.as_tensor((rng.standard_normal((B, R, V)) * 3).astype(np.float32), device="cuda")
        tokens = torch.zeros(B, R, dtype=torch.int32, device="cuda")
        tokens[:, 1:] = logits.topk(2, 2).indices[:, :-1, int(rng.integers(0, 2))]
        n_rows = dev_i32(rng.integers(0, R + 1, B))
        prm = L.make_params(K=R - 1, mode=L.MODE_RELAXED, topk=2, p=0.02)
        want = L.accept_commit(None, None, logits, tokens, n_rows, prm)
        for _ in range(2):
            out = [torch.full(s, -7, dtype=torch.int32, device="cuda") for s in ((B,), (B, R), (B,))]
            got = L.accept_commit_noalloc(None, None, logits, tokens, n_rows, prm, out)
            assert all(torch.equal(g, w) for g, w in zip(got, want)), (B, R, V)
