"""The row pass of the acceptance kernels (csrc/verdict.cuh): rows of any length and alignment, the estimated probability near
its threshold (where the fp64 sum decides), and values at the ends of the range, against the oracle's rule."""
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


def _check(L, logits, tokens, n_rows, mode, k, p):
    prm = L.make_params(K=logits.shape[1] - 1, mode=mode, topk=k, p=p)
    got = L.accept_commit(None, None, torch.as_tensor(logits, device="cuda"), dev_i32(tokens), dev_i32(n_rows), prm)
    want = A.accept_batch(logits, tokens, n_rows, mode, k, float(np.float32(p)))
    for g, w in zip(got, want):
        assert (g.cpu().numpy() == w).all(), (mode, k, p)


# lengths around the vector body, one batch of a CTA (8192 values) and the second; odd ones shift every row's alignment
@pytest.mark.parametrize("V", [1, 2, 3, 5, 7, 1001, 8191, 8192, 8193, 8197, 16385, 50257])
def test_lengths_and_alignments(L, V):
    rng = np.random.default_rng(V)
    B, R = 6, 4
    logits = (rng.standard_normal((B, R, V)) * 3).astype(np.float32)
    logits[1:3] = np.round(logits[1:3])                 # many ties
    order = np.argsort(-logits, axis=2, kind="stable")
    tokens = rng.integers(0, V, (B, R)).astype(np.int32)
    for b in range(B):
        for i in range(1, R):
            tokens[b, i] = order[b, i - 1, min(V - 1, int(rng.integers(0, 3)))]
    n_rows = np.array([4, 4, 3, 4, 1, 4], dtype=np.int32)
    for mode, k, p in [(A.STRICT, 1, 0.0), (A.RELAXED, 2, 0.01), (A.TOPK, 3, 0.0), (A.TOPP, 1, 0.02), (A.RELAXED_ARGMAX, 2, 0.05)]:
        _check(L, logits, tokens, n_rows, mode, k, p)


def test_thresholds_next_to_the_probability(L):
    rng = np.random.default_rng(9)
    for scale in (1.0, 8.0, 300.0):                     # flat, peaked, and large logits whose differences still matter
        logits = (rng.standard_normal((1, 2, 32000)) * scale).astype(np.float32)
        order = np.argsort(-logits[0, 0], kind="stable")
        for rank in (0, 1, 2):
            tokens = np.array([[0, order[rank]]], dtype=np.int32)
            q = A.prob_of(logits[0, 0], int(order[rank]))
            for d in (-1e-2, -1e-4, -1e-5, -1e-6, 1e-6, 1e-5, 1e-4, 1e-2):
                _check(L, logits, tokens, np.array([2], dtype=np.int32), A.RELAXED, 3, float(np.float32(q * (1 + d))))


def test_ends_of_the_range(L):
    V = 9000
    logits = np.full((3, 2, V), -np.inf, dtype=np.float32)
    logits[0, 0, 8500] = -5.0                           # one finite value: probability 1
    logits[1, 0, [3, 8999]] = 3e38                      # two equal, far above the rest
    tokens = np.array([[0, 8500], [0, 8999], [0, 0]], dtype=np.int32)
    for mode, k, p in [(A.STRICT, 1, 0.0), (A.RELAXED, 2, 0.4), (A.RELAXED, 1, 0.4), (A.TOPP, 1, 0.6)]:
        _check(L, logits[:2], tokens[:2], np.array([2, 2], dtype=np.int32), mode, k, p)
    out = L.accept_commit(None, None, torch.as_tensor(logits[2:], device="cuda"), dev_i32(tokens[2:]), dev_i32([1]),
                          L.make_params(K=1, mode=L.MODE_STRICT))
    assert out[1].cpu().tolist() == [[0, -1]]           # nothing above -inf: the smallest id


# A masked draft token (-inf) ranks behind every finite logit and behind the masked tokens of smaller id, and nothing else: the
# lanes' padding past a part's end must not count.  Whole rows and rows in parts, masks of all but one token and of every second.
@pytest.mark.parametrize("V", [5, 6, 7, 1003, 8195, 16390, 32003])
def test_rank_of_a_masked_token(L, V):
    logits = np.full((2, 2, V), -np.inf, dtype=np.float32)
    logits[0, 0, V // 2] = 1.0
    logits[1, 0, ::2] = np.arange((V + 1) // 2, dtype=np.float32) * 1e-3
    for t in sorted({0, 1, V // 3 | 1, V - 3, V - 2, V - 1}):
        tokens = np.array([[0, t], [0, t]], dtype=np.int32)
        for b in range(2):
            row = logits[b, 0]
            rank = int((row > row[t]).sum() + (row[:t] == row[t]).sum())
            for k in (rank, rank + 1):
                if k >= 1:
                    _check(L, logits[b:b + 1], tokens[b:b + 1], np.array([2], dtype=np.int32), A.TOPK, k, 0.0)


# One NaN anywhere in a row makes every probability on it NaN, which exceeds no p: at the ends that are read singly, in a batch
# of its own among masked tokens, and in another part than the rest.
@pytest.mark.parametrize("V", [7, 8195, 16390, 32003])
def test_a_nan_leaves_no_probability(L, V):
    rng = np.random.default_rng(V)
    for masked in (False, True):
        for at in sorted({0, 1, 2, 3, V // 2, V - 3, V - 2, V - 1}):
            for shift in range(4):                       # the row's distance from a 16-byte boundary
                row = np.full(V, -np.inf, dtype=np.float32) if masked else rng.standard_normal(V).astype(np.float32)
                top = (at + V // 3 + 1) % V
                row[top] = 20.0
                row[at] = np.nan
                logits = torch.zeros(shift + 2 * V, device="cuda")[shift:].view(1, 2, V)
                logits[0, 0] = torch.as_tensor(row)
                for mode in (L.MODE_RELAXED, L.MODE_TOPP):
                    tokens = dev_i32([[0, top if mode == L.MODE_RELAXED else (top + 1) % V]])
                    n = L.accept_commit(None, None, logits, tokens, dev_i32([2]), L.make_params(K=1, mode=mode, topk=2, p=1e-6))[0]
                    assert int(n[0]) == 0, (masked, at, shift, mode)


def test_thresholds_below_the_normal_range(L):
    """Probabilities of a few of the smallest fp32 steps (2^-149): exponentials in fp32 have lost their digits there."""
    logits = np.zeros((600, 2, 3), dtype=np.float32)
    logits[:, 0, 1] = -2.0
    logits[:, 0, 2] = np.linspace(-104.0, -101.0, 600, dtype=np.float32)
    tokens = np.tile(np.array([[0, 2]], dtype=np.int32), (600, 1))
    for j in (1, 2, 3, 5, 7):
        for mode in (A.TOPP, A.RELAXED):
            _check(L, logits, tokens, np.full(600, 2, dtype=np.int32), mode, 3, j * 2.0 ** -149)


# Rows with nothing above -inf: the smallest id that is -inf is the arg max, also behind NaN and in any part
@pytest.mark.parametrize("V", [3, 9, 1003, 16390, 32003])
def test_arg_max_of_masked_rows(L, V):
    for first in sorted({0, 1, V // 2, V - 2, V - 1}):
        row = np.full(V, -np.inf, dtype=np.float32)
        row[:first] = np.nan
        logits = torch.as_tensor(np.stack([row, row])[None], device="cuda")
        out = L.accept_commit(None, None, logits, dev_i32([[0, first]]), dev_i32([2]), L.make_params(K=1, mode=L.MODE_STRICT))
        assert out[1].cpu().tolist() == [[first, first]], first
