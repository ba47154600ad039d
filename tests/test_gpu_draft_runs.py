"""Long runs of the retrieval index (csrc/pool.cu): lookups whose occurrences fill one warp, overflow to the kernel with the
vocabulary histogram, overflow that kernel's list for one or several depths, or are cut by max_occ anywhere on the way."""
import numpy as np
import pytest

from helpers import dev_i32, ensure_built
from oracle import retrieval as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    ensure_built()
    from paper_2408_05676_b200 import binding
    return binding


def _compare(L, toks, offs, tails, gids, n_max, **prm):
    pool = L.pool_build(toks, offs, 1, n_max)
    p = L.make_params(n_min=1, n_max=n_max, **prm)
    B = len(tails)
    tails, lens, gids = np.asarray(tails, np.int32), np.full(B, n_max, np.int32), np.asarray(gids, np.int32)
    want = R.draft_batch(toks, offs, tails, lens, gids, p.K, 1, n_max, p.min_draft, p.max_occ)
    for _ in range(2):                         # the work list is left empty by the first call
        got = L.draft(pool, dev_i32(tails), dev_i32(lens), dev_i32(gids), p)
        for g, w in zip(got, want):
            assert (g.cpu().numpy() == w).all()


# vocabulary sizes that leave about `run` occurrences of a token in 20 thousand; 2 keeps thousands alive for several depths
@pytest.mark.parametrize("vocab,n_max,K,max_occ,min_draft", [
    (2, 2, 20, 0, 1), (2, 3, 64, 5000, 1), (4, 1, 9, 4097, 1), (5, 2, 16, 0, 16), (40, 2, 8, 65, 1), (310, 1, 16, 0, 1), (310, 3, 33, 64, 4),
])
def test_runs_of_every_length(L, vocab, n_max, K, max_occ, min_draft):
    rng = np.random.default_rng(vocab * 100 + K)
    toks = rng.integers(0, vocab, 20000, dtype=np.int64).astype(np.int32)
    toks[rng.integers(0, 20000, 12)] = -1                     # documents
    offs = np.array([0, 15000, 15000, 20000], dtype=np.int64)  # one group is empty
    B = 6
    at = rng.integers(10, 14000, B)
    tails = np.stack([np.maximum(toks[a:a + n_max], 0) for a in at]).astype(np.int32)
    gids = np.array([0, 0, 2, 0, 1, 2])
    _compare(L, toks, offs, tails, gids, n_max, K=K, max_occ=max_occ, min_draft=min_draft)


@pytest.mark.parametrize("copies", [31, 32, 33, 63, 64, 65, 66])
def test_a_run_around_one_warp(L, copies):
    # `copies` documents "7 7 a ..": the winner is decided by counts that span both of a lane's occurrences
    rng = np.random.default_rng(copies)
    toks = []
    for c in range(copies):
        toks += [7, 8, 20 + c % 3, 30 + c % 2] + rng.integers(40, 60, int(rng.integers(0, 12))).tolist() + [-1]
    toks = np.array(toks + list(range(100, 140)), dtype=np.int32)
    offs = np.array([0, len(toks)], dtype=np.int64)
    for max_occ in (0, 33, 64):
        _compare(L, toks, offs, np.array([[7, 8], [8, 20], [3, 7]], dtype=np.int32), np.zeros(3, dtype=np.int64), 2, K=12, max_occ=max_occ,
                 min_draft=1)


# Runs on both sides of what a team of 256 threads holds (2048 positions) and a CTA (16384), among them the last run of the position array; tokens up
# to the largest vocabulary; a longer suffix whose draft is too short, so that the CTA goes on with the shorter ones
@pytest.mark.parametrize("copies", [65, 255, 257, 2047, 2048, 2049, 4100, 16384, 16385])
def test_a_run_around_a_team(L, copies):
    rng = np.random.default_rng(copies)
    toks = []
    for c in range(copies):
        toks += [7, 8] + (51199 - rng.integers(0, 3, int(rng.integers(0, 6)))).tolist() + [-1]
    for c in range(90):
        toks += [9, 7, 8, -1]                   # "9 7 8" is never continued, "7 8" is
    toks = np.array(toks + [50] * 70, dtype=np.int32)
    offs = np.array([0, len(toks)], dtype=np.int64)
    tails = np.array([[5, 7, 8], [9, 7, 8], [50, 50, 50], [7, 8, 51199]], dtype=np.int32)
    for max_occ in (0, 65, copies - 1, copies + 1):
        for min_draft in (1, 6):
            _compare(L, toks, offs, tails, np.zeros(4, dtype=np.int64), 3, K=7, max_occ=max_occ, min_draft=min_draft)


# Runs beyond what a CTA holds in registers: their occurrences fit the list of a small vocabulary (more of them than its walk takes
# at once, before and after the first vote), or do not
@pytest.mark.parametrize("copies,spread", [(17000, 2), (17000, 40), (60000, 3)])
def test_a_run_beyond_a_cta(L, copies, spread):
    rng = np.random.default_rng(copies + spread)
    doc = np.full((copies, 5), -1, np.int32)
    doc[:, 0] = 7
    doc[:, 1:4] = 10 + np.minimum(rng.integers(0, spread, (copies, 3)), rng.integers(0, spread, (copies, 3)))
    toks = np.concatenate([doc.reshape(-1), np.arange(100, 140, dtype=np.int32)])
    offs = np.array([0, len(toks)], dtype=np.int64)
    for max_occ in (0, 16500):
        _compare(L, toks, offs, np.array([[7], [10]], dtype=np.int32), np.zeros(2, dtype=np.int64), 1, K=6, max_occ=max_occ, min_draft=1)


# More queries than the large-run kernel has teams (4 on each of 148 CTAs) whose longest suffix occurs often and gives no draft, or one
# that is too short, so that they are handed on to the shorter suffixes; among them runs beyond a team, queries that a team finishes and
# queries that the warp kernel does.  The outputs hold other values before the call.
@pytest.mark.parametrize("B", [592, 593, 700, 4096])
@pytest.mark.parametrize("min_draft,max_occ", [(1, 0), (1, 500), (8, 0), (8, 500)])
def test_more_queries_handed_on_than_teams(L, B, min_draft, max_occ):
    rng = np.random.default_rng(B + 10 * min_draft + max_occ)
    toks = []
    for c in range(70):
        toks += [9, 7, 8, -1]                                   # "9 7 8" is never continued, "7 8" is
    for c in range(90):
        toks += [7, 8] + rng.integers(40, 43, int(rng.integers(0, 6))).tolist() + [-1]
    for c in range(80):
        toks += [1, 2, 3] + rng.integers(50, 52, 12).tolist() + [-1]
    for c in range(2100):
        toks += [20, 21 + c % 2, -1]                            # beyond a team, and never continued
    toks = np.array(toks + list(range(100, 140)), dtype=np.int32)
    offs = np.array([0, len(toks)], dtype=np.int64)
    kinds = np.array([[9, 7, 8], [1, 2, 3], [5, 5, 20], [4, 20, 21], [101, 102, 103], [6, 40, 41], [60, 60, 60]], dtype=np.int32)
    pick = np.where(rng.random(B) < 0.8, 0, rng.integers(0, len(kinds), B))
    pool = L.pool_build(toks, offs, 1, 3)
    p = L.make_params(K=10, n_min=1, n_max=3, min_draft=min_draft, max_occ=max_occ)
    n = len(kinds)
    want = [w[pick] for w in R.draft_batch(toks, offs, kinds, np.full(n, 3, np.int32), np.zeros(n, np.int32), 10, 1, 3, min_draft, max_occ)]
    tails, lens, gids = dev_i32(kinds[pick]), dev_i32(np.full(B, 3)), dev_i32(np.zeros(B))
    out = [dev_i32(np.full(w.shape, -77)) for w in want]
    for _ in range(2):                         # the work list is left empty by the first call
        for o in out:
            o.fill_(-77)
        L.draft(pool, tails, lens, gids, p, *out)
        for g, w in zip(out, want):
            assert (g.cpu().numpy() == w).all()


# A few occurrences that agree up to a depth, with one or several of them parting there (a majority stays, or the smallest of equals): on
# both sides of what a step reads along, of the depths requested together and of the 32 that a warp's lanes hold; a document ends there too
@pytest.mark.parametrize("copies", [1, 2, 3, 4, 5, 8, 9, 33, 64])
def test_occurrences_that_part(L, copies):
    rng = np.random.default_rng(copies)
    toks, offs, K = [], [0], 64
    depths = [1, 2, 8, 9, 16, 31, 32, 33, 34, 63, 64, 65]
    for d in depths:
        line = rng.integers(10, 5000, 70).tolist()
        for c in range(copies):
            own = list(line)
            if c % 3 == 1:
                own[d - 1:] = rng.integers(10, 5000, 71 - d).tolist()
            if c % 5 == 4:
                own = own[:d - 1]
            if c % 4 == 3 and d + 4 < len(own):
                own[d + 4] = 6000 + c
            toks += [7, 8] + own + [-1]
        offs.append(len(toks))
    tails = np.tile(np.array([[7, 8]], dtype=np.int32), (len(depths), 1))
    _compare(L, np.array(toks, dtype=np.int32), np.array(offs, dtype=np.int64), tails, np.arange(len(depths)), 2, K=K, max_occ=64, min_draft=1)


# max_occ on both sides of what bounds the list of the large-run kernel (4096), on runs that it cuts there and on one that it does not
@pytest.mark.parametrize("max_occ", [4095, 4096, 4097, 0])
def test_a_list_at_its_limit(L, max_occ):
    rng = np.random.default_rng(max_occ)
    doc = np.full((17000, 5), -1, np.int32)
    doc[:, 0] = 7
    doc[:, 1:4] = 10 + np.minimum(rng.integers(0, 3, (17000, 3)), rng.integers(0, 3, (17000, 3)))
    doc[4090::4, 0] = 8
    toks = np.concatenate([doc.reshape(-1), np.arange(100, 140, dtype=np.int32)])
    offs = np.array([0, len(toks)], dtype=np.int64)
    tails = np.array([[7], [8], [10], [11], [12]], dtype=np.int32)
    for min_draft in (1, 4):
        _compare(L, toks, offs, tails, np.zeros(5, dtype=np.int64), 1, K=6, max_occ=max_occ, min_draft=min_draft)
