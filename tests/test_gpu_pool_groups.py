"""The index build by group size (csrc/pool.cu): groups that fit shared memory, at the edges of the classes that the build
sorts them into, beside groups that take the slot sort; runs with none to all of a block's positions; sentinels, empty groups, and groups of one token only.  Whatever the way, the same retrieval and the same key count."""
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


def _n_keys(toks, offs, n_min, n_max):
    total = 0
    for lo, hi in zip(offs[:-1], offs[1:]):
        t = toks[lo:hi]
        for n in range(n_min, n_max + 1):
            if len(t) >= n:
                w = np.lib.stride_tricks.sliding_window_view(t, n)
                w = w[(w >= 0).all(axis=1)]
                total += len(np.unique(w, axis=0)) if len(w) else 0
    return total


@pytest.mark.parametrize("sizes,vocab,n_min,n_max", [
    ([0, 1, 2, 3, 31, 32, 33, 0, 64, 500], 5, 1, 4),
    ([4899, 4900, 4901, 7600, 7601], 400, 1, 3),
    ([15400, 15401, 40], 3000, 1, 2),
    ([15401, 100, 40000, 0, 16000], 50000, 2, 5),            # large groups around small ones
    ([15400, 20000, 5000], 1, 1, 2),                               # one token: one run of the whole group
    ([6000, 6000], 47, 1, 1),                                # many positions of a run in a block
    ([700, 15000], 60000, 1, 8),
])
def test_build_by_group_size(L, sizes, vocab, n_min, n_max):
    rng = np.random.default_rng(sum(sizes) + vocab)
    N = sum(sizes)
    toks = (rng.random(N) ** 2 * vocab).astype(np.int32)     # small ids are frequent
    if vocab > 1:
        toks[rng.integers(0, N, N // 200)] = -1
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pool = L.pool_build(toks, offs, n_min, n_max)
    info = pool.info()
    assert info["n_tokens"] == N and info["n_keys"] == _n_keys(toks, offs, n_min, n_max)
    B = 4 * len(sizes)
    gids = np.arange(B, dtype=np.int32) % len(sizes)
    at = offs[gids] + (rng.random(B) * np.maximum(offs[gids + 1] - offs[gids] - n_max, 1)).astype(np.int64)
    at = np.minimum(at, max(N - n_max, 0))
    tails = np.zeros((B, n_max), np.int32)
    for b in range(B):
        t = toks[at[b]:at[b] + n_max]
        tails[b, n_max - len(t):] = np.maximum(t, 0)
    lens = np.full(B, n_max, np.int32)
    for max_occ in (64, 0):
        if max_occ == 0 and vocab > 50000:
            continue                                         # (the histogram of the unlimited path holds 51,200 tokens)
        p = L.make_params(K=10, n_min=n_min, n_max=n_max, max_occ=max_occ)
        want = R.draft_batch(toks, offs, tails, lens, gids, 10, n_min, n_max, 1, max_occ)
        got = L.draft(pool, dev_i32(tails), dev_i32(lens), dev_i32(gids), p)
        for g, w in zip(got, want):
            assert (g.cpu().numpy() == w).all()


def test_freed_pools_are_given_back(L):
    """What freed pools leave with the library is bounded, serves the next build, and goes back to the device on request."""
    import torch

    toks = np.random.default_rng(3).integers(0, 5000, 4_000_000).astype(np.int32)
    offs = np.linspace(0, len(toks), 401).astype(np.int64)
    L.pool_build(toks[:1000], np.array([0, 1000]), 1, 2).free()    # (whatever the first use loads)
    L.trim()
    free0 = torch.cuda.mem_get_info()[0]
    keep = L.pool_build(toks[:1000], np.array([0, 1000]), 1, 2)
    pool = L.pool_build(toks, offs, 1, 4)
    size = pool.info()["device_bytes"]
    pool.free()
    assert free0 - torch.cuda.mem_get_info()[0] < (2 << 30) + (64 << 20)
    L.trim()
    assert free0 - torch.cuda.mem_get_info()[0] < size / 2         # (a block beside the small pool's may stay)
    got = L.draft(keep, dev_i32([toks[10:12]]), dev_i32([2]), dev_i32([0]), L.make_params(K=4, n_min=1, n_max=2, max_occ=64))
    want = R.draft_batch(toks[:1000], np.array([0, 1000]), toks[None, 10:12], np.array([2]), np.array([0]), 4, 1, 2, 1, 64)
    for g, w in zip(got, want):
        assert (g.cpu().numpy() == w).all()
    keep.free()
    L.trim()
    assert torch.cuda.mem_get_info()[0] >= free0


def test_many_tiny_groups(L):
    """Tiny groups that are many are sorted together with the large ones, beside groups of shared memory, on both sides of either
    limit; more groups than a grid's second dimension holds."""
    rng = np.random.default_rng(12)
    sizes = np.concatenate([rng.integers(0, 12, 66000), [15401, 3000, 255, 256, 257, 0, 5000]])
    rng.shuffle(sizes)
    N, n_max, vocab = int(sizes.sum()), 3, 30
    toks = rng.integers(0, vocab, N).astype(np.int32)
    toks[rng.integers(0, N, N // 50)] = -1
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pool = L.pool_build(toks, offs, 1, n_max)
    assert pool.info()["n_keys"] == _n_keys(toks, offs, 1, n_max)
    gids = np.concatenate([np.flatnonzero(sizes >= 200), rng.integers(0, len(sizes), 300)]).astype(np.int32)
    tails = np.zeros((len(gids), n_max), np.int32)
    for b, g in enumerate(gids):
        at = offs[g] + int(rng.integers(0, max(1, sizes[g] - n_max)))
        t = np.maximum(toks[at:min(at + n_max, N)], 0)
        tails[b, n_max - len(t):] = t
    lens = np.full(len(gids), n_max, np.int32)
    for max_occ in (64, 0):
        want = R.draft_batch(toks, offs, tails, lens, gids, 6, 1, n_max, 2, max_occ)
        got = L.draft(pool, dev_i32(tails), dev_i32(lens), dev_i32(gids), L.make_params(K=6, n_min=1, n_max=n_max, min_draft=2, max_occ=max_occ))
        for g, w in zip(got, want):
            assert (g.cpu().numpy() == w).all()


@pytest.mark.parametrize("sizes", ["tiny", "large"])
def test_pools_of_sorted_groups_alone(L, sizes):
    rng = np.random.default_rng(5)
    sizes = rng.integers(0, 4, 70000) if sizes == "tiny" else np.array([16000, 15401, 20000])
    N, n_max = int(sizes.sum()), 2
    toks = rng.integers(0, 6, N).astype(np.int32)
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pool = L.pool_build(toks, offs, 1, n_max)
    assert pool.info()["n_keys"] == _n_keys(toks, offs, 1, n_max)
    gids = rng.integers(0, len(sizes), 200).astype(np.int32)
    tails = rng.integers(0, 6, (200, n_max)).astype(np.int32)
    lens = np.full(200, n_max, np.int32)
    want = R.draft_batch(toks, offs, tails, lens, gids, 3, 1, n_max, 1, 64)
    got = L.draft(pool, dev_i32(tails), dev_i32(lens), dev_i32(gids), L.make_params(K=3, n_min=1, n_max=n_max, max_occ=64))
    for g, w in zip(got, want):
        assert (g.cpu().numpy() == w).all()
