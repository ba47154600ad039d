"""The calls of a decoding step hand plain addresses to the library, so the binding has to refuse what is not a GPU tensor of the
asked type: a host address would be read as a device one.  Nothing is launched here: the library is a stand-in, and its "GPU
tensors" are host tensors that say they are on the GPU."""
import numpy as np
import pytest
import torch

from helpers import ensure_built


class _OnGpu(torch.Tensor):
    is_cuda = True


class _Recorder:
    def __init__(self):
        self.calls = []

    def __getattr__(self, name):
        def call(*args):
            self.calls.append((name, args))
            return 0
        return call


def _gpu(shape, dtype=torch.int32):
    return torch.zeros(shape, dtype=dtype).as_subclass(_OnGpu)


B, K, V = 2, 3, 8


def _calls(L):
    """name -> (arguments by name, the call of them, the checked ones)"""
    prm = L.make_params(K=K)
    i32 = lambda *s: _gpu(s)
    out = lambda: tuple(i32(B) for _ in range(3))
    pool = type("P", (), dict(handle=None))()
    step = dict(logits=_gpu((B, K + 1, V), torch.float32), tokens=i32(B, K + 1), n_rows=i32(B))
    query = dict(tails=i32(B, prm.n_max), tail_len=i32(B), group_id=i32(B))
    rows = dict(last=i32(B), draft=i32(B, K), dlen=i32(B))
    return {
        "draft": (query, lambda a: L.draft(pool, a["tails"], a["tail_len"], a["group_id"], prm, i32(B, K), i32(B), i32(B), stream=0)),
        "draft_tree": (dict(query, hist=i32(B, 5), hist_len=i32(B)),
                       lambda a: L.draft_tree(pool, a["tails"], a["tail_len"], a["group_id"], prm, hist=a["hist"], hist_len=a["hist_len"], stream=0)),
        "make_rows": (rows, lambda a: L.make_rows(a["last"], a["draft"], a["dlen"], K, i32(B, K + 1), i32(B), stream=0)),
        "make_rows_tree": (dict(rows, parents=i32(B, K)), lambda a: L.make_rows_tree(a["last"], a["draft"], a["parents"], a["dlen"], K, stream=0)),
        "accept_commit": (step, lambda a: L.accept_commit(None, None, a["logits"], a["tokens"], a["n_rows"], prm, out=out(), stream=0)),
        "accept_commit_noalloc": (step, lambda a: L.accept_commit_noalloc(None, None, a["logits"], a["tokens"], a["n_rows"], prm, out(), stream=0)),
    }


@pytest.mark.parametrize("name", ["draft", "draft_tree", "make_rows", "make_rows_tree", "accept_commit", "accept_commit_noalloc"])
def test_only_gpu_tensors_of_the_type_reach_the_library(monkeypatch, name):
    ensure_built()
    from paper_2408_05676_b200 import binding as L
    rec = _Recorder()
    monkeypatch.setattr(L, "lib", rec)
    args, call = _calls(L)[name]
    call(args)
    assert [n for n, _ in rec.calls] == ["laser_" + name]
    for arg, t in args.items():
        host = t.as_subclass(torch.Tensor)
        for other in (host.numpy(), host, t.to(torch.int64), None):
            if other is None and arg == "hist":
                continue                       # (without a history: a call of its own)
            with pytest.raises((AssertionError, AttributeError, TypeError)):
                call(dict(args, **{arg: other}))
    assert len(rec.calls) == 1
