"""What this library's performance is measured on: calls of its public entry points, the way a decoding
program makes them.

Five kinds of case, which share the input recipes below:

    step      one decoding step: draft from the pool, build the rows, verify forward, accept and commit
              (as two calls, with acceptance fused into the LM head, or with a token tree)
    generate  laser_generate: prefill of ragged prompts, then steps until every text is finished
    draft     retrieval alone: many queries against a large pool
    accept    acceptance alone, on stored logits
    build     the index of a new pool, and a first batch of queries against it

Inputs are drawn on the GPU from the seed alone.  Weights are random but shaped like a trained model's in the
two respects that decide what the loop does: the residual stream carries the token's embedding past layers
whose output projections are small (std 0.02 / sqrt(2 layers)), and the LM head points from each token to one
successor, so that the next-token distribution is peaked and the text of a prompt is known without running the
model.  Drafts agree with it per position with probability 0.6.
"""
import math

import numpy as np
import torch

from paper_2408_05676_b200 import binding as L
from paper_2408_05676_b200 import synth

DEV = "cuda"
AGREE = 0.6            # share of draft tokens that equal the target's own choice
MODES = {"strict": L.MODE_STRICT, "relaxed": L.MODE_RELAXED, "topk": L.MODE_TOPK, "topp": L.MODE_TOPP}


def listed():
    return [
        # the smallest model end to end (configuration C1): 2 layers, a few sequences; launches and waits, no bandwidth
        dict(name="tiny-generate-b4", kind="generate", shape="tiny", layers=2, kv_heads=4, batch=4, prompt_lo=64, prompt_hi=64,
             new=64, draft=8, pool=20000, groups=4, mode="strict", form="chain"),
        # one user waiting for one text: 9 rows, every weight read for them
        dict(name="7b-step-b1", kind="step", shape="7b", layers=32, kv_heads=32, batch=1, draft=8, ctx_lo=512, ctx_hi=512,
             mode="strict", form="chain", precise=0, pool=5000000, groups=1000),
        # the headline step (configuration C3): batch 16, 512 cached tokens, 1 + 8 rows each
        dict(name="7b-step-b16", kind="step", shape="7b", layers=32, kv_heads=32, batch=16, draft=8, ctx_lo=512, ctx_hi=512,
             mode="strict", form="chain", precise=0, pool=5000000, groups=1000),
        # offline generation with many texts in flight (batch of configuration C4): ragged contexts and draft lengths,
        # Relaxed Verification fused into the LM head
        dict(name="7b-fused-b64-ragged", kind="step", shape="7b", layers=32, kv_heads=32, batch=64, draft=8, ctx_lo=256,
             ctx_hi=768, mode="relaxed", form="fused", precise=0, pool=5000000, groups=1000),
        # token trees instead of chains: 17 rows a sequence, tree attention, path compaction
        dict(name="7b-tree-b16", kind="step", shape="7b", layers=32, kv_heads=32, batch=16, draft=16, ctx_lo=384, ctx_hi=640,
             mode="strict", form="tree", precise=0, pool=5000000, groups=1000),
        # the mode for users who need logits close to an exact forward's: operands as hi + lo pairs
        dict(name="7b-precise-b16", kind="step", shape="7b", layers=32, kv_heads=32, batch=16, draft=8, ctx_lo=512, ctx_hi=512,
             mode="strict", form="chain", precise=1, pool=5000000, groups=1000),
        # the scale-up shape (configuration C5): 1088 rows of the 13B layers; 8 of its 40 layers, so that a few states fit
        dict(name="13b-step-b64", kind="step", shape="13b", layers=8, kv_heads=40, batch=64, draft=16, ctx_lo=256, ctx_hi=1024,
             mode="relaxed", form="chain", precise=0, pool=5000000, groups=1000),
        # prompts of 256 to 1024 tokens (configuration C4) prefilled, then a short text for each
        dict(name="7b-generate-b16", kind="generate", shape="7b", layers=32, kv_heads=32, batch=16, prompt_lo=256, prompt_hi=1024,
             new=32, draft=8, pool=2000000, groups=16, mode="relaxed", form="chain"),
        # retrieval at full size (configuration C2), occurrences cut to 64 ...
        dict(name="draft-q4096-occ64", kind="draft", queries=4096, draft=16, n_max=4, max_occ=64, pool=50000000, groups=10000),
        # ... and with all of them, what the paper's trie returns
        dict(name="draft-q4096-all", kind="draft", queries=4096, draft=16, n_max=4, max_occ=0, pool=50000000, groups=10000),
        # acceptance of a step whose logits the caller keeps
        dict(name="accept-b64-relaxed", kind="accept", batch=64, draft=8, vocab=32000, mode="relaxed", topk=2),
        # the corpus of a day's knowledge generation becomes a pool
        dict(name="build-10m", kind="build", pool=10000000, groups=2000, n_max=4, queries=1024, draft=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "generate", "draft", "draft", "accept", "build"])
    mode = rng.choice(["strict", "relaxed", "topk", "topp"])
    if kind == "step":
        shape = rng.choice(["tiny", "7b", "7b", "7b", "13b"])
        form = rng.choice(["chain", "chain", "fused", "tree"])
        layers = {"tiny": 2, "7b": _log_int(rng, 4, 32), "13b": _log_int(rng, 2, 8)}[shape]
        heads = synth.MODEL_SHAPES[shape]["n_heads"]
        lo = _log_int(rng, 20, 700)
        return dict(kind=kind, shape=shape, layers=layers, kv_heads=rng.choice([heads, heads, heads // 4]), batch=_log_int(rng, 1, 64),
                    draft=rng.randint(3, 16), ctx_lo=lo, ctx_hi=min(1000, lo + _log_int(rng, 1, 400)), mode=mode, form=form,
                    precise=int(rng.random() < 0.2), pool=_log_int(rng, 200000, 5000000), groups=_log_int(rng, 100, 1000))
    if kind == "generate":
        shape = rng.choice(["tiny", "7b"])
        lo = _log_int(rng, 17, 500)
        return dict(kind=kind, shape=shape, layers=2 if shape == "tiny" else _log_int(rng, 4, 16), kv_heads=4 if shape == "tiny" else 32,
                    batch=_log_int(rng, 1, 16), prompt_lo=lo, prompt_hi=lo + _log_int(rng, 1, 400), new=_log_int(rng, 8, 64),
                    draft=rng.randint(3, 12), pool=_log_int(rng, 20000, 2000000), groups=rng.randint(1, 16), mode=rng.choice(["strict", "relaxed"]),
                    form=rng.choice(["chain", "chain", "fused", "tree", "temp"]))
    if kind == "draft":
        pool = _log_int(rng, 100000, 50000000)
        return dict(kind=kind, queries=_log_int(rng, 1, 4096), draft=rng.randint(4, 32), n_max=rng.randint(2, 5),
                    max_occ=rng.choice([0, 0, 16, 64, 64, 500]), pool=pool, groups=max(1, pool // _log_int(rng, 2000, 50000)))
    if kind == "accept":
        return dict(kind=kind, batch=_log_int(rng, 1, 128), draft=rng.randint(1, 16), vocab=rng.choice([4096, 32000, 32003, 50257]),
                    mode=mode, topk=rng.randint(1, 4))
    pool = _log_int(rng, 50000, 10000000)
    return dict(kind=kind, pool=pool, groups=max(1, pool // _log_int(rng, 2000, 50000)), n_max=rng.randint(2, 4),
                queries=_log_int(rng, 16, 1024), draft=rng.randint(4, 16))


# ---- inputs -----------------------------------------------------------------------------------------------

def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1009 + salt) & 0x7fffffff)
    return g


def _normal(g, rows, cols, std):
    return torch.empty(rows, cols, dtype=torch.bfloat16, device=DEV).normal_(0.0, std, generator=g)


def _weights(cfg, g):
    """Random weights in the layout of synth.make_weights, and the successor of every token."""
    d, f, V, n = cfg["d_model"], cfg["d_ffn"], cfg["vocab"], cfg["n_layers"]
    dq, dkv = cfg["n_heads"] * cfg["head_dim"], cfg["n_kv_heads"] * cfg["head_dim"]
    out_std = 0.02 / math.sqrt(2 * n)
    succ = torch.randperm(V, generator=g, device=DEV)
    emb = _normal(g, V, d, 1.0)
    head = torch.empty_like(emb)
    head[succ] = (34.0 / d) * emb
    head += _normal(g, V, d, 0.02)
    W = dict(tok_emb=emb, lm_head=head, final_norm=torch.ones(d, dtype=torch.bfloat16, device=DEV), layers=[])
    for _ in range(n):
        wqkv, wgu = _normal(g, dq + 2 * dkv, d, 0.02), _normal(g, 2 * f, d, 0.02)
        ones = torch.ones(2, d, dtype=torch.bfloat16, device=DEV)
        W["layers"].append(dict(wq=wqkv[:dq], wk=wqkv[dq:dq + dkv], wv=wqkv[dq + dkv:], wo=_normal(g, d, dq, out_std),
                                w_gate=wgu[:f], w_up=wgu[f:], w_down=_normal(g, d, f, out_std), attn_norm=ones[0], ffn_norm=ones[1]))
    return W, succ


def _chain(first, succ, n):
    """first, its successor, the successor's successor, ..: int64 [B, n]."""
    out = [first]
    for _ in range(n - 1):
        out.append(succ[out[-1]])
    return torch.stack(out, 1)


def _zipf(g, n, vocab, perm):
    """n draws from Zipf(1.1) over the ranks of `perm`."""
    cdf = torch.arange(1, vocab + 1, dtype=torch.float64, device=DEV).pow(-1.1).cumsum(0)
    u = torch.rand(n, generator=g, device=DEV) * float(cdf[-1])
    return perm[torch.searchsorted(cdf.float(), u).clamp_(max=vocab - 1)]


def _pool_text(g, seed, n_tokens, n_groups, vocab, least=128):
    """The token stream of synth.make_zipf_pool, drawn on the GPU: Zipf tokens, 30 % of them copies of 200 templates
    of 20 to 60 tokens, in groups of log-normal size, `least` tokens or more.  Returns the int32 tokens on the GPU, the
    int64 offsets on the host and the tokens by rank."""
    perm = torch.randperm(vocab, generator=g, device=DEV).to(torch.int32)
    tok = _zipf(g, n_tokens, vocab, perm)
    t_len = torch.randint(20, 61, (200,), generator=g, device=DEV)
    tmpl = _zipf(g, 200 * 60, vocab, perm).view(200, 60)
    step = 134                                   # one template of 40 tokens on average in every 134
    n_copies = max(0, n_tokens // step - 1)
    if n_copies:
        which = torch.randint(0, 200, (n_copies,), generator=g, device=DEV)
        start = torch.arange(n_copies, device=DEV) * step + torch.randint(0, step - 60, (n_copies,), generator=g, device=DEV)
        at = start[:, None] + torch.arange(60, device=DEV)
        keep = torch.arange(60, device=DEV) < t_len[which][:, None]
        tok[at[keep]] = tmpl[which][keep]
    rng = np.random.default_rng(seed)
    sizes = synth.group_sizes_lognormal(n_tokens, n_groups, rng, min_size=min(least, n_tokens // n_groups))
    offs = np.zeros(n_groups + 1, dtype=np.int64)
    np.cumsum(sizes, out=offs[1:])
    return tok, offs, perm


def _put(tok, offs, groups, docs):
    """Overwrites the head of each listed group with the documents [B, n] (several of one group follow one another)."""
    B, n = docs.shape
    seen = {}
    at = np.empty(B, dtype=np.int64)
    for b, g in enumerate(groups):
        k = seen.get(int(g), 0)
        seen[int(g)] = k + 1
        at[b] = offs[int(g)] + k * (n + 1)
        assert at[b] + n + 1 <= offs[int(g) + 1], "group too small for its documents"
    at = torch.from_numpy(at).to(DEV)
    tok[at[:, None] + torch.arange(n, device=DEV)] = docs.to(torch.int32)
    tok[at + n] = -1


def _queries(g, tok, offs, perm, n, n_tail, vocab):
    """Tails as synth.make_queries draws them: groups by size, 70 % consecutive tokens of the group, 30 % Zipf."""
    o = torch.from_numpy(offs).to(DEV)
    p = torch.randint(0, int(offs[-1]), (n,), generator=g, device=DEV)
    gid = torch.searchsorted(o, p, right=True) - 1
    room = o[gid + 1] - o[gid] - n_tail + 1
    st = o[gid] + (torch.rand(n, generator=g, device=DEV) * room).long().clamp_(min=0)
    own = tok[(st[:, None] + torch.arange(n_tail, device=DEV)).clamp_(max=len(tok) - 1)]
    other = _zipf(g, n * n_tail, vocab, perm).view(n, n_tail)
    use = (torch.rand(n, generator=g, device=DEV) < 0.7) & (room > 0)
    tails = torch.where(use[:, None], own, other).to(torch.int32).contiguous()
    return tails, torch.full((n,), n_tail, dtype=torch.int32, device=DEV), gid.to(torch.int32)


def _cfg(case):
    return synth.model_cfg(case["shape"], n_layers=case["layers"], n_kv_heads=case["kv_heads"], max_draft=case["draft"],
                           precise=case.get("precise", 0))


def _corrupt(g, chain, vocab, agree=AGREE):
    bad = torch.rand(chain.shape, generator=g, device=DEV) >= agree
    return torch.where(bad, torch.randint(0, vocab, chain.shape, generator=g, device=DEV), chain)


def _prepare_step(case, seed):
    g = _gen(seed, 1)
    cfg = _cfg(case)
    B, K, V = case["batch"], case["draft"], cfg["vocab"]
    W, succ = _weights(cfg, g)
    model = L.model_create(cfg, W, max_batch=B)
    pages = -(-(case["ctx_hi"] + K + 1) // 16)
    kv = L.kv_create(model, B, B * pages)
    lens = torch.randint(case["ctx_lo"], case["ctx_hi"] + 1, (B,), generator=g, device=DEV).to(torch.int32)
    width = cfg["n_kv_heads"] * cfg["head_dim"]
    n_of = lens.tolist()
    for layer in range(cfg["n_layers"]):
        kvs = torch.empty(2, B, max(n_of), width, dtype=torch.bfloat16, device=DEV).normal_(generator=g)
        for b in range(B):
            L.kv_import(kv, b, layer, 0, kvs[0, b, :n_of[b]], kvs[1, b, :n_of[b]])
    # the text so far ends in four tokens of the chain; the group's pool holds them with a draft that goes wrong
    # at some positions (three such documents where a tree is drafted)
    tok, offs, perm = _pool_text(g, seed, case["pool"], case["groups"], V)
    first = torch.randint(0, V, (B,), generator=g, device=DEV)
    text = _chain(first, succ, 4 + K)
    tree = case["form"] == "tree"
    size = np.diff(offs)
    big = np.argsort(-size, kind="stable")[:max(1, len(size) // 2)]
    gid = big[np.random.default_rng(seed + 1).permutation(len(big))[np.arange(B) % len(big)]]
    docs = []
    for _ in range(3 if tree else 1):
        doc = text.clone()
        doc[:, 4:] = _corrupt(g, text[:, 4:], V)
        docs.append(doc)
    docs = torch.stack(docs, 1).reshape(-1, 4 + K)
    if case["form"] == "fused":                 # a retrieved draft may also be short, or missing
        cut = torch.randint(0, K + 1, (B,), generator=g, device=DEV)
        docs = torch.where(torch.arange(4 + K, device=DEV) < 4 + cut[:, None], docs, -1)
    _put(tok, offs, np.repeat(gid, 3 if tree else 1), docs)
    pool = L.pool_build(tok, offs, 1, 4)
    prm = L.make_params(K=K, n_min=1 if case["form"] != "fused" else 2, n_max=4, max_occ=64, mode=MODES[case["mode"]], topk=2, p=0.1)
    dev = dict(dtype=torch.int32, device=DEV)
    st = dict(case=case, model=model, kv=kv, pool=pool, prm=prm, K=K, lens=lens, ids=torch.arange(B, **dev),
              tails=text[:, :4].to(torch.int32).contiguous(), tail_len=torch.full((B,), 4, **dev),
              gid=torch.from_numpy(gid.astype(np.int32)).to(DEV), last=text[:, 3].to(torch.int32).contiguous(),
              draft=(torch.empty(B, K, **dev), torch.empty(B, **dev), torch.empty(B, **dev)),
              rows=(torch.empty(B, K + 1, **dev), torch.empty(B, **dev)),
              out=(torch.empty(B, **dev), torch.empty(B, K + 1, **dev), torch.empty(B, **dev)))
    if case["form"] != "fused":
        st["logits"] = torch.zeros(B, K + 1, V, dtype=torch.float32, device=DEV)
    return st


def _run_step(s):
    L.kv_set_len_dev(s["kv"], s["lens"])        # (a pass starts from the same text; a program goes on with the longer one)
    if s["case"]["form"] == "tree":
        d, par, n, m = L.draft_tree(s["pool"], s["tails"], s["tail_len"], s["gid"], s["prm"])
        tokens, parents, n_rows = L.make_rows_tree(s["last"], d, par, n, s["K"])
        L.verify_step_tree(s["model"], s["kv"], s["ids"], tokens, parents, n_rows, logits=s["logits"])
        out = L.accept_tree(s["kv"], s["ids"], s["logits"], tokens, parents, n_rows, s["prm"])
        return dict(draft=d, parents=par, draft_len=n, match_n=m, logits=s["logits"], accept=out)
    d, n, m = L.draft(s["pool"], s["tails"], s["tail_len"], s["gid"], s["prm"], *s["draft"])
    tokens, n_rows = L.make_rows(s["last"], d, n, s["K"], *s["rows"])
    if s["case"]["form"] == "fused":
        out = L.verify_accept(s["model"], s["kv"], s["ids"], tokens, n_rows, s["prm"], out=s["out"])
        return dict(draft=d, draft_len=n, match_n=m, accept=out)
    L.verify_step(s["model"], s["kv"], s["ids"], tokens, n_rows, logits=s["logits"])
    out = L.accept_commit(s["kv"], s["ids"], s["logits"], tokens, n_rows, s["prm"], out=s["out"])
    return dict(draft=d, draft_len=n, match_n=m, logits=s["logits"], accept=out)


def _prepare_generate(case, seed):
    g = _gen(seed, 2)
    cfg = _cfg(case)
    B, K, V = case["batch"], case["draft"], cfg["vocab"]
    W, succ = _weights(cfg, g)
    model = L.model_create(cfg, W, max_batch=B)
    rng = np.random.default_rng(seed)
    lens = rng.integers(case["prompt_lo"], case["prompt_hi"] + 1, B)
    prompts = [rng.integers(0, V, n).astype(np.int32) for n in lens]
    pages = -(-(case["prompt_hi"] + case["new"] + K + 1) // 16)
    kv = L.kv_create(model, B, B * pages)
    tok, offs, perm = _pool_text(g, seed, case["pool"], case["groups"], V, least=-(-B // case["groups"]) * (case["new"] + 2))
    gid = np.arange(B, dtype=np.int32) % case["groups"]
    last = torch.tensor([int(p[-1]) for p in prompts], device=DEV)
    text = _chain(last, succ, case["new"] + 1)
    doc = _corrupt(g, text, V, 0.85)            # what other texts of the group say, in part
    doc[:, 0] = text[:, 0]
    _put(tok, offs, gid, doc)
    pool = L.pool_build(tok, offs, 1, 4)
    form = case["form"]
    prm = L.make_params(K=K, n_min=1, n_max=4, max_occ=64, mode=MODES[case["mode"]], topk=2, p=0.1, max_new=case["new"],
                        temp_branches=int(form == "temp"), tree=int(form == "tree"), fused_accept=int(form == "fused"))
    return dict(case=case, model=model, kv=kv, pool=pool, prm=prm, prompts=prompts, gid=gid)


def _run_generate(s):
    r = L.generate(s["model"], s["kv"], s["pool"], s["prompts"], s["gid"], s["prm"])
    return dict(out=np.asarray(r["out"], dtype=np.int32), out_len=r["out_len"])


def _prepare_draft(case, seed):
    g = _gen(seed, 3)
    tok, offs, perm = _pool_text(g, seed, case["pool"], case["groups"], 32000)
    tails, tail_len, gid = _queries(g, tok, offs, perm, case["queries"], case["n_max"], 32000)
    prm = L.make_params(K=case["draft"], n_min=1, n_max=case["n_max"], max_occ=case.get("max_occ", 64))
    st = dict(case=case, prm=prm, q=(tails, tail_len, gid))
    if case["kind"] == "draft":
        st["pool"] = L.pool_build(tok, offs, 1, case["n_max"])
    else:
        st["text"] = (tok, offs)
    return st


def _run_draft(s):
    return dict(zip(("draft", "draft_len", "match_n"), L.draft(s["pool"], *s["q"], s["prm"])))


def _run_build(s):
    pool = L.pool_build(*s["text"], 1, s["case"]["n_max"])
    out = dict(zip(("draft", "draft_len", "match_n"), L.draft(pool, *s["q"], s["prm"])))
    info = pool.info()
    pool.free()
    return dict(out, n_tokens=info["n_tokens"], n_keys=info["n_keys"])


def _prepare_accept(case, seed):
    """Logits as synth.make_accept_case shapes them (the top token's mass uniform in 0.05 .. 0.9, drafts among the first
    ranks), but for the ties and for masses within 1e-3 of the threshold, drawn on the GPU."""
    g = _gen(seed, 4)
    B, R, V = case["batch"], case["draft"] + 1, case["vocab"]
    x = torch.empty(B * R, V, dtype=torch.float32, device=DEV).normal_(generator=g)
    mass = torch.rand(B * R, 1, generator=g, device=DEV) * 0.85 + 0.05
    mass = torch.where((mass - 0.1).abs() < 1e-3, mass + 0.01, mass)
    at = torch.randint(0, V, (B * R, 1), generator=g, device=DEV)
    x.scatter_(1, at, -math.inf)
    x.scatter_(1, at, (mass / (1 - mass)).log() + torch.logsumexp(x, 1, keepdim=True))
    top = x.topk(3, 1).indices
    c = torch.rand(B * R, generator=g, device=DEV)
    rank = (c >= 0.65).long() + (c >= 0.85).long()
    pick = top.gather(1, rank[:, None])[:, 0].view(B, R)
    tokens = torch.randint(0, V, (B, R), generator=g, device=DEV)
    tokens[:, 1:] = pick[:, :-1]
    n_rows = torch.randint(1, R + 1, (B,), generator=g, device=DEV).to(torch.int32)
    prm = L.make_params(K=R - 1, mode=MODES[case["mode"]], topk=case["topk"], p=0.1)
    dev = dict(dtype=torch.int32, device=DEV)
    return dict(case=case, logits=x.view(B, R, V), tokens=tokens.to(torch.int32), n_rows=n_rows, prm=prm,
                out=(torch.empty(B, **dev), torch.empty(B, R, **dev), torch.empty(B, **dev)))


def _run_accept(s):
    return L.accept_commit(None, None, s["logits"], s["tokens"], s["n_rows"], s["prm"], out=s["out"])


_PREPARE = dict(step=_prepare_step, generate=_prepare_generate, draft=_prepare_draft, build=_prepare_draft, accept=_prepare_accept)
_RUN = dict(step=_run_step, generate=_run_generate, draft=_run_draft, build=_run_build, accept=_run_accept)


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def run(state):
    return _RUN[state["case"]["kind"]](state)


# ---- what a pass cannot do without ----------------------------------------------------------------------------

def _model_work(case, rows, ctx_tokens, head_rows, stored_rows):
    """One forward of `rows` token rows that attend to `ctx_tokens` cached tokens in all, `head_rows` of them through the
    LM head and `stored_rows` rows of logits kept."""
    c = _cfg(case)
    d, f, V, n = c["d_model"], c["d_ffn"], c["vocab"], c["n_layers"]
    dkv, dq = c["n_kv_heads"] * c["head_dim"], c["n_heads"] * c["head_dim"]
    layers = n * (d * (dq + 2 * dkv) + dq * d + 3 * d * f)
    head = d * V if head_rows else 0
    byte = 2 * (layers + head) + 4 * n * dkv * (ctx_tokens + rows) + 4 * V * stored_rows
    return byte, 2 * rows * layers + 2 * head_rows * head


def work(case):
    kind = case["kind"]
    if kind == "step":
        B, R = case["batch"], case["draft"] + 1
        ctx = B * (case["ctx_lo"] + case["ctx_hi"]) / 2
        byte, flop = _model_work(case, B * R, ctx, B * R, 0 if case["form"] == "fused" else B * R)
        return dict(bytes=byte, flops=flop + 4 * R * ctx * case["layers"] * synth.MODEL_SHAPES[case["shape"]]["d_model"])
    if kind == "generate":
        # prompts once; then steps of about 1 + sum of 0.85^i tokens, each of which reads the weights and the cache
        B, R = case["batch"], case["draft"] + 1
        mean = (case["prompt_lo"] + case["prompt_hi"]) / 2
        steps = math.ceil(case["new"] / sum(0.85 ** i for i in range(R)))
        b0, f0 = _model_work(case, B * mean, 0, 0, 0)
        b1, f1 = _model_work(case, B * R, B * (mean + case["new"] / 2), B * R, 0)
        attn = 2 * B * mean * mean * case["layers"] * synth.MODEL_SHAPES[case["shape"]]["d_model"]
        return dict(bytes=b0 + steps * b1, flops=f0 + attn + steps * f1)
    if kind == "accept":
        rows = case["batch"] * (case["draft"] + 2) / 2          # n_rows is uniform in 1 .. K + 1
        return dict(bytes=4 * rows * case["vocab"], flops=4 * rows * case["vocab"])
    # a query reads its tail, one table entry per suffix length and, where it matches, some continuations
    q = case["queries"] * (4 * case["n_max"] + 32 * case["n_max"] + 8 * 4 * case["draft"])
    if kind == "draft":
        return dict(bytes=q, flops=0)
    # per suffix length the tokens in, the positions and the distinct keys' entries out
    return dict(bytes=case["pool"] * case["n_max"] * (4 + 4 + 16 * 0.5) + q, flops=0)


def tolerance(case):
    if case["kind"] in ("draft", "build", "accept"):
        return "exact"
    if case["kind"] == "generate":
        return dict(rel=0.0, max=0.0, differ=0.0)
    # Logits; the tokens beside them have margins of several logits and stay the same.  Another split of the
    # contractions' sums moves 32 layers of the default mode by rel 5.7e-3, max 3.2e-2 (bf16 operands round
    # differently) and of the precise mode by 1.4e-5 and 1.5e-4.
    if case.get("precise"):
        return dict(rel=1e-4, max=1e-3, differ=0.0)
    return dict(rel=2.3e-2, max=0.12, differ=0.0)
