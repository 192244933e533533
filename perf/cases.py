"""The measured cases: what a search on this library has it do, call by call.

Five kinds of case, each through the public calls of ``paper_2608_08020_gb300``:

* ``step``    one decode step of every layer over a beam tree that is already there (the inner
              loop of a search, and where nearly all of its time goes).  The tree is grown by the
              schedule's own rounds: append a thought, push the scores, prune and branch.  Each
              pass appends one token to every beam, as a search does; a search that has used up
              its room ends and the next one begins.
* ``search``  a whole short search from ``gb_pool_init`` on: seed the prompt, then rounds of
              thoughts (appended at once or decoded token by token), scores and tournaments.
* ``rows``    ``gb_paged_decode_noalloc``: decode attention over a serving program's own pages.
* ``scorer``  the sequence scorer over the thought boundaries of a search, its step pool forked
              at every tournament.
* ``boundary`` one thought boundary of a running search: hidden states to scores and running means.

Every input is drawn from the case's seed alone.  ``exact`` replays a case in 64 bits with plain
torch and numpy.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_08020_gb300 import binding as B
from paper_2608_08020_gb300.pool import BeamPool, TORCH_DT
from paper_2608_08020_gb300.seqscorer import SeqScorer

CHUNK = 256          # tokens appended by one call while a tree is grown


# --------------------------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------------------------

def _step(name, **kw):
    c = {"name": name, "kind": "step", "beams": 64, "prompt": 512, "context": 4000, "interval": 512, "K": 32,
         "fanout": 2, "layers": 36, "q_heads": 32, "kv_heads": 8, "page": 16, "path": "auto", "head_scale": False,
         "room": 512}
    c.update(kw)
    return c


def _search(name, **kw):
    c = {"name": name, "kind": "search", "dtype": "bf16", "layers": 1, "beams": 8, "q_heads": 32, "kv_heads": 8,
         "head_dim": 128, "page": 16, "prompt": 64, "rounds": 2, "thought": 0, "steps": 8, "K": 4, "fanout": 2,
         "finish": 0, "scorer": "probe", "hidden": 256, "path": "auto", "graph": False}
    c.update(kw)
    return c


def listed():
    return [
        # The smallest search (8 beams, fp32, contexts 64 to 256, two tournaments), its decode steps
        # replayed from a CUDA graph as a launch-bound loop is run: latency and launches only.
        _search("tiny_fp32", dtype="f32", q_heads=4, kv_heads=2, head_dim=64, steps=96, graph=True),
        # A small interactive search: 13 beams over an odd prompt, 64-token pages, 8 query heads per
        # KV head, a few layers, eager calls, ragged tails and copy-on-write at every round.
        _search("small_search", layers=8, beams=13, q_heads=64, kv_heads=8, page=64, prompt=333, rounds=3, steps=8,
                K=5, hidden=1024),
        # Thoughts of 200 tokens appended at once, then scored, pruned and branched; traces that
        # complete are released and their slots branched again (page accounting and tournaments).
        _search("thoughts_256", layers=2, beams=256, prompt=300, rounds=6, thought=199, steps=1, K=128, finish=24,
                scorer="push"),
        # The decode step of a 36-layer model over 64 beams at 4K tokens: an ordinary search.
        _step("step_64x4k"),
        # Parallel sampling: 512 beams, one in four kept and branched four ways, per-head KV scales.
        _step("step_512x16k", beams=512, prompt=1024, context=16000, interval=1024, K=384, fanout=4, layers=4,
              head_scale=True),
        # Long contexts over a long shared prompt, 32-token pages.
        _step("step_256x32k", beams=256, prompt=4096, context=32000, interval=2048, K=128, layers=2, page=32),
        # The memory-capped search: as many beams as a fixed pool holds, every layer (the largest).
        _step("step_198x8k", beams=198, context=8000, K=99, room=192),
        # Independent traces that share nothing, every beam reading its own context.
        _step("step_unshared_64x16k", prompt=1, context=16000, interval=0, K=0, layers=4, path="per_beam"),
        # A serving program's own pages and tables, ragged lengths up to 8K, pages scattered.
        {"name": "rows_96", "kind": "rows", "dtype": "bf16", "rows": 96, "shortest": 1, "longest": 8192, "q_heads": 32,
         "kv_heads": 8, "head_dim": 128, "page": 16},
        # A handful of short rows of the same: what one small request costs.
        {"name": "rows_5", "kind": "rows", "dtype": "bf16", "rows": 5, "shortest": 17, "longest": 700, "q_heads": 16,
         "kv_heads": 4, "head_dim": 128, "page": 32},
        # A thought boundary of 512 beams scored by the two-layer MLP.
        {"name": "boundary_mlp_512", "kind": "boundary", "scorer": "mlp", "beams": 512, "hidden": 4096,
         "hidden_dtype": "bf16", "width": 512},
        # The sequence scorer over ten thought boundaries of 64 traces, forked at each.
        {"name": "scorer_64", "kind": "scorer", "beams": 64, "hidden": 4096, "layers": 2, "q_heads": 4, "kv_heads": 2,
         "ffn": 1024, "steps": 10, "page": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "search", "search", "rows", "rows", "boundary", "scorer"])
    if kind == "step":
        kvh = rng.choice([4, 8])
        c = _step("", beams=_log(rng, 16, 512), prompt=_log(rng, 1, 4096), interval=_log(rng, 128, 2048),
                  q_heads=kvh * rng.choice([2, 4, 8]), kv_heads=kvh, page=rng.choice([16, 32, 64]),
                  fanout=rng.choice([2, 2, 4]), path=rng.choice(["auto", "auto", "auto", "per_beam"]),
                  head_scale=rng.random() < 0.3, room=1024)
        c["K"] = c["beams"] // 2 if c["fanout"] == 2 else 3 * c["beams"] // 4
        c["context"] = min(32000, c["prompt"] + 2 * c["interval"] + _log(rng, 1, 12000))
        # As many layers as make a pass of a few milliseconds, at most a 36-layer model.
        per_layer = 25.0 + _tree_tokens(c)[0] * kvh * 512 / 5.5e6          # microseconds
        c["layers"] = max(1, min(36, int(2500 / per_layer) + 1))
    elif kind == "search":
        kvh = rng.choice([2, 4, 8])
        f32 = rng.random() < 0.3
        c = _search("", dtype="f32" if f32 else "bf16", layers=rng.choice([1, 2, 4]), beams=_log(rng, 4, 256),
                    q_heads=kvh * rng.choice([2, 4, 8]), kv_heads=kvh, head_dim=64 if f32 else 128,
                    page=rng.choice([16, 32, 64]), prompt=_log(rng, 1, 1024), rounds=rng.randint(2, 5),
                    thought=rng.choice([0, 0, _log(rng, 8, 256)]), steps=rng.randint(1, 12),
                    fanout=rng.choice([2, 3, 4]), scorer="push", path=rng.choice(["auto", "auto", "per_beam"]),
                    graph=rng.random() < 0.3)
        c["K"] = c["beams"] // 2
        c["finish"] = rng.choice([0, c["beams"] // 8])
        if c["graph"]:
            c["finish"] = 0
    elif kind == "rows":
        f32 = rng.random() < 0.3
        kvh = rng.choice([1, 2, 4, 8])
        longest = _log(rng, 64, 16384)
        c = {"kind": "rows", "dtype": "f32" if f32 else "bf16", "rows": _log(rng, 1, 192),
             "shortest": _log(rng, 1, longest), "longest": longest, "q_heads": kvh * rng.choice([2, 4, 8]),
             "kv_heads": kvh, "head_dim": 64 if f32 else 128, "page": rng.choice([16, 32, 64])}
    elif kind == "boundary":
        mlp = rng.random() < 0.6
        c = {"kind": "boundary", "scorer": "mlp" if mlp else "probe", "beams": _log(rng, 8, 1024),
             "hidden": 64 * _log(rng, 4, 128), "hidden_dtype": "bf16" if mlp else rng.choice(["bf16", "f32"]),
             "width": _log(rng, 64, 2048) if mlp else 0}
    else:
        kvh = rng.choice([1, 2, 4])
        c = {"kind": "scorer", "beams": _log(rng, 8, 512), "hidden": rng.choice([1024, 2560, 4096, 5120]),
             "layers": rng.randint(1, 3), "q_heads": kvh * rng.choice([2, 4]), "kv_heads": kvh,
             "ffn": 64 * rng.randint(4, 32), "steps": rng.randint(4, 16), "page": rng.choice([16, 32])}
    c.pop("name", None)
    return c


# --------------------------------------------------------------------------------------------
# The tournament and the tree in numpy (sizes of the pools, the work, and the exact replay)
# --------------------------------------------------------------------------------------------

class _Tree:
    """Which slot holds what: running means and the routing of Algorithm 1's tournament."""

    def __init__(self, C):
        self.C = C
        self.active = np.ones(C, bool)
        self.mean = np.zeros(C, np.float32)
        self.n = np.zeros(C, np.int64)
        self.lineage = np.arange(1, C + 1, dtype=np.int64)
        self.next_lineage = C + 1

    def push(self, scores):
        for b in np.flatnonzero(self.active):
            self.n[b] += 1
            d = np.float32(np.float32(scores[b]) - self.mean[b])
            self.mean[b] = np.float32(self.mean[b] + np.float32(d / np.float32(self.n[b])))

    def prune(self, K, fanout):
        """(parent_of, pruned) of one round; every active slot is eligible."""
        C, act = self.C, self.active.copy()
        order = [int(b) for b in sorted(np.flatnonzero(act), key=lambda b: (-float(self.mean[b]), b))]
        N = len(order)
        parent = np.where(act, np.arange(C), -1).astype(np.int32)
        pruned = np.zeros(C, np.uint8)
        if N < C:
            per, nchild = 1, min(C - N, N)
            parents, slots = order, np.flatnonzero(~act)[:nchild]
        else:
            per = fanout - 1
            Kc = min(K, N)
            parents = order[:N - Kc]
            nchild = min(Kc, per * len(parents))
            slots = np.sort(np.array(order[N - nchild:], dtype=np.int64))
            pruned[slots] = 1
        for k, s in enumerate(slots):
            p = parents[k // per]
            parent[s] = p
        for k, s in enumerate(slots):
            p = parent[s]
            self.mean[s], self.n[s], self.active[s] = self.mean[p], self.n[p], True
            self.lineage[s] = self.next_lineage + k
        self.next_lineage += len(slots)
        return parent, pruned

    def release(self, slots):
        self.active[slots] = False


def _round_scores(seed, rounds, C):
    return np.random.RandomState(seed & 0x7fffffff).uniform(0.0, 1.0, (max(rounds, 1), C)).astype(np.float32)


def _round_lengths(case):
    """Context lengths at which a tree's tournaments run."""
    if not case["interval"]:
        return []
    return list(range(case["prompt"] + case["interval"], case["context"], case["interval"]))


def _tree_tokens(case, seed=0):
    """(distinct tokens held at the context, the most pages held on the way there)."""
    C, P = case["beams"], case["page"]
    rounds = _round_lengths(case)
    scores = _round_scores(seed, len(rounds), C)
    tree = _Tree(C)
    ends = rounds + [case["context"]]
    hist = np.zeros((C, len(ends)), np.int64)      # slot that wrote the beam's i-th interval
    at, most, tokens = case["prompt"], 0, 0
    lengths = []
    for i, end in enumerate(ends):
        hist[:, i] = np.arange(C)
        lengths.append(end - at)
        at = end
        nodes = [len(np.unique(hist[:, j])) for j in range(i + 1)]
        tokens = case["prompt"] + sum(n * m for n, m in zip(nodes, lengths))
        pages = -(-case["prompt"] // P) + sum(n * (-(-m // P) + 1) for n, m in zip(nodes, lengths))
        most = max(most, pages)
        if i < len(rounds):
            tree.push(scores[i])
            parent, _ = tree.prune(case["K"], case["fanout"])
            hist = hist[parent]
    return tokens, most


def _seed_of(*parts):
    x = 0x9E3779B9
    for p in parts:
        x = (x * 1000003 + int(p) + 12345) & 0x7fffffffffff
    return x


def _randn(shape, dtype, *key, scale=None):
    g = torch.Generator(device="cuda")
    g.manual_seed(_seed_of(*key))
    x = torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=g)
    return x if scale is None else x.mul_(scale)


# --------------------------------------------------------------------------------------------
# step: one decode step of every layer over a grown tree
# --------------------------------------------------------------------------------------------

def _head_scale(case, seed):
    if not case["head_scale"]:
        return None
    s = np.random.RandomState(_seed_of(seed, 7) & 0x7fffffff).uniform(0.5, 2.0, case["kv_heads"]).astype(np.float32)
    return torch.from_numpy(s).cuda().to(torch.bfloat16).view(-1, 1)


def _tree_kv(case, seed, layer, chunk, tokens, prompt=False):
    """K and V of `tokens` tokens of every slot (or of the prompt)."""
    rows = (tokens,) if prompt else (tokens, case["beams"])
    shape = rows + (case["kv_heads"], 128)
    hs = _head_scale(case, seed)
    return [_randn(shape, torch.bfloat16, seed, 1 + w, layer, chunk, int(prompt), scale=hs) for w in (0, 1)]


def _chunks(case):
    """The growth of a tree: (chunk number, tokens, round that follows or None)."""
    out, at, n = [], case["prompt"], 0
    rounds = _round_lengths(case)
    for i, end in enumerate(rounds + [case["context"]]):
        while at < end:
            m = min(CHUNK, end - at)
            at += m
            out.append((n, m, i if at == end and i < len(rounds) else None))
            n += 1
    return out


def _grow(st):
    """Begin a search and grow its tree to the context."""
    case, seed, pool = st["case"], st["seed"], st["pool"]
    if st["grown"]:
        B.gb_pool_destroy(pool.handle)
        pool.handle = B.gb_pool_init(pool.cfg, pool.kv, pool.meta)
    st["grown"] = True
    L = case["layers"]
    kv = [_tree_kv(case, seed, l, -1, case["prompt"], True) for l in range(L)]
    k, v = (torch.stack([x[w] for x in kv]) for w in (0, 1))
    pool.seed(case["beams"], case["prompt"], k, v)
    for n, m, rnd in _chunks(case):
        for l in range(L):
            k, v = _tree_kv(case, seed, l, n, m)
            pool.append_kv(l, m, k, v)
        if rnd is not None:
            pool.push_scores(st["scores"][rnd])
            pool.prune_branch(case["K"], case["fanout"])
    st["left"] = case["room"]
    assert pool.status() == 0


def _prepare_step(case, seed):
    C, L, Hq, Hkv, P = case["beams"], case["layers"], case["q_heads"], case["kv_heads"], case["page"]
    _, pages = _tree_tokens(case, seed)
    pages += C * (-(-case["room"] // P) + 2) + 64
    pool = BeamPool(num_layers=L, num_q_heads=Hq, num_kv_heads=Hkv, head_dim=128, page_size=P, kv_dtype="bf16",
                    num_pages=pages, max_beams=C, max_pages_per_beam=-(-(case["context"] + case["room"]) // P) + 1)
    st = {"case": case, "seed": seed, "pool": pool, "grown": False,
          "scores": torch.from_numpy(_round_scores(seed, len(_round_lengths(case)), C)).cuda(),
          "q": [_randn((C, Hq, 128), torch.bfloat16, seed, 11, l) for l in range(L)],
          "kv": [_tree_kv(case, seed, l, -2, 1) for l in range(L)],
          "out": [torch.empty((C, Hq, 128), dtype=torch.float32, device="cuda") for _ in range(L)],
          "flags": B.GB_PATH_PER_BEAM if case["path"] == "per_beam" else B.GB_PATH_AUTO}
    _grow(st)
    return st


def _run_step(st):
    if st["left"] == 0:
        _grow(st)
    st["left"] -= 1
    pool, flags, scale = st["pool"], st["flags"], 1.0 / math.sqrt(128)
    for l, (q, (k, v), out) in enumerate(zip(st["q"], st["kv"], st["out"])):
        pool.decode_attention(l, q, k, v, scale, out, flags)
    return st["out"]


def _attend(q, K, V, L, scale):
    """64-bit decode attention of every beam: q [C][Hq][D] over K, V [C][>= L][Hkv][D]."""
    C, Hq, D = q.shape
    Hkv = K.shape[2]
    out = torch.empty((C, Hq, D), dtype=torch.float64, device=q.device)
    for b in range(C):
        k, v = (x[b, :L].double().transpose(0, 1) for x in (K, V))            # [Hkv][L][D]
        s = torch.bmm(q[b].double().view(Hkv, Hq // Hkv, D), k.transpose(1, 2)) * scale
        out[b] = torch.bmm(torch.softmax(s, -1), v).reshape(Hq, D)
    return out


def _exact_step(case, seed):
    C, L, Hq, Hkv = case["beams"], case["layers"], case["q_heads"], case["kv_heads"]
    scores = _round_scores(seed, len(_round_lengths(case)), C)
    outs = [None] * L
    for l in sorted({0, L - 1}):
        K, V = (torch.empty((C, case["context"] + 1, Hkv, 128), dtype=torch.bfloat16, device="cuda") for _ in (0, 1))
        tree, at = _Tree(C), case["prompt"]
        for X, p in zip((K, V), _tree_kv(case, seed, l, -1, at, True)):
            X[:, :at] = p
        for n, m, rnd in _chunks(case):
            for X, x in zip((K, V), _tree_kv(case, seed, l, n, m)):
                X[:, at:at + m] = x.transpose(0, 1)
            at += m
            if rnd is not None:
                tree.push(scores[rnd])
                parent, _ = tree.prune(case["K"], case["fanout"])
                for s in np.flatnonzero(parent != np.arange(C)):
                    for X in (K, V):
                        X[s, :at] = X[int(parent[s]), :at]
        for X, x in zip((K, V), _tree_kv(case, seed, l, -2, 1)):
            X[:, at] = x[0]
        outs[l] = _attend(_randn((C, Hq, 128), torch.bfloat16, seed, 11, l), K, V, at + 1, 1.0 / math.sqrt(128))
        del K, V
    return outs


# --------------------------------------------------------------------------------------------
# search: a whole short search
# --------------------------------------------------------------------------------------------

def _search_tokens(case):
    return case["prompt"] + case["rounds"] * (case["thought"] + case["steps"])


def _search_inputs(case, seed):
    dt = TORCH_DT[case["dtype"]]
    C, L, Hq, Hkv, D, R = (case[k] for k in ("beams", "layers", "q_heads", "kv_heads", "head_dim", "rounds"))
    qs = 0.125 if case["dtype"] == "f32" else None
    x = {"prompt": [_randn((L, case["prompt"], Hkv, D), dt, seed, 21 + w) for w in (0, 1)],
         "q": _randn((R, case["steps"], L, C, Hq, D), dt, seed, 23, scale=qs),
         "kv": [_randn((R, case["steps"], L, C, Hkv, D), dt, seed, 24 + w) for w in (0, 1)],
         "scores": _round_scores(seed, R, C)}
    if case["thought"]:
        x["thought"] = [_randn((R, L, case["thought"], C, Hkv, D), dt, seed, 26 + w) for w in (0, 1)]
    if case["scorer"] == "probe":
        x["hidden"] = _randn((R, C, case["hidden"]), dt, seed, 28)
        x["w"] = _randn((case["hidden"],), torch.float32, seed, 29, scale=1.0 / math.sqrt(case["hidden"]))
    r = np.random.RandomState(_seed_of(seed, 30) & 0x7fffffff)
    x["done"] = [np.sort(r.choice(C, case["finish"], replace=False)).astype(np.int32)
                 if case["finish"] and i % 3 == 1 else None for i in range(R)]
    return x


def _scale_of(case):
    return 1.0 if case["dtype"] == "f32" else 1.0 / math.sqrt(case["head_dim"])


def _prepare_search(case, seed):
    C, L, Hq, Hkv, D, R, P = (case[k] for k in ("beams", "layers", "q_heads", "kv_heads", "head_dim", "rounds", "page"))
    width = -(-_search_tokens(case) // P) + 1
    pool = BeamPool(num_layers=L, num_q_heads=Hq, num_kv_heads=Hkv, head_dim=D, page_size=P, kv_dtype=case["dtype"],
                    num_pages=C * (width + 1) + 64, max_beams=C, max_pages_per_beam=width)
    x = _search_inputs(case, seed)
    dev = lambda shape, dt: torch.zeros(shape, dtype=dt, device="cuda")
    st = {"case": case, "pool": pool, "prompt": x["prompt"], "thoughts": x.get("thought"), "graph": None,
          "flags": B.GB_PATH_PER_BEAM if case["path"] == "per_beam" else B.GB_PATH_AUTO,
          "out": dev((R, case["steps"], L, C, Hq, D), torch.float32), "probe": dev((R, C), torch.float32),
          "parent": dev((R, C), torch.int32), "pruned": dev((R, C), torch.uint8), "lineage": dev((R, C), torch.int32),
          "scores": torch.from_numpy(x["scores"]).cuda(), "w": x.get("w"), "hidden": x.get("hidden"),
          "done": [None if d is None else torch.from_numpy(d).cuda() for d in x["done"]]}
    # One call's arguments each, kept as the views a program would hold.
    st["calls"] = [[[(l, x["q"][r, t, l], x["kv"][0][r, t, l], x["kv"][1][r, t, l], st["out"][r, t, l])
                     for l in range(L)] for t in range(case["steps"])] for r in range(R)]
    if case["graph"]:
        _begin_search(st)
        _search_rounds(st)
        torch.cuda.synchronize()
        _begin_search(st)
        torch.cuda.synchronize()
        st["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st["graph"]):
            _search_rounds(st)
    return st


def _begin_search(st):
    """The buffers are kept; the pool on them is initialised anew for the search's prompt."""
    pool, case = st["pool"], st["case"]
    B.gb_pool_destroy(pool.handle)
    pool.handle = B.gb_pool_init(pool.cfg, pool.kv, pool.meta)
    pool.seed(case["beams"], case["prompt"], *st["prompt"])


def _search_rounds(st):
    pool, case, flags, scale = st["pool"], st["case"], st["flags"], _scale_of(st["case"])
    for r in range(case["rounds"]):
        if case["thought"]:
            for l in range(case["layers"]):
                pool.append_kv(l, case["thought"], st["thoughts"][0][r, l], st["thoughts"][1][r, l])
        for layers in st["calls"][r]:
            for l, q, k, v, out in layers:
                pool.decode_attention(l, q, k, v, scale, out, flags)
        if case["scorer"] == "probe":
            pool.score_probe(st["hidden"][r], case["dtype"], st["w"], 0.0, None, st["probe"][r])
        else:
            pool.push_scores(st["scores"][r])
        pool.prune_branch(case["K"], case["fanout"], 0, None, st["parent"][r], st["pruned"][r], st["lineage"][r])
        if st["done"][r] is not None:
            pool.release(st["done"][r])


def _run_search(st):
    _begin_search(st)
    if st["graph"] is not None:
        st["graph"].replay()
    else:
        _search_rounds(st)
    return {k: st[k] for k in ("out", "probe", "parent", "pruned", "lineage")}


def _exact_search(case, seed):
    C, L, Hq, Hkv, D, R = (case[k] for k in ("beams", "layers", "q_heads", "kv_heads", "head_dim", "rounds"))
    x, tree, total = _search_inputs(case, seed), _Tree(C), _search_tokens(case)
    K, V = (torch.zeros((L, C, total, Hkv, D), dtype=TORCH_DT[case["dtype"]], device="cuda") for _ in (0, 1))
    at = case["prompt"]
    for X, p in zip((K, V), x["prompt"]):
        X[:, :, :at] = p[:, None]
    out = torch.zeros((R, case["steps"], L, C, Hq, D), dtype=torch.float64, device="cuda")
    probe = torch.zeros((R, C), dtype=torch.float64, device="cuda")
    parents, pruneds, lineages = [], [], []
    for r in range(R):
        if case["thought"]:
            for X, t in zip((K, V), x["thought"]):
                X[:, :, at:at + case["thought"]] = t[r].transpose(1, 2)
            at += case["thought"]
        for t in range(case["steps"]):
            for X, n in zip((K, V), x["kv"]):
                X[:, :, at] = n[r, t]
            at += 1
            act = torch.from_numpy(tree.active).cuda()
            for l in range(L):
                out[r, t, l] = _attend(x["q"][r, t, l], K[l], V[l], at, _scale_of(case)) * act[:, None, None]
        if case["scorer"] == "probe":
            probe[r] = torch.sigmoid(x["hidden"][r].double() @ x["w"].double())
            tree.push(probe[r].float().cpu().numpy())
        else:
            tree.push(x["scores"][r])
        parent, pruned = tree.prune(case["K"], case["fanout"])
        for s in np.flatnonzero((parent >= 0) & (parent != np.arange(C))):
            for X in (K, V):
                X[:, s, :at] = X[:, int(parent[s]), :at]
        parents.append(parent)
        pruneds.append(pruned)
        lineages.append(tree.lineage.astype(np.int32))
        if x["done"][r] is not None:
            tree.release(x["done"][r])
    whole = lambda a: torch.from_numpy(np.stack(a))
    return {"out": out, "probe": probe, "parent": whole(parents), "pruned": whole(pruneds), "lineage": whole(lineages)}


# --------------------------------------------------------------------------------------------
# rows: decode attention over the caller's own pages
# --------------------------------------------------------------------------------------------

def _row_lengths(case, seed):
    r = np.random.RandomState(_seed_of(seed, 41) & 0x7fffffff)
    n = np.exp(r.uniform(math.log(case["shortest"]), math.log(case["longest"] + 0.999), case["rows"])).astype(np.int32)
    n = np.clip(n, case["shortest"], case["longest"])
    n[0] = case["longest"]
    return n


def _rows_inputs(case, seed):
    P, Hkv, D, dt = case["page"], case["kv_heads"], case["head_dim"], TORCH_DT[case["dtype"]]
    lens = _row_lengths(case, seed)
    width = -(-case["longest"] // P)
    pages = -(-lens // P)
    ids = np.random.RandomState(_seed_of(seed, 42) & 0x7fffffff).permutation(int(pages.sum())).astype(np.int32)
    tables = np.zeros((case["rows"], width), np.int32)
    at = 0
    for b, n in enumerate(pages):
        tables[b, :n] = ids[at:at + n]
        at += n
    kv = _randn((int(pages.sum()), 2, Hkv, P, D), dt, seed, 43)
    q = _randn((case["rows"], case["q_heads"], D), dt, seed, 44)
    return lens, tables, kv, q


def _prepare_rows(case, seed):
    lens, tables, kv, q = _rows_inputs(case, seed)
    out = torch.empty((case["rows"], case["q_heads"], case["head_dim"]), dtype=torch.float32, device="cuda")
    st = {"kv": kv, "q": q, "out": out, "tables": torch.from_numpy(tables).cuda(), "lens": torch.from_numpy(lens).cuda()}
    st["args"] = B.GbPagedDecodeArgs(
        kv.data_ptr(), st["tables"].data_ptr(), st["lens"].data_ptr(), q.data_ptr(), out.data_ptr(), case["rows"],
        case["q_heads"], case["kv_heads"], case["head_dim"], case["page"],
        B.GB_F32 if case["dtype"] == "f32" else B.GB_BF16, tables.shape[1], kv.shape[0],
        1.0 / math.sqrt(case["head_dim"]))
    return st


def _run_rows(st):
    B.gb_paged_decode_noalloc(st["args"])
    return st["out"]


def _exact_rows(case, seed):
    lens, tables, kv, q = _rows_inputs(case, seed)
    P, Hq, Hkv, D = case["page"], case["q_heads"], case["kv_heads"], case["head_dim"]
    out = torch.empty((case["rows"], Hq, D), dtype=torch.float64, device="cuda")
    for b, n in enumerate(lens):
        pages = kv[torch.from_numpy(tables[b, :-(-int(n) // P)].astype(np.int64)).cuda()]      # [n][2][Hkv][P][D]
        k, v = (pages[:, w].permute(1, 0, 2, 3).reshape(Hkv, -1, D)[:, :int(n)].double() for w in (0, 1))
        s = torch.bmm(q[b].double().view(Hkv, Hq // Hkv, D), k.transpose(1, 2)) / math.sqrt(D)
        out[b] = torch.bmm(torch.softmax(s, -1), v).reshape(Hq, D)
    return out


# --------------------------------------------------------------------------------------------
# boundary: the scorers of one thought boundary
# --------------------------------------------------------------------------------------------

def _boundary_inputs(case, seed):
    C, H, W = case["beams"], case["hidden"], case["width"]
    x = {"hidden": _randn((C, H), TORCH_DT[case["hidden_dtype"]], seed, 51)}
    if case["scorer"] == "mlp":
        x["w1"] = _randn((W, H), torch.bfloat16, seed, 52, scale=1.0 / math.sqrt(H))
        x["b1"] = _randn((W,), torch.float32, seed, 53, scale=0.1)
        x["w2"] = _randn((W,), torch.float32, seed, 54, scale=1.0 / math.sqrt(W))
    else:
        x["w"] = _randn((H,), torch.float32, seed, 55, scale=1.0 / math.sqrt(H))
    return x


def _prepare_boundary(case, seed):
    C = case["beams"]
    pool = BeamPool(num_layers=1, num_q_heads=32, num_kv_heads=8, head_dim=128, page_size=16, kv_dtype="bf16",
                    num_pages=16, max_beams=C, max_pages_per_beam=2)
    kp = torch.zeros((1, 1, 8, 128), dtype=torch.bfloat16, device="cuda")
    pool.seed(C, 1, kp, kp)
    return {"case": case, "pool": pool, "score": torch.zeros(C, dtype=torch.float32, device="cuda"),
            **_boundary_inputs(case, seed)}


def _run_boundary(st):
    pool = st["pool"]
    if st["case"]["scorer"] == "mlp":
        pool.score_mlp(st["hidden"], st["w1"], st["b1"], st["w2"], 0.1, None, st["score"])
    else:
        pool.score_probe(st["hidden"], st["case"]["hidden_dtype"], st["w"], 0.1, None, st["score"])
    return st["score"]


def _exact_boundary(case, seed):
    x = _boundary_inputs(case, seed)
    h = x["hidden"].double()
    if case["scorer"] == "mlp":
        z = torch.relu(h @ x["w1"].double().T + x["b1"].double()) @ x["w2"].double()
    else:
        z = h @ x["w"].double()
    return torch.sigmoid(z + 0.1)


# --------------------------------------------------------------------------------------------
# scorer: the sequence scorer over a search's thought boundaries
# --------------------------------------------------------------------------------------------

def _scorer_weights(case, seed):
    r = np.random.RandomState(_seed_of(seed, 61) & 0x7fffffff)
    H, F, d, hd = case["hidden"], case["ffn"], case["q_heads"] * 128, 128

    def mat(rows, cols):     # bf16 values held as fp32
        x = torch.from_numpy(r.standard_normal((rows, cols)).astype(np.float32) / np.float32(math.sqrt(cols)))
        return x.to(torch.bfloat16).float().numpy()

    def norm(n):
        return (1 + 0.1 * r.standard_normal(n)).astype(np.float32), (0.1 * r.standard_normal(n)).astype(np.float32)

    w = {"n_q_heads": case["q_heads"], "n_kv_heads": case["kv_heads"], "ln_in": norm(H), "w_in": mat(d, H), "layers": []}
    for _ in range(case["layers"]):
        w["layers"].append({"ln1": norm(d), "wq": mat(d, d), "wk": mat(case["kv_heads"] * hd, d),
                            "wv": mat(case["kv_heads"] * hd, d), "wo": mat(d, d), "ln2": norm(d), "w1": mat(F, d),
                            "w3": mat(F, d), "w2": mat(d, F)})
    w["ln_out"] = norm(d)
    w["w_out"] = (r.standard_normal(d) / math.sqrt(d)).astype(np.float32)
    w["b_out"] = 0.05
    return w


def _scorer_forks(case, seed):
    """parent_of after each boundary: the lower half of the scores takes the upper half's parents."""
    tree, scores = _Tree(case["beams"]), _round_scores(seed, case["steps"], case["beams"])
    out = []
    for t in range(case["steps"]):
        tree.push(scores[t])
        out.append(tree.prune(case["beams"] // 2, 2)[0])
    return np.stack(out)


def _scorer_hidden(case, seed):
    return (_randn((case["hidden"],), torch.bfloat16, seed, 62),
            _randn((case["steps"], case["beams"], case["hidden"]), torch.bfloat16, seed, 63))


def _prepare_scorer(case, seed):
    sc = SeqScorer(_scorer_weights(case, seed), hidden_dim=case["hidden"], ffn_dim=case["ffn"],
                   max_beams=case["beams"], max_steps=case["steps"] + 1, page_size=case["page"])
    h0, hidden = _scorer_hidden(case, seed)
    return {"case": case, "scorer": sc, "h0": h0, "hidden": list(hidden.unbind(0)),
            "parent": list(torch.from_numpy(_scorer_forks(case, seed)).cuda().unbind(0)),
            "scores": torch.zeros((case["steps"], case["beams"]), dtype=torch.float32, device="cuda")}


def _run_scorer(st):
    sc, case = st["scorer"], st["case"]
    pool = sc.pool
    B.gb_pool_destroy(pool.handle)
    pool.handle = B.gb_pool_init(pool.cfg, pool.kv, pool.meta)
    sc.seed(st["h0"], case["beams"])
    for hidden, score, parent in zip(st["hidden"], st["scores"].unbind(0), st["parent"]):
        sc.step(hidden, score)
        sc.fork(parent)
    return st["scores"]


def _exact_scorer(case, seed):
    w, forks = _scorer_weights(case, seed), _scorer_forks(case, seed)
    h0, hidden = _scorer_hidden(case, seed)
    C, Hq, Hkv, d = case["beams"], case["q_heads"], case["kv_heads"], case["q_heads"] * 128
    f64 = lambda a: torch.from_numpy(np.asarray(a, np.float64)).cuda()
    inv = 10000.0 ** (-torch.arange(64, dtype=torch.float64, device="cuda") / 64)

    def ln(x, gb):
        mu = x.mean(-1, keepdim=True)
        return (x - mu) / torch.sqrt(((x - mu) ** 2).mean(-1, keepdim=True) + 1e-5) * f64(gb[0]) + f64(gb[1])

    def rope(x, pos):
        c, s = torch.cos(pos * inv), torch.sin(pos * inv)
        a, b = x[..., :64], x[..., 64:]
        return torch.cat([a * c - b * s, a * s + b * c], -1)

    cache = [[None, None] for _ in w["layers"]]              # K, V of each slot's history: [C][t][Hkv][128]
    scores = torch.zeros((case["steps"], C), dtype=torch.float64, device="cuda")
    for t in range(case["steps"] + 1):
        h = h0.expand(C, -1) if t == 0 else hidden[t - 1]
        z = ln(h.double(), w["ln_in"]) @ f64(w["w_in"]).T
        x = 0.5 * z * (1 + torch.erf(z / math.sqrt(2)))
        for i, Lw in enumerate(w["layers"]):
            u = ln(x, Lw["ln1"])
            q = rope((u @ f64(Lw["wq"]).T).view(C, Hq, 128), t)
            k = rope((u @ f64(Lw["wk"]).T).view(C, 1, Hkv, 128), t)
            v = (u @ f64(Lw["wv"]).T).view(C, 1, Hkv, 128)
            for j, new in enumerate((k, v)):
                cache[i][j] = new if cache[i][j] is None else torch.cat([cache[i][j], new], 1)
            K, V = cache[i]
            s = torch.einsum("chgd,cthd->chgt", q.view(C, Hkv, Hq // Hkv, 128), K) / math.sqrt(128)
            a = torch.einsum("chgt,cthd->chgd", torch.softmax(s, -1), V).reshape(C, d)
            x = x + a @ f64(Lw["wo"]).T
            u = ln(x, Lw["ln2"])
            g = u @ f64(Lw["w1"]).T
            x = x + (g * torch.sigmoid(g) * (u @ f64(Lw["w3"]).T)) @ f64(Lw["w2"]).T
        if t > 0:
            scores[t - 1] = torch.sigmoid(ln(x, w["ln_out"]) @ f64(w["w_out"]) + w["b_out"])
            src = torch.from_numpy(forks[t - 1].astype(np.int64)).cuda()
            cache = [[X[src] for X in kv] for kv in cache]
    return scores


# --------------------------------------------------------------------------------------------
# What the measurement calls
# --------------------------------------------------------------------------------------------

_PREPARE = {"step": _prepare_step, "search": _prepare_search, "rows": _prepare_rows, "boundary": _prepare_boundary,
            "scorer": _prepare_scorer}
_RUN = {"step": _run_step, "search": _run_search, "rows": _run_rows, "boundary": _run_boundary, "scorer": _run_scorer}
_EXACT = {"step": _exact_step, "search": _exact_search, "rows": _exact_rows, "boundary": _exact_boundary,
          "scorer": _exact_scorer}


def prepare(case, seed):
    return {"kind": case["kind"], "state": _PREPARE[case["kind"]](case, seed)}


def run(state):
    return _RUN[state["kind"]](state["state"])


def exact(case, seed):
    return _EXACT[case["kind"]](case, seed)


def work(case):
    """Bytes and operations one pass cannot do without: distinct K/V once, inputs and outputs once."""
    kind, C = case["kind"], case.get("beams", 0)
    if kind == "step":
        tokens, _ = _tree_tokens(case)
        Hq, Hkv = case["q_heads"], case["kv_heads"]
        per_layer = (tokens + 2 * C) * Hkv * 512 + C * Hq * 128 * (2 + 4)
        return {"bytes": case["layers"] * per_layer, "flops": case["layers"] * C * case["context"] * Hq * 512}
    if kind == "search":
        Hq, Hkv, D, L, R = (case[k] for k in ("q_heads", "kv_heads", "head_dim", "layers", "rounds"))
        es = 4 if case["dtype"] == "f32" else 2
        row = 2 * Hkv * D * es
        sim = {"beams": C, "page": case["page"], "prompt": case["prompt"], "K": case["K"], "fanout": case["fanout"],
               "interval": case["thought"] + case["steps"]}
        nbytes = case["prompt"] * row * 2 * L
        flops = 0
        for r in range(R):
            end = case["prompt"] + (r + 1) * sim["interval"]
            tokens, _ = _tree_tokens({**sim, "context": end})
            nbytes += L * C * case["thought"] * row * 2
            nbytes += L * case["steps"] * (tokens * row + C * Hq * D * (es + 4) + 2 * C * row)
            flops += L * case["steps"] * C * end * Hq * D * 4
            nbytes += C * case["hidden"] * es if case["scorer"] == "probe" else 4 * C
        return {"bytes": nbytes, "flops": flops}
    if kind == "rows":
        es = 4 if case["dtype"] == "f32" else 2
        tokens = int(_row_lengths(case, 0).sum())
        return {"bytes": tokens * 2 * case["kv_heads"] * case["head_dim"] * es +
                case["rows"] * case["q_heads"] * case["head_dim"] * (es + 4),
                "flops": tokens * case["q_heads"] * case["head_dim"] * 4}
    if kind == "boundary":
        es, H, W = (4 if case["hidden_dtype"] == "f32" else 2), case["hidden"], case["width"]
        return {"bytes": C * H * es + (W * H * 2 + W * 8 if W else 4 * H) + 4 * C, "flops": 2 * C * H * max(W, 1)}
    H, F, d, T, L = case["hidden"], case["ffn"], case["q_heads"] * 128, case["steps"], case["layers"]
    nqkv = (case["q_heads"] + 2 * case["kv_heads"]) * 128
    params = d * H + L * (nqkv * d + d * d + 3 * F * d)
    history = C * T * (T + 1) // 2 * 2 * case["kv_heads"] * 128 * 2 * L
    return {"bytes": T * (2 * params + 2 * C * H) + history, "flops": 2 * T * C * params}


def tolerance(case):
    """About four times the error against 64 bits: fp32 sums over exact products (1e-7 for scores and
    rows, whose probabilities stay in fp32), and bf16 operands of a second product (probabilities, and
    every product's inputs in the scorer: 1.3e-3 to 2.3e-3)."""
    if case["kind"] == "boundary":
        return {"rel": 2e-6, "max": 2e-5}
    if case["kind"] == "scorer":
        return {"rel": 1e-2, "max": 5e-2}
    if case["kind"] == "rows" or case.get("dtype") == "f32":
        return {"rel": 1e-5, "max": 1e-3}
    return {"rel": 7e-3, "max": 6e-2}
