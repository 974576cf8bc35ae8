"""The work that users of the chordality test have it do, as measurable cases.

A case is a plain dict; `listed` names the fixed ones, `draw` gives others of
the same ranges.  `prepare` makes the inputs on the GPU from the seed alone
(graphs of the families the test is used on: subtree-intersection graphs,
which are chordal, with or without a planted chordless cycle; G(n, p); trees;
cliques; sparse chordal graphs grown along an elimination order), `run` is one
pass through the public entry points, `exact` the same in plain numpy.
"""
import math

import numpy as np
import torch

from paper_1508_06329_gb300 import binding as B

DEV = "cuda:0"
_ctx = None


def context():
    """One library context for the process, as a program that tests graphs keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = B.Context(0)
    return _ctx


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: a graph of a hundred vertices, where launches and step latency are all there is
        {"name": "dense_n100", "kind": "test", "family": "subtree", "n": 100, "tree": 50, "cycle": True},
        # the configuration of one dense graph of 1,000 vertices (500-node tree)
        {"name": "dense_n1000", "kind": "test", "family": "subtree", "n": 1000, "tree": 500, "cycle": False},
        # the headline: the N = 16,384 pair at density 0.1, chordal and with a chordless cycle, in one call
        {"name": "pair_n16384", "kind": "pair", "family": "subtree", "n": 16384, "tree": 562},
        # dense random graphs of the paper's Section 7.2
        {"name": "gnp_n10000", "kind": "test", "family": "gnp", "n": 10000, "p": 0.5},
        # a large CSR query dense enough for the bit-row kernels (the serving stream's slow tail);
        # 41,003 vertices: ragged rows, state beyond one CTA's shared memory
        {"name": "csr_dense_n41003", "kind": "csr", "family": "subtree", "n": 41003, "tree": 2800, "cycle": True},
        # sparse CSR graphs, about 10.5 edges per vertex, shuffled ids, a few edges that close cycles
        {"name": "csr_sparse_n65536", "kind": "csr", "family": "peo", "n": 65536, "smax": 20, "extra": 4},
        {"name": "csr_sparse_n262143", "kind": "csr", "family": "peo", "n": 262143, "smax": 20, "extra": 0},
        # many small graphs at once, N log-uniform in [16, 2048], half with a planted cycle, as a kept plan
        {"name": "batch_4096", "kind": "batch", "count": 4096, "nmin": 16, "nmax": 2048},
        # a burst of queries through the serving queue, N log-uniform in [64, 8192]
        {"name": "queue_64", "kind": "queue", "count": 64, "nmin": 64, "nmax": 8192},
        # the same test by Maximum Cardinality Search
        {"name": "mcs_n16384", "kind": "mcs", "family": "subtree", "n": 16384, "tree": 562, "cycle": True},
        # one LexBFS+ sweep (the building block of the multi-sweep algorithms)
        {"name": "sweep_n12000", "kind": "sweep", "family": "subtree", "n": 12000, "tree": 560, "cycle": False},
        # the perfect-elimination check of a given order alone
        {"name": "check_n16384", "kind": "check", "family": "subtree", "n": 16384, "tree": 562, "cycle": False},
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def _dense_family(rng, n):
    f = rng.choice(["subtree", "subtree", "subtree", "gnp", "tree", "clique"])
    if f == "subtree":   # densities of about 0.01 to 0.2, or the half-size tree of the small configurations
        tree = max(2, n // 2) if n <= 2048 and rng.random() < 0.5 else max(2, int(56 / rng.uniform(0.01, 0.2)))
        return {"family": f, "tree": tree, "cycle": rng.random() < 0.5}
    if f == "gnp":
        return {"family": f, "p": rng.choice([0.5, 0.2, min(0.5, 40.0 / n)])}
    return {"family": f}


def draw(rng):
    kind = rng.choice(["test", "test", "test", "pair", "csr", "csr", "batch", "queue", "mcs", "sweep", "check"])
    if kind == "batch":
        return {"kind": kind, "count": _log_int(rng, 32, 2048), "nmin": 16, "nmax": _log_int(rng, 128, 2048)}
    if kind == "queue":
        return {"kind": kind, "count": _log_int(rng, 8, 64), "nmin": 64, "nmax": _log_int(rng, 512, 8192)}
    if kind == "csr" and rng.random() < 0.7:
        return {"kind": kind, "family": "peo", "n": _log_int(rng, 4097, 200000), "smax": rng.randint(3, 20),
                "extra": rng.choice([0, 0, 1, 5])}
    if kind == "csr":
        n = _log_int(rng, 300, 30000)
        return {"kind": kind, "family": "subtree", "n": n, "tree": int(56 / rng.uniform(0.03, 0.15)),
                "cycle": rng.random() < 0.5}
    if kind == "pair":
        n = _log_int(rng, 4097, 16384)
        return {"kind": kind, "family": "subtree", "n": n, "tree": int(56 / rng.uniform(0.01, 0.2))}
    n = _log_int(rng, 64, 16384)
    return {"kind": kind, "n": n, **_dense_family(rng, n)}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 1508)
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV)


def _randint(g, high):
    """Uniform integers below each entry of `high`."""
    high = high.to(torch.int64)
    return torch.minimum((_rand(g, *high.shape).double() * high).long(), high - 1)


def _forest_subtrees(sizes, trees, g, smax=20):
    """For each graph k: sizes[k] random subtrees of one random recursive tree of
    trees[k] nodes, each grown from a uniform root by uniform frontier nodes to a
    size uniform in 1..smax.  Returns [sum sizes, smax] node ids (-1: none), the
    ids local to the graph's tree."""
    sizes, trees = (torch.tensor(x, device=DEV, dtype=torch.int64) for x in (sizes, trees))
    tbase = torch.cumsum(trees, 0) - trees
    total = int(trees.sum())
    tid = torch.repeat_interleave(torch.arange(len(trees), device=DEV), trees)
    local = torch.arange(total, device=DEV) - tbase[tid]
    child = local.nonzero()[:, 0]
    par = _randint(g, local[child]) + tbase[tid[child]]
    a, b = torch.cat([child, par]), torch.cat([par, child])
    b = b[torch.sort(a, stable=True)[1]]
    deg = torch.bincount(a, minlength=total)
    rp = torch.cumsum(deg, 0) - deg
    vid = torch.repeat_interleave(torch.arange(len(sizes), device=DEV), sizes)
    V = vid.numel()
    nodes = torch.full((V, smax), -1, device=DEV, dtype=torch.int64)
    nodes[:, 0] = tbase[vid] + _randint(g, trees[vid])
    size = torch.ones(V, device=DEV, dtype=torch.int64)
    target = 1 + _randint(g, torch.full((V,), smax, device=DEV))
    sub = torch.arange(V, device=DEV)
    for _ in range(2000):
        nd = nodes[sub]
        d = torch.where(nd >= 0, deg[nd.clamp(min=0)], 0)
        cum = torch.cumsum(d, 1)
        # a tree node outside a subtree touches it by exactly one edge: draw an edge, keep it if it leads out
        live = (size[sub] < target[sub]) & (cum[:, -1] > 2 * (size[sub] - 1))
        sub, nd, d, cum = sub[live], nd[live], d[live], cum[live]
        if not sub.numel():
            break
        r = _randint(g, cum[:, -1])
        slot = (cum <= r[:, None]).sum(1)
        u = nd.gather(1, slot[:, None])[:, 0]
        off = r - (cum - d).gather(1, slot[:, None])[:, 0]
        v = b[rp[u] + off]
        ok = ~(nd == v[:, None]).any(1)
        w = sub[ok]
        nodes[w, size[w]] = v[ok]
        size[w] += 1
    return torch.where(nodes >= 0, nodes - tbase[vid][:, None], -1)


def _pack(adj):
    """Bit rows (int32 words, least significant bit first) of a boolean matrix."""
    r, n = adj.shape
    words = (n + 31) // 32
    if n % 32:
        adj = torch.nn.functional.pad(adj, (0, words * 32 - n))
    w = torch.tensor([1, 2, 4, 8, 16, 32, 64, 128], device=DEV, dtype=torch.uint8)
    return (adj.view(r, words * 4, 8).to(torch.uint8) * w).sum(2, dtype=torch.uint8).view(torch.int32)


def _blocks(nodes, n, tree):
    """Row blocks (first row, boolean rows) of the intersection graph of `nodes`' subtrees."""
    inc = torch.zeros(n, tree + 1, device=DEV, dtype=torch.float16)
    inc.scatter_(1, torch.where(nodes >= 0, nodes, tree), 1.0)
    inc = inc[:, :tree]
    step = max(1, min(n, (1 << 28) // n))
    for a in range(0, n, step):
        adj = inc[a:a + step] @ inc.T > 0
        k = torch.arange(adj.shape[0], device=DEV)
        adj[k, a + k] = False
        yield a, adj


def _plant(rows, n, rng):
    """The subgraph induced by k uniform vertices becomes the chordless cycle C_k, k in 5..8."""
    k = min(int(rng.integers(5, 9)), n)
    if k < 4:
        return
    v = rng.choice(n, k, replace=False)
    at = torch.from_numpy(v).to(DEV)
    sub = rows[at].cpu().numpy().view(np.uint32)
    for i in range(k):
        for j in range(k):
            bit = np.uint32(1 << int(v[j] & 31))
            if (i - j) % k in (1, k - 1):
                sub[i, v[j] >> 5] |= bit
            else:
                sub[i, v[j] >> 5] &= ~bit
    rows[at] = torch.from_numpy(sub.view(np.int32)).to(DEV)


def _dense_rows(case, seed):
    n, g, rng = case["n"], _gen(seed), np.random.default_rng(seed)
    f = case["family"]
    if f == "subtree":
        nodes = _forest_subtrees([n], [case["tree"]], g)
        rows = torch.cat([_pack(adj) for _, adj in _blocks(nodes, n, case["tree"])])
        if case.get("cycle"):
            _plant(rows, n, rng)
        return rows
    if f == "gnp":
        adj = torch.triu(_rand(g, n, n) < case["p"], 1)
        return _pack(adj | adj.T)
    adj = torch.zeros(n, n, device=DEV, dtype=torch.bool)
    if f == "tree":   # a random recursive tree with shuffled ids
        v = torch.arange(1, n, device=DEV)
        perm = torch.randperm(n, generator=g, device=DEV)
        a, b = perm[v], perm[_randint(g, v)]
        adj[a, b] = True
        adj[b, a] = True
    else:             # clique with one edge missing in every second seed
        adj.fill_(True)
        adj.fill_diagonal_(False)
        i = int(rng.integers(0, n))
        j = (i + int(rng.integers(1, n))) % n
        adj[i, j] = adj[j, i] = False
    return _pack(adj)


def _csr_of_rows(rows, n):
    cols, counts = [], []
    step = max(1, (1 << 27) // max(n, 1))
    bit = torch.arange(32, device=DEV, dtype=torch.int32)
    for a in range(0, n, step):
        adj = ((rows[a:a + step, :, None] >> bit) & 1).reshape(-1, rows.shape[1] * 32) != 0
        cols.append(adj.nonzero()[:, 1].to(torch.int32))
        counts.append(adj.sum(1))
    rp = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
    rp[1:] = torch.cumsum(torch.cat(counts), 0)
    return rp, torch.cat(cols)


def _peo_csr(case, seed):
    """Sparse chordal graph grown along a reversed elimination order: vertex t joins a clique of
    s ~ U{1..smax} earlier vertices (an earlier w and s - 1 of the vertices w joined); ids shuffled;
    `extra` random edges on top."""
    n, smax, g = case["n"], case["smax"], _gen(seed)
    s = 1 + _randint(g, torch.full((n,), smax, device=DEV))
    first, top = s[:4096].tolist(), 0
    first[0] = 0
    for v in range(1, len(first)):   # the first vertices find only smaller cliques
        first[v] = min(first[v], top + 1)
        top = max(top, first[v])
    s[:len(first)] = torch.tensor(first, device=DEV)
    t = torch.arange(n, device=DEV)
    w = torch.zeros(n, device=DEV, dtype=torch.int64)
    todo = t[1:]
    while todo.numel():   # w uniform among the earlier vertices that joined enough
        c = _randint(g, todo)
        w[todo] = c
        todo = todo[s[c] < s[todo] - 1]
    level = torch.zeros(n, device=DEV, dtype=torch.int64)
    for _ in range(200):
        nl = torch.where(t > 0, level[w] + 1, 0)
        if torch.equal(nl, level):
            break
        level = nl
    by = torch.sort(level, stable=True)[1]
    ends = torch.cumsum(torch.bincount(level), 0).tolist()
    ln = torch.full((n, smax), -1, device=DEV, dtype=torch.int64)
    for a, b in zip(ends[:-1], ends[1:]):
        v = by[a:b]
        base = ln[w[v]]
        score = torch.where(base >= 0, _rand(g, *base.shape), 2.0)
        pick = base.gather(1, torch.argsort(score, 1))[:, :smax - 1]
        keep = torch.arange(smax - 1, device=DEV)[None] < s[v][:, None] - 1
        ln[v, 0] = w[v]
        ln[v, 1:] = torch.where(keep, pick, -1)
    a, k = (ln >= 0).nonzero(as_tuple=True)
    b = ln[a, k]
    perm = torch.randperm(n, generator=g, device=DEV)
    a, b = perm[a], perm[b]
    if case["extra"]:
        a = torch.cat([a, _randint(g, torch.full((case["extra"],), n, device=DEV))])
        b = torch.cat([b, _randint(g, torch.full((case["extra"],), n, device=DEV))])
    keep = a != b
    a, b = a[keep], b[keep]
    key = torch.unique(torch.cat([a * n + b, b * n + a]))
    rp = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
    rp[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return rp, (key % n).to(torch.int32)


def _many(case, seed):
    """`count` subtree graphs (tree of n/2 nodes), n log-uniform, every second one with a planted cycle."""
    rng = np.random.default_rng(seed)
    lo, hi = math.log(case["nmin"]), math.log(case["nmax"] + 1)
    u = np.random.default_rng(case["count"]).uniform(lo, hi, case["count"])   # the sizes belong to the case
    ns = np.minimum(np.exp(u).astype(int), case["nmax"]).tolist()
    trees = [max(1, n // 2) for n in ns]
    nodes = _forest_subtrees(ns, trees, _gen(seed))
    graphs, at = [], 0
    for i, n in enumerate(ns):
        rows = torch.cat([_pack(adj) for _, adj in _blocks(nodes[at:at + n], n, trees[i])])
        at += n
        if i % 2:
            _plant(rows, n, rng)
        graphs.append((rows, n))
    return graphs


def _ints(*shape):
    return torch.full(shape, -7, device=DEV, dtype=torch.int32)


def prepare(case, seed):
    kind, ctx = case["kind"], context()
    s = {"kind": kind, "ctx": ctx}
    if kind in ("batch", "queue"):
        s["graphs"] = _many(case, seed)
        if kind == "queue":
            s["queue"] = B.Queue(ctx, mem_budget_bytes=1 << 30)
            return s
        s["res"] = _ints(case["count"], 4)
        s["orders"] = _ints(sum(n for _, n in s["graphs"]))
        s["plan"] = B.BatchPlan(ctx, s["graphs"], s["res"], s["orders"])
        return s
    n = s["n"] = case["n"]
    s["order"] = _ints(n)
    s["res"] = _ints(4)
    if kind == "csr":
        s["rp"], s["col"] = _peo_csr(case, seed) if case["family"] == "peo" else _csr_of_rows(_dense_rows(case, seed), n)
        return s
    s["rows"] = _dense_rows(case, seed)
    if kind == "pair":
        h = s["rows"].clone()
        _plant(h, n, np.random.default_rng(seed))
        s["graphs"] = [(s["rows"], n), (h, n)]
        s["res"], s["order"] = _ints(2, 4), _ints(2 * n)
    elif kind in ("sweep", "check"):   # the order that a first LexBFS gave
        s["given"] = _ints(n)
        B.lexbfs_order_dense(ctx, s["rows"], n, s["given"])
        s["parent"] = _ints(n)
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "test":
        B.chordal_test_dense(ctx, s["rows"], s["n"], s["res"], s["order"])
    elif kind == "pair":
        B.chordal_test_batch(ctx, s["graphs"], s["res"], s["order"])
    elif kind == "csr":
        B.chordal_test_csr(ctx, s["rp"], s["col"], s["n"], s["res"], s["order"])
    elif kind == "mcs":
        B.chordal_test_mcs_dense(ctx, s["rows"], s["n"], s["res"], s["order"])
    elif kind == "sweep":
        B.lexbfs_plus_dense(ctx, s["rows"], s["n"], s["given"], s["order"])
        return [s["order"]]
    elif kind == "check":
        B.peo_check_dense(ctx, s["rows"], s["n"], s["given"], s["res"], s["parent"])
        return [s["res"], s["parent"]]
    elif kind == "batch":
        s["plan"].run()
        return [s["res"], s["orders"]]
    else:
        q = s["queue"]
        tickets = [q.submit_dense(rows, n) for rows, n in s["graphs"]]
        q.drain()
        return [np.array([q.poll(t)[1] for t in tickets], dtype=np.int32)]
    return [s["res"], s["order"]]


def work(case):
    """Each input read once, each output written once; the work is on whole numbers, so no flops."""
    def dense(n):
        return 4.0 * n * ((n + 31) // 32) + 4 * n + 16

    kind = case["kind"]
    if kind in ("batch", "queue"):   # the mean over n log-uniform in [nmin, nmax]
        lo, hi = case["nmin"], case["nmax"]
        span = math.log(hi / lo)
        per = (hi ** 2 - lo ** 2) / (16 * span) + 8 * (hi - lo) / span
        return {"bytes": case["count"] * per, "flops": 0.0}
    n = case["n"]
    if kind == "csr":
        deg = case["smax"] + 1.0 if case["family"] == "peo" else 56.0 / case["tree"] * n
        return {"bytes": 8.0 * (n + 1) + 4.0 * deg * n + 4.0 * n + 16, "flops": 0.0}
    return {"bytes": dense(n) * (2 if kind == "pair" else 1) + (4.0 * n if kind in ("sweep", "check") else 0.0),
            "flops": 0.0}


# ------------------------------------------------------------------ the same in plain numpy

def _matrix(rows, n):
    return np.unpackbits(rows.cpu().numpy().view(np.uint8), axis=1, bitorder="little")[:, :n].astype(bool)


def _np_lexbfs(adj):
    n = adj.shape[0]
    lab, order = np.zeros(n, np.int64), np.empty(n, np.int64)
    for i in range(n):
        x = order[i] = int(np.argmax(lab))   # the lowest id among the largest labels
        lab = 2 * lab + adj[x]
        lab[order[:i + 1]] = -1
        if i % 40 == 39:
            lab = np.unique(lab, return_inverse=True)[1].astype(np.int64)
            lab -= lab[x]
            lab[order[:i + 1]] = -1
    return order


def _np_mcs(adj):
    n = adj.shape[0]
    cnt, order = np.zeros(n, np.int64), np.empty(n, np.int64)
    for i in range(n):
        x = order[i] = int(np.argmax(cnt))
        cnt += adj[x]
        cnt[x] = -2 * n
    return order


def _np_check(adj, order):
    n = len(order)
    pos = np.empty(n, np.int64)
    pos[order] = np.arange(n)
    parent, res = np.full(n, -1), None
    for i, v in enumerate(order):
        early = adj[v] & (pos < i)
        if not early.any():
            continue
        p = parent[v] = int(order[np.max(pos[early])])
        bad = early & ~adj[p]
        bad[p] = False
        if res is None and bad.any():
            res = [0, int(v), p, int(np.argmax(bad))]
    return np.array(res or [1, -1, -1, -1]), parent


def exact(case, seed):
    if case["kind"] in ("batch", "queue", "csr"):
        return None
    n = case["n"]
    rows = _dense_rows(case, seed)
    adj = _matrix(rows, n)
    if case["kind"] == "mcs":
        order = _np_mcs(adj)
        return [_np_check(adj, order)[0], order]
    order = _np_lexbfs(adj)
    if case["kind"] == "test":
        return [_np_check(adj, order)[0], order]
    if case["kind"] == "check":
        return list(_np_check(adj, order))
    if case["kind"] == "sweep":   # ties to the vertex latest in the given order
        last = order[::-1]
        return [last[_np_lexbfs(adj[np.ix_(last, last)])]]
    res, orders = [_np_check(adj, order)[0]], [order]
    _plant(rows, n, np.random.default_rng(seed))
    adj = _matrix(rows, n)
    orders.append(_np_lexbfs(adj))
    res.append(_np_check(adj, orders[1])[0])
    return [np.stack(res), np.concatenate(orders)]
