"""CSR LexBFS on narrow sparse graphs, whose next vertex is known only after the
one before: the panels of steps against the oracle (order, verdict and witness)
where they begin, end early (rows of more than 32 entries, more met vertices
than lanes) and alternate with windows, with and without shared-memory links,
and their time.  The bound on the time is four latencies of a barrier pair and
an L2 load per vertex, measured by the library on the same device: on GB300 one
step per vertex took 2.7 to 3.8 of them on such graphs, windows alone 7 to 13."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_1508_06329_gb300 import binding as B  # noqa: E402

pytestmark = pytest.mark.gpu


def narrow(name, n):
    rng = np.random.Generator(np.random.PCG64(n))
    v = np.arange(n)
    if name == "path":
        e = [(v[:-1], v[1:])]
    elif name == "matching":
        e = [(v[0:n - 1:2], v[1:n:2])]
    elif name.startswith("power"):     # of a path
        e = [(v[:-j], v[j:]) for j in range(1, int(name[5:]) + 1)]
    elif name.startswith("cliques"):   # disjoint
        k = int(name[7:])
        e = [(v[:-j][v[:-j] % k + j < k], v[j:][v[:-j] % k + j < k]) for j in range(1, k)]
    elif name == "combs":              # a path whose vertices have 1 to 40 leaves
        s = np.flatnonzero(rng.random(n) < 0.1)
        s[0] = 0
        own = s[np.searchsorted(s, v, side="right") - 1]
        e = [(s[:-1], s[1:]), (own[own != v], v[own != v])]
    elif name == "spider":             # long legs on one vertex, and chords
        e = [(np.where(v[1:] % 25 == 1, 0, v[1:] - 1), v[1:]), (rng.integers(0, n, n // 30), rng.integers(0, n, n // 30))]
    else:                              # "mixed": a path, then a random graph, then a path
        a, b = n // 3, 2 * n // 3
        e = [(v[:-1], v[1:]), (rng.integers(a, b, 4 * n), rng.integers(a, b, 4 * n))]
    x, y = (np.concatenate(k) for k in zip(*e))
    p = rng.permutation(n)
    x, y = p[x[x != y]], p[y[x != y]]
    key = np.unique(np.minimum(x, y) * n + np.maximum(x, y))
    return gg.csr_from_edges(n, key // n, key % n)


def to_dev(g):
    return (torch.from_numpy(np.ascontiguousarray(g.row_ptr, dtype=np.int64)).cuda(),
            torch.from_numpy(np.ascontiguousarray(g.col, dtype=np.int32)).cuda())


KINDS = ("path", "matching", "power3", "power9", "power17", "cliques4", "cliques11", "cliques33", "cliques34", "combs",
         "spider", "mixed")


@pytest.mark.parametrize("name,n", [(k, n) for k in KINDS for n in (4097, 33000)] + [("mixed", 150001), ("spider", 150001)])
def test_narrow_sparse_graphs_match_the_oracle(name, n):
    g = narrow(name, n)
    assert g.nnz < 64 * n
    want = oracle.chordal_test(g)
    res = torch.full((4,), -7, dtype=torch.int32, device="cuda")
    order = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    with B.Context(0) as ctx:
        B.chordal_test_csr(ctx, *to_dev(g), n, res, order)
    assert np.array_equal(order.cpu().numpy(), want.order)
    assert tuple(res.cpu().tolist()) == want.witness


@pytest.mark.parametrize("name", ["path", "matching", "cliques4"])
def test_a_narrow_sparse_graph_costs_a_few_latencies_per_vertex(name):
    n = 65536
    with B.Context(0) as ctx:
        floor = B.step_floor(ctx)
        dev = to_dev(narrow(name, n))
        res = torch.empty(4, dtype=torch.int32, device="cuda")
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            B.chordal_test_csr(ctx, *dev, n, res)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e6)
    assert min(times[1:]) < 4 * (floor["barrier_pair_ns"] + floor["load_ns"]) * n
