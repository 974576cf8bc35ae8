"""Dense LexBFS on narrow graphs, whose next vertex is known only after the one
before: the panels of steps against the oracle (order, verdict and witness) at
the edges of their reach (32 met vertices, classes of more than 32 members, rows
read by one warp or by all threads, the state layouts), alone and in a batch;
and their time.  The bound on the time is four latencies of a barrier pair and
an L2 load per vertex, measured by the library on the same device: on GB300 one
step per vertex took 2.7 to 4.1 of them on such graphs, windows alone 5 to 24."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_1508_06329_gb300 import binding as B  # noqa: E402

from gpu_util import run_dense, to_dev  # noqa: E402

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
    elif name.startswith("blocks"):    # a path of complete bipartite joints, k vertices each
        k = int(name[6:])
        e = [(v[:-j][v[:-j] // k + 1 == v[j:] // k], v[j:][v[:-j] // k + 1 == v[j:] // k]) for j in range(1, 2 * k)]
    elif name == "spider":             # long legs on one vertex, and chords
        e = [(np.where(v[1:] % 25 == 1, 0, v[1:] - 1), v[1:]), (rng.integers(0, n, n // 30), rng.integers(0, n, n // 30))]
    else:                              # "mixed": a path, then a random graph, then a path
        a, b = n // 3, 2 * n // 3
        e = [(v[:-1], v[1:]), (rng.integers(a, b, 4 * n), rng.integers(a, b, 4 * n))]
    x, y = (np.concatenate(k) for k in zip(*e))
    words = (n + 31) // 32
    m = np.zeros((n, words), np.uint32)
    p = rng.permutation(n)
    x, y = p[x[x != y]], p[y[x != y]]
    for s, d in ((x, y), (y, x)):
        np.bitwise_or.at(m, (s, d >> 5), np.uint32(1) << (d & 31).astype(np.uint32))
    return gg.DenseGraph(n, m)


CASES = [(k, n) for k in ("path", "matching", "power3", "cliques4", "spider", "mixed") for n in (33, 300, 2500)]
CASES += [("cliques33", 900), ("cliques34", 900), ("blocks16", 1000), ("blocks33", 1400), ("blocks40", 5000),
          ("power9", 4096), ("path", 4097), ("spider", 9000), ("mixed", 16385), ("cliques5", 19905), ("spider", 20500),
          ("path", 43000), ("mixed", 43000)]


@pytest.mark.parametrize("name,n", CASES)
def test_narrow_graphs_match_the_oracle(name, n):
    g = narrow(name, n)
    want = oracle.chordal_test(g)
    with B.Context(0) as ctx:
        got_w, got_o = run_dense(ctx, g)
    assert np.array_equal(got_o, want.order)
    assert got_w == want.witness


def test_narrow_graphs_in_a_batch():
    graphs = [narrow(k, n) for n in (17, 64, 257, 1030, 2049, 4096) for k in ("path", "power3", "cliques4", "spider")]
    want = [oracle.chordal_test(g) for g in graphs]
    with B.Context(0) as ctx:
        res = torch.full((len(graphs), 4), -7, dtype=torch.int32, device="cuda")
        order = torch.full((sum(g.n for g in graphs),), -7, dtype=torch.int32, device="cuda")
        B.chordal_test_batch(ctx, [(to_dev(g), g.n) for g in graphs], res, order)
        torch.cuda.synchronize()
    assert np.array_equal(order.cpu().numpy(), np.concatenate([w.order for w in want]))
    assert [tuple(r) for r in res.tolist()] == [w.witness for w in want]


@pytest.mark.parametrize("name,n", [("path", 4096), ("cliques4", 4096), ("path", 16384), ("cliques4", 16384)])
def test_a_narrow_graph_costs_a_few_latencies_per_vertex(name, n):
    g = narrow(name, n)
    with B.Context(0) as ctx:
        floor = B.step_floor(ctx)
        rows = to_dev(g)
        res = torch.empty(4, dtype=torch.int32, device="cuda")
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            B.chordal_test_dense(ctx, rows, n, res)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e6)
    assert min(times[1:]) < 4 * (floor["barrier_pair_ns"] + floor["load_ns"]) * n
