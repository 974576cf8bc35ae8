"""The CSR search's panels where they can go wrong, against the CPU oracle
(order, verdict and witness bit for bit): windows of one vertex, windows cut
inside a class, classes too large for the front, components, rows at the limit
of a panel's entries and beyond it, panels with many moved vertices (ranked by
counting and by the network), and an arena that is packed several times."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_1508_06329_gb300 import binding as B  # noqa: E402

pytestmark = pytest.mark.gpu
N = 4801   # beyond the sizes that are expanded to bit rows


def _random(n, deg, rng):
    m = n * deg // 2
    return rng.integers(0, n, m), rng.integers(0, n, m)


def _edges(kind):
    rng = np.random.Generator(np.random.PCG64(sum(map(ord, kind))))
    n, v = N, np.arange(1, N)
    if kind == "path":
        return v - 1, v
    if kind == "matching":
        return np.arange(0, n - 1, 2), np.arange(1, n, 2)
    if kind == "tree":
        return (rng.random(n - 1) * v).astype(int), v
    if kind == "cliques":         # disjoint cliques of 10
        a, b = np.triu_indices(10, 1)
        base = 10 * np.arange(n // 10)[:, None]
        return (a + base).ravel(), (b + base).ravel()
    if kind == "grid":
        k = np.arange(69 * 69).reshape(69, 69)
        return np.r_[k[:, :-1].ravel(), k[:-1].ravel()], np.r_[k[:, 1:].ravel(), k[1:].ravel()]
    if kind == "bipartite":       # 20 long rows; one class of thousands without edges inside
        return np.repeat(np.arange(20), n - 20), np.tile(np.arange(20, n), 20)
    if kind.startswith("hub"):    # a row of exactly this many entries, and a sparse rest
        k = int(kind[3:])
        a, b = _random(n, 3, rng)
        return np.r_[np.zeros(k, int), a + (a == 0)], np.r_[1 + np.arange(k), b + (b == 0)]
    if kind == "longs":            # several long rows over the same vertices
        e = [(np.full(3000, h), 100 + rng.choice(n - 100, 3000, replace=False)) for h in range(8)]
        e.append(_random(n, 4, rng))
        return np.concatenate([x for x, _ in e]), np.concatenate([y for _, y in e])
    return _random(n, int(kind[6:]), rng)   # "randomD"


KINDS = ["path", "matching", "tree", "cliques", "grid", "bipartite", "hub2047", "hub2048", "hub2049", "longs",
         "random1", "random3", "random16", "random60"]


@pytest.mark.parametrize("kind", KINDS)
def test_csr_panels(kind):
    a, b = _edges(kind)
    keep = a != b
    key = np.unique(np.minimum(a, b)[keep] * N + np.maximum(a, b)[keep])
    g = gg.csr_from_edges(N, (key // N).astype(np.int64), (key % N).astype(np.int64))
    perm = np.random.Generator(np.random.PCG64(len(kind))).permutation(N)
    with B.Context(0) as ctx:
        for h in (g, gg.relabel_csr(g, perm)):
            assert h.nnz < 64 * N
            want = oracle.chordal_test(h)
            rp = torch.from_numpy(np.ascontiguousarray(h.row_ptr, dtype=np.int64)).cuda()
            col = torch.from_numpy(np.ascontiguousarray(h.col, dtype=np.int32)).cuda()
            res = torch.full((4,), -7, dtype=torch.int32, device="cuda")
            order = torch.full((N,), -7, dtype=torch.int32, device="cuda")
            B.chordal_test_csr(ctx, rp, col, N, res, order)
            assert np.array_equal(order.cpu().numpy(), want.order)
            assert tuple(res.cpu().tolist()) == want.witness
