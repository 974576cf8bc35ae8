"""CSR LexBFS on graphs with a few hubs over the same leaves, a leaf first: most
of a hub's long row lies in one class.  Order, verdict and witness against the
oracle where the class starts are kept as bits (up to 196,608 sorted
neighbours) and beyond, and the time: a hub's row must cost in proportion to
its length, so twenty of them are bounded by six times the search on the same
number of vertices without edges (measured on GB300 at n = 65,536: 127 ms
against 7.8 where every member walked back through its class, 79 against 53
with one step per vertex)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_1508_06329_gb300 import binding as B  # noqa: E402

pytestmark = pytest.mark.gpu


def hubs(n, h, seed, share=1.0):
    rng = np.random.Generator(np.random.PCG64(seed))
    a, b = np.repeat(np.arange(h), n - h), np.tile(np.arange(h, n), h)
    keep = rng.random(a.size) < share
    perm = rng.permutation(n)
    perm[[0, int(np.argmax(perm == n - 1))]] = perm[[int(np.argmax(perm == n - 1)), 0]]   # (a hub is last)
    a, b = perm[a[keep]], perm[b[keep]]
    key = np.unique(np.minimum(a, b) * n + np.maximum(a, b))
    return gg.csr_from_edges(n, key // n, key % n)


def to_dev(g):
    return (torch.from_numpy(np.ascontiguousarray(g.row_ptr, dtype=np.int64)).cuda(),
            torch.from_numpy(np.ascontiguousarray(g.col, dtype=np.int32)).cuda())


def search(ctx, dev, n):
    order = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    res = torch.full((4,), -7, dtype=torch.int32, device="cuda")
    B.chordal_test_csr(ctx, *dev, n, res, order)
    return order, res


@pytest.mark.parametrize("n,h,share", [(4700, 3, 1.0), (9000, 20, 0.7), (70000, 20, 1.0), (190000, 5, 0.8),
                                       (260000, 4, 1.0), (300000, 3, 0.9)])
def test_hubs_match_the_oracle(n, h, share):
    g = hubs(n, h, n, share)
    want = oracle.chordal_test(g)
    with B.Context(0) as ctx:
        order, res = search(ctx, to_dev(g), n)
        assert np.array_equal(order.cpu().numpy(), want.order)
        assert tuple(res.cpu().tolist()) == want.witness


def test_a_hub_costs_its_row():
    n = 65536

    def best(ctx, g):
        dev = to_dev(g)
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            search(ctx, dev, n)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times[1:])

    with B.Context(0) as ctx:
        empty = gg.csr_from_edges(n, np.zeros(0, np.int64), np.zeros(0, np.int64))
        assert best(ctx, hubs(n, 20, 1)) < 6 * best(ctx, empty)
