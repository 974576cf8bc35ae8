"""GPU parity of the MCS order's panels where a window goes wrong or the bound
of the next one does: all counts equal, cliques and stars, neighbouring ids
with neighbouring counts, vertices that come into the window in mid-panel
(random graphs, where the panels give way to steps), and the sizes around the
first and the last that begin in panels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_1508_06329_gb300 import binding as B  # noqa: E402

from gpu_util import DEV, to_dev  # noqa: E402

pytestmark = pytest.mark.gpu


def _graph(name, n):
    if name == "bipartite":
        return gg.dense_from_edges(n, [(a, b) for a in range(9) for b in range(9, n)])
    if name in ("half", "sparse", "cosparse"):
        return gg.random_dense(n, {"half": 0.5, "sparse": 3.0 / n, "cosparse": 0.99}[name], n)
    return {"empty": gg.empty_dense, "clique": gg.clique, "star": gg.star, "path": gg.path,
            "interval": lambda k: gg.interval_graph(k, 7, span=k, max_len=60),
            "tree": lambda k: gg.random_tree(k, 9)}[name](n)


@pytest.mark.parametrize("name,n", [
    ("empty", 8191), ("empty", 8192), ("clique", 8200), ("star", 9001), ("path", 8222), ("bipartite", 9049),
    ("interval", 9001), ("half", 8193), ("sparse", 12001), ("cosparse", 8300), ("tree", 36608), ("tree", 36609)])
def test_mcs_panels(name, n):
    g = _graph(name, n)
    order = torch.empty(n, dtype=torch.int32, device=DEV)
    pos = torch.empty(n, dtype=torch.int32, device=DEV)
    with B.Context(0) as ctx:
        B.mcs_order_dense(ctx, to_dev(g), n, order, pos)
        got = order.cpu().numpy()
    assert np.array_equal(got, oracle.mcs(g))
    assert np.array_equal(np.argsort(got), pos.cpu().numpy())
