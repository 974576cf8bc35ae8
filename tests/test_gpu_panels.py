"""GPU parity of the dense LexBFS's panels where a panel goes another way than
32 pivots in window order: large independent sets and matchings (the class that
goes on beyond the window), long paths with random ids (few pivots per panel),
dense random and co-sparse graphs (more moved members than the split sort
holds), and the sizes around the limits of the state layouts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_1508_06329_gb300 import binding as B  # noqa: E402

from gpu_util import run_dense  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    c.close()


def _graph(name, n):
    perm = np.random.Generator(np.random.PCG64(n)).permutation(n)
    if name == "star":
        return gg.star(n)
    if name == "matching":
        return gg.dense_from_edges(n, [(perm[k], perm[k + 1]) for k in range(0, n - 1, 2)])
    if name == "path":
        return gg.dense_from_edges(n, [(perm[k], perm[k + 1]) for k in range(n - 1)])
    if name == "interval":
        return gg.relabel_dense(gg.interval_graph(n, n, span=2000, max_len=40), perm)
    return gg.random_dense(n, {"half": 0.5, "cosparse": 0.995, "sparse": 3.0 / n}[name], n)


@pytest.mark.parametrize("name,n", [
    ("star", 1000), ("star", 9000), ("matching", 515), ("matching", 5001), ("path", 300), ("path", 2049),
    ("interval", 1500), ("sparse", 4097), ("sparse", 12345), ("half", 6000), ("half", 17000), ("cosparse", 1025),
    ("cosparse", 6000)])
def test_panels_off_the_common_path(ctx, name, n):
    g = _graph(name, n)
    want = oracle.chordal_test(g)
    got_w, got_o = run_dense(ctx, g)
    assert np.array_equal(got_o, want.order)
    assert got_w == want.witness


@pytest.mark.parametrize("n", [19800, 20100, 41900, 42800])
def test_state_layout_limits(ctx, n):
    """perm leaves shared memory just below 20,000 vertices, the keys above 42,000."""
    g = gg.subtree_dense(n, n // 4, n)
    h, _ = gg.plant_cycle(g, 6, n)
    for G in (g, h):
        want = oracle.chordal_test(G)
        got_w, got_o = run_dense(ctx, G)
        assert np.array_equal(got_o, want.order) and got_w == want.witness
