"""The window rule of the dense LexBFS on the CPU: how many window vertices are
visited in window order, as panel_in_order of lexbfs_dense.cuh decides it (one
comparison per vertex, the breakers against all before them, the class that
goes on beyond the window against the largest label out there), compared with
LexBFS steps on the whole graph."""
import numpy as np
import pytest


def _loses(a, b, z):
    d = (a ^ b) & ((1 << z) - 1)
    return d != 0 and not (a & d & -d)


def _in_order(adj, starts, w2, straddle, ub):
    cls = np.cumsum([(starts >> k) & 1 for k in range(w2)])
    fail = [k for k in range(w2) if straddle and cls[k] == cls[-1] and _loses(adj[k], ub, k)]
    for z in range(w2 - 1):
        if cls[z] == cls[z + 1] and _loses(adj[z], adj[z + 1], z):
            fail += [k for k in range(z + 1) if cls[k] == cls[z + 1] and _loses(adj[k], adj[z + 1], k)]
    return min(fail, default=w2)


@pytest.mark.parametrize("p", [0.03, 0.2, 0.5, 0.9])
def test_in_order_prefix_matches_lexbfs_steps(p):
    rng = np.random.Generator(np.random.PCG64(int(100 * p)))
    for _ in range(150):
        n, w = int(rng.integers(2, 40)), int(rng.integers(1, 13))
        m = np.triu(rng.random((n, n)) < p, 1)
        m = m | m.T
        cuts = np.sort(rng.choice(np.arange(1, n), int(rng.integers(0, min(n - 1, 6) + 1)), replace=False))
        cls = np.zeros(n, int)
        cls[cuts] = 1
        cls = np.cumsum(cls)      # class of each position, ids ascending by position
        w2 = min(w, n)
        adj = [int(sum(1 << j for j in range(w2) if m[k, j])) for k in range(n)]
        starts = sum(1 << k for k in range(w2) if k == 0 or cls[k] != cls[k - 1])
        straddle = w2 < n and cls[w2] == cls[w2 - 1]
        out = [adj[k] for k in range(w2, n) if cls[k] == cls[w2 - 1]]
        ub = 0
        for a in out:
            ub |= a
        label = [()] * n
        steps = 0                 # LexBFS on all n vertices from this partition
        for z in range(w2):
            best = min((k for k in range(n) if k >= z), key=lambda k: (cls[k], tuple(-x for x in label[k]), k))
            if best != z:
                break
            steps += 1
            for k in range(n):
                label[k] = label[k] + (int(m[z, k]),)
        exact = _in_order(adj, starts, w2, straddle, ub)
        assert exact <= steps     # never more than LexBFS visits in this order
        if not straddle:
            assert exact == steps
        assert _in_order(adj, starts, w2, straddle, (1 << 32) - 1) <= steps
