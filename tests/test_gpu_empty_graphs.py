"""Graphs without vertices in a batch and in the queue.  They own no slot of the
packed per-vertex arrays: the slot at their offset is the next graph's first
(another CTA's), or lies past the end.  Run against the bounds-checking build,
which reports a write there as an error of the call."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CALLS = r"""
import sys
sys.path.insert(0, "tests")
import numpy as np, torch
import graphgen as gg, oracle
from gpu_util import to_dev
from paper_1508_06329_gb300 import binding as B
assert b"bounds-checking" in B.cg_version(), B.cg_version()
e = gg.empty_dense(0)
sets = [[e], [e, e], [e, gg.cycle(4), e], [gg.subtree_dense(50, 10, 1), e], [e, gg.subtree_dense(700, 90, 2), e, e]]
with B.Context(0) as ctx:
    for graphs in sets:
        want = [oracle.chordal_test(g) for g in graphs]
        dev = [(to_dev(g), g.n) for g in graphs]
        res = torch.full((len(graphs), 4), -7, dtype=torch.int32, device="cuda")
        order = torch.full((sum(g.n for g in graphs) + 1,), -7, dtype=torch.int32, device="cuda")
        B.chordal_test_batch(ctx, dev, res, order)
        torch.cuda.synchronize()
        assert [tuple(r) for r in res.tolist()] == [w.witness for w in want]
        assert np.array_equal(order[:-1].cpu().numpy(), np.concatenate([w.order for w in want]))
        assert int(order[-1]) == -7
        q = B.Queue(ctx, mem_budget_bytes=1 << 28)
        tickets = [q.submit_dense(rows, n) for rows, n in dev]
        q.drain()
        assert [tuple(q.poll(t)[1]) for t in tickets] == [w.witness for w in want]
        q.close()
print("empty ok")
"""


@pytest.mark.gpu
def test_graphs_without_vertices_own_no_slot():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1508_06329_gb300 import build
    env = dict(os.environ, CG_LIBCHORDAL=build.build(debug=True))
    r = subprocess.run([sys.executable, "-c", CALLS], cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "empty ok" in r.stdout, r.stdout + r.stderr
