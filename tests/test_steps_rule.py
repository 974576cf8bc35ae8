"""The rule of the searches' panels of steps on the CPU: up to 32 pivots from the
classes as they are when the panel starts, a label per vertex that meets one, at
most 32 of these at any time; the next pivot is the class at hand's vertex of
the largest label, else its first member without one; the classes are split when
the panel ends.  Panels of steps alone give the oracle's order and the parents
of the perfect-elimination check, whatever ends a panel."""
import numpy as np
import pytest

import graphgen as gg
import oracle


def steps(adj, lanes, pivots):
    n = len(adj)
    classes = [[-1, list(range(n))]]   # top first: last adjacent pivot, members in id order
    order, parent = [], []
    while len(order) < n:
        label, taken, at, first = {}, [], 0, len(order)   # met and not numbered: bits, the first pivot's highest
        while len(taken) < pivots and len(order) < n:
            while all(y in taken for y in classes[at][1]):
                at += 1
            own, members = classes[at]
            left = [y for y in members if y not in taken]
            x = max(left, key=lambda y: (label.get(y, 0), -y))
            fresh = [y for y in adj[x] if y not in label and y not in taken and y not in order[:first]]
            if len(label) - (x in label) + len(fresh) > lanes and taken:
                break                                      # the panel ends before x
            bits = label.pop(x, 0)
            parent.append(taken[pivots - (bits & -bits).bit_length()] if bits else own)
            for y in adj[x]:
                if y in label or y in fresh:
                    label[y] = label.get(y, 0) | 1 << (pivots - 1 - len(taken))
            taken.append(x)
            order.append(x)
        split = []
        for own, members in classes:
            met = sorted((-label.get(y, 0), y) for y in members if y not in taken)
            for bits in sorted({b for b, _ in met}):
                last = taken[pivots - (-bits & bits).bit_length()] if bits else own
                split.append([last, [y for b, y in met if b == bits]])
        classes = split
    return order, parent


@pytest.mark.parametrize("lanes,pivots", [(32, 32), (4, 32), (32, 5), (6, 7), (100, 1)])
def test_panels_of_steps_match_the_oracle(lanes, pivots):
    rng = np.random.Generator(np.random.PCG64(lanes * 100 + pivots))
    graphs = [gg.path(40), gg.cycle(33), gg.star(30), gg.clique(12), gg.empty_dense(9), gg.random_tree(70, 3),
              gg.subtree_dense(60, 40, 2)] + [gg.random_dense(n, p, n) for n, p in ((25, .1), (45, .05), (30, .4))]
    for g in graphs:
        g = gg.relabel_dense(g, rng.permutation(g.n))
        adj = [sorted(int(y) for y in nb) for nb in gg.adjacency_lists(g)]
        order, parent = steps(adj, lanes, pivots)
        assert order == oracle.chordal_test(g).order.tolist()
        pos = {v: i for i, v in enumerate(order)}
        for i, v in enumerate(order):
            early = [pos[u] for u in adj[v] if pos[u] < i]
            assert parent[i] == (order[max(early)] if early else -1)
