"""Plans of one structure search for their execution tree once (host side, no GPU).

A plan that reuses another's tree (the projector networks of an answer string, for one)
gets the same execution tree, without a search of its own: the copy is at least three
times faster than a search (about twenty times here)."""

import time

import paper_1709_03636_gb300 as q
from synth import random_regular_graph


def test_reused_plans_share_the_search():
    n = 22
    circ = q.Circuit.qaoa(n, random_regular_graph(n, 7, 3), 1)

    def projector(bits):
        return q.Network(circ, "projector", bits=bits + [2] * (n - len(bits)), lightcone=False)

    def timed(plan):
        start = time.perf_counter()
        tree = plan.execution_tree("c128")
        return time.perf_counter() - start, tree.steps()

    search, copies = [], []
    for seed in range(4):
        first = q.Plan(projector([0]), "lg", seed=seed)
        t, steps = timed(first)
        search.append(t)
        assert steps != first.steps()
        for bits in ([1], [0, 1], [1, 0, 0]):
            plan = q.Plan(projector(bits), like=first)
            t, again = timed(plan)
            copies.append(t)
            assert again == steps
            assert plan.steps() == first.steps()
    assert min(copies) < min(search) / 3
