"""Execution trees of plans that are too wide for any device (host side, no GPU).

The search's tables end at 64 labels per step, so a plan with a wider step keeps
its tree; one whose steps stay below is still searched."""

import pytest

import paper_1709_03636_gb300 as q
from synth import random_regular_graph


@pytest.mark.parametrize("n,d,wide", [(56, 4, False), (104, 6, True), (108, 6, True),
                                      (116, 6, True), (200, 6, True)])
def test_plans_with_steps_above_64_labels_keep_their_tree(n, d, wide):
    edges = random_regular_graph(n, d, n)
    plan = q.Plan(q.Network(q.Circuit.qaoa(n, edges, 1), edge=edges[0], lightcone=False), "lg")
    assert (max(sum(s) for s in plan.step_shapes()) > 64) == wide
    tree = plan.execution_tree("c128")
    assert (tree.steps() == plan.steps()) == wide
