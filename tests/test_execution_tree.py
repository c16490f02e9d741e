"""The trees the graph executor contracts (host side, no GPU).

A plan's execution tree is another binary tree over the same leaves: its
scalar equals the state vector's to rounding (1e-12 on values of order one),
its graph program passes the host validation and its grouped row steps equal
the plain contraction (1e-11, as for the plans' own trees), and a large network's
takes fewer multiply-adds.  Networks whose tensors stay at rank 10, and
single precision, keep their plan.
"""

import ctypes

import pytest

import paper_1709_03636_gb300 as q
from oracle import statevector as sv
from paper_1709_03636_gb300 import _lib
from synth import random_regular_graph
from test_host_plans import run_plan


@pytest.mark.parametrize("ordering", ["lg", "stoch"])
@pytest.mark.parametrize("diag", [True, False])
@pytest.mark.parametrize("n,d,p,lightcone", [(13, 4, 2, True), (14, 5, 1, False), (8, 3, 1, True)])
def test_execution_tree_gives_the_same_scalar(n, d, p, lightcone, diag, ordering):
    edges = random_regular_graph(n, d, n)
    params = [0.7, 0.45][:p] + [0.3, 1.1][:p]
    ref = sv.edge_zz(n, edges, params[:p], params[p:])
    circ = q.Circuit.qaoa(n, edges, p)
    for i in (0, len(edges) - 1):
        net = q.Network(circ, edge=edges[i], lightcone=lightcone, diag=diag)
        plan = q.Plan(net, ordering, seed=i)
        if plan.stats()["max_rank"] > 20:
            continue   # too large for the einsum evaluation below
        for dtype in ("c64", "c128"):
            tree = plan.execution_tree(dtype)
            assert sorted(x for s in tree.steps() for x in s) == list(
                range(2 * len(tree.steps())))
            value = run_plan(net, tree, params)
            assert abs(value - ref[i]) < 1e-12
            before, after = plan.stats(), tree.stats()
            if before["max_rank"] <= 10 or dtype == "c64":
                assert tree.steps() == plan.steps()
            elif before["max_rank"] > 12:
                assert after["cmacs"] < before["cmacs"]


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_execution_trees_lower_to_valid_programs(dtype):
    edges = random_regular_graph(14, 5, 2)
    for kw in (dict(lightcone=False), dict(lightcone=False, diag=False), dict(ordering="stoch")):
        batch = q.Batch(q.Circuit.qaoa(14, edges, 1 if "lightcone" in kw else 2), edges[:6], **kw)
        trees = batch.execution_trees(dtype)
        assert trees.stats()["n_networks"] == 6 and trees.edges == batch.edges
        for small, grad in ((3, 1), (8, 1), (10, 0)):
            assert trees.program_info(dtype, grad, force_graph=True, small_rank=small)["graph"]
            err, count = ctypes.c_double(), ctypes.c_int32()
            _lib.check(_lib.lib.qtc_selftest_tile_steps(
                trees.ptr, q.DTYPES[dtype], grad, 1, small, 0, 16, ctypes.byref(err),
                ctypes.byref(count)))
            assert err.value < 1e-11
