"""Shared-memory programs run level by level by a team of warps: one network
per CTA (warp teams off), and subtree tasks of the graph executor, against the
state-vector oracle.  The shapes reach the ends of the op forms: ops of 1 to
2^10 outputs and 1 to 2^9 summed values, narrow and team ops, leaf adjoints,
long adjoint sums shared by lanes.  Bounds of the element types: complex128
1e-11, complex64 2e-6 per edge and 1e-4 relative on the gradient."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

import paper_1709_03636_gb300 as q  # noqa: E402
from oracle import statevector as sv  # noqa: E402
from synth import random_regular_graph  # noqa: E402


@pytest.mark.parametrize("dtype,tol,gtol", [("c128", 1e-11, 1e-9), ("c64", 2e-6, 1e-4)])
@pytest.mark.parametrize("n,d,p,diag,lightcone,ordering", [
    (4, 3, 1, True, True, "lg"),         # a handful of ops
    (13, 4, 2, True, False, "lg"),       # ranks up to 11 and more
    (12, 3, 2, False, True, "lg"),       # rank-4 gates: sums over several labels
    (10, 3, 2, False, False, "stoch"),   # long sums over few outputs
    (9, 4, 3, True, True, "stoch"),      # six gradient slots
])
def test_team_programs_match_the_state_vector(n, d, p, diag, lightcone, ordering, dtype, tol,
                                              gtol):
    edges = random_regular_graph(n, d, 10 * n + p)
    g, b = [0.4 + 0.3 * k for k in range(p)], [0.9 - 0.2 * k for k in range(p)]
    batch = q.Batch(q.Circuit.qaoa(n, edges, p), lightcone=lightcone, diag=diag,
                    ordering=ordering, seed=3)
    ref = sv.edge_zz(n, edges, g, b)
    _, ref_grad = sv.gradient(n, edges, g, b)
    for graph, small_rank in ((False, 0), (True, 10), (True, 5)):
        engine = q.Engine(0, arena_bytes=1 << 30)
        engine.set_task_options(warp_teams=0)
        engine.set_graph_options(graph, small_rank)
        for want_grad in (False, True):
            _, zz, grad = q.qaoa_expectation(engine, batch, g, b, dtype, want_grad=want_grad)
            assert np.max(np.abs(np.array(zz) - ref)) < tol
        assert np.max(np.abs(np.array(grad) - ref_grad)) < gtol * max(1, np.max(np.abs(ref_grad)))
