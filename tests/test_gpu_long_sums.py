"""Long sums over few outputs in the graph executor (rows staged through shared
memory in batches of summed values) against the state-vector oracle.

Forced graph programs whose tensors leave shared memory at a low rank reach
rows of 1 to 256 outputs and sums of 64 to 4096 values in each order of
addition (sequential, eight accumulators, four of pairs).  Bounds: complex128
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
@pytest.mark.parametrize("n,d,p,diag,ordering,small_rank", [
    (14, 5, 1, True, "stoch", 5), (14, 5, 1, False, "stoch", 3), (12, 3, 2, False, "lg", 4),
    (16, 6, 1, True, "lg", 2), (13, 4, 2, True, "stoch", 6)])
def test_long_sums_match_the_state_vector(n, d, p, diag, ordering, small_rank, dtype, tol, gtol):
    edges = random_regular_graph(n, d, n + d)
    g, b = [0.5 + 0.35 * k for k in range(p)], [0.8 - 0.25 * k for k in range(p)]
    ref = sv.edge_zz(n, edges, g, b)
    _, ref_grad = sv.gradient(n, edges, g, b)
    engine = q.Engine(0, arena_bytes=8 << 30)
    engine.set_graph_options(True, small_rank)
    batch = q.Batch(q.Circuit.qaoa(n, edges, p), lightcone=False, diag=diag, ordering=ordering,
                    seed=1)
    _, zz, grad = q.qaoa_expectation(engine, batch, g, b, dtype, want_grad=True)
    assert np.max(np.abs(np.array(zz) - ref)) < tol
    assert np.max(np.abs(np.array(grad) - ref_grad)) < gtol * max(1, np.max(np.abs(ref_grad)))
    # one network alone: its steps are cut finest
    one = batch.subset([len(edges) // 2])
    _, zz1, _ = q.qaoa_expectation(engine, one, g, b, dtype)
    assert abs(zz1[0] - ref[len(edges) // 2]) < tol
